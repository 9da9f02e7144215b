// Cyclic reduction of (s + i delta) x = f, s real symmetric tridiagonal: the
// block solve of the P-space preconditioner, s = theta - T.
//
// The block inverse is bounded: 1 / d of an eigenvalue of the block at distance
// d = theta - lambda is taken as d / (d^2 + delta^2), the real part of
// 1 / (d + i delta), at most 1 / (2 delta) = 1e4.  (theta passes the block's
// lowest eigenvalue from above on its way and may stop on one; beyond that
// bound FP32 leaves nothing of the Olsen correction's difference of two
// parallel vectors.)  s + i delta needs no pivoting: cyclic reduction divides by
// diagonal elements of its Schur complements, and those of a symmetric s,
//   s_11 + i delta - B (s_22 + i delta)^{-1} B^T,
// have the imaginary part delta (1 + B (s_22^2 + delta^2)^{-1} B^T) >= delta.
// A real reduction with pivots clamped at 1e-6 amplified by up to 5e6 where
// theta met an eigenvalue; over 600 solves with a second state 5e-4 to 3e-3 Eh
// above the lowest (7 orbitals) it took 8,755 iterations, this one 7,710.
// Host and device code.
#pragma once

#ifdef __CUDACC__
#define TRI_FN __host__ __device__ __forceinline__
#else
#define TRI_FN inline
#endif

constexpr int TRI_MAX = 128;
constexpr float TRI_DELTA = 5e-5f;

struct TriC {
  float re, im;
};

TRI_FN TriC tri_div(TriC a, TriC b) {
  const float n = b.re * b.re + b.im * b.im;
#ifdef __CUDA_ARCH__
  const float s = __fdividef(1.f, n);
#else
  const float s = 1.f / n;
#endif
  return TriC{(a.re * b.re + a.im * b.im) * s, (a.im * b.re - a.re * b.im) * s};
}
// a - k b
TRI_FN TriC tri_sub(TriC a, TriC k, TriC b) {
  return TriC{a.re - (k.re * b.re - k.im * b.im), a.im - (k.re * b.im + k.im * b.re)};
}

// Row i of one level, distance st between the rows that are still coupled:
// o[0..2] the elements left of, on and right of the diagonal, o[3], o[4] two
// right-hand sides; w the next level.  After the last level (st >= n) the
// unknowns are o[3] / o[1] and o[4] / o[1].
TRI_FN void tri_level(const TriC (*o)[TRI_MAX], TriC (*w)[TRI_MAX], int i, int st, int n) {
  const int lo = i - st, hi = i + st;
  TriC b = o[1][i], f = o[3][i], g = o[4][i], a = {0.f, 0.f}, c = {0.f, 0.f};
  if (lo >= 0) {
    const TriC k = tri_div(o[0][i], o[1][lo]);
    b = tri_sub(b, k, o[2][lo]);
    f = tri_sub(f, k, o[3][lo]);
    g = tri_sub(g, k, o[4][lo]);
    a = tri_sub(a, k, o[0][lo]);
  }
  if (hi < n) {
    const TriC k = tri_div(o[2][i], o[1][hi]);
    b = tri_sub(b, k, o[0][hi]);
    f = tri_sub(f, k, o[3][hi]);
    g = tri_sub(g, k, o[4][hi]);
    c = tri_sub(c, k, o[2][hi]);
  }
  w[0][i] = a;
  w[1][i] = b;
  w[2][i] = c;
  w[3][i] = f;
  w[4][i] = g;
}
