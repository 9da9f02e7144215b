// Lowest eigenpair of the Davidson subspace matrix (the Rayleigh-Ritz step),
// one CTA of 256 threads per tuple.
//
// GB300 issues FP64 at a small fraction of its FP32 rate, so the O(m^3)
// diagonalisation runs in FP32 and only O(m^2) work per step is FP64:
//   1. cyclic Jacobi in FP32 with the round-robin (tournament) ordering: the
//      m/2 rotations of one step touch disjoint index pairs and are applied
//      together, rows and columns at once;
//   2. the lowest FP32 eigenvector z_k is refined in FP64 by Newton steps in
//      the approximate eigenbasis: with s = G y - theta y (FP64),
//        y <- y - sum_{j != k} z_j (z_j . s) / (lambda_j - theta),
//      each step multiplying the error by ~ (FP32 residual of Z) / gap, and
//      theta = y.G.y is the FP64 Rayleigh quotient of the normalised y.
// m <= 32; G is symmetric.
//
// The step is a chain of short dependent phases, so its latency is what
// counts.  A thread owns column (lane) and four rows of A and Z; it forms the
// rotation of its own column's pair itself, takes those of its rows from the
// other lanes by shuffles and writes into the other buffer: one barrier per
// Jacobi step.  When the subspace has grown by one vector since the last call
// the sweeps start from Z^T G Z, an arrow matrix whose border is small near
// convergence (2-3 sweeps instead of 6), Z the kept vectors after one
// Newton-Schulz step, Z + Z (1 - Z^T Z) / 2: kept over 30 calls as they are,
// they leave orthonormality by 1e-5, an error of |theta| 1e-5 in every
// lambda_j - theta, and a root 1e-3 above the lowest cost up to half as many
// iterations again.  FP64 sums run in one warp: an FP64 instruction of a warp
// takes 64 cycles of its sub-partition's unit, a division or root about 1,200.
// So the refinement stops once its update is below 2e-10 (mostly the second,
// the fifth at a gap of 1e-3 below theta = -24; the error left is that times
// the ratio above) or no longer halves (a gap lost in FP32), y.Gy and y.y share
// one reduction, and y.y, 1 to about 1e-6, is inverted by a series.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

constexpr int RITZ_THREADS = 256;
constexpr int RITZ_UPDATES = 12;   // of the FP64 refinement at most

struct RitzShared {
  double G[32][33];
  double y[32], gy[32];
  float A[2][32][33];
  float Z[2][32][33];
  float lam[32], s32[32], coef[32], wmax[8], theta;
};

__device__ __forceinline__ double ritz_warp_sum(double v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float ritz_warp_sumf(float v) {
  for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Called by all RITZ_THREADS threads of a block.  Gb: row-major, leading
// dimension M.  Zk: the eigenvectors kept between calls (32 x 32), read when
// `warm` (they then belong to the leading m - 1 rows of G) and written.
static __device__ void ritz_lowest(const double* __restrict__ Gb, int m, int M, RitzShared& S,
                                   float* __restrict__ Zk, bool warm, double* theta_out,
                                   double* y_out) {
  const int tid = threadIdx.x, r = tid & 31, w = tid >> 5;
  for (int i = w; i < 32; i += 8) {
    double g = 0.0;
    if (i < m && r < m) g = Gb[(int64_t)i * M + r];
    S.G[i][r] = g;
    S.A[0][i][r] = (float)g;
    S.Z[0][i][r] = warm && i < m - 1 && r < m - 1 ? Zk[i * 32 + r] : (i == r) ? 1.f : 0.f;
  }
  __syncthreads();
  int cur = 0;
  if (warm) {
    // Z[1] <- Z + Z (1 - Z^T Z) / 2, then A[1] <- Z^T A Z (the product A Z in Z[0])
    for (int i = w; i < m; i += 8) {
      float v = i == r ? 1.f : 0.f;
      for (int j = 0; j < m; j++) v = fmaf(-S.Z[0][j][i], S.Z[0][j][r], v);
      S.A[1][i][r] = v;
    }
    __syncthreads();
    for (int i = w; i < m; i += 8) {
      float v = 0.f;
      for (int j = 0; j < m; j++) v = fmaf(S.Z[0][i][j], S.A[1][j][r], v);
      S.Z[1][i][r] = fmaf(0.5f, v, S.Z[0][i][r]);
    }
    __syncthreads();
    for (int i = w; i < m; i += 8) {
      float v = 0.f;
      for (int j = 0; j < m; j++) v = fmaf(S.A[0][i][j], S.Z[1][j][r], v);
      S.Z[0][i][r] = v;
    }
    __syncthreads();
    for (int i = w; i < m; i += 8) {
      float v = 0.f;
      for (int j = 0; j < m; j++) v = fmaf(S.Z[1][j][i], S.Z[0][j][r], v);
      S.A[1][i][r] = v;
    }
    __syncthreads();
    cur = 1;
  }
  // ---- 1. FP32 tournament Jacobi
  const int n2 = m + (m & 1);
  for (int sweep = 0; sweep < 12 && m > 1; sweep++) {
    // every warp sums the whole matrix: the decision is the same in all
    float off = 0.f, dia = 0.f;
    for (int j = 0; j < m; j++) {
      const float a = r < m ? S.A[cur][j][r] : 0.f;
      if (j != r) off += a * a;
      else dia += a * a;
    }
    off = ritz_warp_sumf(off);
    dia = ritz_warp_sumf(dia);
    if (off <= 1e-12f * dia) break;
    for (int step = 0; step < n2 - 1; step++) {
      const float(*A)[33] = S.A[cur];
      const float(*Z)[33] = S.Z[cur];
      // the partner of index r in this step and the rotation of their pair:
      // new column r = cr * column r + sr * column pr
      int pr = r;
      float cr = 1.f, sr = 0.f;
      if (r < m) {
        int k = 0;
        if (r != 0) {
          k = r - step;
          if (k < 1) k += n2 - 1;
        }
        const int kp = n2 - 1 - k;
        int q = 0;
        if (kp != 0) {
          q = kp + step;
          if (q > n2 - 1) q -= n2 - 1;
        }
        if (q < m) {
          pr = q;
          const int lo = min(r, q), hi = max(r, q);
          const float apq = A[lo][hi];
          if (fabsf(apq) > 1e-30f) {
            // an approximate angle does (c and s stay normalised to an ulp)
            const float th = __fdividef(A[hi][hi] - A[lo][lo], 2.f * apq);
            const float h = fmaf(th, th, 1.f);
            // |th| above 2^63 (h infinite): t = 1 / (2 th) underflows to 0
            const float t = h < 3e38f
                                ? copysignf(__fdividef(1.f, fabsf(th) + h * rsqrtf(h)), th) : 0.f;
            cr = rsqrtf(fmaf(t, t, 1.f));
            sr = r == lo ? -t * cr : t * cr;
          }
        }
      }
#pragma unroll
      for (int k = 0; k < 4; k++) {
        const int i = w + 8 * k;
        const int pi = __shfl_sync(0xffffffffu, pr, i);
        const float ci = __shfl_sync(0xffffffffu, cr, i), si = __shfl_sync(0xffffffffu, sr, i);
        if (i < m && r < m) {
          const float x = fmaf(cr, A[i][r], sr * A[i][pr]);
          const float y = fmaf(cr, A[pi][r], sr * A[pi][pr]);
          S.A[cur ^ 1][i][r] = fmaf(ci, x, si * y);
          S.Z[cur ^ 1][i][r] = fmaf(cr, Z[i][r], sr * Z[i][pr]);
        }
      }
      __syncthreads();
      cur ^= 1;
    }
  }
  const float(*Z)[33] = S.Z[cur];
  for (int i = w; i < m; i += 8)
    if (r < m) Zk[i * 32 + r] = Z[i][r];
  // the lowest eigenvalue (the first of equal ones), known to every lane
  int k = r;
  {
    float v = r < m ? S.A[cur][r][r] : 3.4e38f;
    for (int o = 16; o; o >>= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, v, o);
      const int ok = __shfl_xor_sync(0xffffffffu, k, o);
      if (ov < v || (ov == v && ok < k)) {
        v = ov;
        k = ok;
      }
    }
  }
  // ---- 2. FP64 Newton refinement of the lowest pair (y unnormalised; warp 0
  // keeps it, lane = component); row products are spread over 8 threads
  double y = r < m ? (double)Z[r][k] : 0.0;
  double theta = 0.0, n = 1.0;
  const int row = tid >> 3, part = tid & 7;
  // s (FP32) drives the update; an update of c leaves an error of c times the
  // ratio of the last two in y, and its square in theta and |y|^2
  float cprev = 0.f;
  bool last = false;   // the update before was the last one: theta and |y| only
  for (int it = 0;; it++) {
    if (w == 0) S.y[r] = y;
    __syncthreads();
    if (4 * w < m) {   // the warps that hold rows below m
      double gy = 0.0;
      for (int j = part; j < m; j += 8) gy = fma(S.G[row][j], S.y[j], gy);
      for (int o = 4; o; o >>= 1) gy += __shfl_xor_sync(0xffffffffu, gy, o);
      if (part == 0) S.gy[row] = gy;
    }
    __syncthreads();
    if (w == 0) {
      const double g = r < m ? S.gy[r] : 0.0;
      // lanes below 16 sum y.gy, the others y.y
      const double a0 = y * g, n0 = y * y;
      double v = r < 16 ? a0 : n0;
      v += __shfl_xor_sync(0xffffffffu, r < 16 ? n0 : a0, 16);
      for (int o = 8; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
      const double a = __shfl_sync(0xffffffffu, v, 0);
      n = __shfl_sync(0xffffffffu, v, 16);
      const double d = n - 1.0;
      if (fabs((float)d) < 1e-4f)   // 1 / (1 + d), to d^5
        theta = a * fma(-d, fma(-d, fma(-d, 1.0 - d, 1.0), 1.0), 1.0);
      else
        theta = a / n;
      S.s32[r] = (float)(g - theta * y);
      if (r == 0) S.theta = (float)theta;
    }
    if (last) break;
    __syncthreads();
    if (4 * w < m) {
      float d = 0.f;
      for (int j = part; j < m; j += 8) d = fmaf(Z[j][row], S.s32[j], d);
      for (int o = 4; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
      float cf = 0.f;
      if (row < m && row != k) {
        const float th = S.theta, den = S.A[cur][row][row] - th;
        if (fabsf(den) > 1e-6f * fmaxf(1.f, fabsf(th))) cf = d / den;
      }
      if (part == 0) S.coef[row] = cf;
      // largest of the warp's four rows (bits of |x| order like |x|, NaN above)
      const uint32_t c = __reduce_max_sync(0xffffffffu, __float_as_uint(fabsf(cf)));
      if (r == 0) S.wmax[w] = __uint_as_float(c);
    }
    __syncthreads();
    float cm = 0.f;
    for (int j = 0; 4 * j < m; j++) cm = S.wmax[j] <= cm ? cm : S.wmax[j];
    const bool go = !(cm < 2e-10f);
    last = it + 1 == RITZ_UPDATES || (it >= 2 && !(cm < 0.5f * cprev));
    cprev = cm;
    if (4 * w < m) {
      float c = 0.f;
      for (int j = part; j < m; j += 8) c = fmaf(Z[row][j], S.coef[j], c);
      for (int o = 4; o; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
      if (part == 0) S.lam[row] = c;
    }
    __syncthreads();
    if (w == 0) {
      const double c = r < m ? (double)S.lam[r] : 0.0;
      if (!go) n -= 2.0 * (double)ritz_warp_sumf((float)y * (float)c);   // |y - c|^2, c^2 < 1e-18
      y -= c;
    }
    if (!go) break;
  }
  if (w == 0) {   // y / |y|
    const double d = n - 1.0;
    if (fabs((float)d) < 1e-4f)   // (1 + d)^(-1/2), to d^5
      y *= fma(d, fma(d, fma(d, fma(d, 35.0 / 128.0, -5.0 / 16.0), 3.0 / 8.0), -0.5), 1.0);
    else
      y /= sqrt(n);
  }
  if (tid == 0) *theta_out = theta;
  if (w == 0 && r < m) y_out[r] = y;
}
