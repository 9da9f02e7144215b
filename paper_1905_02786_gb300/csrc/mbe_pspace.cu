// P-space preconditioner of the mixed-precision Davidson iteration.
//
// The diagonal (Davidson) preconditioner t_I = r_I / (theta - A_II) treats
// every determinant alone.  The determinants of lowest diagonal energy are
// the ones that couple most strongly to the solution and among themselves,
// so for a set P of them the correction is taken with the exact block:
//   t_P = (theta - A_PP)^{-1} r_P,     t_I = r_I / (theta - A_II) elsewhere,
// A = H + lambda S^2 (the operator of the Davidson iteration, core energy
// excluded).  Every Davidson vector is alpha-beta symmetric, so P is a set
// of symmetric basis functions: a canonical determinant pair (a, b), a <= b,
// stands for (|a b> + |b a>) / sqrt(2) (or |a a>), and A_PP is A in that
// basis.  Per tuple, once:
//   k_psp_select  the npp canonical pairs of lowest diagonal (FP32, ties
//                 broken by index), in index order, and the lowest of them
//                 (the start vector);
//   k_psp_tri     A_PP from the Slater-Condon rules (one-electron h_eff with
//                 the core folded in, (pq|rs) of the active orbitals, the
//                 spin-exchange couplings of lambda S^2), reduced to
//                 tridiagonal form A_PP = Q T Q^T by Householder reflections
//                 in shared memory, FP32 (a preconditioner needs no more);
// per iteration:
//   k_psp_apply   t_P = Q (theta - T)^{-1} Q^T r_P, the inverse bounded by 1e4
//                 (mbe_tridiag.cuh; r_P recovered from the diagonal
//                 correction as t_I (theta - A_II)), written
//                 back into the packed vector; the same for M^-1 x, x the
//                 Ritz vector; and the first Gram-Schmidt pass's
//                 coefficients from the residual kernel's partial dots and
//                 the changed elements.
// With an exact block M^-1 r = -x on P whenever x lies in P and does not
// couple out of it (the lowest-diagonal start vector of a small space does),
// which the orthogonalisation removes, so the Davidson iteration takes
// Olsen's combination t = M^-1 r - eps M^-1 x, eps = x.M^-1 r / x.M^-1 x
// (J. Olsen, P. Jorgensen, J. Simons, Chem. Phys. Lett. 169, 463 (1990)),
// an inverse-iteration step in that case.  npp is capped at half the
// canonical pairs.
#include "mbe_internal.cuh"
#include "mbe_tridiag.cuh"
#include <algorithm>

namespace {

constexpr int PSP_MAX = 128;
static_assert(PSP_MAX == TRI_MAX, "rows of the tridiagonal solve");
constexpr int SEL_THREADS = 1024;
constexpr int TRI_THREADS = 8 * PSP_MAX;
constexpr int APPLY_THREADS = 4 * PSP_MAX;

// FP32 bit pattern mapped to an unsigned key with the same order
__device__ __forceinline__ uint32_t order_key(float x) {
  const uint32_t u = __float_as_uint(x);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// packed position p of the diagonal -> linear index a nstr + c, a <= c
__device__ __forceinline__ int linear_of(int64_t p, int nstr) {
  const int nd = sym_nd(nstr);
  if (p < nd) return (int)p * nstr + (int)p;
  const int64_t t = p - nd;   // row a starts at a (2 nstr - a - 1) / 2
  int a = (int)(((2.0f * nstr - 1.0f) - sqrtf((2.0f * nstr - 1.0f) * (2.0f * nstr - 1.0f) - 8.0f * (float)t)) * 0.5f);
  a = max(0, min(a, nstr - 2));
  while (a > 0 && (int64_t)a * (2 * nstr - a - 1) / 2 > t) a--;
  while ((int64_t)(a + 1) * (2 * nstr - a - 2) / 2 <= t) a++;
  return a * nstr + (int)(t - (int64_t)a * (2 * nstr - a - 1) / 2) + a + 1;
}

// psel[b][0..npp) = linear indices a nstr + c (a <= c) of the npp canonical
// pairs of lowest diagonal, in increasing index order; gidx[b] the lowest one
// (ties: the lower index).  One CTA per tuple, three passes over the packed
// diagonal (contiguous 16-byte loads): the smallest and largest value, a
// histogram on the linear scale between them, and the elements up to the bin
// of the npp-th, which are sorted in shared memory.  Bins near the lowest
// determinants hold few elements; where they hold more than SEL_CAP (a
// diagonal with many equal values) the threshold is found by bisection on the
// ordered keys instead, 64 more passes.  (10e/13o, 829,000 elements: 0.26 ms;
// a four-pass radix select over all pairs with the index arithmetic per
// element took 2.6 ms.)
constexpr int SEL_BINS = 4096, SEL_CAP = 2048;
struct SelShared {
  union {
    int hist[SEL_BINS];
    unsigned long long cand[SEL_CAP];   // key, then linear index
  };
};
__global__ void __launch_bounds__(SEL_THREADS)
    k_psp_select(const float* __restrict__ hd_all, int nstr, int64_t ld, int npp,
                 int32_t* __restrict__ psel, int32_t* __restrict__ gidx) {
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const float* hd = hd_all + (int64_t)b * ld;
  const int nd = sym_nd(nstr);
  const int64_t len = (int64_t)nd + (int64_t)nstr * (nstr - 1) / 2;   // the last element, + 1
  __shared__ SelShared S;
  __shared__ float s_lo[32], s_hi[32];
  __shared__ int s_n, s_bin, s_scan[32];
  // fn(value, position) over the diagonal's elements
  auto each = [&](auto fn) {
    for (int64_t q = tid; q < (ld >> 2); q += SEL_THREADS) {
      const float4 v = reinterpret_cast<const float4*>(hd)[q];
      const float x[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; e++) {
        const int64_t p = 4 * q + e;
        if (p < len && (p < nstr || p >= nd)) fn(x[e], p);
      }
    }
  };
  float lo = 3.4e38f, hi = -3.4e38f;
  each([&](float x, int64_t) {
    lo = fminf(lo, x);
    hi = fmaxf(hi, x);
  });
  for (int o = 16; o; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (lane == 0) {
    s_lo[warp] = lo;
    s_hi[warp] = hi;
  }
  for (int i = tid; i < SEL_BINS; i += SEL_THREADS) S.hist[i] = 0;
  if (tid == 0) s_n = 0;
  __syncthreads();
  for (int w = 0; w < SEL_THREADS / 32; w++) {
    lo = fminf(lo, s_lo[w]);
    hi = fmaxf(hi, s_hi[w]);
  }
  const float scale = hi > lo ? (float)(SEL_BINS - 1) / (hi - lo) : 0.f;
  auto bin = [&](float x) { return min(SEL_BINS - 1, max(0, (int)((x - lo) * scale))); };
  each([&](float x, int64_t) { atomicAdd(&S.hist[bin(x)], 1); });
  __syncthreads();
  {
    // the bin of the npp-th element: 4 bins per thread, scanned over the block
    constexpr int PER = SEL_BINS / SEL_THREADS;
    int c[PER], s = 0;
    for (int j = 0; j < PER; j++) s += c[j] = S.hist[tid * PER + j];
    int inc = s;
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) s_scan[warp] = inc;
    __syncthreads();
    int base = inc - s;
    for (int w = 0; w < warp; w++) base += s_scan[w];
    for (int j = 0; j < PER; j++) {
      if (base < npp && base + c[j] >= npp) s_bin = base + c[j] <= SEL_CAP ? tid * PER + j : -1;
      base += c[j];
    }
  }
  __syncthreads();
  uint32_t kmax = 0xffffffffu;   // key of the npp-th element (many equal values)
  const int tbin = s_bin;
  if (tbin < 0) {
    // smallest key with at least npp elements up to it
    uint32_t k0 = 0, k1 = 0xffffffffu;
    while (k0 < k1) {
      const uint32_t mid = k0 + (k1 - k0) / 2;
      int n = 0;
      each([&](float x, int64_t) { n += order_key(x) <= mid; });
      __syncthreads();
      if (tid == 0) s_n = 0;
      __syncthreads();
      atomicAdd(&s_n, n);
      __syncthreads();
      if (s_n >= npp) k1 = mid;
      else k0 = mid + 1;
    }
    kmax = k0;
    __syncthreads();
    if (tid == 0) s_n = 0;
    __syncthreads();
  }
  // candidates: below kmax all, of those equal to it the lowest indices (they
  // can be many: kept by a bound on the index, halved until they fit)
  auto put = [&](float x, int64_t p) {
    const int at = atomicAdd(&s_n, 1);
    if (at < SEL_CAP)
      S.cand[at] = ((unsigned long long)order_key(x) << 32) | (unsigned)linear_of(p, nstr);
  };
  if (tbin >= 0) {
    each([&](float x, int64_t p) {
      if (bin(x) <= tbin) put(x, p);
    });
  } else {
    // index bound such that at least npp and at most SEL_CAP elements qualify
    int i0 = 0, i1 = nstr * nstr - 1;
    while (i0 < i1) {
      const int mid = i0 + (i1 - i0) / 2;
      int n = 0;
      each([&](float x, int64_t p) {
        const uint32_t k = order_key(x);
        n += k < kmax || (k == kmax && linear_of(p, nstr) <= mid);
      });
      __syncthreads();
      if (tid == 0) s_n = 0;
      __syncthreads();
      atomicAdd(&s_n, n);
      __syncthreads();
      if (s_n >= npp) i1 = mid;
      else i0 = mid + 1;
    }
    __syncthreads();
    if (tid == 0) s_n = 0;
    __syncthreads();
    each([&](float x, int64_t p) {
      const uint32_t k = order_key(x);
      if (k < kmax || (k == kmax && linear_of(p, nstr) <= i0)) put(x, p);
    });
  }
  __syncthreads();
  // rank of every candidate by (key, index); the npp lowest, then their rank
  // by index
  const int n = min(s_n, SEL_CAP);
  __shared__ int s_sel[PSP_MAX];
  for (int i = tid; i < n; i += SEL_THREADS) {
    const unsigned long long v = S.cand[i];
    int r = 0;
    for (int j = 0; j < n; j++) r += S.cand[j] < v;
    if (r < npp) s_sel[r] = (int)(unsigned)v;
  }
  __syncthreads();
  if (tid < npp) {
    const int v = s_sel[tid];
    int r = 0;
    for (int j = 0; j < npp; j++) r += s_sel[j] < v;
    psel[(int64_t)b * PSP_MAX + r] = v;
    if (tid == 0) gidx[b] = v;
  }
}

__device__ __forceinline__ int pair_index(int p, int q) {
  return p >= q ? p * (p + 1) / 2 + q : q * (q + 1) / 2 + p;
}

// phase of a+_p a_q on the string m (q occupied, p empty): the parity of the
// occupied orbitals strictly between p and q
__device__ __forceinline__ float exc_sign(uint32_t m, int p, int q) {
  const int lo = min(p, q), hi = max(p, q);
  const uint32_t between = m & ((1u << hi) - 1u) & ~((2u << lo) - 1u);
  return (__popc(between) & 1) ? -1.f : 1.f;
}

// <na nb| H + lam S^2 |ma mb> for two different determinants (Slater-Condon
// rules; g holds (pq|rs) packed by orbital pairs, heff the one-electron
// operator with the core folded in)
__device__ float psp_offdiag(uint32_t ma, uint32_t mb, uint32_t na, uint32_t nb,
                             const float* heff, const float* g, int n, int npair, float lam) {
  const uint32_t da = ma ^ na, db = mb ^ nb;
  const int ea = __popc(da) >> 1, eb = __popc(db) >> 1;
  if (ea + eb > 2 || ea + eb == 0) return 0.f;
  auto G = [&](int p, int q, int r, int s) { return g[pair_index(p, q) * npair + pair_index(r, s)]; };
  if (ea + eb == 1) {
    // single excitation q -> p in one spin; the other spin's occupied
    // orbitals enter through the Coulomb term only
    const uint32_t m = ea ? ma : mb, nm = ea ? na : nb, d = ea ? da : db;
    const uint32_t other = ea ? mb : ma;
    const int q = __ffs(m & d) - 1, p = __ffs(nm & d) - 1;
    float v = heff[p * n + q];
    for (uint32_t k = m; k; k &= k - 1) {
      const int o = __ffs(k) - 1;
      v += G(p, q, o, o) - G(p, o, o, q);
    }
    for (uint32_t k = other; k; k &= k - 1) {
      const int o = __ffs(k) - 1;
      v += G(p, q, o, o);
    }
    return exc_sign(m, p, q) * v;
  }
  if (ea == 1 && eb == 1) {
    const int q = __ffs(ma & da) - 1, p = __ffs(na & da) - 1;
    const int s = __ffs(mb & db) - 1, r = __ffs(nb & db) - 1;
    const float sg = exc_sign(ma, p, q) * exc_sign(mb, r, s);
    float v = sg * G(p, q, r, s);
    if (p == s && q == r) v -= lam * sg;   // spin exchange (S^2 coupling)
    return v;
  }
  // same-spin double: holes q < s, particles p < r
  const uint32_t m = ea ? ma : mb, nm = ea ? na : nb, d = ea ? da : db;
  const uint32_t hm = m & d, pm = nm & d;
  const int q = __ffs(hm) - 1, s = 31 - __clz(hm);
  const int p = __ffs(pm) - 1, r = 31 - __clz(pm);
  const float s1 = exc_sign(m, p, q);
  const uint32_t m1 = m ^ (1u << p) ^ (1u << q);
  const float s2 = exc_sign(m1, r, s);
  return s1 * s2 * (G(p, q, r, s) - G(p, s, r, q));
}

constexpr int TRI_PITCH = PSP_MAX + 8;   // 8 columns of 4 rows: 32 banks

struct TriShared {
  uint32_t a_off, g_off, h_off, total;
};

__host__ __device__ inline TriShared tri_layout(int n) {
  const int npair = n * (n + 1) / 2;
  TriShared s;
  uint32_t o = 0;
  s.a_off = o;
  o += PSP_MAX * TRI_PITCH * 4;
  s.g_off = o;
  o += (uint32_t)npair * npair * 4;
  s.h_off = o;
  o += (uint32_t)n * n * 4;
  s.total = o;
  return s;
}

// A_PP in the symmetric basis and its tridiagonal form A_PP = Q T Q^T:
// tri[b] = diagonal (PSP_MAX) then subdiagonal, Qt[b][k][u] = Q[u][k].
// One CTA per tuple, eight lanes per row: a reflection is a row product, one
// barrier, the rank-two update and another; the transformation is accumulated
// backwards on Q^T, whose rows never meet, in registers.  128 functions:
// 0.40 ms for one tuple, 0.54 ms per batch of the 8e/23o expansion to order 3
// (up to 544 tuples), A_PP included; the eigenvectors by cyclic Jacobi, 1,270
// rounds of three barriers over the matrix and its rotations, took 3.7 and 5.1
// ms (22 % of that expansion).
__global__ void __launch_bounds__(TRI_THREADS)
    k_psp_tri(const uint32_t* __restrict__ masks, int nstr, int n, int nsig,
              const double* __restrict__ heff_all, const double* __restrict__ hp_all,
              const double* __restrict__ gp_all, const float* __restrict__ hd_all, int64_t ld,
              float lam, int npp, const int32_t* __restrict__ psel, float* __restrict__ tri,
              float* __restrict__ Qt) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int b = blockIdx.x;
  const int npair = n * (n + 1) / 2;
  const TriShared L = tri_layout(n);
  float* A = (float*)(smem + L.a_off);
  float* g = (float*)(smem + L.g_off);
  float* heff = (float*)(smem + L.h_off);
  __shared__ uint32_t s_ma[PSP_MAX], s_mb[PSP_MAX];
  __shared__ int s_diag[PSP_MAX];
  __shared__ float s_hd[PSP_MAX], s_p[PSP_MAX], s_beta[PSP_MAX];
  __shared__ uint8_t s_op[128], s_oq[128];
  const int tid = threadIdx.x, lane = tid & 31;
  for (int p = tid; p < n; p += blockDim.x)
    for (int q = 0; q <= p; q++) {
      s_op[p * (p + 1) / 2 + q] = (uint8_t)p;
      s_oq[p * (p + 1) / 2 + q] = (uint8_t)q;
    }
  __syncthreads();
  // (pq|rs) = g'_PQ - (h'_pq d_rs + d_pq h'_rs) / N_active (the definition of g')
  const double* gp = gp_all + (int64_t)b * npair * npair;
  const double* hp = hp_all + (int64_t)b * n * n;
  const double inv = nsig > 0 ? 1.0 / (2 * nsig) : 0.0;
  for (int t = tid; t < npair * npair; t += blockDim.x) {
    const int P = t / npair, Q = t - P * npair;
    const int p = s_op[P], q = s_oq[P], r = s_op[Q], s = s_oq[Q];
    double v = gp[t];
    if (r == s) v -= hp[p * n + q] * inv;
    if (p == q) v -= hp[r * n + s] * inv;
    g[t] = (float)v;
  }
  for (int t = tid; t < n * n; t += blockDim.x) heff[t] = (float)heff_all[(int64_t)b * n * n + t];
  // basis functions: canonical pairs (a, c), a <= c
  for (int u = tid; u < npp; u += blockDim.x) {
    const int i = psel[(int64_t)b * PSP_MAX + u];
    const int a = i / nstr, c = i - a * nstr;
    s_ma[u] = masks[a];
    s_mb[u] = masks[c];
    s_diag[u] = a == c;
    s_hd[u] = hd_all[(int64_t)b * ld + sym_index(a, c, nstr)];
  }
  for (int t = tid; t < PSP_MAX * TRI_PITCH; t += blockDim.x) A[t] = 0.f;
  __syncthreads();
  const float r2 = 0.70710678118654752f;
  for (int t = tid; t < npp * npp; t += blockDim.x) {
    const int u = t / npp, v = t - u * npp;
    if (v < u) continue;
    // |u> = c_u (|a b> + |b a>) (one term when a == b), c_u = 1/sqrt(2) or 1
    const uint32_t ua = s_ma[u], ub = s_mb[u], va = s_ma[v], vb = s_mb[v];
    float x;
    if (u == v) {
      x = s_diag[u] ? s_hd[u] : s_hd[u] + psp_offdiag(ua, ub, ub, ua, heff, g, n, npair, lam);
    } else {
      float sum = psp_offdiag(ua, ub, va, vb, heff, g, n, npair, lam);
      if (!s_diag[v]) sum += psp_offdiag(ua, ub, vb, va, heff, g, n, npair, lam);
      if (!s_diag[u]) {
        sum += psp_offdiag(ub, ua, va, vb, heff, g, n, npair, lam);
        if (!s_diag[v]) sum += psp_offdiag(ub, ua, vb, va, heff, g, n, npair, lam);
      }
      x = sum * (s_diag[u] ? 1.f : r2) * (s_diag[v] ? 1.f : r2);
    }
    A[u * TRI_PITCH + v] = x;
    A[v * TRI_PITCH + u] = x;
  }
  __syncthreads();
  const int m = npp, row = tid >> 3, l = tid & 7;
  // reflection k: v = row k right of the diagonal with its first element
  // replaced by x0 - mu, H = 1 - beta v v^T, mu the new subdiagonal element.
  // Every warp forms the sums over v itself (no barrier for them).
  for (int k = 0; k + 2 < m; k++) {
    const float* vk = A + k * TRI_PITCH;
    float s = 0.f;
    for (int j = k + 2 + lane; j < m; j += 32) s = fmaf(vk[j], vk[j], s);
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float x0 = vk[k + 1];
    const float nrm = sqrtf(fmaf(x0, x0, s));
    const float mu = x0 > 0.f ? -nrm : nrm;
    const float v0 = x0 - mu;
    const float beta = s > 1e-30f ? 2.f / fmaf(v0, v0, s) : 0.f;   // s ~ 0: H = 1
    // p = beta A v
    if (row > k && row < m) {
      float acc = 0.f;
      for (int j = k + 1 + l; j < m; j += 8)
        acc = fmaf(A[row * TRI_PITCH + j], j == k + 1 ? v0 : vk[j], acc);
      for (int o = 4; o; o >>= 1) acc += __shfl_xor_sync(0xffu << (lane & 24), acc, o);
      if (l == 0) s_p[row] = beta * acc;
    }
    __syncthreads();
    // q = p - (beta/2 p.v) v, A <- A - v q^T - q v^T
    float pv = 0.f;
    for (int j = k + 1 + lane; j < m; j += 32) pv = fmaf(s_p[j], j == k + 1 ? v0 : vk[j], pv);
    for (int o = 16; o; o >>= 1) pv += __shfl_xor_sync(0xffffffffu, pv, o);
    const float kk = 0.5f * beta * pv;
    if (row > k && row < m) {
      const float vi = row == k + 1 ? v0 : vk[row], qi = s_p[row] - kk * vi;
      for (int j = k + 1 + l; j < m; j += 8) {
        const float vj = j == k + 1 ? v0 : vk[j];
        A[row * TRI_PITCH + j] -= vi * (s_p[j] - kk * vj) + qi * vj;
      }
    }
    __syncthreads();
    if (tid == 0) {
      // row k now keeps v; its diagonal is final
      tri[(int64_t)b * 2 * PSP_MAX + k] = vk[k];
      tri[(int64_t)b * 2 * PSP_MAX + PSP_MAX + k] = beta != 0.f ? mu : x0;
      A[k * TRI_PITCH + k + 1] = v0;
      s_beta[k] = beta;
    }
    // (row k is read again only below)
  }
  __syncthreads();
  if (tid == 0) {
    for (int k = max(0, m - 2); k < m; k++) {
      tri[(int64_t)b * 2 * PSP_MAX + k] = A[k * TRI_PITCH + k];
      if (k + 1 < m) tri[(int64_t)b * 2 * PSP_MAX + PSP_MAX + k] = A[k * TRI_PITCH + k + 1];
    }
  }
  // Q^T = H_{m-3} .. H_0, row by row: R <- R - beta (R v) v^T
  float R[PSP_MAX / 8];
#pragma unroll
  for (int t = 0; t < PSP_MAX / 8; t++) R[t] = l + 8 * t == row ? 1.f : 0.f;
  for (int k = m - 3; k >= 0; k--) {
    const float* vk = A + k * TRI_PITCH;
    const float beta = s_beta[k];
    float v[PSP_MAX / 8], d = 0.f;
#pragma unroll
    for (int t = 0; t < PSP_MAX / 8; t++) {
      const int j = l + 8 * t;
      v[t] = j > k && j < m ? vk[j] : 0.f;
      d = fmaf(R[t], v[t], d);
    }
    for (int o = 4; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
    d *= beta;
#pragma unroll
    for (int t = 0; t < PSP_MAX / 8; t++) R[t] = fmaf(-d, v[t], R[t]);
  }
  float* Qb = Qt + (int64_t)b * PSP_MAX * PSP_MAX;
#pragma unroll
  for (int t = 0; t < PSP_MAX / 8; t++)
    if (row < m && l + 8 * t < m) Qb[row * PSP_MAX + l + 8 * t] = R[t];
}

// What an iteration does between the residual and the Gram-Schmidt passes,
// one CTA per tuple still iterating:
//   t_P = Q Re (theta - T + i delta)^{-1} Q^T r_P (npp = 0: no P-space), the
//   tridiagonal system by cyclic reduction, all unknowns at once (seven steps);
//   with olsen the same block solve turns u = x / (theta - A_II) (Uo, from the
//   residual kernel) into M^-1 x on P;
//   the dots x.t, x.u (xpart) and, with dots, V.t (dpart) and V.u (upart) are
//   summed over their chunks, with the changes of t and u on P;
//   Olsen's eps = x.t / x.u and the first Gram-Schmidt pass's coefficients
//   coef = V.t - eps V.u.
// Q^T comes from L2 twice (by rows for Q^T r, a warp per row; by columns for
// Q z, a quarter of a column per thread); the whole is a latency chain of a
// few thousand cycles (19-22 us a call; eigenvectors staged in shared memory,
// two of 256 threads' warps busy, took 37-47 us and four more launches for
// the sums).
__global__ void __launch_bounds__(APPLY_THREADS)
    k_psp_apply(float* __restrict__ T, const float* __restrict__ hd_all, int nstr, int64_t ld,
                const double* __restrict__ theta, int npp, const int32_t* __restrict__ psel,
                const float* __restrict__ Qt, const float* __restrict__ tri,
                const float* __restrict__ V, int m, int M, int nchunks,
                const double* __restrict__ dpart, int dots, const int32_t* __restrict__ active,
                int olsen, float* __restrict__ Uo, const float* __restrict__ X,
                const double* __restrict__ upart, const double* __restrict__ xpart,
                const double* __restrict__ y, double* __restrict__ yp, double* __restrict__ coef,
                float* __restrict__ eps) {
  const int b = blockIdx.x;
  if (!active[b]) return;
  __shared__ float s_r[PSP_MAX], s_x[PSP_MAX];
  __shared__ float s_del[PSP_MAX], s_delu[PSP_MAX], s_xv[PSP_MAX];
  __shared__ float s_pr[4][PSP_MAX], s_px[4][PSP_MAX];
  __shared__ TriC s_t[2][5][TRI_MAX];   // a, b, c and the two right-hand sides
  __shared__ int s_i[PSP_MAX];
  __shared__ double s_c[32], s_c2[32], s_xs[2];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int NW = APPLY_THREADS / 32;
  if (yp)
    for (int i = tid; i < M; i += APPLY_THREADS)
      yp[(int64_t)b * M + i] = i < m ? y[(int64_t)b * M + i] : 0.0;
  if (npp) {
    float* Tb = T + (int64_t)b * ld;
    float* Ob = olsen ? Uo + (int64_t)b * ld : nullptr;
    const float* Xb = olsen ? X + (int64_t)b * ld : nullptr;
    const float* hb = hd_all + (int64_t)b * ld;
    const float* Qb = Qt + (int64_t)b * PSP_MAX * PSP_MAX;
    const float th = (float)theta[b];
    const float sq2 = 1.41421356237309505f, r2 = 0.70710678118654752f;
    if (tid < npp) {
      const int u = tid;
      const int i0 = psel[(int64_t)b * PSP_MAX + u];
      const int a = i0 / nstr, c = i0 - a * nstr;
      const int i = (int)sym_index(a, c, nstr);          // packed position
      // the diagonal correction's denominator, exactly as the residual kernel
      float d = th - hb[i];
      if (fabsf(d) < 1e-4f) d = d < 0.f ? -1e-4f : 1e-4f;
      const float r = Tb[i] * d;
      s_r[u] = a == c ? r : sq2 * r;
      const float x = olsen ? Xb[i] : 0.f;
      s_xv[u] = x;
      s_x[u] = a == c ? x : sq2 * x;
      s_i[u] = i;
    }
    __syncthreads();
    // Q^T r and Q^T x
    for (int k = warp; k < npp; k += NW) {
      float v = 0.f, vx = 0.f;
#pragma unroll
      for (int q = 0; q < PSP_MAX / 32; q++) {
        const int u = lane + 32 * q;
        if (u < npp) {
          const float uk = Qb[k * PSP_MAX + u];
          v = fmaf(uk, s_r[u], v);
          vx = fmaf(uk, s_x[u], vx);
        }
      }
      for (int o = 16; o; o >>= 1) {
        v += __shfl_xor_sync(0xffffffffu, v, o);
        vx += __shfl_xor_sync(0xffffffffu, vx, o);
      }
      if (lane == 0) {
        s_t[0][3][k] = {v, 0.f};
        s_t[0][4][k] = {vx, 0.f};
      }
    }
    if (tid < npp) {
      const float* tb = tri + (int64_t)b * 2 * PSP_MAX;
      s_t[0][0][tid] = {tid > 0 ? -tb[PSP_MAX + tid - 1] : 0.f, 0.f};
      s_t[0][1][tid] = {th - tb[tid], TRI_DELTA};
      s_t[0][2][tid] = {tid + 1 < npp ? -tb[PSP_MAX + tid] : 0.f, 0.f};
    }
    __syncthreads();
    int cur = 0;
    for (int st = 1; st < npp; st <<= 1, cur ^= 1) {
      if (tid < npp) tri_level(s_t[cur], s_t[cur ^ 1], tid, st, npp);
      __syncthreads();
    }
    if (tid < npp) {
      s_r[tid] = tri_div(s_t[cur][3][tid], s_t[cur][1][tid]).re;
      s_x[tid] = tri_div(s_t[cur][4][tid], s_t[cur][1][tid]).re;
    }
    __syncthreads();
    {
      // Q z: thread -> u and a quarter of the k
      const int u = tid & (PSP_MAX - 1), part = tid / PSP_MAX;
      float w = 0.f, wx = 0.f;
      if (u < npp) {
        const int k1 = npp * (part + 1) / 4;
#pragma unroll 8
        for (int k = npp * part / 4; k < k1; k++) {
          const float uk = Qb[k * PSP_MAX + u];
          w = fmaf(uk, s_r[k], w);
          wx = fmaf(uk, s_x[k], wx);
        }
      }
      s_pr[part][u] = w;
      s_px[part][u] = wx;
    }
    __syncthreads();
    if (tid < npp) {
      const int u = tid, i = s_i[u];
      const float v = (s_pr[0][u] + s_pr[1][u]) + (s_pr[2][u] + s_pr[3][u]);
      const float vx = (s_px[0][u] + s_px[1][u]) + (s_px[2][u] + s_px[3][u]);
      const bool diag = i < sym_nd(nstr);
      const float f = diag ? 1.f : 2.f;   // both elements of a pair change alike
      const float tn = diag ? v : v * r2;
      s_del[u] = (tn - Tb[i]) * f;
      Tb[i] = tn;
      if (olsen) {
        const float un = diag ? vx : vx * r2;
        s_delu[u] = (un - Ob[i]) * f;
        Ob[i] = un;
      }
    }
    __syncthreads();
  }
  if (!olsen && !dots) return;
  // the sums: a warp per value
  const float* Vb = V + (int64_t)b * M * ld;
  const int nv = dots ? m : 0;
  const int ntask = olsen ? 2 * nv + 2 : nv;
  for (int t = warp; t < ntask; t += NW) {
    const bool xs = t >= 2 * nv && olsen, second = xs ? t == 2 * nv + 1 : t >= nv;
    const int i = xs ? 0 : second ? t - nv : t;
    const double* p = xs ? xpart + ((int64_t)b * 2 + (second ? 1 : 0)) * nchunks
                         : (second ? upart : dpart) + ((int64_t)b * M + i) * nchunks;
    double s = 0.0;
    for (int c = lane; c < nchunks; c += 32) s += p[c];
    for (int u = lane; u < npp; u += 32) {
      const float v = xs ? s_xv[u] : Vb[(int64_t)i * ld + s_i[u]];
      s += (double)v * (double)(second ? s_delu[u] : s_del[u]);
    }
    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) (xs ? s_xs : second ? s_c2 : s_c)[xs ? (second ? 1 : 0) : i] = s;
  }
  __syncthreads();
  double e = 0.0;
  if (olsen) {
    const double xu = s_xs[1];
    e = s_xs[0] / xu;
    if (!(xu != 0.0) || !isfinite(e)) e = 0.0;
    if (tid == 0) eps[b] = (float)e;
  }
  if (tid < nv) coef[(int64_t)b * M + tid] = olsen ? s_c[tid] - e * s_c2[tid] : s_c[tid];
}

}  // namespace

int pspace_size(const BinProblem& bp, int requested) {
  if (requested <= 0) return 0;
  const int64_t ncan = (int64_t)bp.nstr * (bp.nstr + 1) / 2;
  const int64_t cap = std::min<int64_t>({(int64_t)requested, (int64_t)PSP_MAX, ncan / 2});
  if (cap < 2) return 0;
  return (int)cap;
}

void pspace_setup(mbe_ctx* ctx, BinProblem& bp, const float* hd, int64_t ld, double shift,
                  int npp, PspaceWork& w) {
  w.npp = npp;
  if (!npp) return;
  const int B = bp.B;
  w.sel.reset(&ctx->pool, (size_t)B * PSP_MAX);
  w.low.reset(&ctx->pool, B);
  w.tri.reset(&ctx->pool, (size_t)B * 2 * PSP_MAX);
  w.Qt.reset(&ctx->pool, (size_t)B * PSP_MAX * PSP_MAX);
  cudaStream_t st = ctx->stream;
  k_psp_select<<<B, SEL_THREADS, 0, st>>>(hd, bp.nstr, ld, npp, w.sel.ptr, w.low.ptr);
  CU_LAUNCH_CHECK();
  static bool attr_set[MBE_MAX_DEVICES] = {false};
  once_per_device(attr_set, ctx->device, [] {
    CU_CHECK(cudaFuncSetAttribute(k_psp_tri, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)tri_layout(15).total));
  });
  k_psp_tri<<<B, TRI_THREADS, tri_layout(bp.n).total, st>>>(
      bp.tab->masks.ptr, bp.nstr, bp.n, bp.nsig, bp.heff.ptr, bp.hp.ptr, bp.gp.ptr, hd, ld,
      (float)shift, npp, w.sel.ptr, w.tri.ptr, w.Qt.ptr);
  CU_LAUNCH_CHECK();
}

void pspace_apply(mbe_ctx* ctx, const BinProblem& bp, const PspaceWork& w, float* T,
                  const float* hd, int64_t ld, const double* theta, const float* V, int m, int M,
                  int nchunks, const double* dpart, bool dots, const int32_t* active, bool olsen,
                  float* Uo, const float* X, const double* upart, const double* xpart,
                  const double* y, double* yp, double* coef, float* eps) {
  k_psp_apply<<<bp.B, APPLY_THREADS, 0, ctx->stream>>>(
      T, hd, bp.nstr, ld, theta, w.npp, w.sel.ptr, w.Qt.ptr, w.tri.ptr, V, m, M, nchunks, dpart,
      dots ? 1 : 0, active, olsen ? 1 : 0, Uo, X, upart, xpart, y, yp, coef, eps);
  CU_LAUNCH_CHECK();
}
