// FP64-grade sigma vector for the exact points of the mixed-precision
// Davidson iteration, fused like the tensor-core sigma: gather, contraction
// and scatter in one kernel, with no D or E intermediate in HBM.  Requires
// c = c^T with FP32 values and |c_i| <= 1 (normalised exact-point vectors).
//
// The exact point vector c is FP32 (its values are taken as exact), so
//   D_P(a,k) = s_a c(J_a, k) + s_k c(a, J_k)
// is the exact sum of two FP32 numbers.  Per determinant m = (a, k) of a
// tile, e_m bounds |d_1| + |d_2| over all pairs P (|.| < 2^e_m): from the
// largest |c| of row k and of row a (|d_1| <= max_j |c(j, k)|, |d_2| <=
// max_j |c(a, j)|, c = c^T; k_rowmax), and
//   F_P(m) = round(d_1 2^(39 - e_m)) + round(d_2 2^(39 - e_m))   (|F| <= 2^39)
// is cut into five balanced 8-bit digits, exact in bf16; g' is cut the same
// way per row with exponent e_P (once per batch, k_slice_gp_exact).  Every
// digit product is an integer below 2^14, and each group s = i + j (i, j
// slice indices, s <= 5) of at most five such products summed over K <= 80
// stays below 2^24, so its FP32 accumulator in tensor memory is exact
// (error-free slicing: Ozaki, Ogita, Oishi & Rump, Numer. Algorithms 59, 95
// (2012)).  The six group accumulators (6 x kpad <= 480 TMEM columns) give
// the exact integer I = sum_s acc_s 2^(8 (5 - s)) with E_P(m) =
// I 2^(e_P + e_m - 54).  The scatter X(a, J) += 1/2 s E is accumulated in
// 64-bit fixed point in shared memory: units 2^Z with Z = max_P e_P + 2 - 48
// (|c| <= 1 gives e_m <= 2, so |X| < 2^60 units and each contribution is I
// shifted right by at least 7 bits, rounded).  The rows of X are written in
// FP64; sigma = X + X^T + shift S^2 c follows in k_finish_sym_fp64.  Each
// term carries an error of at most 2^-38 (2^(e_m - 40)) of the largest |g'|.
//
// Layout of a tile, as in the tensor-core sigma: M = 128 determinants
// (R rows a of X per CTA, W = 128 / R column strings k), N = kpad pairs,
// A = D digits (K-major), B = g' digits (K-major), accumulator = E^T.
//
// Instruction issue and shared-memory atomics bound it (75 MMAs are a third of
// a tile's time), so: digits by FP32 additions and byte permutes instead of
// 64-bit shifts and conversions, the small groups' integers likewise, 64-bit
// sums as two 32-bit atomics, and the next tile's global reads behind the MMAs.
// 64 x 8e/12o: 10.19 -> 7.31 ms, 8 x 10e/12o 4.06 -> 3.18 ms per call.
#include "mbe_internal.cuh"
#include "mbe_tcgen05.cuh"
#include <cuda_bf16.h>
#include <algorithm>

namespace {

using namespace tc5;

constexpr int EX_THREADS = 640;
constexpr int EX_M = 128;
constexpr int EX_SLICES = 5;
constexpr int EX_GROUPS = 6;
constexpr int EX_MAXK = 80;            // 6 groups x kpad columns <= 512: up to 12 orbitals
constexpr int EX_R = 2;                // rows a of X per CTA
constexpr uint32_t EX_TMEM_COLS = 512;

__host__ __device__ inline int ex_link_stride(int kpad) { return 8 * ((kpad >> 3) | 1); }

// frexp exponent of an FP64 value (|x| < 2^e); -1022 for zero
__device__ __forceinline__ int exp_f64(double x) {
  const int be = (int)((__double_as_longlong(x) >> 52) & 0x7FF);
  return be == 0 ? -1022 : be - 1022;
}

// frexp exponent of an FP32 value; -1000 for zero (subnormals count as zero)
__device__ __forceinline__ int exp_f32(float x) {
  const int be = (int)((__float_as_uint(x) >> 23) & 0xFF);
  return be == 0 ? -1000 : be - 126;
}

// Digits of F = round(d1 2^(39 - e)) + round(d2 2^(39 - e)), |d| < 2^e, without
// conversions (16 per clock and SM against 128 additions): with sc = 2^(39 - e)
// and y = d sc (exact), y = h 2^20 + l, |h| <= 2^19, |l| <= 2^19, and adding
// 1.5 2^23 rounds h and l to integers that stand in the low bits of the sum.
// F + 0x80808080 then has the balanced digits plus 128 as its low four bytes,
// the first digit above them; a byte u becomes the float 2^23 + u by PRMT and
// u - 128 by one addition (exact, and its upper half is the bf16 value).
__device__ __forceinline__ void split39(float d, float sc, uint32_t& h, uint32_t& l) {
  constexpr float M = 12582912.f;   // 1.5 2^23, 0x4B400000
  const float y = d * sc, t = fmaf(y, 0x1p-20f, M);
  h += __float_as_uint(t);
  l += __float_as_uint(fmaf(t - M, -0x1p20f, y) + M);
}
__device__ __forceinline__ void digits_f32(float d1, float d2, float sc, float* f) {
  uint32_t h = 0u - 2u * 0x4B400000u, l = 0x80808080u - 2u * 0x4B400000u;
  split39(d1, sc, h, l);
  split39(d2, sc, h, l);
  const long long G = (long long)(int)h * (1 << 20) + (long long)l;
  const uint32_t u = (uint32_t)G;
#pragma unroll
  for (int i = 1; i < EX_SLICES; i++)
    f[i] = __uint_as_float(__byte_perm(u, 0x4B000000u, 0x7440 | (4 - i))) - 8388736.f;
  f[0] = __int_as_float((int)(G >> 32) + 0x4B400000) - 12582912.f;
}

// round(x 2^(39 - e)) for an FP64 x, |x| < 2^e (integer ops)
__device__ __forceinline__ long long fixed39_f64(double x, int e) {
  const unsigned long long bits = (unsigned long long)__double_as_longlong(x);
  const int be = (int)((bits >> 52) & 0x7FF);
  if (be == 0) return 0;
  const long long M = (long long)((bits & 0xFFFFFFFFFFFFFull) | (1ull << 52));
  const int sh = be - 1075 + 39 - e;
  long long F = 0;
  if (sh >= 0) F = M << sh;
  else if (sh > -60) F = (M + (1LL << (-sh - 1))) >> (-sh);
  return (bits >> 63) ? -F : F;
}

// the five balanced base-256 digits of F (|F| <= 2^39), most significant first
__device__ __forceinline__ void digits5(long long F, __nv_bfloat16* s) {
#pragma unroll
  for (int i = EX_SLICES - 1; i >= 1; i--) {
    const int d = (int)(signed char)(F & 0xFF);
    s[i] = __int2bfloat16_rn(d);
    F = (F - d) >> 8;
  }
  s[0] = __int2bfloat16_rn((int)F);
}

// g' of every tuple of the batch cut into digit planes: out[b] = 5 planes of
// kpad x kpad bf16 (K-major core-matrix layout), ge[b][P] = row exponents
__global__ void k_slice_gp_exact(const double* __restrict__ gp_all, int npair, int kpad,
                                 uint8_t* __restrict__ out, int32_t* __restrict__ ge) {
  const int b = blockIdx.y;
  const double* g = gp_all + (int64_t)b * npair * npair;
  const uint32_t plane = (uint32_t)kpad * kpad * 2;
  uint8_t* o = out + (int64_t)b * EX_SLICES * plane;
  __shared__ int sE[128];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  for (int P = warp; P < kpad; P += blockDim.x >> 5) {
    double mx = 0.0;
    if (P < npair)
      for (int Q = lane; Q < npair; Q += 32) mx = fmax(mx, fabs(g[(int64_t)P * npair + Q]));
    int e = exp_f64(mx);
    for (int off = 16; off; off >>= 1) e = max(e, __shfl_xor_sync(0xffffffffu, e, off));
    if (lane == 0) {
      sE[P] = e;
      ge[(int64_t)b * kpad + P] = e;
    }
  }
  __syncthreads();
  for (int it = threadIdx.x; it < kpad * (kpad >> 3); it += blockDim.x) {
    const int row = it / (kpad >> 3), kb = (it % (kpad >> 3)) * 8;
    __align__(16) __nv_bfloat16 sl[EX_SLICES][8];
#pragma unroll
    for (int j = 0; j < 8; j++) {
      const int q = kb + j;
      const double x = (row < npair && q < npair) ? g[(int64_t)row * npair + q] : 0.0;
      __nv_bfloat16 d[EX_SLICES];
      digits5(fixed39_f64(x, sE[row]), d);
#pragma unroll
      for (int i = 0; i < EX_SLICES; i++) sl[i][j] = d[i];
    }
    const uint32_t off = kmajor_offset(row, kb, kpad);
#pragma unroll
    for (int i = 0; i < EX_SLICES; i++) *(uint4*)(o + i * plane + off) = *(uint4*)sl[i];
  }
}

// rmax[b][a] = max_k |c(a, k)| (one warp per row)
__global__ void k_rowmax(const float* __restrict__ c, int64_t c_stride, int nstr,
                         const int32_t* __restrict__ active, float* __restrict__ rmax) {
  const int b = blockIdx.y;
  if (active && !active[b]) return;
  const int a = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (a >= nstr) return;
  const float* row = c + (int64_t)b * c_stride + (int64_t)a * nstr;
  float m = 0.f;
  for (int k = lane; k < nstr; k += 32) m = fmaxf(m, fabsf(row[k]));
  for (int o = 16; o; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
  if (lane == 0) rmax[(int64_t)b * nstr + a] = m;
}

struct ExShared {
  uint32_t g, d, c_rows, x_rows, link_k, link_a, ep, em, total;
};

__host__ __device__ inline ExShared ex_layout(int kpad, int nstr) {
  constexpr int R = EX_R, W = EX_M / R;
  ExShared s;
  uint32_t o = 0;
  auto take = [&](uint32_t bytes) {
    const uint32_t r = o;
    o += (bytes + 127u) & ~127u;
    return r;
  };
  s.g = take((uint32_t)EX_SLICES * kpad * kpad * 2);
  s.d = take((uint32_t)EX_SLICES * EX_M * kpad * 2);
  s.c_rows = take((uint32_t)R * (nstr + 1) * 4);
  s.x_rows = take((uint32_t)R * (nstr + 1) * 8);
  s.link_k = take((uint32_t)2 * W * ex_link_stride(kpad) * 2);
  s.link_a = take((uint32_t)R * kpad * 4);
  s.ep = take((uint32_t)kpad * 4);
  s.em = take((uint32_t)EX_M * 4);
  s.total = o;
  return s;
}

__global__ void __launch_bounds__(EX_THREADS, 1)
k_sigma_exact(const int32_t* __restrict__ link, int nstr, int npair, int kpad,
              const uint8_t* __restrict__ gslices, const int32_t* __restrict__ ge,
              const float* __restrict__ c, int64_t c_stride, const float* __restrict__ rmax,
              const int32_t* __restrict__ active, double* __restrict__ X, int64_t x_stride,
              long long wait_limit, int32_t* __restrict__ err) {
  constexpr int R = EX_R, W = EX_M / R;
  const int LS = ex_link_stride(kpad);
  const int b = blockIdx.y;
  if (active && !active[b]) return;
  const int a0 = blockIdx.x * R;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  extern __shared__ __align__(1024) uint8_t smem[];
  __shared__ uint64_t mbar;
  __shared__ uint32_t tmem_base_sh;
  __shared__ int s_maxep;
  const ExShared L = ex_layout(kpad, nstr);
  const uint32_t gplane = (uint32_t)kpad * kpad * 2, dplane = (uint32_t)EX_M * kpad * 2;
  uint8_t* sG = smem + L.g;
  uint8_t* sD = smem + L.d;
  float* sC = (float*)(smem + L.c_rows);
  // X rows, nstr + 1 words of the low and as many of the high halves
  uint32_t* sX = (uint32_t*)(smem + L.x_rows);
  uint16_t* sLk = (uint16_t*)(smem + L.link_k);
  int32_t* sLa = (int32_t*)(smem + L.link_a);
  int* sEP = (int*)(smem + L.ep);
  int* sEm = (int*)(smem + L.em);
  const float* cb = c + (int64_t)b * c_stride;

  // ---- setup: g' digit planes, row exponents, rows a of c (zero pad), X
  {
    const uint4* src = (const uint4*)(gslices + (int64_t)b * EX_SLICES * gplane);
    uint4* dst = (uint4*)sG;
    const int n16 = (int)((EX_SLICES * gplane) >> 4);
    for (int i = tid; i < n16; i += EX_THREADS) dst[i] = src[i];
  }
  if (tid == 0) s_maxep = -1022;
  __syncthreads();
  for (int P = tid; P < kpad; P += EX_THREADS) {
    const int e = ge[(int64_t)b * kpad + P];
    sEP[P] = e;
    if (P < npair) atomicMax(&s_maxep, e);
  }
  for (int it = tid; it < R * (nstr + 1); it += EX_THREADS) {
    const int r = it / (nstr + 1), k = it - r * (nstr + 1);
    const int a = a0 + r;
    sC[it] = (a < nstr && k < nstr) ? cb[a * nstr + k] : 0.f;
  }
  for (int it = tid; it < 2 * R * (nstr + 1); it += EX_THREADS) sX[it] = 0;
  for (int it = tid; it < R * kpad; it += EX_THREADS) {
    const int r = it / kpad, P = it - r * kpad;
    const int a = a0 + r;
    const int t = (a < nstr && P < npair) ? link[a * npair + P] : -1;
    sLa[it] = t < 0 ? -1 : (((t >> 1) * nstr) << 1) | (t & 1);
  }
  if (warp == 0) tmem_alloc(&tmem_base_sh, EX_TMEM_COLS);
  if (tid == 0) {
    mbar_init(&mbar, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_base_sh;
  const int Z = s_maxep + 2 - 48;
  const uint32_t idesc = make_idesc(EX_M, kpad);
  const uint32_t sbo = (uint32_t)(kpad >> 3) * 128u;
  const int nkb = kpad >> 3;
  uint32_t phase = 0;
  bool ok = true;

  // thread -> determinant m = tid % 128 and P-blocks tid / 128 + 5 i (gather),
  // warp -> TMEM lanes 32 (w mod 4) and 8-column chunks w / 4 + 5 i (epilogue):
  // the ten blocks and chunks of kpad = 80 in two even rounds
  const int gm = tid & (EX_M - 1);
  const int gr = gm / W, gj = gm % W;
  const int ga = a0 + gr;
  const int32_t* la = sLa + gr * kpad;
  const float* crow = sC + gr * (nstr + 1);
  const int em_ = 32 * (warp & 3) + lane;
  const int er = em_ / W, ej = em_ % W;
  uint32_t* xlo = sX + er * (nstr + 1);
  int* xhi = (int*)(xlo + R * (nstr + 1));

  // What a tile reads from global memory is fetched while the MMAs of the one
  // before it run: the elements c(J_a, k) of this thread's blocks and the row
  // maximum of k into registers, the link rows into the other of two buffers
  constexpr int NB = (EX_MAXK / 8 + EX_THREADS / EX_M - 1) / (EX_THREADS / EX_M);
  float xa[NB][8], rk;
  auto fetch = [&](int k0, uint16_t* lk) {
    const int k = k0 + gj;
    const bool col_ok = ga < nstr && k < nstr;
    const float* ccol = cb + (col_ok ? k : 0);   // column 0 stands in for an invalid one
    rk = col_ok ? rmax[(int64_t)b * nstr + k] : 0.f;
#pragma unroll
    for (int i = 0; i < NB; i++) {
      const int kb = (tid >> 7) + i * (EX_THREADS / EX_M);
#pragma unroll
      for (int q = 0; q < 8; q++) {
        const int t = kb < nkb ? la[kb * 8 + q] : -1;
        xa[i][q] = ccol[t >= 0 ? (t >> 1) : 0];
      }
    }
    // link rows of the tile's column strings (pad-encoded, as in the
    // tensor-core sigma)
    for (int j = warp; j < W; j += EX_THREADS / 32) {
      uint16_t* dst = lk + j * LS;
      const int32_t* src = link + (int64_t)(k0 + j) * npair;
      for (int P = lane; P < kpad; P += 32) {
        const int t = (k0 + j < nstr && P < npair) ? src[P] : -1;
        dst[P] = (uint16_t)(t < 0 ? nstr : ((t >> 1) | ((t & 1) << 15)));
      }
    }
  };
  // the two FP32 terms of D_P(m) for the 8 pairs of block pb
  auto terms = [&](const float* x1, bool col_ok, int pb, const uint16_t* lkg, float* d1,
                   float* d2) {
    const int4 a0v = *reinterpret_cast<const int4*>(la + pb);
    const int4 a1v = *reinterpret_cast<const int4*>(la + pb + 4);
    const int4 kv = *reinterpret_cast<const int4*>(lkg + pb);
    const int ta[8] = {a0v.x, a0v.y, a0v.z, a0v.w, a1v.x, a1v.y, a1v.z, a1v.w};
    const uint32_t kw[4] = {(uint32_t)kv.x, (uint32_t)kv.y, (uint32_t)kv.z, (uint32_t)kv.w};
#pragma unroll
    for (int q = 0; q < 8; q++) {
      d1[q] = (col_ok && ta[q] >= 0) ? ((ta[q] & 1) ? -x1[q] : x1[q]) : 0.f;
      const uint32_t e = (kw[q >> 1] >> (16 * (q & 1))) & 0xFFFFu;
      const float x = crow[e & 0x7FFFu];
      d2[q] = (e & 0x8000u) ? -x : x;
    }
  };
  const float ra = ga < nstr ? rmax[(int64_t)b * nstr + ga] : 0.f;
  fetch(0, sLk);
  __syncthreads();

  for (int k0 = 0; k0 < nstr && ok; k0 += W) {
    const int k = k0 + gj;
    const bool col_ok = ga < nstr && k < nstr;
    uint16_t* lk = sLk + (k0 / W & 1) * W * LS;
    const uint16_t* lkg = lk + gj * LS;
    // ---- digit planes of D (A operand), e_m from the row maxima of c
    {
      // (below 2^-80 the terms round to zero units of X; d = 0 where !col_ok)
      const int e = max(col_ok ? exp_f32(ra + rk) : -80, -80);
      const float sc = __int_as_float((39 - e + 127) << 23);   // 2^(39 - e), e >= -80
      if (tid < EX_M) sEm[gm] = e;
#pragma unroll
      for (int r = 0; r < NB; r++) {
        const int kb = (tid >> 7) + r * (EX_THREADS / EX_M);
        if (kb >= nkb) break;
        float d1[8], d2[8];
        terms(xa[r], col_ok, kb * 8, lkg, d1, d2);
        __align__(16) uint32_t sl[EX_SLICES][4];
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
          float f0[EX_SLICES], f1[EX_SLICES];
          digits_f32(d1[q], d2[q], sc, f0);
          digits_f32(d1[q + 1], d2[q + 1], sc, f1);
#pragma unroll
          for (int i = 0; i < EX_SLICES; i++)
            sl[i][q >> 1] = __byte_perm(__float_as_uint(f0[i]), __float_as_uint(f1[i]), 0x7632);
        }
        const uint32_t off = kmajor_offset(gm, kb * 8, kpad);
#pragma unroll
        for (int i = 0; i < EX_SLICES; i++) *(uint4*)(sD + i * dplane + off) = *(uint4*)sl[i];
      }
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // ---- group accumulators: acc_s = sum_{i + j = s} D_i g'_j^T (columns s kpad)
    if (warp == 0 && elect_one()) {
      const uint32_t d0 = smem_u32(sD), g0 = smem_u32(sG);
      for (int ks = 0; ks < (kpad >> 4); ks++) {
        const uint32_t koff = (uint32_t)ks * 256u;
        for (int s = 0; s < EX_GROUPS; s++) {
          bool first = true;
          for (int i = 0; i < EX_SLICES; i++) {
            const int j = s - i;
            if (j < 0 || j >= EX_SLICES) continue;
            mma_bf16(tmem + (uint32_t)(s * kpad), make_desc(d0 + i * dplane + koff, 128, sbo),
                     make_desc(g0 + j * gplane + koff, 128, sbo), idesc,
                     (ks > 0 || !first) ? 1u : 0u);
            first = false;
          }
        }
      }
      mma_commit(&mbar);
    }
    if (k0 + W < nstr) fetch(k0 + W, sLk + ((k0 / W & 1) ^ 1) * W * LS);
    const int timed_out = mbar_wait(&mbar, phase, wait_limit) ? 0 : 1;
    if (__syncthreads_or(timed_out)) {
      ok = false;
      if (tid == 0) {
        atomicExch(err, MBE_ETIMEOUT);
        // the issued MMAs end before the accumulators are freed
        mbar_wait(&mbar, phase, SPIN_LIMIT);
      }
    }
    phase ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // ---- epilogue: exact integers I, then X(a, J) += 1/2 s I 2^(e_P + e_m - 54)
    // in units of 2^Z (a right shift by >= 7 bits, rounded)
    if (ok) {
      const int e_m = sEm[em_];
      const uint16_t* lke = lk + ej * LS;
      const uint32_t lane_off = (uint32_t)(32 * (warp & 3)) << 16;
#pragma unroll 1
      for (int ch = warp >> 2; ch < nkb; ch += EX_THREADS / EX_M) {
        uint32_t u[EX_GROUPS][8];
#pragma unroll
        for (int s = 0; s < EX_GROUPS; s++)
          tmem_ld8_nowait(tmem + lane_off + (uint32_t)(s * kpad + ch * 8), u[s]);
        const int4 kv = *reinterpret_cast<const int4*>(lke + ch * 8);
        const uint32_t kw[4] = {(uint32_t)kv.x, (uint32_t)kv.y, (uint32_t)kv.z, (uint32_t)kv.w};
        tmem_wait_ld();
#pragma unroll
        for (int s = 0; s < EX_GROUPS; s++)
#pragma unroll
          for (int q = 0; q < 8; q++) asm volatile("" : "+r"(u[s][q]));
        uint32_t lo[8], J[8];
        int hi[8];
#pragma unroll
        for (int q = 0; q < 8; q++) {
          // the groups of at most three products stay below 2^22 (3 x 80 x 2^14):
          // adding 1.5 2^23 leaves the integer in the low bits
          long long I = 0;
#pragma unroll
          for (int s = 0; s < EX_GROUPS; s++) {
            const float a = __uint_as_float(u[s][q]);
            const int v = s < 3 ? __float_as_int(a + 12582912.f) - 0x4B400000 : __float2int_rn(a);
            I += (long long)v * (1LL << (8 * (EX_GROUPS - 1 - s)));
          }
          const uint32_t t = (kw[q >> 1] >> (16 * (q & 1))) & 0xFFFFu;
          J[q] = t & 0x7FFFu;
          // >= 7; 63 and more: zero
          const int sh = min(63, Z + 54 + 1 - (sEP[ch * 8 + q] + e_m));
          long long v = ((I >> (sh - 1)) + 1) >> 1;
          if (t & 0x8000u) v = -v;
          lo[q] = (uint32_t)v;
          hi[q] = (int)(v >> 32);
        }
        // 64-bit sums as two 32-bit atomics: the low words wrap, and each wrap
        // adds one to the high word, in whatever order (a 64-bit shared atomic
        // is a compare-and-swap loop); unlinked pairs (J = nstr) are predicated
        // off (adding them to a spare column serialises on its one address)
#pragma unroll
        for (int q = 0; q < 8; q++) {
          const uint32_t old = J[q] < (uint32_t)nstr ? atomicAdd(&xlo[J[q]], lo[q]) : 0u;
          hi[q] += old + lo[q] < old ? 1 : 0;
        }
#pragma unroll
        for (int q = 0; q < 8; q++)
          if (J[q] < (uint32_t)nstr) atomicAdd(&xhi[J[q]], hi[q]);
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  }
  // ---- X rows in FP64: sX 2^Z
  const double scale = __longlong_as_double((long long)(Z + 1023) << 52);
  for (int it = tid; it < R * nstr; it += EX_THREADS) {
    const int r = it / nstr, kk = it - r * nstr;
    const int a = a0 + r;
    const int at = r * (nstr + 1) + kk;
    const long long v = (long long)(((unsigned long long)sX[R * (nstr + 1) + at] << 32) | sX[at]);
    if (a < nstr) X[(int64_t)b * x_stride + (int64_t)a * nstr + kk] = (double)v * scale;
  }
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, EX_TMEM_COLS);
}

}  // namespace

bool sigma_exact_supported(int npair, int nstr) {
  const int kpad = ((npair + 15) / 16) * 16;
  if (kpad > EX_MAXK) return false;
  return ex_layout(kpad, nstr).total + 2048 <= 227 * 1024;
}

void sigma_exact_prepare(mbe_ctx* ctx, BinProblem& bp, SigmaWork& w) {
  const int npair = bp.npair, nstr = bp.nstr;
  const int kpad = ((npair + 15) / 16) * 16;
  const ExShared L = ex_layout(kpad, nstr);
  if (kpad > EX_MAXK || L.total + 2048 > 227 * 1024)
    throw MbeError{MBE_EINVAL, "active space too large for the fused exact sigma"};
  if (!w.err.ptr) {
    w.err.reset(&ctx->pool, 1);
    CU_CHECK(cudaMemsetAsync(w.err.ptr, 0, sizeof(int32_t), ctx->stream));
  }
  // g' digit planes once per batch (g' is constant over the iteration)
  const size_t gbytes = (size_t)bp.B * EX_SLICES * kpad * kpad * 2;
  if (w.gex.n != gbytes) {
    w.gex.reset(&ctx->pool, gbytes);
    w.gexp.reset(&ctx->pool, (size_t)bp.B * kpad);
    k_slice_gp_exact<<<dim3(1, bp.B), 256, 0, ctx->stream>>>(bp.gp.ptr, npair, kpad, w.gex.ptr,
                                                             w.gexp.ptr);
    CU_LAUNCH_CHECK();
  }
  if (w.rmax.n < (size_t)bp.B * nstr) w.rmax.reset(&ctx->pool, (size_t)bp.B * nstr);
  static bool attr_done[MBE_MAX_DEVICES] = {false};
  once_per_device(attr_done, ctx->device, [] {
    CU_CHECK(cudaFuncSetAttribute(k_sigma_exact, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  227 * 1024 - 1024));
  });
}

void sigma_exact(mbe_ctx* ctx, BinProblem& bp, SigmaWork& w, const float* c, int64_t c_stride,
                 double* X, int64_t x_stride, const int32_t* active) {
  const int npair = bp.npair, nstr = bp.nstr;
  const int kpad = ((npair + 15) / 16) * 16;
  const ExShared L = ex_layout(kpad, nstr);
  // one-time set-up of the batch (allocations, g' digit planes)
  sigma_exact_prepare(ctx, bp, w);
  const dim3 grid((unsigned)((nstr + EX_R - 1) / EX_R), bp.B);
  cudaEvent_t ev;
  ctx->fp64_timer.begin(ctx->stream, ctx->opt.timing != 0, &ev);
  k_rowmax<<<dim3((unsigned)((nstr + 7) / 8), bp.B), 256, 0, ctx->stream>>>(c, c_stride, nstr,
                                                                          active, w.rmax.ptr);
  CU_LAUNCH_CHECK();
  k_sigma_exact<<<grid, EX_THREADS, L.total, ctx->stream>>>(
      bp.tab->link.ptr, nstr, npair, kpad, w.gex.ptr, w.gexp.ptr, c, c_stride, w.rmax.ptr, active,
      X, x_stride, ctx->opt.wait_limit, w.err.ptr);
  CU_LAUNCH_CHECK();
  ctx->fp64_timer.end(ctx->stream, ev);
  ctx->stats.fp64_launches += 1;
}
