// Two-spin part of the mixed-precision sigma vector over pairs of
// (N-1)-electron strings, on the tensor cores.
//
// With K a string of nsig - 1 electrons, sg(q, K) the parity of its electrons
// below orbital q, and
//   T_qs(Ka, Kb) = sg(q, Ka) sg(s, Kb) c(Ka + q, Kb + s)   (0 if q in Ka or s in Kb)
//   U_pr(Ka, Kb) = sum_qs M[pr][qs] T_qs(Ka, Kb),
//   M[pr][qs] = g'_{pq,rs} - shift d_ps d_qr,
// the two-spin operator sum_PQ g'_PQ L_P x L_Q and the off-diagonal part of
// the spin term (S^2 = nsig - sum_pq E^a_qp E^b_pq) together are
//   Z(a, b) = sum_{p in a} sum_{r in b} sg(p, a-p) sg(r, b-r) U_pr(a-p, b-r).
// (Zarrabian, Sarma & Paldus, Chem. Phys. Lett. 155, 183 (1989).)  For c = c^T
// U_pr(Ka, Kb) = U_rp(Kb, Ka), so only the pairs Ka <= Kb are formed, with
// weight 1/2 for Ka = Kb, and Z is the result plus its transpose.  Beyond the
// default shift the spin term would carry more rounding into M and c than g'
// does (k_sigma_nm1_finish adds it in FP32 there).
//
// This is one dense GEMM per tuple: rows = the nK (nK + 1) / 2 pairs, K = N =
// n^2 orbital pairs, and its operand M is the same for every row.  Against
// the rows-of-c form (k_sigma_ab: 128 column strings per row a, K = links of a,
// N = pairs) 8e/12o takes 190 tiles of 128 rows per tuple instead of 1,980,
// and the accumulator values that have to leave tensor memory, which bound
// that kernel, are 2.7e6 instead of 2.0e7.  Measured over the iterations of a
// solve (both two-spin kernels, then the finish): 64 x 8e/12o 804 -> 326 us and
// 222 -> 68, 96 x 6e/12o 219 -> 80 and 50 -> 27, 8 x 10e/12o 452 -> 249 and
// 119 -> 38.  Errors against FP64 are those of k_sigma_ab (rms 4.7e-6 of rms
// sigma, 7 to 12 orbitals).
//
// One persistent CTA per SM, warp-specialised.  It owns a contiguous range of
// Ka (over all tuples still iterating; equal costs) and walks its pairs
// in tiles of 128 rows, a tile covering at most G values of Ka:
//   warp 0       one thread issues the MMAs (M = 128 pairs, N = NP, split
//                bf16x3) with A in tensor memory and B = M^T in shared memory;
//   warps 1-2    the nv rows Ka + q of c of every Ka (bf16 hi | lo words), into
//                a ring of GR > G shared-memory slots;
//   warp 3       B, once per tuple;
//   warps 4-7    A: a thread owns a pair (TMEM lane) and gathers its T_qs from
//                the slot's rows (its column offsets come from a table per K
//                string), in chunks of CS k-steps through a ring of NST TMEM
//                slots;
//   warps 8-23   add the accumulator rows into shared row sums, one per (Ka, p):
//                sum(Ka, p)[Kb + r] += sg(r, Kb) U_pr.  Lanes of a warp hit
//                distinct elements for one r; NC copies of the sums and 4 / NC
//                barrier-separated phases keep the warps apart, so there are
//                no atomics and the order is fixed.  A finished Ka is written
//                to its slot (nK nv rows per tuple); k_sigma_nm1_finish sums
//                the nsig slots of each row.
// The row sums bound it (8e/12o: 6,000 of 11,000 cycles per tile add, 3,000 copy
// finished rows out): each step is a shared-memory load, add and store whose
// lanes hit about two banks' worth of columns, in a serial chain over r.  So an
// orbital that every lane's Ka holds is skipped (a quarter at 4 of 12), sixteen
// warps share the sums and four build A (eight and eight: 435 us at 8e/12o), and
// finished rows leave 16 bytes at a time.  The tables are 16-bit, 32 bytes per
// string, two loads per lane (one word per orbital: 358 us).  CTAs get equal
// costs, not equal rows: a tile holds at most G strings, so a tuple's last ones
// fill few of its rows (equal rows: 435 -> 389 us, 10e/12o 402 -> 304 us).
// Every wait is bounded as in k_sigma_ab.
#include "mbe_internal.cuh"
#include "mbe_tcgen05.cuh"
#include <cuda_bf16.h>
#include <algorithm>
#include <type_traits>

namespace {

using namespace tc5;
typedef __nv_bfloat16 bf16;

constexpr int NM_CWARPS = 2, NM_BWARP = 3, NM_BUILD0 = 4, NM_EPI0 = 8, NM_THREADS = 768;
constexpr int NM_GR_MAX = 20;
constexpr int NM_EPI = NM_THREADS - 32 * NM_EPI0;   // epilogue threads
constexpr int NM_EH = NM_EPI / 128;                 // its warps per TMEM quadrant
constexpr uint32_t NM_HINT_NS = 1000, NM_SLEEP = 64;
constexpr uint32_t NM_SMEM_MAX = 222 * 1024;
constexpr uint32_t NM_SMEM_MIN = 116 * 1024;   // one CTA per SM (512 TMEM columns)

template <int N>
struct Shape {
  static constexpr int NS = (N + 1) & ~1;                      // s padded to even
  static constexpr int CQ = N <= 6 ? N : N == 9 ? 3 : N == 10 ? 5 : 4;   // q per chunk
  static constexpr int CH = (N + CQ - 1) / CQ;                 // chunks per tile
  static constexpr int CK = (CQ * NS + 15) / 16 * 16;          // k of a chunk, zero padded
  static constexpr int CS = CK / 16;                           // its k-steps
  static constexpr int KP = CH * CK;
  static constexpr int NP = (N * N + 15) / 16 * 16;
  static constexpr int ACOLS = CK;                             // TMEM columns of a slot (hi, lo)
  static constexpr int NST = (512 - 2 * NP) / ACOLS < 4 ? (512 - 2 * NP) / ACOLS : 4;
};

struct NmPlan {
  int cq, ck, KP, NP;
  int G, GR, NC, NB, nst, nv, nK, R, ldw;   // ldw: words per row of the operand
  uint32_t b_bytes, acc, rows, zero, list, total;
};

__device__ __forceinline__ void bar_sync_n(int id, int n) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(n) : "memory");
}
__device__ __forceinline__ bool bar_red_or(int id, int n, bool pred) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 q, %1, 0;\n\t"
      "bar.red.or.pred p, %2, %3, q;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)pred), "r"(id), "r"(n)
      : "memory");
  return r != 0;
}
// W consecutive columns from W registers
template <int W>
__device__ __forceinline__ void tmem_st(uint32_t taddr, const uint32_t* r) {
  if constexpr (W >= 4) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x4.b32 [%0], {%1,%2,%3,%4};" ::"r"(taddr),
                 "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3])
                 : "memory");
    tmem_st<W - 4>(taddr + 4, r + 4);
  } else if constexpr (W >= 2) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x2.b32 [%0], {%1,%2};" ::"r"(taddr), "r"(r[0]),
                 "r"(r[1])
                 : "memory");
    tmem_st<W - 2>(taddr + 2, r + 2);
  } else if constexpr (W == 1) {
    asm volatile("tcgen05.st.sync.aligned.32x32b.x1.b32 [%0], {%1};" ::"r"(taddr), "r"(r[0])
                 : "memory");
  }
}
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ float lds(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ uint32_t lds_u(uint32_t a) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts(uint32_t a, float v) {
  asm volatile("st.shared.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}
// A from tensor memory (row = lane, two consecutive k per column), B from
// shared memory
__device__ __forceinline__ void mma_bf16_ta(uint32_t tmem_d, uint32_t tmem_a, uint64_t db,
                                            uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(tmem_d),
      "r"(tmem_a), "l"(db), "r"(idesc), "r"(accumulate));
}

// row length of the sums and of the rows of c in shared memory: a spare element
// at column ldw (an absent column adds there and reads zero), 16-byte rows
__host__ __device__ inline int nm_ars(int nstr) { return ((nstr + 3) & ~3) + 4; }

// the table of columns by K string: (column << 1 | parity) of K + s as 16-bit
// words, 16 per string, `ldw` for an s in K
template <int N>
__device__ __forceinline__ void nm_columns(const uint4* __restrict__ kcol, int kb, uint32_t* w) {
  const uint4 a = kcol[2 * kb];
  w[0] = a.x;
  w[1] = a.y;
  w[2] = a.z;
  if (N > 6) w[3] = a.w;
  if (N > 8) {
    const uint2 c = *reinterpret_cast<const uint2*>(&kcol[2 * kb + 1]);
    w[4] = c.x;
    if (N > 10) w[5] = c.y;
  }
}
// byte offset of column x, and its parity in bit 31
__device__ __forceinline__ uint32_t nm_off(const uint32_t* w, int x) {
  return ((x & 1 ? w[x >> 1] >> 16 : w[x >> 1]) & 0xfffeu) << 1;
}
__device__ __forceinline__ uint32_t nm_par(const uint32_t* w, int x) {
  return (x & 1 ? w[x >> 1] << 15 : w[x >> 1] << 31) & 0x80000000u;
}

// cost of the Ka before k, in rows: Ka has nK - Ka pairs, but a tile holds at
// most G of them, so the last ones cost 128 / G rows each whatever they hold
__host__ __device__ inline long long nm_start(long long k, long long nK, int G) {
  const long long w = 128 / G, kx = nK > w ? nK - w : 0, ke = k < kx ? k : kx;
  return ke * nK - ke * (ke - 1) / 2 + (k - ke) * w;
}

// position x in the cost of all tuples -> the next start of a Ka at or
// after it: (tuple, Ka)
__device__ inline void nm_locate(long long x, long long R, int nK, int G, int& t,
                                 int& k) {
  t = (int)(x / R);
  const long long y = x - (long long)t * R;
  int lo = 0, hi = nK;
  while (lo < hi) {
    const int mid = (lo + hi) >> 1;
    if (nm_start(mid, nK, G) < y) lo = mid + 1;
    else hi = mid;
  }
  k = lo;
  if (k == nK) {
    t++;
    k = 0;
  }
}

// a walk over the pairs of one tuple: the pair `rem` rows after (k, o),
// k < klim (k = klim: past the tile's last Ka)
__device__ __forceinline__ void nm_walk(int& k, int& o, int rem, int klim, int nK) {
  while (k < klim && rem >= nK - k - o) {
    rem -= nK - k - o;
    k++;
    o = 0;
  }
  if (k < klim) o += rem;
}

template <int N>
__global__ void __launch_bounds__(NM_THREADS, 1)
k_sigma_nm1(const int32_t* __restrict__ krow, const uint4* __restrict__ kcol,
            const uint32_t* __restrict__ kmask,
            const int32_t* __restrict__ kj0, const uint8_t* __restrict__ bop,
            const uint32_t* __restrict__ cw, int nstr, int ldS, const int32_t* __restrict__ active,
            int B, NmPlan L, float* __restrict__ slots, long long wait_limit,
            int32_t* __restrict__ err) {
  using S = Shape<N>;
  extern __shared__ uint8_t dsm[];
  uint8_t* sm = dsm + ((1024u - (smem_u32(dsm) & 1023u)) & 1023u);
  __shared__ uint64_t full_a[4], empty_a[4], full_b[2], empty_b[2], acc_full[2], acc_empty[2],
      full_c[NM_GR_MAX], empty_c[NM_GR_MAX], mdone;
  __shared__ uint32_t tmem_sh;
  __shared__ int abort_sh, s_nact, s_cnt[NM_THREADS / 32];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  volatile int* abort_v = &abort_sh;
  float* sAcc = reinterpret_cast<float*>(sm + L.acc);
  uint16_t* sList = reinterpret_cast<uint16_t*>(sm + L.list);
  const int nK = L.nK, nv = L.nv, G = L.G, GR = L.GR, NC = L.NC, NB = L.NB, nst = L.nst;
  const int ldw = L.ldw;
  // every row has a spare element past its end (an absent column adds there;
  // in the rows of c it is a zero word), and one spare row each (an absent
  // orbital): the inner loops need no branches
  const int ars = nm_ars(nstr), crs = ars;
  for (uint32_t i = L.acc / 4 + tid; i < L.list / 4; i += NM_THREADS)
    reinterpret_cast<uint32_t*>(sm)[i] = 0u;
  if (tid == 0) {
    for (int s = 0; s < 4; s++) {
      mbar_init(&full_a[s], 4);
      mbar_init(&empty_a[s], 1);
    }
    for (int s = 0; s < 2; s++) {
      mbar_init(&full_b[s], 1);
      mbar_init(&empty_b[s], 1);
      mbar_init(&acc_full[s], 1);
      mbar_init(&acc_empty[s], NM_EPI / 32);
    }
    for (int s = 0; s < L.GR; s++) {
      mbar_init(&full_c[s], 1);
      mbar_init(&empty_c[s], 4);
    }
    mbar_init(&mdone, 1);
    abort_sh = 0;
    s_nact = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) tmem_alloc(&tmem_sh, 512);
  __syncthreads();
  // the tuples still iterating, in order
  for (int b0 = 0; b0 < B; b0 += NM_THREADS) {
    const int b = b0 + tid;
    const bool on = b < B && (!active || active[b]);
    const unsigned m = __ballot_sync(0xffffffffu, on);
    if (lane == 0) s_cnt[warp] = __popc(m);
    __syncthreads();
    int at = s_nact;
    for (int w = 0; w < warp; w++) at += s_cnt[w];
    if (on) sList[at + __popc(m & ((1u << lane) - 1u))] = (uint16_t)b;
    __syncthreads();
    if (tid == 0)
      for (int w = 0; w < NM_THREADS / 32; w++) s_nact += s_cnt[w];
    __syncthreads();
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_sh;
  // this CTA's range: from (t0, k0) up to (t1, k1), exclusive
  int t0, k0, t1, k1;
  const long long R = L.R, total = R * s_nact;
  nm_locate(total * blockIdx.x / gridDim.x, R, nK, G, t0, k0);
  nm_locate(total * (blockIdx.x + 1) / gridDim.x, R, nK, G, t1, k1);
  const int tend = k1 > 0 ? t1 + 1 : t1;
  // the range of Ka of tuple position t
  auto kbeg = [&](int t) { return t == t0 ? k0 : 0; };
  auto kend = [&](int t) { return t == t1 ? k1 : nK; };

  if (warp == 0) {
    // ------------------------------------------------ MMA issue
    if (elect_one()) {
      constexpr uint32_t idesc = make_idesc(128, S::NP);
      constexpr uint32_t sbo = (uint32_t)(S::KP >> 3) * 128u;
      uint32_t j = 0, it = 0, ib = 0;
      bool ok = true;
      for (int t = t0; t < tend && ok; t++) {
        const int sbb = (int)(ib % (uint32_t)NB);
        ok = mbar_wait_or_abort(&full_b[sbb], (ib / (uint32_t)NB) & 1u, wait_limit, abort_v,
                                NM_HINT_NS, NM_SLEEP);
        if (!ok) break;
        const uint32_t bh = smem_u32(sm + (uint32_t)sbb * L.b_bytes), bl = bh + L.b_bytes / 2;
        const int ke = kend(t);
        int k = kbeg(t), o = 0;
        while (k < ke && ok) {
          nm_walk(k, o, 128, min(ke, k + G), nK);
          const int sb = (int)(it & 1u);
          ok = mbar_wait_or_abort(&acc_empty[sb], ((it >> 1) & 1u) ^ 1u, wait_limit, abort_v,
                                  NM_HINT_NS, NM_SLEEP);
          if (!ok) break;
          const uint32_t d = tmem + (uint32_t)(sb * S::NP);
          for (int ci = 0; ci < S::CH; ci++, j++) {
            const int sa = (int)(j % (uint32_t)nst);
            ok = mbar_wait_or_abort(&full_a[sa], (j / (uint32_t)nst) & 1u, wait_limit, abort_v,
                                    NM_HINT_NS, NM_SLEEP);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t ah = tmem + (uint32_t)(2 * S::NP + sa * S::ACOLS);
            const uint32_t al = ah + (uint32_t)(S::CS * 8);
            for (int kk = 0; kk < S::CS; kk++) {
              const uint32_t ko = (uint32_t)(ci * S::CS + kk) * 256u;
              const uint64_t dh = make_desc(bh + ko, 128, sbo), dl = make_desc(bl + ko, 128, sbo);
              mma_bf16_ta(d, ah + (uint32_t)(kk * 8), dh, idesc, (ci | kk) ? 1u : 0u);
              mma_bf16_ta(d, al + (uint32_t)(kk * 8), dh, idesc, 1u);
              mma_bf16_ta(d, ah + (uint32_t)(kk * 8), dl, idesc, 1u);
            }
            mma_commit(&empty_a[sa]);
          }
          if (!ok) break;
          mma_commit(&acc_full[sb]);
          it++;
        }
        if (!ok) break;
        mma_commit(&empty_b[sbb]);
        ib++;
      }
      if (!ok) {
        *abort_v = 1;
        atomicExch(err, MBE_ETIMEOUT);
      }
      // every MMA issued here ends before the tensor memory is freed
      mma_commit(&mdone);
      mbar_wait(&mdone, 0, SPIN_LIMIT);
    }
  } else if (warp == NM_BWARP) {
    // ------------------------------------------------ B: M^T of the tuple
    uint32_t ib = 0;
    bool ok = true;
    for (int t = t0; t < tend && ok; t++, ib++) {
      const int sbb = (int)(ib % (uint32_t)NB);
      const bool got = lane == 0 ? mbar_wait_or_abort(&empty_b[sbb], ((ib / (uint32_t)NB) & 1u) ^ 1u,
                                                      wait_limit, abort_v, NM_HINT_NS, 256)
                                 : true;
      ok = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
      if (!ok) break;
      const uint8_t* src = bop + (int64_t)sList[t] * L.b_bytes;
      const uint32_t dst = smem_u32(sm + (uint32_t)sbb * L.b_bytes);
      for (uint32_t i = (uint32_t)lane * 16u; i < L.b_bytes; i += 512u)
        cp_async16(dst + i, src + i, 16u);
      cp_async_commit();
      cp_async_wait<0>();
      fence_async_smem();
      __syncwarp();
      if (lane == 0) mbar_arrive(&full_b[sbb]);
    }
    if (!ok && lane == 0) {
      *abort_v = 1;
      atomicExch(err, MBE_ETIMEOUT);
    }
  } else if (warp <= NM_CWARPS) {
    // ------------------------------------------------ rows Ka + q of c
    // the CTA's Ka in order; this warp takes every other one
    uint32_t x = 0;
    bool ok = true;
    for (int t = t0; t < tend && ok; t++) {
      const uint32_t* cb = cw + (int64_t)sList[t] * nstr * ldw;
      for (int k = kbeg(t); k < kend(t); k++, x++) {
        if ((int)(x & 1u) != warp - 1) continue;
        const int sl = (int)(x % (uint32_t)GR);
        const bool got =
            lane == 0 ? mbar_wait_or_abort(&empty_c[sl], ((x / (uint32_t)GR) & 1u) ^ 1u, wait_limit,
                                           abort_v, NM_HINT_NS, 256)
                      : true;
        ok = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
        if (!ok) break;
        const uint32_t dst = smem_u32(sm + L.rows) + (uint32_t)(sl * nv * crs) * 4u;
        // the strings Ka + q, q ascending (lane: q)
        const int e = lane < 16 ? krow[k * 16 + lane] : -1;
        unsigned on = __ballot_sync(0xffffffffu, e >= 0);
        for (int pi = 0; on; pi++, on &= on - 1) {
          const int row = __shfl_sync(0xffffffffu, e, __ffs(on) - 1) >> 1;
          const uint32_t* src = cb + (int64_t)row * ldw;
          for (int i = lane * 4; i < ldw; i += 128)
            cp_async16(dst + (uint32_t)(pi * crs + i) * 4u, src + i, 16u);
        }
        cp_async_commit();
        cp_async_wait<0>();
        __syncwarp();
        if (lane == 0) mbar_arrive(&full_c[sl]);
      }
    }
    cp_async_wait<0>();
    if (!ok && lane == 0) {
      *abort_v = 1;
      atomicExch(err, MBE_ETIMEOUT);
    }
  } else if (warp < NM_EPI0) {
    // ------------------------------------------------ A: T rows
    const int m = 32 * (warp & 3) + lane;
    const uint32_t ta = tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)(2 * S::NP);
    const uint32_t sRows = smem_u32(sm + L.rows), zrow = smem_u32(sm + L.zero);
    uint32_t j = 0, xt = 0;   // xt: position of the tuple's first Ka in the row ring
    bool ok = true;
    // the pad columns of the slots stay zero
    for (int c = 0; c < nst * S::ACOLS; c += 4) {
      const uint32_t z[4] = {0u, 0u, 0u, 0u};
      tmem_st<4>(ta + (uint32_t)c, z);
    }
    tmem_wait_st();
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    bar_sync_n(2, 128);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    for (int t = t0; t < tend && ok; xt += (uint32_t)(kend(t) - kbeg(t)), t++) {
      const int ke = kend(t), kb0 = kbeg(t);
      int k = kb0, o = 0;
      while (k < ke && ok) {
        const int klim = min(ke, k + G), kfirst = k;
        int ka = k, kb = o;
        nm_walk(ka, kb, m, klim, nK);
        const bool valid = ka < klim;
        kb = valid ? ka + kb : 0;
        if (!valid) ka = kfirst;
        nm_walk(k, o, 128, klim, nK);
        // column offsets and signs of this pair's s (absent, also a row past the
        // tile's end: the zero word)
        uint32_t cs[6], off[S::NS], sg[S::NS];
        nm_columns<N>(kcol, kb, cs);
#pragma unroll
        for (int q = 0; q < S::NS; q++) {
          off[q] = q < N && valid ? nm_off(cs, q) : (uint32_t)ldw * 4u;
          sg[q] = q < N ? (nm_par(cs, q) >> 31) * 0x80008000u : 0u;
        }
        // the rows of the tile's Ka: kfirst up to the last one it touches
        const int klast = min(klim - 1, o > 0 ? k : k - 1);
        for (int kc = kfirst; kc <= klast && ok; kc++) {
          const uint32_t x = xt + (uint32_t)(kc - kb0);
          const bool got = lane == 0 ? mbar_wait_or_abort(&full_c[x % (uint32_t)GR],
                                                          (x / (uint32_t)GR) & 1u, wait_limit,
                                                          abort_v, NM_HINT_NS, NM_SLEEP)
                                     : true;
          ok = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
        }
        if (!ok) break;
        const uint32_t ma = kmask[ka];
        const uint32_t mine =
            sRows + (uint32_t)((int)((xt + (uint32_t)(ka - kb0)) % (uint32_t)GR) * nv * crs) * 4u;
        for (int ci = 0; ci < S::CH; ci++, j++) {
          const int sa = (int)(j % (uint32_t)nst);
          const bool got =
              lane == 0 ? mbar_wait_or_abort(&empty_a[sa], ((j / (uint32_t)nst) & 1u) ^ 1u,
                                             wait_limit, abort_v, NM_HINT_NS, NM_SLEEP)
                        : true;
          ok = __shfl_sync(0xffffffffu, got ? 1 : 0, 0) != 0;
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t ts = ta + (uint32_t)(sa * S::ACOLS);
          const int q1 = min(N, ci * S::CQ + S::CQ);
          for (int q = ci * S::CQ, qi = 0; qi < S::CQ; q++, qi++) {
            // (q past the last orbital: zeros, in the last chunk only)
            const uint32_t below = (uint32_t)__popc(ma & ((1u << q) - 1u));
            const bool in = q < q1 && !((ma >> q) & 1u);
            const uint32_t row = in ? mine + (uint32_t)(q - (int)below) * (uint32_t)crs * 4u : zrow;
            const uint32_t sq = (below & 1u) ? 0x80008000u : 0u;
            uint32_t w[S::NS], hi[S::NS / 2], lo[S::NS / 2];
            if (__any_sync(0xffffffffu, in)) {
#pragma unroll
              for (int x = 0; x < S::NS; x++) w[x] = lds_u(row + off[x]);
#pragma unroll
              for (int x = 0; x < S::NS; x++) w[x] ^= sq ^ sg[x];
            } else {
#pragma unroll
              for (int x = 0; x < S::NS; x++) w[x] = 0u;
            }
#pragma unroll
            for (int x = 0; x < S::NS / 2; x++) {
              hi[x] = __byte_perm(w[2 * x], w[2 * x + 1], 0x5410);
              lo[x] = __byte_perm(w[2 * x], w[2 * x + 1], 0x7632);
            }
            tmem_st<S::NS / 2>(ts + (uint32_t)(qi * (S::NS / 2)), hi);
            tmem_st<S::NS / 2>(ts + (uint32_t)(S::CK / 2 + qi * (S::NS / 2)), lo);
          }
          tmem_wait_st();
          asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
          __syncwarp();
          if (lane == 0) mbar_arrive(&full_a[sa]);
        }
        if (!ok) break;
        // the rows of the finished Ka are free
        __syncwarp();
        if (lane == 0)
          for (int kc = kfirst; kc < k; kc++)
            mbar_arrive(&empty_c[(xt + (uint32_t)(kc - kb0)) % (uint32_t)GR]);
      }
    }
    if (!ok && lane == 0) {
      *abort_v = 1;
      atomicExch(err, MBE_ETIMEOUT);
    }
  } else {
    // ------------------------------------------------ row sums
    const int e = warp - NM_EPI0, qd = warp & 3, h = e >> 2, et = tid - NM_EPI0 * 32;
    const int m = 32 * qd + lane;
    const int PH = 4 / NC;
    const uint32_t cls = NC == 1 ? 1u : NC == 2 ? 0x0101u : 0x1111u;   // every NM_EH PH-th p
    const uint32_t copy = smem_u32(sAcc + (int64_t)(qd * NC / 4) * G * nv * ars);
    const uint32_t spare = smem_u32(sAcc + (int64_t)NC * G * nv * ars);
    const int cstride = G * nv * ars;
    uint32_t it = 0;
    bool ok = true;
    for (int t = t0; t < tend && ok; t++) {
      float* sl = slots + (int64_t)sList[t] * nK * nv * ldS;
      const int ke = kend(t);
      int k = kbeg(t), o = 0;
      // a tile's table entries are loaded while the tile before it is flushed
      int ka, kb, j0v, slot = k % G;   // slot: of the sums of Ka = k
      uint32_t ma, cs[6];
      bool valid;
      auto fetch = [&]() {
        const int klim = min(ke, k + G);
        ka = k;
        kb = o;
        nm_walk(ka, kb, m, klim, nK);
        valid = ka < klim;
        kb = valid ? ka + kb : 0;
        if (!valid) ka = k;
        nm_columns<N>(kcol, kb, cs);
        ma = valid ? kmask[ka] : 0xffffffffu;
        j0v = kj0[min(k + lane, nK - 1)];   // lane i: the tile's i-th Ka
      };
      if (k < ke) fetch();
      while (k < ke) {
        const int klim = min(ke, k + G), kfirst = k, j0s = j0v;
        int ks = slot + ka - kfirst;
        if (ks >= G) ks -= G;
        nm_walk(k, o, 128, klim, nK);
        // column offsets and signs of this pair's r (absent: the spare element)
        uint32_t off[N];
        float f[N];
        const float wgt = ka == kb ? 0.5f : 1.f;
#pragma unroll
        for (int r = 0; r < N; r++) {
          off[r] = nm_off(cs, r);
          f[r] = __uint_as_float(__float_as_uint(wgt) ^ nm_par(cs, r));
        }
        const int sb = (int)(it & 1u);
        const bool got = lane == 0 ? mbar_wait_or_abort(&acc_full[sb], (it >> 1) & 1u, wait_limit,
                                                        abort_v, NM_HINT_NS, NM_SLEEP)
                                   : true;
        // also: the last flush is done before this tile adds to its slots
        if (bar_red_or(1, NM_EPI, !got)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t td = tmem + ((uint32_t)(32 * qd) << 16) + (uint32_t)(sb * S::NP);
        const uint32_t rows = copy + (uint32_t)(ks * nv * ars) * 4u;
        // the rows of p = x, x + NG, .. (those some lane has), two at a time:
        // their updates interleave.  A lane whose Ka holds p adds to the spare row
        auto update = [&](auto nx, const int* p) {
          constexpr int X = decltype(nx)::value;
          uint32_t u[X][16], ro[X];
#pragma unroll
          for (int x = 0; x < X; x++) {
            ro[x] = !((ma >> p[x]) & 1u)
                        ? rows + (uint32_t)((p[x] - __popc(ma & ((1u << p[x]) - 1u))) * ars) * 4u
                        : spare;
            // (p N + 16 <= 2 NP: the reads stay inside the accumulators)
            tmem_ld8_nowait(td + (uint32_t)(p[x] * N), u[x]);
            if (N > 8) tmem_ld4_nowait(td + (uint32_t)(p[x] * N + 8), u[x] + 8);
          }
          tmem_wait_ld();
#pragma unroll
          for (int x = 0; x < X; x++)
#pragma unroll
            for (int r = 0; r < N; r++) asm volatile("" : "+r"(u[x][r]));
#pragma unroll
          for (int r = 0; r < N; r++) {
            float y[X];
#pragma unroll
            for (int x = 0; x < X; x++) y[x] = lds(ro[x] + off[r]);
#pragma unroll
            for (int x = 0; x < X; x++)
              sts(ro[x] + off[r], fmaf(f[r], __uint_as_float(u[x][r]), y[x]));
            __syncwarp();   // another lane may take this element at the next r
          }
        };
        const uint32_t todo = ~__reduce_and_sync(0xffffffffu, ma) & ((1u << N) - 1u);
        for (int ph = 0; ph < PH; ph++) {
          uint32_t mine = todo & (cls << (h * PH + ((qd + ph) & (PH - 1))));
          while (mine) {
            int p[2];
            p[0] = __ffs(mine) - 1;
            mine &= mine - 1;
            if (mine) {
              p[1] = __ffs(mine) - 1;
              mine &= mine - 1;
              update(std::integral_constant<int, 2>(), p);
            } else {
              update(std::integral_constant<int, 1>(), p);
            }
          }
          if (ph + 1 < PH) bar_sync_n(1, NM_EPI);
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) mbar_arrive(&acc_empty[sb]);
        it++;
        if (k < ke) fetch();
        if (k > kfirst) {
          // Ka = kfirst .. k - 1 are complete: to their slots, sums cleared
          // (nothing was added left of kj0; 16 bytes at a time)
          bar_sync_n(1, NM_EPI);
          for (int kc = kfirst; kc < k; kc++) {
            const int j0 = __shfl_sync(0xffffffffu, j0s, kc - kfirst) & ~3;
            float* src = sAcc + slot * nv * ars + j0;
            if (++slot == G) slot = 0;
            float* dst = sl + (int64_t)kc * nv * ldS + j0;
            const int w4 = (nstr - j0 + 3) >> 2;
            int pi = 0, c = et;
            while (c >= w4 && pi < nv) {
              c -= w4;
              pi++;
            }
            while (pi < nv) {
              float4* q = reinterpret_cast<float4*>(src + pi * ars) + c;
              float4 x = *q;
              *q = make_float4(0.f, 0.f, 0.f, 0.f);
              for (int cp = 1; cp < NC; cp++) {
                q += cstride / 4;
                const float4 y = *q;
                *q = make_float4(0.f, 0.f, 0.f, 0.f);
                x.x += y.x;
                x.y += y.y;
                x.z += y.z;
                x.w += y.w;
              }
              *reinterpret_cast<float4*>(dst + (int64_t)pi * ldS + 4 * c) = x;
              c += NM_EPI;
              while (c >= w4 && pi < nv) {
                c -= w4;
                pi++;
              }
            }
          }
        }
      }
    }
    if (!ok && et == 0) {
      *abort_v = 1;
      atomicExch(err, MBE_ETIMEOUT);
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  if (warp == 0) tmem_dealloc(tmem, 512);
}

// B operand of every tuple: rows (p, r) of M, K-major core matrices, hi then
// lo halves
__global__ void k_nm1_operand(const double* __restrict__ gp_all, int n, int npair, int ns, int cq,
                              int ck, int KP, int NP, double shift, uint8_t* __restrict__ out) {
  const int b = blockIdx.y;
  const double* g = gp_all + (int64_t)b * npair * npair;
  const uint32_t half = (uint32_t)KP * NP * 2;
  uint8_t* o = out + (int64_t)b * 2 * half;
  auto pr = [](int p, int q) { return p >= q ? p * (p + 1) / 2 + q : q * (q + 1) / 2 + p; };
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < KP * NP; t += gridDim.x * blockDim.x) {
    const int row = t / KP, k = t - row * KP;
    const int p = row / n, r = row - p * n, kc = k % ck, qi = kc / ns;
    const int q = k / ck * cq + qi, s = kc - qi * ns;
    double v = 0.0;
    if (p < n && qi < cq && q < n && s < n) {
      v = g[(int64_t)pr(p, q) * npair + pr(r, s)];
      if (p == s && q == r) v -= shift;
    }
    const bf16 h = __double2bfloat16(v);
    const uint32_t off = kmajor_offset(row, k, KP);
    *reinterpret_cast<bf16*>(o + off) = h;
    *reinterpret_cast<bf16*>(o + half + off) = __double2bfloat16(v - (double)__bfloat162float(h));
  }
}

// K strings (nsig - 1 electrons): krow[K][o] = (index of K + o << 1) | parity
// of K's electrons below o, -1 if o is in K (16 per string); kcol the same for
// nm_columns; kj0[K] the first
// string with a larger mask; and for every string a and electron e (the p-th
// orbital) srow[a][e] = ((slot row of (a - p, p)) << 1 | parity, kj0[a - p])
__global__ void k_nm1_ktables(const uint32_t* __restrict__ masks, int nstr, int n, int nsig, int nK,
                              const uint32_t* __restrict__ kmask, int32_t* __restrict__ krow,
                              uint16_t* __restrict__ kcol, int32_t* __restrict__ kj0,
                              int2* __restrict__ srow) {
  auto find = [](const uint32_t* v, int len, uint32_t m) {   // first element >= m
    int lo = 0, hi = len;
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (v[mid] < m) lo = mid + 1;
      else hi = mid;
    }
    return lo;
  };
  const int nv = n - nsig + 1;
  const int tot = nK * 17 + nstr * nsig;
  for (int t = blockIdx.x * blockDim.x + threadIdx.x; t < tot; t += gridDim.x * blockDim.x) {
    if (t < nK * 16) {
      const int K = t >> 4, o = t & 15;
      const uint32_t m = kmask[K];
      const int v =
          o < n && !((m >> o) & 1u)
              ? (find(masks, nstr, m | (1u << o)) << 1) | (__popc(m & ((1u << o) - 1u)) & 1)
              : -1;
      krow[t] = v;
      kcol[t] = (uint16_t)(v >= 0 ? v : ((nstr + 3) & ~3) << 1);
    } else if (t < nK * 17) {
      kj0[t - nK * 16] = find(masks, nstr, kmask[t - nK * 16] + 1u);
    } else {
      const int x = t - nK * 17, a = x / nsig, e = x - a * nsig;
      uint32_t m = masks[a];
      uint32_t u = m;
      for (int i = 0; i < e; i++) u &= u - 1;
      const int p = __ffs(u) - 1;
      m ^= 1u << p;
      const int K = find(kmask, nK, m), below = __popc(m & ((1u << p) - 1u));
      srow[x] = make_int2(((K * nv + p - below) << 1) | (below & 1), find(masks, nstr, m + 1u));
    }
  }
}

// The spin term goes through the split operand M up to the default shift: its
// rms error against FP64 is then that of the FP32 term within 2 % (0.98-1.02 over
// six shapes, 12 seeds each); at shifts of 1, 2 and 4 it would be 1.10, 1.34
// and 2.04 times that, and worse in proportion beyond.
inline bool nm_spin_in_operand(double shift) { return shift >= 0.0 && shift <= 0.5; }

// sigma(a, b) = X(a, b) + X(b, a) + shift nsig c(a, b), X = W + the slots of
// row a (SPIN: + shift (S^2 c)(a, b) in FP32 instead, M without the spin term).
// One CTA per 32 x 32 tile pair (I, J), I <= J; a warp reads 32
// consecutive columns of W and of each slot.  packed: c and sigma in the packed
// symmetric layout, only tile (I, J) is written.
template <bool SPIN>
__global__ void __launch_bounds__(256)
k_sigma_nm1_finish(const float* __restrict__ W, int64_t w_stride, const float* __restrict__ slots,
                   int64_t s_stride, int ldS, const int2* __restrict__ srow,
                   const int32_t* __restrict__ link, const uint32_t* __restrict__ masks, int npair,
                   int nstr, int nsig, const float* __restrict__ c, int64_t c_stride, float shift,
                   const int32_t* __restrict__ active, float* __restrict__ out, int64_t out_stride,
                   int packed) {
  const int b = blockIdx.y;
  if (active && !active[b]) return;
  const int nt = (nstr + 31) / 32;
  int t = blockIdx.x, I = 0;
  while (t >= nt - I) {
    t -= nt - I;
    I++;
  }
  const int J = I + t;
  __shared__ float sX[2][32][33];
  const float* Wb = W + (int64_t)b * w_stride;
  const float* sb = slots + (int64_t)b * s_stride;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int h = 0; h < (I == J ? 1 : 2); h++) {
    const int r0 = (h ? J : I) * 32, col = (h ? I : J) * 32 + tx;
#pragma unroll
    for (int i = ty; i < 32; i += 8) {
      const int row = r0 + i;
      float x = 0.f;
      if (row < nstr && col < nstr) {
        x = Wb[(int64_t)row * nstr + col];
#pragma unroll 4
        for (int e = 0; e < nsig; e++) {
          const int2 s = srow[row * nsig + e];
          if (col >= s.y) {
            const float v = sb[(int64_t)(s.x >> 1) * ldS + col];
            x += (s.x & 1) ? -v : v;
          }
        }
      }
      sX[h][i][tx] = x;
    }
  }
  __syncthreads();
  const float* cb = c + (int64_t)b * c_stride;
  float* ob = out + (int64_t)b * out_stride;
  const float(*sT)[33] = sX[I == J ? 0 : 1];
  float v[4];
#pragma unroll
  for (int k = 0; k < 4; k++) {
    const int i = ty + 8 * k, ia = I * 32 + i, ib = J * 32 + tx;
    v[k] = 0.f;
    if (ia < nstr && ib < nstr) {
      const int64_t at = packed ? sym_index(ia, ib, nstr) : (int64_t)ia * nstr + ib;
      const float x = sX[0][i][tx] + sT[tx][i];
      if constexpr (SPIN)
        v[k] = fmaf(shift, spin_square_sym(link, masks, nstr, npair, nsig, cb, packed, ia, ib), x);
      else
        v[k] = fmaf(shift * (float)nsig, cb[at], x);
      if (!packed || ia <= ib) ob[at] = v[k];
    }
  }
  if (I == J || packed) return;                      // the tile was its own transpose
  __syncthreads();
#pragma unroll
  for (int k = 0; k < 4; k++) sX[0][ty + 8 * k][tx] = v[k];
  __syncthreads();
  for (int i = ty; i < 32; i += 8) {
    const int ia = J * 32 + i, ib = I * 32 + tx;
    if (ia < nstr && ib < nstr) ob[(int64_t)ia * nstr + ib] = sX[0][tx][i];
  }
}

// tiles of one tuple when a tile covers at most G values of Ka
inline int nm_tiles(int nK, int G) {
  int tiles = 0, k = 0, o = 0;
  while (k < nK) {
    const int klim = std::min(nK, k + G);
    int rem = 128;
    while (k < klim && rem >= nK - k - o) {
      rem -= nK - k - o;
      k++;
      o = 0;
    }
    if (k < klim) o += rem;
    tiles++;
  }
  return tiles;
}

template <int N>
bool nm_plan_n(int nsig, int nstr, int B, NmPlan& L) {
  using S = Shape<N>;
  L.nv = N - nsig + 1;
  L.nK = (int)string_count(N, nsig - 1);
  L.b_bytes = (uint32_t)S::KP * S::NP * 4;
  L.NB = L.b_bytes * 2 <= 80 * 1024 ? 2 : 1;
  L.nst = S::NST;
  L.cq = S::CQ;
  L.ck = S::CK;
  L.KP = S::KP;
  L.NP = S::NP;
  L.ldw = (nstr + 3) & ~3;
  const uint32_t list = ((uint32_t)std::max(B, 1) * 2 + 127) & ~127u;
  const uint32_t row = (uint32_t)L.nv * nm_ars(nstr) * 4, crow = row;
  const uint32_t spare = ((uint32_t)nm_ars(nstr) * 4 + 127) & ~127u;
  const uint32_t zero = spare;
  const int64_t room =
      (int64_t)NM_SMEM_MAX - 1024 - 256 - L.b_bytes * L.NB - list - spare - zero;
  // fewest cycles: tiles times what one takes, about 4,500 + 300 per phase of
  // its row sums.  More copies shorten a tile, more strings per tile make fewer
  // tiles (10e/12o: one copy, G = 2: 249 us; weighing the copies more takes two
  // copies, G = 1: 1.2 times slower)
  double best = 1e300;
  for (int NC = 1; NC <= 4; NC *= 2)
    for (int G = 1; G <= 17; G++) {
      const int64_t left = room - (int64_t)row * NC * G;
      const int GR = (int)std::min<int64_t>(left / crow, G + 2);
      if (left < 0 || GR < G + 1) break;
      const double cost = nm_tiles(L.nK, G) * (4500.0 + 300.0 * (4 / NC));
      if (cost < best) {
        best = cost;
        L.G = G;
        L.GR = GR;
        L.NC = NC;
      }
    }
  if (best > 1e299) return false;
  L.R = (int)nm_start(L.nK, L.nK, L.G);
  L.acc = L.b_bytes * L.NB;
  L.rows = L.acc + ((row * L.G * L.NC + 127) & ~127u) + spare;
  L.zero = L.rows + ((crow * L.GR + 127) & ~127u);
  L.list = L.zero + zero;
  L.total = std::max(NM_SMEM_MIN, L.list + list + 1024);
  return L.total <= NM_SMEM_MAX;
}

bool nm_plan(int n, int nsig, int nstr, int B, NmPlan& L) {
  if (nsig < 1 || nsig > n || B > SIGMA_NM1_MAX_BATCH) return false;
  switch (n) {
#define NM_CASE(N) case N: return nm_plan_n<N>(nsig, nstr, B, L);
    NM_CASE(5) NM_CASE(6) NM_CASE(7) NM_CASE(8) NM_CASE(9) NM_CASE(10) NM_CASE(11) NM_CASE(12)
#undef NM_CASE
    default: return false;
  }
}

template <int N>
void nm_launch(mbe_ctx* ctx, int grid, const NmPlan& L, const StringTables* tab, const uint8_t* bop,
               const uint32_t* cw, int ldS, const int32_t* active, int B, float* slots,
               int32_t* err) {
  static bool attr_done[MBE_MAX_DEVICES] = {false};
  once_per_device(attr_done, ctx->device, [] {
    CU_CHECK(cudaFuncSetAttribute(k_sigma_nm1<N>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)NM_SMEM_MAX));
  });
  k_sigma_nm1<N><<<grid, NM_THREADS, L.total, ctx->stream>>>(
      tab->krow.ptr, reinterpret_cast<const uint4*>(tab->krow.ptr + (size_t)L.nK * 16),
      tab->kmask.ptr, tab->kj0.ptr, bop, cw, tab->nstr, ldS, active, B, L, slots,
      ctx->opt.wait_limit, err);
  CU_LAUNCH_CHECK();
}

inline int nm_ld(int nstr) { return (nstr + 7) & ~7; }

}  // namespace

bool sigma_nm1_supported(int n, int nsig, int nstr, int B) {
  NmPlan L;
  return nm_plan(n, nsig, nstr, B, L);
}

int sigma_nm1_tiles(int n, int nsig, int nstr, int B) {
  NmPlan L;
  return nm_plan(n, nsig, nstr, B, L) ? nm_tiles(L.nK, L.G) : 0;
}

int64_t sigma_nm1_slot_floats(int n, int nsig, int nstr) {
  return string_count(n, nsig - 1) * (n - nsig + 1) * nm_ld(nstr);
}

// words per row of the operand
int sigma_nm1_ldw(int nstr) { return (nstr + 3) & ~3; }

int sigma_nm1_stages(int n, int nsig, int nstr, int B) {
  NmPlan L;
  return nm_plan(n, nsig, nstr, B, L) ? L.nst : 0;
}

void sigma_nm1_prepare(mbe_ctx* ctx, BinProblem& bp, SigmaWork& w, double shift) {
  const int n = bp.n, nsig = bp.nsig, nstr = bp.nstr;
  NmPlan L;
  if (!nm_plan(n, nsig, nstr, bp.B, L))
    throw MbeError{MBE_EINVAL, "active space too large for the two-spin kernel"};
  StringTables* t = get_tables(ctx, n, nsig);
  cudaStream_t st = ctx->stream;
  if (!t->nm1_ready) {
    t->kmask.reset(&ctx->pool, L.nK);
    t->kj0.reset(&ctx->pool, L.nK);
    t->srow.reset(&ctx->pool, (size_t)nstr * nsig);
    t->krow.reset(&ctx->pool, (size_t)L.nK * 24);   // krow, then kcol (16-bit)
    uint16_t* kcol = reinterpret_cast<uint16_t*>(t->krow.ptr + (size_t)L.nK * 16);
    launch_string_masks(ctx, n, nsig - 1, L.nK, t->kmask.ptr);
    const int tot = L.nK * 17 + nstr * nsig;
    k_nm1_ktables<<<(tot + 255) / 256, 256, 0, st>>>(t->masks.ptr, nstr, n, nsig, L.nK,
                                                    t->kmask.ptr, t->krow.ptr, kcol, t->kj0.ptr,
                                                    t->srow.ptr);
    CU_LAUNCH_CHECK();
    t->nm1_ready = true;
  }
  const size_t need = (size_t)bp.B * L.b_bytes;
  if (bp.nmop.n != need) {
    bp.nmop.reset(&ctx->pool, need);
    k_nm1_operand<<<dim3(std::max(1, std::min(16, 2432 / bp.B)), bp.B), 256, 0, st>>>(
        bp.gp.ptr, n, bp.npair, (n + 1) & ~1, L.cq, L.ck, L.KP, L.NP,
        nm_spin_in_operand(shift) ? shift : 0.0, bp.nmop.ptr);
    CU_LAUNCH_CHECK();
  }
  const size_t sf = (size_t)bp.B * sigma_nm1_slot_floats(n, nsig, nstr);
  if (w.slots.n < sf) w.slots.reset(&ctx->pool, sf);
  const size_t cwn = (size_t)bp.B * nstr * sigma_nm1_ldw(nstr);
  if (w.cw.n < cwn) w.cw.reset(&ctx->pool, cwn);
}

void sigma_nm1(mbe_ctx* ctx, BinProblem& bp, SigmaWork& w, const int32_t* active, int nsm,
               int stages) {
  NmPlan L;
  nm_plan(bp.n, bp.nsig, bp.nstr, bp.B, L);
  if (stages >= 2 && stages < L.nst) L.nst = stages;
  const int grid = (int)std::min<int64_t>(nsm, (int64_t)bp.B * L.nK);
  const StringTables* t = bp.tab;
  const int ldS = nm_ld(bp.nstr);
  switch (bp.n) {
#define NM_CASE(N)                                                                          \
  case N:                                                                                   \
    nm_launch<N>(ctx, grid, L, t, bp.nmop.ptr, w.cw.ptr, ldS, active, bp.B, w.slots.ptr,     \
                 w.err.ptr);                                                                \
    break;
    NM_CASE(5) NM_CASE(6) NM_CASE(7) NM_CASE(8) NM_CASE(9) NM_CASE(10) NM_CASE(11) NM_CASE(12)
#undef NM_CASE
    default:
      throw MbeError{MBE_EINVAL, "unsupported active space of the two-spin kernel"};
  }
}

void sigma_nm1_finish(mbe_ctx* ctx, const BinProblem& bp, const SigmaWork& w, int64_t w_stride,
                      const float* c, int64_t c_stride, double shift, const int32_t* active,
                      float* out, int64_t out_stride, bool packed) {
  const int ntl = (bp.nstr + 31) / 32;
  auto kernel = nm_spin_in_operand(shift) ? k_sigma_nm1_finish<false> : k_sigma_nm1_finish<true>;
  kernel<<<dim3((unsigned)(ntl * (ntl + 1) / 2), bp.B), 256, 0, ctx->stream>>>(
      w.Xf.ptr, w_stride, w.slots.ptr, sigma_nm1_slot_floats(bp.n, bp.nsig, bp.nstr),
      nm_ld(bp.nstr), bp.tab->srow.ptr, bp.tab->link.ptr, bp.tab->masks.ptr, bp.npair, bp.nstr,
      bp.nsig, c, c_stride, (float)shift, active, out, out_stride, packed ? 1 : 0);
  CU_LAUNCH_CHECK();
}
