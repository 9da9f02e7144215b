// CASCI building blocks of one bin of tuples (same active size n and same
// number of active electrons per spin nsig):
//   K1  string enumeration and the per-(string, orbital pair) link table
//   K2  effective integrals of each tuple (inactive-core fold, Sec. 2/Fig. 2)
//   K3  diagonal of H_active + shift * S^2 (Davidson preconditioner)
//   K4  gather and pull scatter of the emulated-FP64 sigma vector (its (kl|ij)
//       contraction is in mbe_ozaki.cu; the FP64 sigma is in mbe_sigma64.cu),
//       plus the S^2 spin shift
//
// Sigma vector (Knowles & Handy, Chem. Phys. Lett. 111, 315 (1984); Olsen
// et al., J. Chem. Phys. 89, 2185 (1988)): with h'_pq = h_pq - 1/2 sum_r
// (pr|rq) and g'_{pq,rs} = (pq|rs) + (h'_pq d_rs + d_pq h'_rs)/N the active
// Hamiltonian is H = 1/2 sum_{PQ} g'_{PQ} E+_P E+_Q over packed pairs
// P = (p >= q), E+_P = E_pq + E_qp (E_pp on the diagonal).  Hence
//   D_P(K)  = sum_J <K|E+_P|J> c_J            (gather)
//   F_P(K)  = sum_Q g'_{PQ} D_Q(K)            (contraction)
//   sigma_I = 1/2 sum_P sum_K <I|E+_P|K> F_P(K)   (pull scatter)
// E+_P acting on one spin string has at most one non-zero matrix element
// per string, which the link table stores.
#include "mbe_internal.cuh"
#include <algorithm>

namespace {

__constant__ int c_binom[33][33];

bool g_binom_ready[MBE_MAX_DEVICES] = {false};

// the binomial table is copied with a synchronous cudaMemcpyToSymbol on the
// first use on a device (it waits for the device once)
void ensure_binom(int device) {
  once_per_device(g_binom_ready, device, [] {
    int tab[33][33];
    for (int n = 0; n <= 32; n++)
      for (int k = 0; k <= 32; k++) {
        if (k == 0) tab[n][k] = 1;
        else if (n == 0) tab[n][k] = 0;
        else {
          long long v = (long long)tab[n - 1][k - 1] + tab[n - 1][k];
          tab[n][k] = v > 0x7fffffff ? 0x7fffffff : (int)v;
        }
      }
    CU_CHECK(cudaMemcpyToSymbol(c_binom, tab, sizeof(tab)));
  });
}

// colexicographic rank of a k-subset bit mask = its position when all
// k-subsets are sorted by integer value
__device__ __forceinline__ int mask_rank(uint32_t m) {
  int r = 0, i = 1;
  while (m) {
    int p = __ffs(m) - 1;
    r += c_binom[p][i];
    i++;
    m &= m - 1;
  }
  return r;
}

__device__ uint32_t mask_unrank(int r, int n, int k) {
  uint32_t m = 0;
  for (int i = k; i >= 1; i--) {
    int p = i - 1;
    while (p + 1 < n && c_binom[p + 1][i] <= r) p++;
    m |= 1u << p;
    r -= c_binom[p][i];
  }
  return m;
}

__global__ void k_strings(uint32_t* masks, int nstr, int n, int k) {
  int I = blockIdx.x * blockDim.x + threadIdx.x;
  if (I < nstr) masks[I] = mask_unrank(I, n, k);
}

__global__ void k_link(const uint32_t* masks, int32_t* link, int nstr, int n) {
  int npair = n * (n + 1) / 2;
  int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= (int64_t)nstr * npair) return;
  int I = (int)(t / npair), P = (int)(t % npair);
  int p = (int)((sqrtf(8.f * P + 1.f) - 1.f) * 0.5f);
  while (p * (p + 1) / 2 > P) p--;
  while ((p + 1) * (p + 2) / 2 <= P) p++;
  int q = P - p * (p + 1) / 2;
  uint32_t m = masks[I];
  int32_t v = -1;
  int bp = (m >> p) & 1, bq = (m >> q) & 1;
  if (p == q) {
    if (bp) v = I << 1;
  } else if (bp != bq) {
    uint32_t J = m ^ (1u << p) ^ (1u << q);
    // orbitals strictly between q and p (p > q) decide the sign
    uint32_t between = (m & ((1u << p) - 1u)) & ~((2u << q) - 1u);
    int neg = __popc(between) & 1;
    v = (mask_rank(J) << 1) | neg;
  }
  link[t] = v;
}

}  // namespace

int64_t string_count(int n, int nsig) {
  long long nstr = 1;
  for (int i = 0; i < nsig; i++) nstr = nstr * (n - i) / (i + 1);
  return nstr;
}

void launch_string_masks(mbe_ctx* ctx, int n, int nsig, int nstr, uint32_t* masks) {
  ensure_binom(ctx->device);
  k_strings<<<(nstr + 255) / 256, 256, 0, ctx->stream>>>(masks, nstr, n, nsig);
  CU_LAUNCH_CHECK();
}

void build_string_tables(mbe_ctx* ctx, StringTables* t) {
  const int64_t nstr = string_count(t->n, t->nsig);
  if (nstr > (1 << 28)) throw MbeError{MBE_EINVAL, "string space too large"};
  t->nstr = (int)nstr;
  t->npair = t->n * (t->n + 1) / 2;
  t->masks.reset(&ctx->pool, t->nstr);
  t->link.reset(&ctx->pool, (size_t)t->nstr * t->npair);
  launch_string_masks(ctx, t->n, t->nsig, t->nstr, t->masks.ptr);
  const int64_t tot = nstr * t->npair;
  k_link<<<(unsigned)((tot + 255) / 256), 256, 0, ctx->stream>>>(t->masks.ptr, t->link.ptr,
                                                                 t->nstr, t->n);
  CU_LAUNCH_CHECK();
}

// ------------------------------------------------------------------ K2
namespace {

__device__ __forceinline__ int64_t gpair(int p, int q) {
  return p >= q ? (int64_t)p * (p + 1) / 2 + q : (int64_t)q * (q + 1) / 2 + p;
}

// gridDim.y CTAs per tuple, each forming the small parts (a few thousand
// gathers) and writing a slice of g' (B = 1 with one CTA and the pairs decoded
// by an FP64 square root per element took 21 us).  act: n sorted global
// orbital ids, or NULL: the ones in `al` (one tuple).
__global__ void __launch_bounds__(256)
k_effints(const double* __restrict__ h, const double* __restrict__ eri, int norb, int nocc,
          int npair_g, const int32_t* __restrict__ act_all, ActList al, int n, int nel,
          double* ecore_out, double* heff_out, double* hp_out, double* gp_out, double* jk_out) {
  const int b = blockIdx.x;
  extern __shared__ double sm[];
  double* s_heff = sm;            // n*n
  double* s_hp = sm + n * n;      // n*n
  __shared__ int s_core[MBE_MAX_NORB];
  __shared__ int s_ncore;
  __shared__ int s_act[MBE_MAX_ACT];
  __shared__ uint8_t s_p[128], s_q[128];   // orbitals of a packed active pair
  __shared__ int s_g[128];                 // its global pair index
  const int tid = threadIdx.x, nt = blockDim.x;
  const bool lead = blockIdx.y == 0;
  if (tid < n) s_act[tid] = act_all ? act_all[(int64_t)b * n + tid] : al.v[tid];
  const int npair = n * (n + 1) / 2;
  for (int p = tid; p < n; p += nt)
    for (int q = 0; q <= p; q++) {
      s_p[p * (p + 1) / 2 + q] = (uint8_t)p;
      s_q[p * (p + 1) / 2 + q] = (uint8_t)q;
    }
  __syncthreads();
  if (tid < 32) {
    // inactive core: occupied orbitals outside the active space, ascending
    int nc = 0;
    for (int i0 = 0; i0 < nocc; i0 += 32) {
      const int i = i0 + tid;
      bool in = i < nocc;
      for (int j = 0; in && j < n; j++) in = s_act[j] != i;
      const unsigned m = __ballot_sync(0xffffffffu, in);
      if (in) s_core[nc + __popc(m & ((1u << tid) - 1u))] = i;
      nc += __popc(m);
    }
    if (tid == 0) s_ncore = nc;
  }
  for (int P = tid; P < npair; P += nt) s_g[P] = (int)gpair(s_act[s_p[P]], s_act[s_q[P]]);
  __syncthreads();
  const int nc = s_ncore;
  const int64_t NP = npair_g;
  // inactive-core energy (Fig. 2: occupied orbitals outside the active space
  // stay doubly occupied): sum 2 h_ii + sum_ij [2 (ii|jj) - (ij|ji)]
  if (lead && tid < 32) {
    double e = 0.0;
    for (int t = tid; t < nc * nc; t += 32) {
      const int i = s_core[t / nc], j = s_core[t % nc];
      e += 2.0 * eri[gpair(i, i) * NP + gpair(j, j)] - eri[gpair(i, j) * NP + gpair(j, i)];
    }
    for (int x = tid; x < nc; x += 32) e += 2.0 * h[(int64_t)s_core[x] * norb + s_core[x]];
    for (int o = 16; o; o >>= 1) e += __shfl_xor_sync(0xffffffffu, e, o);
    if (tid == 0) ecore_out[b] = e;
  }
  // h_eff_pq = h_pq + sum_i [2 (pq|ii) - (pi|iq)] and
  // h'_pq = h_eff_pq - 1/2 sum_r (pr|rq), r over the active orbitals
  for (int t = tid; t < n * n; t += nt) {
    const int p = t / n, q = t - p * n;
    const int P = s_act[p], Q = s_act[q];
    double v = h[(int64_t)P * norb + Q];
#pragma unroll 4
    for (int x = 0; x < nc; x++) {
      const int i = s_core[x];
      v += 2.0 * eri[gpair(P, Q) * NP + gpair(i, i)] - eri[gpair(P, i) * NP + gpair(i, Q)];
    }
    double x = 0.0;
#pragma unroll 4
    for (int r = 0; r < n; r++) x += eri[gpair(P, s_act[r]) * NP + gpair(s_act[r], Q)];
    s_heff[t] = v;
    s_hp[t] = v - 0.5 * x;
    if (lead) {
      heff_out[(int64_t)b * n * n + t] = v;
      hp_out[(int64_t)b * n * n + t] = v - 0.5 * x;
      jk_out[(int64_t)b * 2 * n * n + t] = eri[gpair(P, P) * NP + gpair(Q, Q)];
      jk_out[(int64_t)b * 2 * n * n + n * n + t] = eri[gpair(P, Q) * NP + gpair(Q, P)];
    }
  }
  __syncthreads();
  // g'_{PQ} = (pq|rs) + (h'_pq d_rs + d_pq h'_rs) / N_active, N_active = nel
  // active electrons of both spins (sum_r E_rr = N_active on the space)
  const double inv = nel > 0 ? 1.0 / nel : 0.0;
  for (int t = blockIdx.y * nt + tid; t < npair * npair; t += gridDim.y * nt) {
    const int P = t / npair, Q = t - P * npair;
    const int p = s_p[P], q = s_q[P], r = s_p[Q], s = s_q[Q];
    double v = eri[(int64_t)s_g[P] * NP + s_g[Q]];
    if (r == s) v += s_hp[p * n + q] * inv;
    if (p == q) v += s_hp[r * n + s] * inv;
    gp_out[(int64_t)b * npair * npair + t] = v;
  }
}

}  // namespace

void launch_effints_raw(mbe_ctx* ctx, const int32_t* act, const ActList* al, int B, int n, int nel,
                        double* ecore, double* heff, double* hp, double* gp, double* jk) {
  size_t smem = 2 * sizeof(double) * n * n;
  // a CTA per 1024 elements of g' while the batch leaves SMs idle
  const int npair = n * (n + 1) / 2;
  const int split = std::max(1, std::min((npair * npair + 1023) / 1024, 304 / B));
  k_effints<<<dim3(B, split), 256, smem, ctx->stream>>>(
      ctx->h.ptr, ctx->eri.ptr, ctx->norb, ctx->nocc, ctx->npair_g, act, al ? *al : ActList{}, n,
      nel, ecore, heff, hp, gp, jk);
  CU_LAUNCH_CHECK();
}

void launch_effints(mbe_ctx* ctx, BinProblem& bp) {
  const int n = bp.n, B = bp.B;
  bp.ecore.reset(&ctx->pool, B);
  bp.heff.reset(&ctx->pool, (size_t)B * n * n);
  bp.hp.reset(&ctx->pool, (size_t)B * n * n);
  bp.gp.reset(&ctx->pool, (size_t)B * bp.npair * bp.npair);
  bp.jk.reset(&ctx->pool, (size_t)B * 2 * n * n);
  const int nel = bp.nsig + (bp.nsigb < 0 ? bp.nsig : bp.nsigb);
  launch_effints_raw(ctx, bp.act.ptr, nullptr, B, n, nel, bp.ecore.ptr, bp.heff.ptr, bp.hp.ptr,
                     bp.gp.ptr, bp.jk.ptr);
}

// ------------------------------------------------------------------ K3
namespace {

// energy of one spin string with itself: sum h_pp + 1/2 sum_{pq} (J - K)
__device__ __forceinline__ double string_self(uint32_t m, const double* heff, const double* J,
                                              const double* K, int n) {
  double e = 0.0, e2 = 0.0;
  for (int p = 0; p < n; p++) {
    if (!((m >> p) & 1)) continue;
    e += heff[p * n + p];
    for (int q = 0; q < n; q++)
      if ((m >> q) & 1) e2 += J[p * n + q] - K[p * n + q];
  }
  return e + 0.5 * e2;
}

// <Ia Ib| H_active + shift S^2 |Ia Ib>, computed symmetrically in (Ia, Ib).
// alpha strings masks[nstr], beta strings masksb[nstrb] (the same table for
// a closed shell); <S^2> diagonal = (beta-only orbitals) + Ms(Ms+1) (msms).
__global__ void k_hdiag(const uint32_t* __restrict__ masks, const uint32_t* __restrict__ masksb,
                        int nstr, int nstrb, int n, int nsigb, double msms,
                        const double* __restrict__ heff_all, const double* __restrict__ jk_all,
                        double shift, double* hd_all, int64_t ld, int packed) {
  const int b = blockIdx.y;
  extern __shared__ double sm[];
  double* s_heff = sm;
  double* s_J = sm + n * n;
  double* s_K = sm + 2 * n * n;
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    s_heff[t] = heff_all[(int64_t)b * n * n + t];
    s_J[t] = jk_all[(int64_t)b * 2 * n * n + t];
    s_K[t] = jk_all[(int64_t)b * 2 * n * n + n * n + t];
  }
  __syncthreads();
  const int64_t ndet = (int64_t)nstr * nstrb;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ndet;
       i += (int64_t)gridDim.x * blockDim.x) {
    int ia = (int)(i / nstrb), ib = (int)(i % nstrb);
    if (packed && ia > ib) continue;
    uint32_t ma = masks[ia], mb = masksb[ib];
    double ea = string_self(ma, s_heff, s_J, s_K, n);
    double eb = string_self(mb, s_heff, s_J, s_K, n);
    double cross = 0.0;
    for (int p = 0; p < n; p++) {
      int ap = (ma >> p) & 1, bpp = (mb >> p) & 1;
      if (ap & bpp) cross += s_J[p * n + p];
      for (int q = 0; q < p; q++) {
        int w = (ap & ((mb >> q) & 1)) + (((ma >> q) & 1) & bpp);
        if (w) cross += w * s_J[p * n + q];
      }
    }
    int ndocc = __popc(ma & mb);
    hd_all[(int64_t)b * ld + (packed ? sym_index(ia, ib, nstr) : i)] =
        (ea + eb) + cross + shift * ((double)(nsigb - ndocc) + msms);
  }
}

}  // namespace

void launch_hdiag(mbe_ctx* ctx, BinProblem& bp, double spin_shift, double* hd, int64_t ld,
                  bool packed) {
  const int n = bp.n;
  size_t smem = 3 * sizeof(double) * n * n;
  int64_t blocks = (bp.ndet + 255) / 256;
  if (blocks > 4096) blocks = 4096;
  dim3 grid((unsigned)blocks, bp.B);
  k_hdiag<<<grid, 256, smem, ctx->stream>>>(bp.tab->masks.ptr, bp.tabb->masks.ptr, bp.nstr,
                                            bp.nstrb, n, bp.nsigb, bp.msms(), bp.heff.ptr,
                                            bp.jk.ptr, spin_shift, hd, ld, packed ? 1 : 0);
  CU_LAUNCH_CHECK();
}

// ------------------------------------------------------------------ K4
namespace {

// D[b][P][Ia*nstr+Ib] = s_a C(Ja, Ib) + s_b C(Ia, Jb)
__global__ void k_gather_fp64(const int32_t* __restrict__ link, const int32_t* __restrict__ linkb,
                              int nstr, int nstrb, int npair,
                              const double* __restrict__ c, int64_t c_stride,
                              const int32_t* __restrict__ active, const int32_t* __restrict__ bmap,
                              double* __restrict__ D) {
  const int bl = blockIdx.y;                 // local index in the sub-batch
  const int b = bmap[bl];
  if (active && !active[b]) return;
  const double* cb = c + (int64_t)b * c_stride;
  const int64_t ndet = (int64_t)nstr * nstrb;
  double* Db = D + (int64_t)bl * npair * ndet;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ndet;
       i += (int64_t)gridDim.x * blockDim.x) {
    int ia = (int)(i / nstrb), ib = (int)(i % nstrb);
    const int32_t* la = link + (int64_t)ia * npair;
    const int32_t* lb = linkb + (int64_t)ib * npair;
    for (int P = 0; P < npair; P++) {
      double v = 0.0;
      int32_t ta = la[P], tb = lb[P];
      if (ta >= 0) {
        double x = cb[(int64_t)(ta >> 1) * nstrb + ib];
        v += (ta & 1) ? -x : x;
      }
      if (tb >= 0) {
        double x = cb[(int64_t)ia * nstrb + (tb >> 1)];
        v += (tb & 1) ? -x : x;
      }
      Db[(int64_t)P * ndet + i] = v;
    }
  }
}

// sigma(Ia,Ib) = 1/2 sum_P [s_a E_P(Ja,Ib) + s_b E_P(Ia,Jb)] + shift (S^2 c)(Ia,Ib)
// S^2 c = (nsig - ndocc) c - sum over pairs {p,q} with Ia holding one of them
// and Ib the other of s_a s_b c(Ja, Jb)   (S^2 = N_beta - sum E^a_qp E^b_pq)
// E element i: the float pair hi + lo written by the sliced tensor-core
// contraction
__device__ __forceinline__ double load_e(const double* __restrict__ Eb, int64_t i) {
  const float2 v = reinterpret_cast<const float2*>(Eb)[i];
  return (double)v.x + (double)v.y;
}

// General (not necessarily symmetric) c, alpha table link/masks (nstr
// strings) and beta table linkb/masksb (nstrb strings, the same table for a
// closed shell); S^2 = S-S+ + Ms(Ms+1): diagonal (beta-only orbitals) + msms,
// off-diagonal the alpha-only / beta-only exchanges.
__global__ void k_scatter_fp64(const int32_t* __restrict__ link, const uint32_t* __restrict__ masks,
                               const int32_t* __restrict__ linkb,
                               const uint32_t* __restrict__ masksb, int nstr, int nstrb, int n,
                               int nsigb, double msms, const double* __restrict__ E,
                               const double* __restrict__ c, int64_t c_stride, double shift,
                               const int32_t* __restrict__ active, const int32_t* __restrict__ bmap,
                               double* __restrict__ out, int64_t out_stride) {
  const int bl = blockIdx.y;
  const int b = bmap[bl];
  if (active && !active[b]) return;
  const int npair = n * (n + 1) / 2;
  const int64_t ndet = (int64_t)nstr * nstrb;
  const double* Eb = E + (int64_t)bl * npair * ndet;
  const double* cb = c + (int64_t)b * c_stride;
  double* ob = out + (int64_t)b * out_stride;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ndet;
       i += (int64_t)gridDim.x * blockDim.x) {
    int ia = (int)(i / nstrb), ib = (int)(i % nstrb);
    const int32_t* la = link + (int64_t)ia * npair;
    const int32_t* lb = linkb + (int64_t)ib * npair;
    double acc = 0.0;
    for (int P = 0; P < npair; P++) {
      int32_t ta = la[P], tb = lb[P];
      if (ta >= 0) {
        double x = load_e(Eb, (int64_t)P * ndet + (int64_t)(ta >> 1) * nstrb + ib);
        acc += (ta & 1) ? -x : x;
      }
      if (tb >= 0) {
        double x = load_e(Eb, (int64_t)P * ndet + (int64_t)ia * nstrb + (tb >> 1));
        acc += (tb & 1) ? -x : x;
      }
    }
    double v = 0.5 * acc;
    if (shift != 0.0) {
      uint32_t ma = masks[ia], mb = masksb[ib];
      double s2 = ((double)(nsigb - __popc(ma & mb)) + msms) * cb[i];
      uint32_t oa = ma & ~mb, ob2 = mb & ~ma;   // open shells of each spin
      for (int q = 0; q < n; q++) {
        if (!((oa >> q) & 1)) continue;
        for (int p = 0; p < n; p++) {
          if (!((ob2 >> p) & 1)) continue;
          int P = p > q ? p * (p + 1) / 2 + q : q * (q + 1) / 2 + p;
          int32_t ta = la[P], tb = lb[P];
          double x = cb[(int64_t)(ta >> 1) * nstrb + (tb >> 1)];
          s2 -= ((ta ^ tb) & 1) ? -x : x;
        }
      }
      v += shift * s2;
    }
    ob[i] = v;
  }
}

// Symmetric c (c(a,b) = c(b,a), the alpha<->beta symmetric Davidson
// vectors): D and E are symmetric in the two strings, so the beta half of
// the scatter is the transpose of the alpha half and
//   sigma = X + X^T + shift S^2 c,  X(a,b) = 1/2 sum_P s_a E_P(J_a, b),
// with every E read coalesced (row J_a, consecutive b).  k_scatter_sym_fp64
// writes X into out; k_finish_sym_fp64 adds the transpose (32 x 32 tile
// pairs in shared memory, in place) and the spin penalty.
__global__ void k_scatter_sym_fp64(const int32_t* __restrict__ link, int nstr, int npair,
                                   const double* __restrict__ E,
                                   const int32_t* __restrict__ active,
                                   const int32_t* __restrict__ bmap, double* __restrict__ out,
                                   int64_t out_stride) {
  const int bl = blockIdx.y;
  const int b = bmap[bl];
  if (active && !active[b]) return;
  const int ndet = nstr * nstr;
  const double* Eb = E + (int64_t)bl * npair * ndet;
  double* ob = out + (int64_t)b * out_stride;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < ndet; i += gridDim.x * blockDim.x) {
    const int ia = i / nstr, ib = i - ia * nstr;
    const int32_t* la = link + (int64_t)ia * npair;
    double acc = 0.0;
    for (int P = 0; P < npair; P++) {
      const int32_t ta = la[P];
      if (ta >= 0) {
        const double x = load_e(Eb, (int64_t)P * ndet + (int64_t)(ta >> 1) * nstr + ib);
        acc += (ta & 1) ? -x : x;
      }
    }
    ob[i] = 0.5 * acc;
  }
}

__global__ void k_finish_sym_fp64(double* __restrict__ out, int64_t out_stride,
                                  const int32_t* __restrict__ link,
                                  const uint32_t* __restrict__ masks, int nstr, int n, int nsig,
                                  const double* __restrict__ c, int64_t c_stride, double shift,
                                  const int32_t* __restrict__ active) {
  const int b = blockIdx.y;
  if (active && !active[b]) return;
  const int nt = (nstr + 31) / 32;
  int t = blockIdx.x, I = 0;
  while (t >= nt - I) {
    t -= nt - I;
    I++;
  }
  const int J = I + t;
  __shared__ double sX[2][32][33];
  double* ob = out + (int64_t)b * out_stride;
  const double* cb = c + (int64_t)b * c_stride;
  const int npair = n * (n + 1) / 2;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5;
  for (int h = 0; h < 2; h++) {
    const int r0 = (h ? J : I) * 32, c0 = (h ? I : J) * 32;
    for (int i = ty; i < 32; i += blockDim.x >> 5) {
      const int row = r0 + i, col = c0 + tx;
      sX[h][i][tx] = (row < nstr && col < nstr) ? ob[(int64_t)row * nstr + col] : 0.0;
    }
  }
  __syncthreads();
  // sigma is symmetric: the values of tile (I, J) are formed once and
  // written to both tiles (the transpose through shared memory)
  const int ny = blockDim.x >> 5;
  double v[4];
  for (int k = 0, i = ty; i < 32; i += ny, k++) {
    const int ia = I * 32 + i, ib = J * 32 + tx;
    double s = sX[0][i][tx] + sX[1][tx][i];
    if (shift != 0.0 && ia < nstr && ib < nstr) {
      // evaluated for (min, max): bitwise the same for both elements
      const int lo = min(ia, ib), hi = max(ia, ib);
      const int32_t* la = link + (int64_t)lo * npair;
      const int32_t* lb = link + (int64_t)hi * npair;
      const uint32_t ma = masks[lo], mb = masks[hi];
      double s2 = (double)(nsig - __popc(ma & mb)) * cb[(int64_t)lo * nstr + hi];
      uint32_t oa = ma & ~mb;
      const uint32_t obm = mb & ~ma;
      while (oa) {
        const int q = __ffs(oa) - 1;
        oa &= oa - 1;
        uint32_t o2 = obm;
        while (o2) {
          const int p = __ffs(o2) - 1;
          o2 &= o2 - 1;
          const int P = p > q ? p * (p + 1) / 2 + q : q * (q + 1) / 2 + p;
          const int32_t ta = la[P], tb = lb[P];
          const double x = cb[(int64_t)(ta >> 1) * nstr + (tb >> 1)];
          s2 -= ((ta ^ tb) & 1) ? -x : x;
        }
      }
      s += shift * s2;
    }
    v[k] = s;
  }
  // every read of tile (I, J) and (J, I) went through shared memory above;
  // the CTA owns both tiles, so the in-place stores race with nothing
  for (int k = 0, i = ty; i < 32; i += ny, k++) {
    const int ia = I * 32 + i, ib = J * 32 + tx;
    if (ia < nstr && ib < nstr) ob[(int64_t)ia * nstr + ib] = v[k];
  }
  if (I == J) return;
  __syncthreads();
  for (int k = 0, i = ty; i < 32; i += ny, k++) sX[0][i][tx] = v[k];
  __syncthreads();
  for (int i = ty; i < 32; i += ny) {
    const int ia = J * 32 + i, ib = I * 32 + tx;
    if (ia < nstr && ib < nstr) ob[(int64_t)ia * nstr + ib] = sX[0][tx][i];
  }
}

__global__ void k_s2(const int32_t* __restrict__ link, const uint32_t* __restrict__ masks,
                     const int32_t* __restrict__ linkb, const uint32_t* __restrict__ masksb,
                     int nstr, int nstrb, int n, int nsigb, double msms,
                     const double* __restrict__ c, int64_t c_stride,
                     const int32_t* __restrict__ active, double* __restrict__ out,
                     int64_t out_stride) {
  const int b = blockIdx.y;
  if (active && !active[b]) return;
  const int npair = n * (n + 1) / 2;
  const int64_t ndet = (int64_t)nstr * nstrb;
  const double* cb = c + (int64_t)b * c_stride;
  double* ob = out + (int64_t)b * out_stride;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < ndet;
       i += (int64_t)gridDim.x * blockDim.x) {
    int ia = (int)(i / nstrb), ib = (int)(i % nstrb);
    const int32_t* la = link + (int64_t)ia * npair;
    const int32_t* lb = linkb + (int64_t)ib * npair;
    uint32_t ma = masks[ia], mb = masksb[ib];
    double s2 = ((double)(nsigb - __popc(ma & mb)) + msms) * cb[i];
    uint32_t oa = ma & ~mb, obm = mb & ~ma;
    for (int q = 0; q < n; q++) {
      if (!((oa >> q) & 1)) continue;
      for (int p = 0; p < n; p++) {
        if (!((obm >> p) & 1)) continue;
        int P = p > q ? p * (p + 1) / 2 + q : q * (q + 1) / 2 + p;
        int32_t ta = la[P], tb = lb[P];
        double x = cb[(int64_t)(ta >> 1) * nstrb + (tb >> 1)];
        s2 -= ((ta ^ tb) & 1) ? -x : x;
      }
    }
    ob[i] = s2;
  }
}

}  // namespace

void sigma_emulated(mbe_ctx* ctx, BinProblem& bp, SigmaWork& w, const double* c, int64_t c_stride,
                    double* out, int64_t out_stride, const int32_t* active, double spin_shift,
                    bool symmetric) {
  const int npair = bp.npair, nstr = bp.nstr, nstrb = bp.nstrb;
  if (!w.err.ptr) {
    w.err.reset(&ctx->pool, 1);
    CU_CHECK(cudaMemsetAsync(w.err.ptr, 0, sizeof(int32_t), ctx->stream));
  }
  const int64_t ndet = bp.ndet;
  // sub-batch so that D and E stay within ~2 GB each
  int64_t per = (int64_t)npair * ndet;
  int64_t sb = (int64_t)(2.0e9 / 8.0) / (per > 0 ? per : 1);
  if (sb < 1) sb = 1;
  if (sb > bp.B) sb = bp.B;
  if (w.sub_batch != sb || w.D.n < (size_t)(sb * per)) {
    w.D.reset(&ctx->pool, sb * per);
    w.E.reset(&ctx->pool, sb * per);
    w.sub_batch = sb;
  }
  std::vector<int32_t> bm(bp.B);
  for (int i = 0; i < bp.B; i++) bm[i] = i;
  DevBuf<int32_t> bmap(&ctx->pool, bp.B);
  CU_CHECK(cudaMemcpyAsync(bmap.ptr, bm.data(), sizeof(int32_t) * bp.B, cudaMemcpyHostToDevice,
                           ctx->stream));
  int64_t blocks = (ndet + 255) / 256;
  if (blocks > 2048) blocks = 2048;
  for (int64_t b0 = 0; b0 < bp.B; b0 += sb) {
    const int nb = (int)std::min<int64_t>(sb, bp.B - b0);
    const dim3 g1((unsigned)blocks, nb);
    const int32_t* bm_d = bmap.ptr + b0;
    k_gather_fp64<<<g1, 256, 0, ctx->stream>>>(bp.tab->link.ptr, bp.tabb->link.ptr, nstr, nstrb,
                                               npair, c, c_stride, active, bm_d, w.D.ptr);
    CU_LAUNCH_CHECK();
    cudaEvent_t ev;
    ctx->fp64_timer.begin(ctx->stream, ctx->opt.timing != 0, &ev);
    contract_ozaki(ctx, bp.gp.ptr, npair, w.D.ptr, ndet, nb, active, bm_d, w.E.ptr, w.err.ptr);
    ctx->fp64_timer.end(ctx->stream, ev);
    ctx->stats.fp64_launches += 1;
    if (symmetric && bp.closed()) {
      k_scatter_sym_fp64<<<g1, 256, 0, ctx->stream>>>(bp.tab->link.ptr, nstr, npair, w.E.ptr,
                                                      active, bm_d, out, out_stride);
      CU_LAUNCH_CHECK();
      // the sub-batch is the contiguous tuple range [b0, b0 + nb)
      const int ntl = (nstr + 31) / 32;
      k_finish_sym_fp64<<<dim3((unsigned)(ntl * (ntl + 1) / 2), nb), 256, 0, ctx->stream>>>(
          out + b0 * out_stride, out_stride, bp.tab->link.ptr, bp.tab->masks.ptr, nstr, bp.n,
          bp.nsig, c + b0 * c_stride, c_stride, spin_shift, active ? active + b0 : nullptr);
      CU_LAUNCH_CHECK();
    } else {
      k_scatter_fp64<<<g1, 256, 0, ctx->stream>>>(
          bp.tab->link.ptr, bp.tab->masks.ptr, bp.tabb->link.ptr, bp.tabb->masks.ptr, nstr, nstrb,
          bp.n, bp.nsigb, bp.msms(), w.E.ptr, c, c_stride, spin_shift, active, bm_d, out,
          out_stride);
      CU_LAUNCH_CHECK();
    }
  }
}

void s2_apply(mbe_ctx* ctx, BinProblem& bp, const double* c, int64_t c_stride, double* out,
              int64_t out_stride, const int32_t* active) {
  int64_t blocks = (bp.ndet + 255) / 256;
  if (blocks > 2048) blocks = 2048;
  dim3 g((unsigned)blocks, bp.B);
  k_s2<<<g, 256, 0, ctx->stream>>>(bp.tab->link.ptr, bp.tab->masks.ptr, bp.tabb->link.ptr,
                                   bp.tabb->masks.ptr, bp.nstr, bp.nstrb, bp.n, bp.nsigb,
                                   bp.msms(), c, c_stride, active, out, out_stride);
  CU_LAUNCH_CHECK();
}

// ------------------------------------------------------------ warm starts
namespace {

__global__ void k_f64_to_f32(const double* __restrict__ src, float* __restrict__ dst, int64_t n) {
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < n;
       k += (int64_t)gridDim.x * blockDim.x)
    dst[k] = (float)src[k];
}

// V[b][0] of the child tuple from the parent's vector: every parent string
// (n - 1 orbitals) gains the added orbital at active position jo -- empty,
// or occupied in both strings, which moves its creation operators past the
// electrons below it: sign (-1)^(n_alpha below + n_beta below).  The child
// row is zeroed first by k_zero_start.
template <typename T>
__global__ void k_zero_start(const int32_t* __restrict__ bidx, int64_t N, T* __restrict__ V,
                             int64_t vstride) {
  T* Vb = V + (int64_t)bidx[blockIdx.y] * vstride;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N;
       k += (int64_t)gridDim.x * blockDim.x)
    Vb[k] = (T)0;
}

template <typename T>
__global__ void k_parent_guess(const float* const* __restrict__ src,
                               const int32_t* __restrict__ bidx, const int32_t* __restrict__ jo,
                               const int32_t* __restrict__ occ,
                               const uint32_t* __restrict__ masks_v, int nstr_v,
                               const uint32_t* __restrict__ masks_o, int nstr_o, int nstr,
                               T* __restrict__ V, int64_t vstride) {
  const int e = blockIdx.y;
  const int o = occ[e], j = jo[e];
  const uint32_t* pm = o ? masks_o : masks_v;
  const int np = o ? nstr_o : nstr_v;
  const int64_t Np = (int64_t)np * np;
  const uint32_t low = (1u << j) - 1u;
  const float* sv = src[e];
  T* Vb = V + (int64_t)bidx[e] * vstride;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < Np;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int ia = (int)(i / np), ib = (int)(i - (int64_t)ia * np);
    const uint32_t ma = pm[ia], mb = pm[ib];
    const uint32_t ca = (ma & low) | ((ma & ~low) << 1) | ((uint32_t)o << j);
    const uint32_t cb = (mb & low) | ((mb & ~low) << 1) | ((uint32_t)o << j);
    const int neg = o ? ((__popc(ma & low) + __popc(mb & low)) & 1) : 0;
    const float v = sv[i];
    Vb[(int64_t)mask_rank(ca) * nstr + mask_rank(cb)] = (T)(neg ? -v : v);
  }
}

// the inserted vectors are FP32 copies: normalise each in FP64 (the
// Rayleigh-Ritz step assumes an orthonormal basis), one block per tuple
template <typename T>
__global__ void k_normalize_start(const int32_t* __restrict__ bidx, int64_t N, T* __restrict__ V,
                                  int64_t vstride) {
  T* Vb = V + (int64_t)bidx[blockIdx.x] * vstride;
  __shared__ double red[32];
  double s = 0.0;
  for (int64_t k = threadIdx.x; k < N; k += blockDim.x) s += (double)Vb[k] * (double)Vb[k];
  for (int off = 16; off; off >>= 1) s += __shfl_down_sync(0xffffffffu, s, off);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  __shared__ double inv;
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) t += red[w];
    inv = t > 0.0 ? 1.0 / sqrt(t) : 1.0;
  }
  __syncthreads();
  for (int64_t k = threadIdx.x; k < N; k += blockDim.x) Vb[k] = (T)((double)Vb[k] * inv);
}

}  // namespace

void launch_parent_guess(mbe_ctx* ctx, const GuessPlan& plan, int n, int nsig, int nstr,
                         float* V32, double* V64, int64_t vstride) {
  const int ne = (int)plan.b.size();
  if (ne == 0 || n < 2) return;
  bool any_o = false, any_v = false;
  for (int e = 0; e < ne; e++) (plan.occ[e] ? any_o : any_v) = true;
  const StringTables* tv = any_v ? get_tables(ctx, n - 1, nsig) : nullptr;
  const StringTables* to = (any_o && nsig >= 1) ? get_tables(ctx, n - 1, nsig - 1) : nullptr;
  if (any_o && !to) throw MbeError{MBE_ESTATE, "occupied added orbital without electrons"};
  DevBuf<int32_t> bidx(&ctx->pool, ne), jo(&ctx->pool, ne), occ(&ctx->pool, ne);
  DevBuf<const float*> src(&ctx->pool, ne);
  cudaStream_t st = ctx->stream;
  CU_CHECK(cudaMemcpyAsync(bidx.ptr, plan.b.data(), sizeof(int32_t) * ne, cudaMemcpyHostToDevice, st));
  CU_CHECK(cudaMemcpyAsync(jo.ptr, plan.jo.data(), sizeof(int32_t) * ne, cudaMemcpyHostToDevice, st));
  CU_CHECK(cudaMemcpyAsync(occ.ptr, plan.occ.data(), sizeof(int32_t) * ne, cudaMemcpyHostToDevice, st));
  CU_CHECK(cudaMemcpyAsync(src.ptr, plan.src.data(), sizeof(const float*) * ne,
                           cudaMemcpyHostToDevice, st));
  const int64_t N = (int64_t)nstr * nstr;
  const dim3 g((unsigned)std::min<int64_t>((N + 255) / 256, 1024), ne);
  const uint32_t* mv = tv ? tv->masks.ptr : nullptr;
  const uint32_t* mo = to ? to->masks.ptr : nullptr;
  const int nv = tv ? tv->nstr : 0, no = to ? to->nstr : 0;
  if (V32) {
    k_zero_start<float><<<g, 256, 0, st>>>(bidx.ptr, N, V32, vstride);
    CU_LAUNCH_CHECK();
    k_parent_guess<float><<<g, 256, 0, st>>>(src.ptr, bidx.ptr, jo.ptr, occ.ptr, mv, nv, mo, no,
                                             nstr, V32, vstride);
    CU_LAUNCH_CHECK();
    k_normalize_start<float><<<ne, 1024, 0, st>>>(bidx.ptr, N, V32, vstride);
  } else {
    k_zero_start<double><<<g, 256, 0, st>>>(bidx.ptr, N, V64, vstride);
    CU_LAUNCH_CHECK();
    k_parent_guess<double><<<g, 256, 0, st>>>(src.ptr, bidx.ptr, jo.ptr, occ.ptr, mv, nv, mo, no,
                                              nstr, V64, vstride);
    CU_LAUNCH_CHECK();
    k_normalize_start<double><<<ne, 1024, 0, st>>>(bidx.ptr, N, V64, vstride);
  }
  CU_LAUNCH_CHECK();
}

void convert_f64_to_f32(mbe_ctx* ctx, const double* src, float* dst, int64_t n) {
  if (n <= 0) return;
  k_f64_to_f32<<<(unsigned)std::min<int64_t>((n + 255) / 256, 4096), 256, 0, ctx->stream>>>(
      src, dst, n);
  CU_LAUNCH_CHECK();
}

void launch_finish_sym_fp64(mbe_ctx* ctx, const BinProblem& bp, double* out, int64_t out_stride,
                            const double* c, int64_t c_stride, double spin_shift,
                            const int32_t* active) {
  const int ntl = (bp.nstr + 31) / 32;
  k_finish_sym_fp64<<<dim3((unsigned)(ntl * (ntl + 1) / 2), bp.B), 256, 0, ctx->stream>>>(
      out, out_stride, bp.tab->link.ptr, bp.tab->masks.ptr, bp.nstr, bp.n, bp.nsig, c, c_stride,
      spin_shift, active);
  CU_LAUNCH_CHECK();
}
