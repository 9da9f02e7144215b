// FP64 sigma vector on the CUDA cores, element by element from the string
// links (no D and E intermediates).
//
// With L_P the matrix of E_pq + E_qp (E_pp for p = q) between strings of one
// spin, H = 1/2 sum_PQ g'_PQ (L_P x 1 + 1 x L_P)(L_Q x 1 + 1 x L_Q) gives
//   sigma(a, b) = sum_a' H^a(a, a') c(a', b) + sum_b' H^b(b, b') c(a, b')
//               + sum_{P in links(a)} sum_{Q in links(b)} g'_PQ s_a(P) s_b(Q)
//                                                         c(J_a(P), J_b(Q))
//               + shift (S^2 c)(a, b),
// H^a = 1/2 sum_PQ g'_PQ L_P L_Q on the alpha strings (single and double
// replacements), H^b the same on the beta strings.
//
// GB300 issues two FP64 FMAs per clock and SM, against 16 doubles of shared
// memory per clock: the number of FP64 operations is what bounds this, not
// the gathers.  The dense route (gather D, E = g' D over all npair pairs,
// scatter) takes npair^2 FMAs per determinant; only the n_off = nsig (n -
// nsig) pairs that link a string contribute, so the sum above takes n_off^2 +
// 2 n_off + 2 nnz (nnz non-zero H^a per row), and half of that when c is
// symmetric (sigma(a, b) for a <= b): 8e/12o 747 against 6084, 6e/9o 252
// against 2025.  Measured per launch: 3 x 8e/11o 0.379 ms (79 % of the FP64
// FMA rate) against 3.94 ms for the dense route's four kernels, 45 tuples of
// 6e/9o and 8e/9o 0.148 against 1.69 ms.
//
// One CTA per (row a, tuple).  The rows J_a(P) of c lie transposed in shared
// memory (a column J is n_off contiguous doubles), the rows P of g' signed by
// s_a(P) likewise (a pair Q is n_off contiguous doubles), so a thread that
// owns the string b walks the links Q of b with two 16-byte loads per two
// FMAs.  Rows that do not fit go through in chunks of NI links.  The links
// of b are split over S parts (one warp takes 32 strings and one part), the
// parts summed in a fixed order.  The spin term is part of the same sum: its
// exchange of a's link with the same pair of b, occupied the other way round,
// is a second copy of that row of g' with -shift added.
#include "mbe_internal.cuh"
#include <algorithm>

namespace {

__device__ __forceinline__ int pair_of(int p, int q) {
  return p >= q ? p * (p + 1) / 2 + q : q * (q + 1) / 2 + p;
}
// position of the i-th set bit
__device__ __forceinline__ int nth_bit(uint32_t m, int i) {
  for (; i > 0; i--) m &= m - 1;
  return __ffs(m) - 1;
}
// parity of the occupied orbitals strictly between p and q
__device__ __forceinline__ int parity_between(uint32_t m, int p, int q) {
  const int lo = min(p, q), hi = max(p, q);
  return __popc(m & ((1u << hi) - 1u) & ~((2u << lo) - 1u)) & 1;
}
// i-th pair (x < y) of 0 .. ny-1 in the order (0,1), (0,2), (1,2), (0,3) ..
__device__ __forceinline__ void pair_decode(int i, int& x, int& y) {
  y = 1;
  while (i >= y) {
    i -= y;
    y++;
  }
  x = i;
}

// replacements of a string: k = 0 the string itself, then the single ones
// (hole-major), then the double ones
struct Repl {
  int kind;          // 0, 1, 2 replaced orbitals
  int q, p, s, r;    // q -> p and s -> r
};
__device__ __forceinline__ Repl repl_of(uint32_t m, int n, int nsig, int k) {
  Repl x = {0, 0, 0, 0, 0};
  if (k == 0) return x;
  const int nv = n - nsig, noff = nsig * nv;
  const uint32_t v = ~m & ((1u << n) - 1u);
  if (k <= noff) {
    x.kind = 1;
    x.q = nth_bit(m, (k - 1) / nv);
    x.p = nth_bit(v, (k - 1) % nv);
    return x;
  }
  const int nvp = nv * (nv - 1) / 2, kk = k - 1 - noff;
  int h0, h1, v0, v1;
  pair_decode(kk / nvp, h0, h1);
  pair_decode(kk % nvp, v0, v1);
  x.kind = 2;
  x.q = nth_bit(m, h0);
  x.s = nth_bit(m, h1);
  x.p = nth_bit(v, v0);
  x.r = nth_bit(v, v1);
  return x;
}

// the ascending (colexicographic) order of the k-subsets of n bits: binomial
// coefficients of up to 15 orbitals
struct Binom {
  uint16_t c[16][16];
};
__device__ __forceinline__ int rank_of(const Binom& t, uint32_t m) {
  int r = 0;
  for (int i = 1; m; i++, m &= m - 1) r += t.c[__ffs(m) - 1][i];
  return r;
}
__device__ __forceinline__ uint32_t unrank(const Binom& t, int r, int n, int k) {
  uint32_t m = 0;
  for (int p = n - 1; p >= 0 && k > 0; p--)
    if (t.c[p][k] <= r) {
      r -= t.c[p][k--];
      m |= 1u << p;
    }
  return m;
}

// per shape: the strings (ascending masks), hidx[k][I] the string of
// replacement k of I, and olnk[x][I] the off-diagonal links
// (J << 9) | (Q << 2) | (dir << 1) | (sign < 0), dir = 1 if I holds the larger
// orbital of the pair Q
__global__ void k_direct_tables(const Binom bn, int nstr, int n, int nsig, int nnz,
                                uint32_t* __restrict__ masks, uint16_t* __restrict__ hidx,
                                uint32_t* __restrict__ olnk) {
  __shared__ Binom sb;
  for (int t = threadIdx.x; t < 256; t += blockDim.x) sb.c[t >> 4][t & 15] = bn.c[t >> 4][t & 15];
  __syncthreads();
  const int noff = nsig * (n - nsig);
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < (int64_t)nnz * nstr;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int k = (int)(t / nstr), I = (int)(t - (int64_t)k * nstr);
    const uint32_t m = unrank(sb, I, n, nsig);
    const Repl x = repl_of(m, n, nsig, k);
    uint32_t m2 = m;
    if (x.kind >= 1) m2 ^= (1u << x.q) ^ (1u << x.p);
    if (x.kind == 2) m2 ^= (1u << x.s) ^ (1u << x.r);
    const int J = x.kind ? rank_of(sb, m2) : I;
    if (k == 0) masks[I] = m;
    hidx[t] = (uint16_t)J;
    if (x.kind == 1 && k <= noff)
      olnk[(int64_t)(k - 1) * nstr + I] = ((uint32_t)J << 9) | ((uint32_t)pair_of(x.p, x.q) << 2) |
                                          (x.q > x.p ? 2u : 0u) |
                                          (uint32_t)parity_between(m, x.p, x.q);
  }
}

// per tuple: hv[k][I] = <I| 1/2 sum_PQ g'_PQ L_P L_Q |replacement k of I> by
// the Slater-Condon rules of one spin (k_ps = 1/2 sum_q g'_{pq,qs} its
// one-body part), and wt[P][I] = sum_{q in I} g'_{P,qq}
__global__ void k_direct_values(const uint32_t* __restrict__ masks, int nstr, int n, int nsig,
                                int nnz, int npair, const double* __restrict__ gp_all,
                                double* __restrict__ hv_all, double* __restrict__ wt_all) {
  const int b = blockIdx.y;
  const double* g = gp_all + (int64_t)b * npair * npair;
  double* hv = hv_all + (int64_t)b * nnz * nstr;
  double* wt = wt_all ? wt_all + (int64_t)b * npair * nstr : nullptr;
  __shared__ double sk[15 * 15];
  for (int t = threadIdx.x; t < n * n; t += blockDim.x) {
    const int p = t / n, s = t - p * n;
    double v = 0.0;
    for (int q = 0; q < n; q++) v += g[(int64_t)pair_of(p, q) * npair + pair_of(q, s)];
    sk[t] = 0.5 * v;
  }
  __syncthreads();
  auto G = [&](int p, int q, int r, int s) {
    return g[(int64_t)pair_of(p, q) * npair + pair_of(r, s)];
  };
  const int64_t nh = (int64_t)nnz * nstr, tot = nh + (wt ? (int64_t)npair * nstr : 0);
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < tot;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t row = (t < nh ? t : t - nh) / nstr;
    const int I = (int)((t < nh ? t : t - nh) - row * nstr);
    const uint32_t m = masks[I];
    if (t >= nh) {
      double v = 0.0;
      for (uint32_t o = m; o; o &= o - 1) {
        const int q = __ffs(o) - 1;
        v += g[row * npair + q * (q + 1) / 2 + q];
      }
      wt[t - nh] = v;
      continue;
    }
    const Repl x = repl_of(m, n, nsig, (int)row);
    double v;
    if (x.kind == 0) {
      v = 0.0;
      double v2 = 0.0;
      for (uint32_t o = m; o; o &= o - 1) {
        const int p = __ffs(o) - 1;
        v += sk[p * n + p];
        for (uint32_t u = m; u; u &= u - 1) {
          const int r = __ffs(u) - 1;
          v2 += G(p, p, r, r) - G(p, r, r, p);
        }
      }
      v += 0.5 * v2;
    } else if (x.kind == 1) {
      v = sk[x.p * n + x.q];
      for (uint32_t o = m & ~(1u << x.q); o; o &= o - 1) {
        const int r = __ffs(o) - 1;
        v += G(x.p, x.q, r, r) - G(x.p, r, r, x.q);
      }
      if (parity_between(m, x.p, x.q)) v = -v;
    } else {
      v = G(x.p, x.q, x.r, x.s) - G(x.p, x.s, x.r, x.q);
      const uint32_t m1 = m ^ (1u << x.p) ^ (1u << x.q);
      if (parity_between(m, x.p, x.q) ^ parity_between(m1, x.r, x.s)) v = -v;
    }
    hv[t] = v;
  }
}

// plan of the main kernel: NI links of a per chunk, row pitch, S parts
struct DirPlan {
  int ni, pitch, nchunk, parts, threads;
  uint32_t g, c, part, crow, wa, coef, total;   // byte offsets in shared memory
};

constexpr uint32_t DIR_SMEM = 220 * 1024;

inline DirPlan direct_plan(int npair, int noff, int nnz, int nstrb) {
  DirPlan p;
  // 8 parts keep the warps of a row evenly loaded (a row of 300 strings is 80
  // tasks for 16 warps); above 512 strings a row has warps enough
  p.parts = nstrb <= 512 ? 8 : nstrb <= 1024 ? 4 : nstrb <= 2048 ? 2 : 1;
  p.threads = nstrb <= 64 ? 128 : nstrb <= 256 ? 256 : 512;
  auto lay = [&](int ni) {
    p.ni = ni;
    // an odd number of 16-byte units per row: columns spread over the banks
    p.pitch = (ni >> 1) & 1 ? ni : ni + 2;
    uint32_t o = 0;
    auto take = [&](uint32_t bytes) {
      const uint32_t r = o;
      o += (bytes + 15u) & ~15u;
      return r;
    };
    p.g = take((uint32_t)(npair + noff) * p.pitch * 8);
    p.c = take((uint32_t)nstrb * p.pitch * 8);
    p.part = take((uint32_t)p.parts * nstrb * 8);
    p.crow = take((uint32_t)nstrb * 8);
    p.wa = take((uint32_t)npair * 8);
    p.coef = take((uint32_t)nnz * 12);
    p.total = o;
    return o <= DIR_SMEM;
  };
  const int full = std::max(2, (noff + 1) & ~1);
  p.nchunk = 1;
  int ni = full;
  while (!lay(ni) && ni > 2) {
    p.nchunk++;
    ni = ((full + p.nchunk - 1) / p.nchunk + 1) & ~1;
  }
  p.nchunk = (full + p.ni - 1) / p.ni;
  return p;
}

__device__ __forceinline__ double flip_if(double x, uint32_t neg) {
  return __hiloint2double(__double2hiint(x) ^ (int)(neg << 31), __double2loint(x));
}

struct DirArgs {
  int n, npair, nstr, nstrb, nsig, nsigb, nnz, nnzb, sym;
  const uint32_t *masks, *masksb, *olnk, *olnkb;
  const uint16_t *hidx, *hidxb;
  const double *hv, *hvb, *wt;
  const double* gp;
  const double* c;
  int64_t c_stride;
  double* out;
  int64_t out_stride;
  const int32_t* active;
  double shift, msms;
};

// (two CTAs of 512 threads per SM, 62 registers: with the 40 registers that the
// compiler takes for three, 3 x 8e/11o is 449 us against 437 and 14e/14o 109 ms
// against 96; 45 of 6e/9o and 8e/9o are 129 us against 135)
__global__ void __launch_bounds__(512, 2)
k_sigma_direct(const DirArgs A, const DirPlan L) {
  const int b = blockIdx.y;
  if (A.active && !A.active[b]) return;
  extern __shared__ __align__(16) unsigned char smem[];
  double* sG = reinterpret_cast<double*>(smem + L.g);
  double* sC = reinterpret_cast<double*>(smem + L.c);
  double* sPart = reinterpret_cast<double*>(smem + L.part);
  double* sRow = reinterpret_cast<double*>(smem + L.crow);
  double* sWa = reinterpret_cast<double*>(smem + L.wa);
  double* sCoef = reinterpret_cast<double*>(smem + L.coef);
  int* sIdx = reinterpret_cast<int*>(sCoef + A.nnz);
  __shared__ uint32_t sLink[64];       // the links of a
  __shared__ uint16_t sSel[2 * 128];   // row of sG for (Q, dir)
  const int a = blockIdx.x, tid = threadIdx.x, nt = blockDim.x;
  const int lane = tid & 31, warp = tid >> 5;
  const int npair = A.npair, nstrb = A.nstrb;
  const int noff = A.nsig * (A.n - A.nsig), noffb = A.nsigb * (A.n - A.nsigb);
  const int pitch = L.pitch, S = L.parts;
  const uint32_t ma = A.masks[a];
  const double* g = A.gp + (int64_t)b * npair * npair;
  const double* cb = A.c + (int64_t)b * A.c_stride;
  const double* hv = A.hv + (int64_t)b * A.nnz * A.nstr;
  const double* hvb = A.hvb + (int64_t)b * A.nnzb * nstrb;
  const double* wt = A.wt + (int64_t)b * npair * nstrb;
  const int b0 = A.sym ? a : 0, nb = nstrb - b0;

  for (int x = tid; x < noff; x += nt) sLink[x] = A.olnk[(int64_t)x * A.nstr + a];
  for (int t = tid; t < 2 * npair; t += nt) sSel[t] = (uint16_t)(t >> 1);
  for (int k = tid; k < A.nnz; k += nt) {
    sCoef[k] = hv[(int64_t)k * A.nstr + a];
    sIdx[k] = A.hidx[(int64_t)k * A.nstr + a];
  }
  for (int k = tid; k < nstrb; k += nt) sRow[k] = cb[(int64_t)a * nstrb + k];
  for (int Q = tid; Q < npair; Q += nt) {
    double v = 0.0;
    for (uint32_t o = ma; o; o &= o - 1) {
      const int p = __ffs(o) - 1;
      v += g[(int64_t)(p * (p + 1) / 2 + p) * npair + Q];
    }
    sWa[Q] = v;
  }
  __syncthreads();
  // the other occupation of a's own pairs takes the row with the spin exchange
  for (int x = tid; x < noff; x += nt) {
    const uint32_t e = sLink[x];
    const int Q = (e >> 2) & 127, dir = (e >> 1) & 1;
    sSel[2 * Q + (dir ^ 1)] = (uint16_t)(npair + x);
  }

  const int nblk = (nb + 31) / 32;
  for (int ch = 0; ch < L.nchunk; ch++) {
    const int i0 = ch * L.ni, ni = min(L.ni, noff - i0);   // ni <= 0: no links
    const int nip = (ni + 1) & ~1;
    __syncthreads();
    // signed rows of g' for this chunk's links, pair-major; the copies of a's
    // own pairs with -shift in their own place
    for (int t = tid; t < nip * (npair + noff); t += nt) {
      const int i = t / (npair + noff), r = t - i * (npair + noff);
      double v = 0.0;
      if (i < ni) {
        const uint32_t e = sLink[i0 + i];
        const int P = (e >> 2) & 127;
        const int Q = r < npair ? r : (int)((sLink[r - npair] >> 2) & 127);
        v = g[(int64_t)P * npair + Q];
        if (r >= npair && r - npair == i0 + i) v -= A.shift;
        v = flip_if(v, e & 1u);
      }
      sG[r * pitch + i] = v;
    }
    // rows J_a(P_i) of c, column-major
    for (int t = tid; t < nip * nstrb; t += nt) {
      const int i = t / nstrb, k = t - i * nstrb;
      sC[k * pitch + i] = i < ni ? cb[(int64_t)(sLink[i0 + i] >> 9) * nstrb + k] : 0.0;
    }
    __syncthreads();
    for (int task = warp; task < nblk * S; task += nt >> 5) {
      const int part = task / nblk, k = (task - part * nblk) * 32 + lane;
      if (k >= nb) continue;
      const int ib = b0 + k;
      double acc0 = ch ? sPart[part * nb + k] : 0.0, acc1 = 0.0;
      const int x0 = noffb * part / S, x1 = noffb * (part + 1) / S;
      if (nip > 0)
        for (int x = x0; x < x1; x++) {
          const uint32_t e = A.olnkb[(int64_t)x * nstrb + ib];
          const double2* cp = reinterpret_cast<const double2*>(sC + (e >> 9) * pitch);
          const double2* gq =
              reinterpret_cast<const double2*>(sG + (int)sSel[(e >> 1) & 255u] * pitch);
          const uint32_t neg = e & 1u;
          acc0 = flip_if(acc0, neg);
          acc1 = flip_if(acc1, neg);
#pragma unroll 4
          for (int i = 0; i < nip >> 1; i++) {
            const double2 u = cp[i], v = gq[i];
            acc0 = fma(u.x, v.x, acc0);
            acc1 = fma(u.y, v.y, acc1);
          }
          acc0 = flip_if(acc0, neg);
          acc1 = flip_if(acc1, neg);
        }
      if (ch == 0) {
        // beta replacements at fixed a: H^b, and a's diagonal with b's links
#pragma unroll 4
        for (int q = A.nnzb * part / S; q < A.nnzb * (part + 1) / S; q++)
          acc0 = fma(hvb[(int64_t)q * nstrb + ib], sRow[A.hidxb[(int64_t)q * nstrb + ib]], acc0);
        for (int x = x0; x < x1; x++) {
          const uint32_t e = A.olnkb[(int64_t)x * nstrb + ib];
          acc1 = fma(flip_if(sWa[(e >> 2) & 127], e & 1u), sRow[e >> 9], acc1);
        }
        // alpha replacements at fixed b: H^a, and a's links with b's diagonal
#pragma unroll 4
        for (int q = A.nnz * part / S; q < A.nnz * (part + 1) / S; q++)
          acc0 = fma(sCoef[q], cb[(int64_t)sIdx[q] * nstrb + ib], acc0);
        for (int x = noff * part / S; x < noff * (part + 1) / S; x++) {
          const uint32_t e = sLink[x];
          acc1 = fma(flip_if(wt[(int64_t)((e >> 2) & 127) * nstrb + ib], e & 1u),
                     cb[(int64_t)(e >> 9) * nstrb + ib], acc1);
        }
        if (part == 0) {
          const uint32_t mb = A.masksb[ib];
          double d = A.shift * ((double)(A.nsigb - __popc(ma & mb)) + A.msms);
          for (uint32_t o = mb; o; o &= o - 1) {
            const int q = __ffs(o) - 1;
            d += sWa[q * (q + 1) / 2 + q];
          }
          acc1 = fma(d, sRow[ib], acc1);
        }
      }
      sPart[part * nb + k] = acc0 + acc1;
    }
  }
  __syncthreads();
  double* ob = A.out + (int64_t)b * A.out_stride;
  for (int k = tid; k < nb; k += nt) {
    double s = sPart[k];
    for (int part = 1; part < S; part++) s += sPart[part * nb + k];
    if (A.sym == 1) {
      ob[sym_index(a, b0 + k, nstrb)] = s;
    } else {
      ob[(int64_t)a * nstrb + b0 + k] = s;
      if (A.sym) ob[(int64_t)(b0 + k) * nstrb + a] = s;
    }
  }
}

}  // namespace

int direct_nnz(int n, int nsig) {
  const int nv = n - nsig;
  return 1 + nsig * nv + nsig * (nsig - 1) / 2 * (nv * (nv - 1) / 2);
}

// flops of one sigma vector: two per element that the kernel multiplies (link
// pairs, one-spin elements, links with the other spin's diagonal), of the upper
// triangle where c = c^T
double direct_flops(int n, int nsig, int nsigb, int64_t nstr, int64_t nstrb, bool symmetric) {
  const double na = (double)nsig * (n - nsig), nb = (double)nsigb * (n - nsigb);
  const double rows = symmetric ? 0.5 * nstr * (nstr + 1) : (double)nstr * nstrb;
  return 2.0 * rows * (na * nb + na + nb + direct_nnz(n, nsig) + direct_nnz(n, nsigb) + 1);
}

void launch_direct_tables(mbe_ctx* ctx, int n, int nsig, int nstr, uint32_t* masks,
                          uint16_t* hidx, uint32_t* olnk) {
  Binom bn;   // C(15, 7) = 6435 at most
  for (int p = 0; p < 16; p++)
    for (int k = 0; k < 16; k++) bn.c[p][k] = k > p ? 0 : (uint16_t)string_count(p, k);
  const int nnz = direct_nnz(n, nsig);
  const int64_t tot = (int64_t)nnz * nstr;
  k_direct_tables<<<(unsigned)std::min<int64_t>((tot + 255) / 256, 4096), 256, 0, ctx->stream>>>(
      bn, nstr, n, nsig, nnz, masks, hidx, olnk);
  CU_LAUNCH_CHECK();
}

void launch_direct_values(mbe_ctx* ctx, int n, int nsig, int nstr, const uint32_t* masks, int B,
                          const double* gp, double* hv, double* wt) {
  const int nnz = direct_nnz(n, nsig), npair = n * (n + 1) / 2;
  const int64_t tot = (int64_t)(nnz + (wt ? npair : 0)) * nstr;
  // about 16 CTAs per SM over the batch at most
  const int64_t most = std::max<int64_t>(1, 2432 / B);
  k_direct_values<<<dim3((unsigned)std::min<int64_t>((tot + 255) / 256, most), B), 256, 0,
                    ctx->stream>>>(masks, nstr, n, nsig, nnz, npair, gp, hv, wt);
  CU_LAUNCH_CHECK();
}

// the kernel's shared memory, once per device (before a capture: an attribute
// loads the kernel)
static void sigma_direct_attributes(int device) {
  static bool attr_done[MBE_MAX_DEVICES] = {false};
  once_per_device(attr_done, device, [] {
    CU_CHECK(cudaFuncSetAttribute(k_sigma_direct, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  (int)DIR_SMEM));
  });
}

void sigma_direct_raw(mbe_ctx* ctx, int n, const DirectSide& al, const DirectSide& be,
                      const double* wt, const double* gp, const double* c, int64_t c_stride,
                      double* out, int64_t out_stride, const int32_t* active,
                      int nb, double spin_shift, int symmetric) {
  DirArgs A;
  A.n = n;
  A.npair = n * (n + 1) / 2;
  A.nstr = al.nstr;
  A.nstrb = be.nstr;
  A.nsig = al.nsig;
  A.nsigb = be.nsig;
  A.nnz = direct_nnz(n, al.nsig);
  A.nnzb = direct_nnz(n, be.nsig);
  A.sym = symmetric;
  A.masks = al.masks;
  A.masksb = be.masks;
  A.olnk = al.olnk;
  A.olnkb = be.olnk;
  A.hidx = al.hidx;
  A.hidxb = be.hidx;
  A.hv = al.hv;
  A.hvb = be.hv;
  A.wt = wt;
  A.gp = gp;
  A.c = c;
  A.c_stride = c_stride;
  A.out = out;
  A.out_stride = out_stride;
  A.active = active;
  A.shift = spin_shift;
  A.msms = 0.25 * (al.nsig - be.nsig) * (al.nsig - be.nsig + 2);   // Ms(Ms+1)
  const DirPlan L = direct_plan(A.npair, al.nsig * (n - al.nsig), A.nnz, be.nstr);
  if (L.total > DIR_SMEM) throw MbeError{MBE_EINVAL, "active space too large for the FP64 sigma"};
  sigma_direct_attributes(ctx->device);
  cudaEvent_t ev;
  ctx->fp64_timer.begin(ctx->stream, ctx->opt.timing != 0, &ev);
  k_sigma_direct<<<dim3((unsigned)al.nstr, (unsigned)nb), L.threads, L.total, ctx->stream>>>(A, L);
  CU_LAUNCH_CHECK();
  ctx->fp64_timer.end(ctx->stream, ev);
  ctx->stats.fp64_launches += 1;
}

// the closed-shell shape fits the kernel's shared memory
bool sigma_direct_supported(int n, int nsig, int nstr) {
  return direct_plan(n * (n + 1) / 2, nsig * (n - nsig), direct_nnz(n, nsig), nstr).total <=
         DIR_SMEM;
}

// the shape's tables (once) and the batch's values (once per batch)
void sigma_direct_prepare(mbe_ctx* ctx, BinProblem& bp) {
  sigma_direct_attributes(ctx->device);
  const int n = bp.n;
  auto tables = [&](const StringTables* ct) {
    StringTables* t = const_cast<StringTables*>(ct);
    if (t->direct_ready) return;
    t->hidx.reset(&ctx->pool, (size_t)direct_nnz(n, t->nsig) * t->nstr);
    t->olnk.reset(&ctx->pool, std::max<size_t>(1, (size_t)t->nsig * (n - t->nsig) * t->nstr));
    launch_direct_tables(ctx, n, t->nsig, t->nstr, t->masks.ptr, t->hidx.ptr, t->olnk.ptr);
    t->direct_ready = true;   // the tables outlive a call that runs out of memory half-way
  };
  tables(bp.tab);
  tables(bp.tabb);
  const size_t need = (size_t)bp.B * direct_nnz(n, bp.nsig) * bp.nstr;
  if (bp.hv.n == need) return;
  bp.hv.reset(&ctx->pool, need);
  bp.wt.reset(&ctx->pool, (size_t)bp.B * bp.npair * bp.nstrb);
  if (bp.closed()) {
    launch_direct_values(ctx, n, bp.nsig, bp.nstr, bp.tab->masks.ptr, bp.B, bp.gp.ptr, bp.hv.ptr,
                         bp.wt.ptr);
  } else {
    bp.hvb.reset(&ctx->pool, (size_t)bp.B * direct_nnz(n, bp.nsigb) * bp.nstrb);
    launch_direct_values(ctx, n, bp.nsig, bp.nstr, bp.tab->masks.ptr, bp.B, bp.gp.ptr, bp.hv.ptr,
                         nullptr);
    launch_direct_values(ctx, n, bp.nsigb, bp.nstrb, bp.tabb->masks.ptr, bp.B, bp.gp.ptr,
                         bp.hvb.ptr, bp.wt.ptr);
  }
}

void sigma_direct(mbe_ctx* ctx, BinProblem& bp, const double* c, int64_t c_stride, double* out,
                  int64_t out_stride, const int32_t* active, double spin_shift, bool symmetric,
                  bool packed) {
  sigma_direct_prepare(ctx, bp);
  const DirectSide al = {bp.nsig, bp.nstr, bp.tab->masks.ptr, bp.tab->olnk.ptr, bp.tab->hidx.ptr,
                         bp.hv.ptr};
  const DirectSide be = {bp.nsigb, bp.nstrb, bp.tabb->masks.ptr, bp.tabb->olnk.ptr,
                         bp.tabb->hidx.ptr, bp.closed() ? bp.hv.ptr : bp.hvb.ptr};
  sigma_direct_raw(ctx, bp.n, al, be, bp.wt.ptr, bp.gp.ptr, c, c_stride, out, out_stride, active,
                   bp.B, spin_shift, !symmetric || !bp.closed() ? 0 : packed ? 1 : 2);
}
