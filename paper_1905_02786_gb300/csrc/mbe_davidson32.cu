// Davidson iteration of the mixed-precision mode, laid out for GB300.
//
// GB300 issues FP64 arithmetic at roughly 1/60 of its FP32 rate, so every
// per-determinant operation here is FP32: the subspace vectors V, their
// sigma vectors AV, residuals and preconditioned corrections are stored and
// combined in FP32, with per-thread FP32 partial sums reduced in FP64 across
// threads.  FP64-grade quantities are formed only where the energy depends
// on them, at "exact points":
//   x      the current Ritz vector (FP32 values, taken as exact),
//   A x    by the FP64-grade sliced tensor-core contraction,
//   x.x    by an error-free FP32 dot (two-product + compensated sum),
//   theta  = x.Ax / x.x, the Rayleigh quotient reported as the energy,
//   r_x    = A x - theta x, its norm in FP64.
// Iteration (Davidson, J. Comput. Phys. 17, 87 (1975)):
//   stage A: tensor-core (split-BF16x3) sigma vectors until the residual is
//            below mixed_stage_tol max(1, |theta|) (default 1e-5, above
//            their precision floor);
//   rounds:  exact point; tuples with |r_x| above the target continue from
//            {x, t_1, ...} where t_j get tensor-core sigma vectors and the
//            couplings x.A t_j = theta (x.t_j) + r_x.t_j use only exact data;
//            the stage stops at max(target, mixed_round_drop |r_x|)
//            (default |r_x| / 100).
// The energy error of the reported Rayleigh quotient is below |r_x|^2 / gap.
#include "mbe_dvec.cuh"
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <limits>

using namespace dvec;

namespace {

// Every FP32 vector of the mixed Davidson iteration is alpha-beta symmetric
// and kept packed (mbe_dvec.cuh): L = sym_len(nstr) elements, about half of
// N_det.

// error-free dot of two packed FP32 vectors: products split exactly
// (p + e = x y), the p terms summed with compensation, all per-thread sums
// combined in FP64
__global__ void __launch_bounds__(RT)
k32_dot_comp(const float* __restrict__ X, int64_t xb, const float* __restrict__ Y, int64_t yb,
             int64_t N, int64_t nd, int ch, int nchunks, const int32_t* __restrict__ active,
             double* __restrict__ partial, int32_t* __restrict__ cnt, double* __restrict__ out) {
  const int b = blockIdx.y;
  if (active && !active[b]) return;
  __shared__ double red[32];
  const int64_t k0 = (int64_t)blockIdx.x * ch, k1 = min(N, k0 + ch);
  const float* x = X + (int64_t)b * xb;
  const float* y = Y + (int64_t)b * yb;
  // (s, lo): s + lo carries the running sum to ~2^-48 relative; every
  // product is split exactly (p + e = a b, fma) and every addition of p to s
  // exactly (TwoSum: s + p = t + err)
  float s = 0.f, lo = 0.f;
  for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
    const float a = x[k] * (k < nd ? 1.f : 2.f), bb = y[k];   // weight: exact
    const float p = a * bb;
    const float e = fmaf(a, bb, -p);
    const float t = s + p;
    const float bp = t - s;
    const float err = (s - (t - bp)) + (p - bp);
    s = t;
    lo += err + e;
  }
  const double tot = block_sum((double)s + (double)lo, red);
  double* pb = partial + (int64_t)b * nchunks;
  if (threadIdx.x == 0) pb[blockIdx.x] = tot;
  if (!last_cta(cnt + b, nchunks)) return;
  if (threadIdx.x < 32) {
    const double v = row_sum(pb, nchunks);
    if (threadIdx.x == 0) out[b] = v;
  }
}

// t = r / (theta - H_II) on the packed vector (the full vector's
// symmetrised correction: r and H_II are symmetric)
__global__ void k32_precondition(float* __restrict__ T, const float* __restrict__ hd, int64_t L,
                                 const double* __restrict__ theta,
                                 const int32_t* __restrict__ active) {
  const int b = blockIdx.y;
  if (!active[b]) return;
  const float th = (float)theta[b];
  float* Tb = T + (int64_t)b * L;
  const float* hb = hd + (int64_t)b * L;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < L;
       k += (int64_t)gridDim.x * blockDim.x) {
    float d = th - hb[k];
    if (fabsf(d) < 1e-4f) d = d < 0.f ? -1e-4f : 1e-4f;
    Tb[k] = Tb[k] / d;
  }
}

// T <- T - eps U (Olsen's combination where the dots are taken afterwards)
__global__ void k32_sub_eps(float* __restrict__ T, const float* __restrict__ U,
                            const float* __restrict__ eps, int64_t N,
                            const int32_t* __restrict__ active) {
  const int b = blockIdx.y;
  if (!active[b]) return;
  const float e = eps[b];
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N;
       k += (int64_t)gridDim.x * blockDim.x)
    T[(int64_t)b * N + k] = fmaf(-e, U[(int64_t)b * N + k], T[(int64_t)b * N + k]);
}

// Diagonal of H + shift S^2 in FP32 for the preconditioner (FP64 where it
// accumulates over a string): e(I) = sum_{p in I} h_pp + 1/2 sum_{p,q in I}
// (J_pq - K_pq) per string, then
//   H_II = e(a) + e(b) + sum_{p in a, q in b} J_pq + shift (nsig - |a & b|)
// with the alpha-beta Coulomb sum taken over pairs p >= q of a | b in a
// fixed order, so that H(a,b) = H(b,a) bitwise.
__global__ void k32_string_energy(const uint32_t* __restrict__ masks, int nstr, int n,
                                  const double* __restrict__ heff_all,
                                  const double* __restrict__ jk_all, float* __restrict__ estr) {
  const int b = blockIdx.y;
  const double* heff = heff_all + (int64_t)b * n * n;
  const double* J = jk_all + (int64_t)b * 2 * n * n;
  const double* K = J + n * n;
  for (int I = blockIdx.x * blockDim.x + threadIdx.x; I < nstr; I += gridDim.x * blockDim.x) {
    const uint32_t m = masks[I];
    double e = 0.0, e2 = 0.0;
    for (uint32_t mp = m; mp; mp &= mp - 1) {
      const int p = __ffs(mp) - 1;
      e += heff[p * n + p];
      for (uint32_t mq = m; mq; mq &= mq - 1) {
        const int q = __ffs(mq) - 1;
        e2 += J[p * n + q] - K[p * n + q];
      }
    }
    estr[(int64_t)b * nstr + I] = (float)(e + 0.5 * e2);
  }
}

__global__ void k32_hdiag(const uint32_t* __restrict__ masks, int nstr, int64_t ld, int n,
                          int nsig, const double* __restrict__ jk_all,
                          const float* __restrict__ estr, float shift, float* __restrict__ hd_all) {
  const int b = blockIdx.y;
  __shared__ float sJ[MBE_MAX_ACT * MBE_MAX_ACT];
  for (int t = threadIdx.x; t < n * n; t += blockDim.x)
    sJ[t] = (float)jk_all[(int64_t)b * 2 * n * n + t];
  __syncthreads();
  const int64_t N = (int64_t)nstr * nstr;
  const float* eb = estr + (int64_t)b * nstr;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < N;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int ia = (int)(i / nstr), ib = (int)(i - (int64_t)ia * nstr);
    if (ia > ib) continue;                      // packed: the upper triangle
    const uint32_t ma = masks[ia], mb = masks[ib], mu = ma | mb;
    float cross = 0.f;
    for (uint32_t mp = mu; mp; mp &= mp - 1) {
      const int p = __ffs(mp) - 1;
      const int ap = (ma >> p) & 1, bp = (mb >> p) & 1;
      for (uint32_t mq = mu & ((2u << p) - 1u); mq; mq &= mq - 1) {
        const int q = __ffs(mq) - 1;
        const int w = q == p ? (ap & bp) : ap * ((mb >> q) & 1) + ((ma >> q) & 1) * bp;
        if (w) cross = fmaf((float)w, sJ[p * n + q], cross);
      }
    }
    hd_all[(int64_t)b * ld + sym_index(ia, ib, nstr)] =
        (eb[ia] + eb[ib]) + cross + shift * (float)(nsig - __popc(ma & mb));
  }
}

// lowest-diagonal determinant a nstr + c, a <= c, of every tuple (without a
// P-space, whose selection finds it too)
__global__ void k32_lowest(const float* __restrict__ hd, int nstr, int64_t ld,
                           int32_t* __restrict__ low) {
  const int b = blockIdx.x;
  const int64_t N = (int64_t)nstr * nstr;
  __shared__ float sv[256];
  __shared__ int64_t si[256];
  float best = 3.4e38f;
  int64_t bi = 0;
  for (int64_t k = threadIdx.x; k < N; k += blockDim.x) {
    const int ia = (int)(k / nstr), ib = (int)(k - (int64_t)ia * nstr);
    if (ia > ib) continue;   // the mirror element has the same value, a larger k
    const float v = hd[(int64_t)b * ld + sym_index(ia, ib, nstr)];
    if (v < best) { best = v; bi = k; }
  }
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = blockDim.x / 2; s; s >>= 1) {
    if (threadIdx.x < s) {
      const float o = sv[threadIdx.x + s];
      const int64_t oi = si[threadIdx.x + s];
      if (o < sv[threadIdx.x] || (o == sv[threadIdx.x] && oi < si[threadIdx.x])) {
        sv[threadIdx.x] = o;
        si[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) low[b] = (int)si[0];
}

// start vectors: (|a b> + |b a>) / sqrt(2) of the lowest determinant (its
// packed element carries both halves), or |a a>; V_0 is zero on entry
__global__ void k32_guess(const int32_t* __restrict__ low, int B, int nstr, int64_t vstride,
                          float* __restrict__ V) {
  for (int b = blockIdx.x * blockDim.x + threadIdx.x; b < B; b += gridDim.x * blockDim.x) {
    const int ia = low[b] / nstr, ib = low[b] - ia * nstr;
    V[(int64_t)b * vstride + sym_index(ia, ib, nstr)] = ia == ib ? 1.f : 0.70710678f;
  }
}

// V0 = X / |X|: packed into V (slot 0), full into F (FP32, input of the
// exact sigma) and C64 (its FP64 copy); Lf is the stride of the full vectors
__global__ void k32_exact_prep(const float* __restrict__ X, const double* __restrict__ xx,
                               float* __restrict__ V, int M, int64_t L, float* __restrict__ F,
                               double* __restrict__ C64, int64_t Lf, int nstr,
                               const int32_t* __restrict__ active) {
  const int b = blockIdx.y;
  if (!active[b]) return;
  __shared__ float s_inv;
  if (threadIdx.x == 0) s_inv = (float)(1.0 / sqrt(xx[b]));   // one FP64 root per block
  __syncthreads();
  const float inv = s_inv;
  const int64_t N = (int64_t)nstr * nstr;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int ia = (int)(k / nstr), ib = (int)(k - (int64_t)ia * nstr);
    const int64_t p = sym_index(ia, ib, nstr);
    const float v = X[(int64_t)b * L + p] * inv;
    F[(int64_t)b * Lf + k] = v;
    C64[(int64_t)b * Lf + k] = (double)v;
    if (ia <= ib) V[(int64_t)b * M * L + p] = v;
  }
}

// start vectors of the tuples in plan_mask: the full FP32 vectors F (stride
// Lf) written by the parent guess, packed into V (slot 0)
__global__ void k32_pack_start(const float* __restrict__ F, int64_t Lf,
                               const int32_t* __restrict__ plan_mask, int nstr, int M, int64_t L,
                               float* __restrict__ V) {
  const int b = blockIdx.y;
  if (!plan_mask[b]) return;
  const int64_t N = (int64_t)nstr * nstr;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int ia = (int)(k / nstr), ib = (int)(k - (int64_t)ia * nstr);
    if (ia <= ib) V[(int64_t)b * M * L + sym_index(ia, ib, nstr)] = F[(int64_t)b * Lf + k];
  }
}

// r_x = A V0 - theta_x V0 (stored FP32), theta_x = xAx / xx, and |r_x|^2 into
// rnorm (C64, S64 full, stride N; RX packed, stride L); the last CTA of a
// tuple leaves theta_x (thx, theta) and G = [[xAx]]
__global__ void __launch_bounds__(RT)
k32_exact_rx(const double* __restrict__ C64, const double* __restrict__ S64,
             const double* __restrict__ xax, const double* __restrict__ xx, int64_t N, int ch,
             int nchunks, const int32_t* __restrict__ active, float* __restrict__ RX, int64_t L,
             int nstr, int M, double* __restrict__ partial, int32_t* __restrict__ cnt,
             double* __restrict__ thx, double* __restrict__ theta, double* __restrict__ G,
             double* __restrict__ rnorm, int32_t* __restrict__ iters) {
  const int b = blockIdx.y;
  if (!active[b]) return;
  __shared__ double red[32], s_th;
  if (threadIdx.x == 0) s_th = xax[b] / xx[b];
  __syncthreads();
  const double th = s_th;
  const int64_t k0 = (int64_t)blockIdx.x * ch, k1 = min(N, k0 + ch);
  double acc = 0.0;
  for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x) {
    const double r = fma(-th, C64[(int64_t)b * N + k], S64[(int64_t)b * N + k]);
    const int ia = (int)(k / nstr), ib = (int)(k - (int64_t)ia * nstr);
    if (ia <= ib && ia < nstr) RX[(int64_t)b * L + sym_index(ia, ib, nstr)] = (float)r;
    acc = fma(r, r, acc);
  }
  const double tot = block_sum(acc, red);
  double* pb = partial + (int64_t)b * nchunks;
  if (threadIdx.x == 0) pb[blockIdx.x] = tot;
  if (!last_cta(cnt + b, nchunks)) return;
  if (threadIdx.x < 32) {
    const double s = row_sum(pb, nchunks);
    if (threadIdx.x == 0) {
      rnorm[b] = s;
      thx[b] = th;
      theta[b] = th;
      G[(int64_t)b * M * M] = xax[b];
      iters[b] += 1;
    }
  }
}

// target of tuple b: max(abs_target, rel_target max(1, |theta_x|)); the FP32
// storage of x puts a floor of a few 1e-8 |A| on its exact residual
// rnorm of the tuples in `mask` arrives as |r_x|^2 and leaves as |r_x|
__global__ void k32_select(double* __restrict__ rnorm, const int32_t* __restrict__ mask,
                           const double* __restrict__ thx, int B, double abs_target,
                           double rel_target, double drop, int32_t* __restrict__ active,
                           double* __restrict__ tolr, int32_t* __restrict__ nactive) {
  __shared__ int cnt;
  if (threadIdx.x == 0) cnt = 0;
  __syncthreads();
  for (int b = threadIdx.x; b < B; b += blockDim.x) {
    const double target = fmax(abs_target, rel_target * fmax(1.0, fabs(thx[b])));
    double r = rnorm[b];
    if (mask[b]) {
      r = sqrt(fmax(0.0, r));
      rnorm[b] = r;
    }
    const int a = (mask[b] && r > target) ? 1 : 0;
    active[b] = a;
    tolr[b] = fmax(target, drop * r);
    if (a) atomicAdd(&cnt, 1);
  }
  __syncthreads();
  if (threadIdx.x == 0) *nactive = cnt;
}

__global__ void k32_copy_i(const int32_t* s, int32_t* d, int n) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) d[i] = s[i];
}

}  // namespace

void davidson_batch_mixed(mbe_ctx* ctx, BinProblem& bp, double* e_out_host, int32_t* status_host,
                          double* x_out_dev, const GuessPlan* plan) {
  const int B = bp.B;
  // Ms: the subspace cap of the first stage and of a refinement round; M: the
  // allocated size (stride), the cap of the rounds after one that ended with
  // its subspace full and tuples still above their targets
  const int Ms = std::max(4, std::min(32, ctx->opt.max_subspace));
  const int M = mixed_subspace_alloc(ctx->opt.max_subspace);
  // N determinants per tuple; every FP32 Davidson vector is packed (L =
  // sym_len elements), the FP64 exact-point vectors and the FP32 input of the
  // exact sigma are full (Lf = N rounded up to a multiple of 4).  Padding
  // stays zero: no kernel writes it, and every combination of zero elements
  // is zero.
  const int64_t N = bp.ndet, L = sym_len(bp.nstr), Lf = (N + 3) / 4 * 4;
  const int64_t nd = sym_nd(bp.nstr);
  const double shift = ctx->opt.spin_shift;
  DevPool* P = &ctx->pool;
  const int nsm = [&] {
    int v = 0;
    CU_CHECK(cudaDeviceGetAttribute(&v, cudaDevAttrMultiProcessorCount, ctx->device));
    return v;
  }();
  const int ch = chunk_of(L, B, nsm, 4);
  const int nchunks = (int)((L + ch - 1) / ch);
  const int nchunks_f = (int)((Lf + ch - 1) / ch);   // chunks of the full FP64 vectors
  DevBuf<float> V(P, (size_t)B * M * L), AV(P, (size_t)B * M * L), hd(P, (size_t)B * L),
      T(P, (size_t)B * L), X(P, (size_t)B * L), RX(P, (size_t)B * L), F(P, (size_t)B * Lf);
  DevBuf<double> C64(P, (size_t)B * Lf), S64(P, (size_t)B * Lf),
      G(P, (size_t)B * M * M), y(P, (size_t)B * M), yp(P, (size_t)B * M), theta(P, B),
      theta_old(P, B), thx(P, B), rnorm(P, B), tolr(P, B), coef(P, (size_t)B * M), inv(P, B),
      xx(P, B), xax(P, B), partial(P, (size_t)B * (M + 2) * nchunks),
      rpart(P, (size_t)B * std::max(nchunks, nchunks_f));
  DevBuf<float> Z(P, (size_t)B * 1024);
  DevBuf<int32_t> active(P, B), iters(P, B), nact(P, 1), mask(P, B), cnt(P, B);
  SigmaWork sw;
  cudaStream_t st = ctx->stream;
  // zero padding (the vectors' tails are read by the streaming kernels)
  CU_CHECK(cudaMemsetAsync(V.ptr, 0, sizeof(float) * B * M * L, st));
  CU_CHECK(cudaMemsetAsync(AV.ptr, 0, sizeof(float) * B * M * L, st));
  CU_CHECK(cudaMemsetAsync(hd.ptr, 0, sizeof(float) * B * L, st));
  CU_CHECK(cudaMemsetAsync(RX.ptr, 0, sizeof(float) * B * L, st));
  if (Lf != N) {
    CU_CHECK(cudaMemsetAsync(F.ptr, 0, sizeof(float) * B * Lf, st));
    CU_CHECK(cudaMemsetAsync(C64.ptr, 0, sizeof(double) * B * Lf, st));
    CU_CHECK(cudaMemsetAsync(S64.ptr, 0, sizeof(double) * B * Lf, st));
  }
  const int64_t eb = std::min<int64_t>((L + 255) / 256, 1024);
  const int64_t ebf = std::min<int64_t>((Lf + 255) / 256, 1024);
  const dim3 ge((unsigned)eb, B), gef((unsigned)ebf, B), gc(nchunks, B), gcf(nchunks_f, B);
  CU_CHECK(cudaMemsetAsync(cnt.ptr, 0, sizeof(int32_t) * B, st));
  set_attributes<float>(ctx->device);
  const int max_iter = std::max(1, ctx->opt.max_iter);
  int total_it = 0;
  int64_t vecs_tc = 0, vecs_ex = 0;

  // diagonal (FP64 kernel shared with the FP64 mode), kept in FP32
  {
    DevBuf<float> estr(P, (size_t)B * bp.nstr);
    k32_string_energy<<<dim3((unsigned)((bp.nstr + 255) / 256), B), 256, 0, st>>>(
        bp.tab->masks.ptr, bp.nstr, bp.n, bp.heff.ptr, bp.jk.ptr, estr.ptr);
    CU_LAUNCH_CHECK();
    k32_hdiag<<<gef, 256, 0, st>>>(bp.tab->masks.ptr, bp.nstr, L, bp.n, bp.nsig, bp.jk.ptr,
                                  estr.ptr, (float)shift, hd.ptr);
    CU_LAUNCH_CHECK();
  }
  // P-space preconditioner: the lowest-diagonal block of A solved exactly,
  // with Olsen's correction (u = M^-1 x in U32, its dot partials in upart,
  // x.M^-1 r and x.M^-1 x in xpart)
  PspaceWork psp;
  pspace_setup(ctx, bp, hd.ptr, L, shift, pspace_size(bp, ctx->opt.pspace), psp);
  const bool olsen = psp.npp > 0;
  DevBuf<float> U32(P, olsen ? (size_t)B * L : 0), epsb(P, olsen ? (size_t)B : 0);
  DevBuf<double> upart(P, olsen ? (size_t)B * M * nchunks : 0),
      xpart(P, olsen ? (size_t)B * 2 * nchunks : 0);
  if (!olsen) {
    psp.low.reset(P, B);
    k32_lowest<<<B, 256, 0, st>>>(hd.ptr, bp.nstr, L, psp.low.ptr);
    CU_LAUNCH_CHECK();
  }
  k32_guess<<<(B + 255) / 256, 256, 0, st>>>(psp.low.ptr, B, bp.nstr, (int64_t)M * L, V.ptr);
  CU_LAUNCH_CHECK();
  if (plan) {
    // the parent guess writes full vectors (into F), packed into V_0 here
    launch_parent_guess(ctx, *plan, bp.n, bp.nsig, bp.nstr, F.ptr, nullptr, Lf);
    std::vector<int32_t> pm(B, 0);
    for (int b : plan->b) pm[b] = 1;
    DevBuf<int32_t> pmask(P, B);
    CU_CHECK(cudaMemcpyAsync(pmask.ptr, pm.data(), sizeof(int32_t) * B, cudaMemcpyHostToDevice, st));
    k32_pack_start<<<gef, 256, 0, st>>>(F.ptr, Lf, pmask.ptr, bp.nstr, M, L, V.ptr);
    CU_LAUNCH_CHECK();
    CU_CHECK(cudaStreamSynchronize(st));   // pm is read by the copy above
  }
  k_fill_i<<<1, 256, 0, st>>>(active.ptr, B, 1);
  CU_LAUNCH_CHECK();
  CU_CHECK(cudaMemsetAsync(iters.ptr, 0, sizeof(int32_t) * B, st));
  CU_CHECK(cudaMemsetAsync(G.ptr, 0, sizeof(double) * B * M * M, st));
  k_fill_d<<<1, 256, 0, st>>>(tolr.ptr, B, ctx->opt.mixed_stage_tol);
  CU_LAUNCH_CHECK();

  auto dot_comp = [&](const float* Xv, int64_t xb, const float* Yv, int64_t yb, double* out,
                      const int32_t* act) {
    k32_dot_comp<<<gc, RT, 0, st>>>(Xv, xb, Yv, yb, L, nd, ch, nchunks, act, partial.ptr, cnt.ptr,
                                    out);
    CU_LAUNCH_CHECK();
  };
  auto count_active = [&]() {
    int32_t n = 0;
    CU_CHECK(cudaMemcpyAsync(&n, nact.ptr, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CU_CHECK(cudaStreamSynchronize(st));
    if (ctx->opt.verbose) {
      std::vector<double> rn(B), th(B);
      CU_CHECK(cudaMemcpy(rn.data(), rnorm.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost));
      CU_CHECK(cudaMemcpy(th.data(), theta.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost));
      double mx = 0.0;
      for (double r : rn) mx = std::max(mx, r);
      fprintf(stderr, "[mbe mixed] n=%d nsig=%d B=%d it=%d active=%d max|r|=%.3e theta0=%.12f\n",
              bp.n, bp.nsig, B, total_it, n, mx, th[0]);
    }
    return n;
  };
  // the correction T orthogonalised against V[0..m) twice (classical
  // Gram-Schmidt), 1 / |T| left in inv (the next head appends it as V[m]).
  // raw: T is an unpreconditioned residual; dots_ready: T is preconditioned
  // and `partial` holds the first pass's V_i . T partials (both from
  // k_residual).  The P-space block of the correction is replaced first, with
  // Olsen's combination (its exact block would return t = -x) except for the
  // exact-point residual (raw), which takes the plain block.
  auto extend = [&](int m, bool raw, bool dots_ready, double* yprev) {
    if (raw) {
      k32_precondition<<<ge, 256, 0, st>>>(T.ptr, hd.ptr, L, theta.ptr, active.ptr);
      CU_LAUNCH_CHECK();
    }
    const bool ols = olsen && !raw;
    pspace_apply(ctx, bp, psp, T.ptr, hd.ptr, L, theta.ptr, V.ptr, m, M, nchunks, partial.ptr,
                 dots_ready, active.ptr, ols, U32.ptr, X.ptr, upart.ptr, xpart.ptr, y.ptr, yprev,
                 coef.ptr, epsb.ptr);
    if (!dots_ready) {
      if (ols) {
        k32_sub_eps<<<ge, 256, 0, st>>>(T.ptr, U32.ptr, epsb.ptr, L, active.ptr);
        CU_LAUNCH_CHECK();
      }
      k_dots<float><<<gc, RT, (size_t)m * RT * sizeof(float), st>>>(
          V.ptr, (int64_t)M * L, L, T.ptr, L, m, M, L, nd, ch, nchunks, active.ptr, partial.ptr,
          cnt.ptr, coef.ptr);
      CU_LAUNCH_CHECK();
    }
    for (int pass = 0; pass < 2; pass++) {
      const bool fold = ols && dots_ready && pass == 0;   // t = t1 - eps u inside the pass
      k_orth<float><<<gc, RT, pass ? 0 : (size_t)m * RT * sizeof(float), st>>>(
          T.ptr, V.ptr, m, M, L, nd, coef.ptr, active.ptr, pass, ch, nchunks, partial.ptr,
          fold ? U32.ptr : nullptr, epsb.ptr, cnt.ptr, inv.ptr, 1e-24);
      CU_LAUNCH_CHECK();
    }
  };
  // Davidson iterations from a subspace of m_start vectors, the newest one's
  // sigma pending; exact0: V_0 is an exact point (no restart: the stage ends
  // when the subspace is full)
  // returns true when an exact0 stage ended because its subspace (mcap
  // vectors) was full with tuples still iterating
  //
  // An iteration is a head (sigma vector of V[m-1], subspace row, Ritz
  // step, residual and correction, convergence flags), one synchronisation
  // (the number of tuples still iterating), then a tail (restart when the
  // subspace is full, the next vector V[m]).  The tail is issued together
  // with the next head, so that with opt.graphs one CUDA graph per
  // iteration carries both: the host makes one launch and one
  // synchronisation per iteration.  The graph's shape depends only on
  // (exact0, tail present, restart); m changes pointers and loop bounds,
  // which the in-place update of the executable graph takes.
  // (the legacy default stream cannot be captured: plain launches there)
  const bool use_graphs = ctx->opt.graphs != 0 && st != nullptr && st != cudaStreamLegacy;
  GraphRunner gr(st);
  auto tail = [&](int m, bool restart) {
    if (restart) {
      k_restart_coef<<<B, 32, 0, st>>>(y.ptr, yp.ptr, m, M, active.ptr, G.ptr);
      CU_LAUNCH_CHECK();
      k_restart_vec<float><<<ge, 256, 0, st>>>(V.ptr, AV.ptr, m, M, L, y.ptr, yp.ptr, active.ptr);
      CU_LAUNCH_CHECK();
      k_restart_yprev<<<B, 32, 0, st>>>(yp.ptr, M, active.ptr);
      CU_LAUNCH_CHECK();
    }
    // after a restart V changed: the first pass's dots are taken again
    extend(restart ? 2 : m, false, !restart, restart ? nullptr : yp.ptr);
  };
  Converge cv = {tolr.ptr,  std::numeric_limits<double>::infinity(), 0, 1, theta_old.ptr, rnorm.ptr,
                 active.ptr, iters.ptr, nact.ptr};
  // append: V[m-1] = T / |T| first; warm: the last Ritz step was on V[0..m-1)
  auto head = [&](int m, bool append, bool warm, bool first, int rel, bool exact0) {
    sigma_tc(ctx, bp, sw, V.ptr + (int64_t)(m - 1) * L, (int64_t)M * L,
             AV.ptr + (int64_t)(m - 1) * L, (int64_t)M * L, active.ptr, shift, true,
             append ? T.ptr : nullptr, inv.ptr);
    k_subspace<float><<<gc, RT, subspace_smem<float>(m), st>>>(
        V.ptr, AV.ptr, L, nd, m, M, ch, nchunks, active.ptr, partial.ptr, cnt.ptr, exact0 ? 1 : 0,
        RX.ptr, thx.ptr, G.ptr, Z.ptr, warm ? 1 : 0, theta.ptr, y.ptr, nact.ptr);
    CU_LAUNCH_CHECK();
    cv.first = first ? 1 : 0;
    cv.rel = rel;
    // without the P-space the kernel itself leaves the coefficients in coef
    k_residual<float><<<gc, RT, (olsen ? 2 : 1) * m * RT * sizeof(float), st>>>(
        V.ptr, AV.ptr, RX.ptr, exact0 ? 1 : 0, m, M, L, nd, y.ptr, theta.ptr, thx.ptr, hd.ptr,
        X.ptr, T.ptr, ch, nchunks, rpart.ptr, partial.ptr, olsen ? 1 : 0, U32.ptr, upart.ptr,
        xpart.ptr, 1e-4f, cnt.ptr, cv, coef.ptr, nullptr);
    CU_LAUNCH_CHECK();
  };
  // round_start: a refinement round's first correction (the preconditioned
  // exact residual, to be V_1) goes with the round's first head
  auto round_start = [&] {
    k32_copy_i<<<1, 256, 0, st>>>(active.ptr, mask.ptr, B);
    CU_LAUNCH_CHECK();
    CU_CHECK(cudaMemcpyAsync(T.ptr, RX.ptr, sizeof(float) * B * L, cudaMemcpyDeviceToDevice, st));
    k_restart_yprev<<<B, 32, 0, st>>>(yp.ptr, M, active.ptr);
    CU_LAUNCH_CHECK();
    extend(1, true, false, nullptr);
  };
  auto stage = [&](int m_start, int cap, int rel, bool exact0, int nact0, int mcap) -> bool {
    int m = m_start, nact_h = nact0;
    bool pending = false, restart = false;   // the tail still to issue
    int m_tail = 0;
    for (int it = 0; it < cap && total_it < max_iter; it++, total_it++) {
      const bool pend = pending, rs = restart, pro = exact0 && it == 0;
      const int mt = m_tail;
      auto body = [&] {
        if (pro) round_start();
        if (pend) tail(mt, rs);
        head(m, pro || pend, pend && !rs, m_start == 1 && it == 0, rel, exact0);
      };
      // the first iteration of a batch runs as plain launches: it makes the
      // one-time set-up of the sigma path (tables, operand plans, the
      // autotuner's timed launches), which synchronises
      if (use_graphs && total_it >= 1)
        gr.run((exact0 ? 1 : 0) | (pend ? 2 : 0) | (pend && rs ? 4 : 0) | (pro ? 8 : 0), body);
      else
        body();
      pending = false;
      vecs_tc += nact_h;
      nact_h = count_active();
      if (nact_h == 0) return false;
      if (exact0 && m == mcap) return true;
      restart = m == mcap;
      m_tail = m;
      pending = true;
      m = (restart ? 2 : m) + 1;
    }
    return false;
  };
  // the exact-point sigma: fused on the tensor cores where it fits (up to 12
  // orbitals: 64 x 8e/12o 7.31 ms against 24.3), beyond that FP64 from the string
  // links (10e/13o: 3.96 ms against 8.5 for the sliced contraction through D and
  // E, which stays where a row of c is too long for the FP64 kernel)
  const bool exact_fused = sigma_exact_supported(bp.npair, bp.nstr);
  const bool exact_direct = !exact_fused && sigma_direct_supported(bp.n, bp.nsig, bp.nstr);
  // exact point of the tuples in `mask` (n_exact of them): V0 = x/|x|, exact A
  // V0, theta_x, r_x and its norm; G = [[V0.AV0]]
  int n_exact = B;
  auto exact_point = [&]() {
    k32_copy_i<<<1, 256, 0, st>>>(mask.ptr, active.ptr, B);
    CU_LAUNCH_CHECK();
    dot_comp(X.ptr, L, X.ptr, L, xx.ptr, active.ptr);
    k32_exact_prep<<<gef, 256, 0, st>>>(X.ptr, xx.ptr, V.ptr, M, L, F.ptr, C64.ptr, Lf, bp.nstr,
                                        active.ptr);
    CU_LAUNCH_CHECK();
    dot_comp(V.ptr, (int64_t)M * L, V.ptr, (int64_t)M * L, xx.ptr, active.ptr);
    if (exact_fused) {
      sigma_exact(ctx, bp, sw, F.ptr, Lf, S64.ptr, Lf, active.ptr);
      launch_finish_sym_fp64(ctx, bp, S64.ptr, Lf, C64.ptr, Lf, shift, active.ptr);
    } else if (exact_direct) {
      sigma_direct(ctx, bp, C64.ptr, Lf, S64.ptr, Lf, active.ptr, shift, true, false);
    } else {
      sigma_emulated(ctx, bp, sw, C64.ptr, Lf, S64.ptr, Lf, active.ptr, shift, true);
    }
    vecs_ex += n_exact;
    k_dot64<<<gcf, RT, 0, st>>>(C64.ptr, S64.ptr, Lf, ch, nchunks_f, active.ptr, rpart.ptr,
                                cnt.ptr, xax.ptr);
    CU_LAUNCH_CHECK();
    k32_exact_rx<<<gcf, RT, 0, st>>>(C64.ptr, S64.ptr, xax.ptr, xx.ptr, Lf, ch, nchunks_f,
                                     active.ptr, RX.ptr, L, bp.nstr, M, rpart.ptr, cnt.ptr, thx.ptr,
                                     theta.ptr, G.ptr, rnorm.ptr, iters.ptr);
    CU_LAUNCH_CHECK();
  };

  // the exact path's set-up before any of its calls is captured
  if (exact_fused) sigma_exact_prepare(ctx, bp, sw);
  if (exact_direct) sigma_direct_prepare(ctx, bp);
  // stage A
  stage(1, 150, 1, false, B, Ms);
  // refinement rounds
  const double abs_target = ctx->opt.conv_tol_r, rel_target = ctx->opt.mixed_rel_tol;
  k_fill_i<<<1, 256, 0, st>>>(mask.ptr, B, 1);
  CU_LAUNCH_CHECK();
  int round_cap = Ms;
  for (int round = 0; round < 12; round++) {
    // the exact point and the selection of the tuples above their targets
    // (one graph; the sliced contraction stages host data and runs plain)
    auto point = [&] {
      exact_point();
      k32_select<<<1, 256, 0, st>>>(rnorm.ptr, mask.ptr, thx.ptr, B, abs_target, rel_target,
                                    ctx->opt.mixed_round_drop, active.ptr, tolr.ptr, nact.ptr);
      CU_LAUNCH_CHECK();
    };
    if (use_graphs && (exact_fused || exact_direct))
      gr.run(16, point);
    else
      point();
    const int na = n_exact = count_active();
    if (ctx->opt.verbose) {
      double t0 = 0.0, r0 = 0.0;
      CU_CHECK(cudaMemcpy(&t0, thx.ptr, sizeof(double), cudaMemcpyDeviceToHost));
      CU_CHECK(cudaMemcpy(&r0, rnorm.ptr, sizeof(double), cudaMemcpyDeviceToHost));
      fprintf(stderr, "[mbe mixed] exact point %d: %d above target; theta_x0=%.15f |r_x0|=%.3e\n",
              round, na, t0, r0);
    }
    if (na == 0 || total_it >= max_iter) break;
    // the exact residual, preconditioned, is the first correction: issued
    // with the round's first iteration (round_start)
    // a round that filled its subspace before its tuples reached the target
    // (near-degenerate spaces) makes the later rounds use all M vectors
    if (stage(2, 40, 0, true, na, round_cap)) round_cap = M;
  }
  if (sigma_tc_error(ctx, sw)) throw MbeError{MBE_ETIMEOUT, "tensor-core sigma wait timed out"};

  // energies: E = E_core + theta_x - shift <S^2> (S^2 of the exact-point vector, FP64)
  s2_apply(ctx, bp, C64.ptr, Lf, S64.ptr, Lf, nullptr);
  std::vector<double> th(B), ec(B), rn(B), s2(B), nx(B);
  std::vector<int32_t> it_h(B);
  {
    // <S^2> = C64.S64 / C64.C64
    k_dot64<<<gcf, RT, 0, st>>>(C64.ptr, S64.ptr, Lf, ch, nchunks_f, nullptr, rpart.ptr, cnt.ptr,
                                coef.ptr);
    CU_LAUNCH_CHECK();
    k_dot64<<<gcf, RT, 0, st>>>(C64.ptr, C64.ptr, Lf, ch, nchunks_f, nullptr, rpart.ptr, cnt.ptr,
                                xax.ptr);
    CU_LAUNCH_CHECK();
  }
  CU_CHECK(cudaMemcpyAsync(th.data(), thx.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaMemcpyAsync(ec.data(), bp.ecore.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaMemcpyAsync(rn.data(), rnorm.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaMemcpyAsync(s2.data(), coef.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaMemcpyAsync(nx.data(), xax.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaMemcpyAsync(it_h.data(), iters.ptr, sizeof(int32_t) * B, cudaMemcpyDeviceToHost, st));
  if (x_out_dev)
    CU_CHECK(cudaMemcpy2DAsync(x_out_dev, sizeof(double) * N, C64.ptr, sizeof(double) * Lf,
                               sizeof(double) * N, B, cudaMemcpyDeviceToDevice, st));
  CU_CHECK(cudaStreamSynchronize(st));

  for (int b = 0; b < B; b++) {
    const double s2n = nx[b] > 0.0 ? s2[b] / nx[b] : 0.0;
    if (ctx->opt.verbose)
      fprintf(stderr, "[mbe mixed] tuple %d: theta_x=%.15f <S^2>=%.3e |r_x|=%.3e E_core=%.12f\n", b,
              th[b], s2n, rn[b], ec[b]);
    if (e_out_host) e_out_host[b] = ec[b] + th[b] - shift * s2n;
    const bool ok = rn[b] <= 10.0 * std::max(abs_target, rel_target * std::max(1.0, std::fabs(th[b])));
    if (status_host) status_host[b] = ok ? MBE_OK : MBE_ENOCONV;
    ctx->stats.iters_total += it_h[b];
    ctx->stats.iters_max = std::max<int64_t>(ctx->stats.iters_max, it_h[b]);
    ctx->stats.noconv += ok ? 0 : 1;
  }
  const double per = 2.0 * (double)N * bp.npair * bp.npair;
  ctx->stats.graph_launches += gr.launched;
  ctx->stats.graph_builds += gr.instantiated;
  ctx->stats.casci += B;
  ctx->stats.sigma_vectors += vecs_tc + vecs_ex;
  ctx->stats.sigma_flops += (double)(vecs_tc + vecs_ex) * per;
  ctx->stats.dom_flops += (double)vecs_tc * per;
  ctx->stats.fp64_flops +=
      (double)vecs_ex *
      (exact_direct ? direct_flops(bp.n, bp.nsig, bp.nsigb, bp.nstr, bp.nstrb, true) : per);
}
