// Batched Davidson iteration (Davidson, J. Comput. Phys. 17, 87 (1975)) for
// the lowest state of every CASCI of one bin in the FP64 and emulated-FP64
// modes (the mixed mode's Davidson is in mbe_davidson32.cu), FP64 throughout.
// The operator is H_active + spin_shift * S^2; a closed shell is restricted to
// the alpha<->beta symmetric vectors, kept packed (half the bytes and half
// the FP64 operations of the full ones).  The start vector is the lowest
// diagonal determinant, symmetrised; the preconditioner t = r / (theta -
// H_II) with |denominator| >= 1e-8; two-pass Gram-Schmidt.  All tuples of a
// batch share the subspace size m; a tuple that has converged is frozen
// (every kernel skips it).
//
// An iteration is six kernels: append (V[m] = T / |T|, expanded to the full
// vector the sigma reads), sigma, subspace row with the Ritz step, residual
// with the preconditioner and the convergence test, two Gram-Schmidt passes
// (mbe_dvec.cuh), issued as one CUDA graph.  Small batches are bound by that
// chain: with a launch for each reduction it was 22 kernels and 330 us per
// iteration on 17 CASCIs of 6e/7o and 8e/7o.
#include "mbe_dvec.cuh"
#include <algorithm>
#include <cmath>
#include <cstdio>
#include <limits>

using namespace dvec;

namespace {

// V[m] = T / |T| of the tuples still iterating, and (closed shell) the full
// vector C from it, one CTA per 32 x 32 tile pair, both halves written
// coalesced.  inv == NULL: C from V[m] as it stands (every tuple).
__global__ void k_append_sym(const double* __restrict__ T, double* __restrict__ V, int64_t vstride,
                             int64_t L, const double* __restrict__ inv, int nstr,
                             const int32_t* __restrict__ active, double* __restrict__ C) {
  const int b = blockIdx.y;
  if (active && !active[b]) return;
  const int nt = (nstr + 31) / 32;
  int t = blockIdx.x, I = 0;
  while (t >= nt - I) {
    t -= nt - I;
    I++;
  }
  const int J = I + t;
  __shared__ double sC[32][33];
  double* Vb = V + (int64_t)b * vstride;
  const double* src = inv ? T + (int64_t)b * L : Vb;
  const double f = inv ? inv[b] : 1.0;
  double* Cb = C + (int64_t)b * nstr * nstr;
  const int tx = threadIdx.x & 31, ty = threadIdx.x >> 5, ny = blockDim.x >> 5;
  for (int i = ty; i < 32; i += ny) {
    const int r = I * 32 + i, k = J * 32 + tx;
    double v = 0.0;
    if (r < nstr && k < nstr && (I < J || r <= k)) {
      const int64_t p = sym_index(r, k, nstr);
      v = src[p] * f;
      if (inv) Vb[p] = v;
      Cb[(int64_t)r * nstr + k] = v;
    }
    sC[i][tx] = v;
  }
  __syncthreads();
  for (int i = ty; i < 32; i += ny) {
    const int r = J * 32 + i, k = I * 32 + tx;
    if (r < nstr && k < nstr && (I < J || r > k)) Cb[(int64_t)r * nstr + k] = sC[tx][i];
  }
}

// open shell: V[m] = T / |T|
__global__ void k_append_full(const double* __restrict__ T, double* __restrict__ V, int64_t vstride,
                              int64_t L, const double* __restrict__ inv,
                              const int32_t* __restrict__ active) {
  const int b = blockIdx.y;
  if (!active[b]) return;
  const double f = inv[b];
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < L;
       k += (int64_t)gridDim.x * blockDim.x)
    V[(int64_t)b * vstride + k] = T[(int64_t)b * L + k] * f;
}

// packed V (stride vstride) from full symmetric vectors C; mask may be NULL
__global__ void k_pack(const double* __restrict__ C, int nstr, const int32_t* __restrict__ mask,
                       double* __restrict__ V, int64_t vstride) {
  const int b = blockIdx.y;
  if (mask && !mask[b]) return;
  const int64_t N = (int64_t)nstr * nstr;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N;
       k += (int64_t)gridDim.x * blockDim.x) {
    const int ia = (int)(k / nstr), ib = (int)(k - (int64_t)ia * nstr);
    if (ia <= ib) V[(int64_t)b * vstride + sym_index(ia, ib, nstr)] = C[(int64_t)b * N + k];
  }
}

// full X (stride N) from open-shell vectors of stride L
__global__ void k_unpad(const double* __restrict__ V, int64_t L, int64_t N, double* __restrict__ X) {
  const int b = blockIdx.y;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < N;
       k += (int64_t)gridDim.x * blockDim.x)
    X[(int64_t)b * N + k] = V[(int64_t)b * L + k];
}

// start vector: lowest diagonal determinant (Ia, Ib), symmetrised for a
// closed shell (packed vectors); for an open shell (nstrb beta strings) the
// determinant itself.  V_0 is zero on entry.
__global__ void k_guess(const double* __restrict__ hd, int nstr, int nstrb, int closed, int64_t L,
                        int64_t vstride, double* __restrict__ V) {
  const int b = blockIdx.x;
  const int64_t N = (int64_t)nstr * nstrb;
  __shared__ double sv[256];
  __shared__ int64_t si[256];
  double best = 1e300;
  int64_t bi = 0;
  for (int64_t k = threadIdx.x; k < N; k += blockDim.x) {
    const int ia = (int)(k / nstrb), ib = (int)(k - (int64_t)ia * nstrb);
    if (closed && ia > ib) continue;   // the mirror element has the same value, a larger k
    const double v = hd[(int64_t)b * L + (closed ? sym_index(ia, ib, nstr) : k)];
    if (v < best) { best = v; bi = k; }
  }
  sv[threadIdx.x] = best;
  si[threadIdx.x] = bi;
  __syncthreads();
  for (int s = blockDim.x / 2; s; s >>= 1) {
    if (threadIdx.x < s) {
      const double o = sv[threadIdx.x + s];
      const int64_t oi = si[threadIdx.x + s];
      if (o < sv[threadIdx.x] || (o == sv[threadIdx.x] && oi < si[threadIdx.x])) {
        sv[threadIdx.x] = o;
        si[threadIdx.x] = oi;
      }
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    const int64_t i0 = si[0];
    const int ia = (int)(i0 / nstrb), ib = (int)(i0 % nstrb);
    double* Vb = V + (int64_t)b * vstride;
    // (|a b> + |b a>) / sqrt(2): its packed element carries both halves
    if (closed) Vb[sym_index(ia, ib, nstr)] = ia == ib ? 1.0 : sqrt(0.5);
    else Vb[i0] = 1.0;
  }
}

}  // namespace

// Davidson for one batch of tuples: one stage with FP64 (or emulated-FP64)
// sigma vectors to conv_tol_r / conv_tol_e.
void davidson_batch(mbe_ctx* ctx, BinProblem& bp, double* e_out_host, int32_t* status_host,
                    double* s2_host, double* x_out_dev, const GuessPlan* plan) {
  const int B = bp.B;
  const int M = std::max(4, std::min(32, ctx->opt.max_subspace));
  const int64_t N = bp.ndet;
  const bool closed = bp.closed();
  const int64_t L = closed ? sym_len(bp.nstr) : (N + 3) & ~(int64_t)3;
  const int64_t nd = closed ? sym_nd(bp.nstr) : L;
  const int64_t vs = (int64_t)M * L;   // stride of a tuple's subspace
  const double shift = ctx->opt.spin_shift;
  DevPool* P = &ctx->pool;
  cudaStream_t st = ctx->stream;
  // sigma vectors: FP64 CUDA cores (MBE_FP64) or the FP64-grade sliced
  // tensor-core contraction (MBE_EMULATED_FP64, and the mixed mode's
  // fallback for spaces the fused tensor-core kernel does not cover)
  const bool emulated = ctx->opt.precision != MBE_FP64 && ozaki_supported(bp.npair);
  int nsm = 0;
  CU_CHECK(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, ctx->device));
  const int ch = chunk_of(L, B, nsm, 4);
  const int nchunks = (int)((L + ch - 1) / ch), nchunks_f = (int)((N + ch - 1) / ch);
  DevBuf<double> V(P, (size_t)B * vs), AV(P, (size_t)B * vs), hd(P, (size_t)B * L),
      T(P, (size_t)B * L), X(P, (size_t)B * L), C(P, (size_t)B * N),
      SF(P, emulated && closed ? (size_t)B * N : 0), G(P, (size_t)B * M * M), y(P, (size_t)B * M),
      yp(P, (size_t)B * M), theta(P, B), theta_old(P, B), rnorm(P, B), tolr(P, B),
      coef(P, (size_t)B * M), inv(P, B), xs2(P, B), xx(P, B),
      partial(P, (size_t)B * (M + 2) * nchunks),
      rpart(P, (size_t)B * std::max(nchunks, nchunks_f));
  DevBuf<float> Z(P, (size_t)B * 1024);
  DevBuf<int32_t> active(P, B), iters(P, B), nact(P, 1), cnt(P, B);
  SigmaWork sw;
  set_attributes<double>(ctx->device);

  // zero padding: no kernel writes it, the streaming kernels read it
  CU_CHECK(cudaMemsetAsync(V.ptr, 0, sizeof(double) * B * vs, st));
  CU_CHECK(cudaMemsetAsync(AV.ptr, 0, sizeof(double) * B * vs, st));
  CU_CHECK(cudaMemsetAsync(hd.ptr, 0, sizeof(double) * B * L, st));
  CU_CHECK(cudaMemsetAsync(iters.ptr, 0, sizeof(int32_t) * B, st));
  CU_CHECK(cudaMemsetAsync(cnt.ptr, 0, sizeof(int32_t) * B, st));
  CU_CHECK(cudaMemsetAsync(G.ptr, 0, sizeof(double) * B * M * M, st));
  launch_hdiag(ctx, bp, shift, hd.ptr, L, closed);
  k_guess<<<B, 256, 0, st>>>(hd.ptr, bp.nstr, bp.nstrb, closed ? 1 : 0, L, vs, V.ptr);
  CU_LAUNCH_CHECK();
  const dim3 gN((unsigned)std::min<int64_t>((N + 255) / 256, 1024), B);
  const dim3 gL((unsigned)std::min<int64_t>((L + 255) / 256, 1024), B);
  if (plan) {
    // the parent guess writes full vectors, packed into V_0 here
    launch_parent_guess(ctx, *plan, bp.n, bp.nsig, bp.nstr, nullptr, C.ptr, N);
    std::vector<int32_t> pm(B, 0);
    for (int b : plan->b) pm[b] = 1;
    DevBuf<int32_t> pmask(P, B);
    CU_CHECK(cudaMemcpyAsync(pmask.ptr, pm.data(), sizeof(int32_t) * B, cudaMemcpyHostToDevice, st));
    k_pack<<<gN, 256, 0, st>>>(C.ptr, bp.nstr, pmask.ptr, V.ptr, vs);
    CU_LAUNCH_CHECK();
    CU_CHECK(cudaStreamSynchronize(st));   // pm is read by the copy above
  }
  k_fill_i<<<1, 256, 0, st>>>(active.ptr, B, 1);
  CU_LAUNCH_CHECK();
  k_fill_d<<<1, 256, 0, st>>>(tolr.ptr, B, ctx->opt.conv_tol_r);
  CU_LAUNCH_CHECK();
  if (!emulated) sigma_direct_prepare(ctx, bp);

  const int nt = (bp.nstr + 31) / 32;
  const dim3 gt((unsigned)(nt * (nt + 1) / 2), B), gc(nchunks, B);
  const int max_iter = std::max(1, ctx->opt.max_iter);
  int64_t vecs = 0;
  Converge cv = {tolr.ptr, ctx->opt.conv_tol_e, 0,          1,        theta_old.ptr,
                 rnorm.ptr, active.ptr,         iters.ptr, nact.ptr};

  // V[m-1] (from T unless it is the start vector) and its sigma vector, the
  // subspace row and Ritz step, the residual and its correction in T
  auto head = [&](int m, bool append, bool warm, bool first) {
    double* Vm = V.ptr + (int64_t)(m - 1) * L;
    double* AVm = AV.ptr + (int64_t)(m - 1) * L;
    if (closed) {
      k_append_sym<<<gt, 256, 0, st>>>(T.ptr, Vm, vs, L, append ? inv.ptr : nullptr, bp.nstr,
                                       append ? active.ptr : nullptr, C.ptr);
      CU_LAUNCH_CHECK();
    } else if (append) {
      k_append_full<<<gL, 256, 0, st>>>(T.ptr, Vm, vs, L, inv.ptr, active.ptr);
      CU_LAUNCH_CHECK();
    }
    if (!emulated) {
      sigma_direct(ctx, bp, closed ? C.ptr : Vm, closed ? N : vs, AVm, vs, active.ptr, shift, closed);
    } else if (closed) {
      sigma_emulated(ctx, bp, sw, C.ptr, N, SF.ptr, N, active.ptr, shift, true);
      k_pack<<<gN, 256, 0, st>>>(SF.ptr, bp.nstr, active.ptr, AVm, vs);
      CU_LAUNCH_CHECK();
    } else {
      sigma_emulated(ctx, bp, sw, Vm, vs, AVm, vs, active.ptr, shift, false);
    }
    k_subspace<double><<<gc, RT, subspace_smem<double>(m), st>>>(
        V.ptr, AV.ptr, L, nd, m, M, ch, nchunks, active.ptr, partial.ptr, cnt.ptr, 0, nullptr,
        nullptr, G.ptr, Z.ptr, warm ? 1 : 0, theta.ptr, y.ptr, nact.ptr);
    CU_LAUNCH_CHECK();
    cv.first = first ? 1 : 0;
    // (a restart follows a full subspace and needs the previous y)
    k_residual<double><<<gc, RT, (size_t)m * RT * sizeof(double), st>>>(
        V.ptr, AV.ptr, nullptr, 0, m, M, L, nd, y.ptr, theta.ptr, nullptr, hd.ptr, X.ptr, T.ptr, ch,
        nchunks, rpart.ptr, partial.ptr, 0, nullptr, nullptr, nullptr, 1e-8, cnt.ptr, cv, coef.ptr,
        m == M ? nullptr : yp.ptr);
    CU_LAUNCH_CHECK();
  };
  // orthogonalise the correction T against V[0..m); after a full subspace
  // restart with {x, x_prev} first
  auto tail = [&](int m, bool restart) {
    if (restart) {
      k_restart_coef<<<B, 32, 0, st>>>(y.ptr, yp.ptr, m, M, active.ptr, G.ptr);
      CU_LAUNCH_CHECK();
      k_restart_vec<double><<<gL, 256, 0, st>>>(V.ptr, AV.ptr, m, M, L, y.ptr, yp.ptr, active.ptr);
      CU_LAUNCH_CHECK();
      k_restart_yprev<<<B, 32, 0, st>>>(yp.ptr, M, active.ptr);
      CU_LAUNCH_CHECK();
      m = 2;
      // V changed: the first pass's dots are taken again
      k_dots<double><<<gc, RT, (size_t)m * RT * sizeof(double), st>>>(
          V.ptr, vs, L, T.ptr, L, m, M, L, nd, ch, nchunks, active.ptr, partial.ptr, cnt.ptr,
          coef.ptr);
      CU_LAUNCH_CHECK();
    }
    for (int pass = 0; pass < 2; pass++) {
      k_orth<double><<<gc, RT, pass ? 0 : (size_t)m * RT * sizeof(double), st>>>(
          T.ptr, V.ptr, m, M, L, nd, coef.ptr, active.ptr, pass, ch, nchunks, partial.ptr, nullptr,
          nullptr, cnt.ptr, inv.ptr, 1e-28);
      CU_LAUNCH_CHECK();
    }
  };
  // Each iteration's tail is issued together with the next one's head, as one
  // CUDA graph (opt.graphs; the emulated sigma stages host data and runs
  // plain, as does the legacy default stream, which cannot be captured); one
  // synchronisation per iteration, for the number of tuples still iterating.
  const bool use_graphs =
      ctx->opt.graphs != 0 && !emulated && st != nullptr && st != cudaStreamLegacy;
  GraphRunner gr(st);
  int m = 1, m_tail = 0, nact_h = B;
  bool restart = false;
  for (int it = 0; it < max_iter; it++) {
    const int mt = m_tail, mc = m;
    const bool rs = restart, pend = it > 0;
    auto body = [&] {
      if (pend) tail(mt, rs);
      head(mc, pend, pend && !rs, it == 0);
    };
    if (use_graphs && it >= 1) gr.run(rs ? 1 : 0, body);
    else body();
    vecs += nact_h;
    CU_CHECK(cudaMemcpyAsync(&nact_h, nact.ptr, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
    CU_CHECK(cudaStreamSynchronize(st));
    if (ctx->opt.verbose) {
      std::vector<double> rn(B), th(B);
      CU_CHECK(cudaMemcpy(rn.data(), rnorm.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost));
      CU_CHECK(cudaMemcpy(th.data(), theta.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost));
      double mx = 0.0;
      for (double r : rn) mx = std::max(mx, r);
      fprintf(stderr, "[mbe davidson] n=%d nsig=%d B=%d it=%d active=%d max|r|=%.3e theta0=%.12f\n",
              bp.n, bp.nsig, B, it, nact_h, mx, th[0]);
    }
    if (nact_h == 0) break;
    restart = m == M;
    m_tail = m;
    m = (restart ? 2 : m) + 1;
  }
  if (emulated && sigma_tc_error(ctx, sw))
    throw MbeError{MBE_ETIMEOUT, "tensor-core contraction wait timed out"};

  // status and energies: eps = E_core + theta - shift <x|S^2|x> / <x|x>
  std::vector<int32_t> it_h(B);
  std::vector<double> rn_h(B);
  CU_CHECK(cudaMemcpyAsync(it_h.data(), iters.ptr, sizeof(int32_t) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaMemcpyAsync(rn_h.data(), rnorm.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  double* XF = x_out_dev ? x_out_dev : C.ptr;   // the converged vectors, full
  if (closed) {
    k_append_sym<<<gt, 256, 0, st>>>(nullptr, X.ptr, L, L, nullptr, bp.nstr, nullptr, XF);
    CU_LAUNCH_CHECK();
  } else {
    k_unpad<<<gN, 256, 0, st>>>(X.ptr, L, N, XF);
    CU_LAUNCH_CHECK();
  }
  double* S2X = V.ptr;   // the subspace is not needed any more (M >= 4 vectors of N / 2)
  s2_apply(ctx, bp, XF, N, S2X, N, nullptr);
  const dim3 gcf(nchunks_f, B);
  k_dot64<<<gcf, RT, 0, st>>>(XF, S2X, N, ch, nchunks_f, nullptr, rpart.ptr, cnt.ptr, xs2.ptr);
  CU_LAUNCH_CHECK();
  k_dot64<<<gcf, RT, 0, st>>>(XF, XF, N, ch, nchunks_f, nullptr, rpart.ptr, cnt.ptr, xx.ptr);
  CU_LAUNCH_CHECK();
  std::vector<double> th(B), s2(B), ec(B), nx(B);
  CU_CHECK(cudaMemcpyAsync(th.data(), theta.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaMemcpyAsync(s2.data(), xs2.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaMemcpyAsync(nx.data(), xx.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaMemcpyAsync(ec.data(), bp.ecore.ptr, sizeof(double) * B, cudaMemcpyDeviceToHost, st));
  CU_CHECK(cudaStreamSynchronize(st));
  const double rtol = ctx->opt.conv_tol_r;
  for (int b = 0; b < B; b++) {
    const double s2n = nx[b] > 0.0 ? s2[b] / nx[b] : 0.0;
    if (e_out_host) e_out_host[b] = ec[b] + th[b] - shift * s2n;
    if (s2_host) s2_host[b] = s2n;
    bool ok = rn_h[b] <= rtol * 10.0 || N == 1;
    if (status_host) status_host[b] = ok ? MBE_OK : MBE_ENOCONV;
    ctx->stats.iters_total += it_h[b];
    ctx->stats.iters_max = std::max<int64_t>(ctx->stats.iters_max, it_h[b]);
    ctx->stats.noconv += ok ? 0 : 1;
  }
  const double per = 2.0 * (double)N * bp.npair * bp.npair;
  ctx->stats.graph_launches += gr.launched;
  ctx->stats.graph_builds += gr.instantiated;
  ctx->stats.casci += B;
  ctx->stats.sigma_vectors += vecs;
  ctx->stats.sigma_flops += (double)vecs * per;
  // exact sigma vectors, by what their route multiplies
  ctx->stats.fp64_flops +=
      (double)vecs *
      (emulated ? per : direct_flops(bp.n, bp.nsig, bp.nsigb, bp.nstr, bp.nstrb, closed));
}
