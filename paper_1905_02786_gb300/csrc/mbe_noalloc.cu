// mbe_sigma_noalloc: the FP64 sigma vector of mbe_sigma with every
// intermediate in one file-scope device array instead of the context's pool.
//
// Callers it serves: code that must not allocate device memory around a
// sigma application -- cudaMalloc and cudaFree can synchronise the whole
// device (stalling every other stream of the process), and a caller running
// under a fixed device-memory budget (the rest of HBM held by another
// allocator) cannot let the pool grow.  This path calls no allocating
// routine; it reads integrals, writes into the caller's device buffers and
// the scratch array below.
//
// Scratch: MBE_NOALLOC_SCRATCH_BYTES per device (the array is part of the
// loaded module, one copy per device).  A problem whose tables, integrals
// and D / E intermediates do not fit is rejected with MBE_EINVAL before
// anything is launched (the limit counts two npair x nstr^2 intermediates of
// a gather / contract / scatter sigma, which this one no longer needs: what
// the call takes stays as documented).  No part of the scratch needs to start
// at zero: every word a kernel reads is written earlier in the same call
// (string tables, effective integrals, one-spin elements).
//
// Calls that overlap on one device race on the single scratch array: a
// caller serialises them (issue them on one stream, or wait for one call to
// finish before issuing the next from another stream or context).
//
// The first call on a device resolves the scratch address with
// cudaGetSymbolAddress and sets the sigma kernel's shared-memory
// attribute; it should come before any stream capture.  The active orbitals
// reach the scratch through a kernel argument (no host-memory copy); with a
// non-NULL e_core the call copies the core energy back and waits for the
// stream.
#include "mbe_internal.cuh"
#include <algorithm>
#include <mutex>

namespace {

static __device__ __align__(256) unsigned char g_sigma_scratch[MBE_NOALLOC_SCRATCH_BYTES];

std::mutex g_scratch_mu;
void* g_scratch_ptr[MBE_MAX_DEVICES] = {nullptr};

unsigned char* scratch_base(int device) {
  if (device < 0 || device >= MBE_MAX_DEVICES) throw MbeError{MBE_EINVAL, "device index out of range"};
  std::lock_guard<std::mutex> lk(g_scratch_mu);
  if (!g_scratch_ptr[device]) {
    void* p = nullptr;
    CU_CHECK(cudaGetSymbolAddress(&p, g_sigma_scratch));
    if (!p) throw MbeError{MBE_ECUDA, "scratch symbol has no device address"};
    g_scratch_ptr[device] = p;
  }
  return (unsigned char*)g_scratch_ptr[device];
}

// byte offsets of the pieces inside the scratch array (256-byte aligned)
struct NoallocLayout {
  size_t masks, ecore, heff, hp, gp, jk, hidx, olnk, hv, wt, c, total;
  size_t limit;   // what MBE_NOALLOC_SCRATCH_BYTES is compared with
};

NoallocLayout noalloc_layout(int n, int nsig, int64_t nstr) {
  const int64_t npair = (int64_t)n * (n + 1) / 2;
  const int64_t ndet = nstr * nstr, nnz = direct_nnz(n, nsig);
  NoallocLayout L;
  size_t o = 0;
  auto take = [&](size_t bytes) {
    const size_t r = o;
    o += (bytes + 255) & ~(size_t)255;
    return r;
  };
  L.masks = take(sizeof(uint32_t) * nstr);
  L.ecore = take(sizeof(double));
  L.heff = take(sizeof(double) * n * n);
  L.hp = take(sizeof(double) * n * n);
  L.gp = take(sizeof(double) * npair * npair);
  L.jk = take(sizeof(double) * 2 * n * n);
  const size_t common = o;
  L.hidx = take(sizeof(uint16_t) * nnz * nstr);
  L.olnk = take(sizeof(uint32_t) * nsig * (n - nsig) * nstr);
  L.hv = take(sizeof(double) * nnz * nstr);
  L.wt = take(sizeof(double) * npair * nstr);
  L.c = take(sizeof(double) * ndet);   // of c, where sigma overwrites it
  L.total = o;
  o = common;
  take(sizeof(int32_t) * n);
  take(sizeof(int32_t) * nstr * npair);
  take(sizeof(int32_t));
  take(sizeof(double) * npair * ndet);
  take(sizeof(double) * npair * ndet);
  L.limit = o;
  return L;
}

}  // namespace

int noalloc_sigma_run(mbe_ctx* ctx, const int* act, int nact, const double* c_dev,
                      double* sigma_dev, int64_t ndet_arg, double* e_core) {
  if (ctx->norb == 0) throw MbeError{MBE_ESTATE, "no integrals loaded"};
  if (nact < 1 || nact > 15 || !act || !c_dev || !sigma_dev)
    throw MbeError{MBE_EINVAL, "bad sigma arguments"};
  if (ctx->two_sz != 0)
    throw MbeError{MBE_EINVAL, "the no-allocation sigma takes closed-shell references only"};
  std::vector<int32_t> a(act, act + nact);
  std::sort(a.begin(), a.end());
  for (int i = 0; i < nact; i++)
    if (a[i] < 0 || a[i] >= ctx->norb || (i && a[i] == a[i - 1]))
      throw MbeError{MBE_EINVAL, "bad active orbital"};
  int nsig = 0;
  for (int o : a) nsig += o < ctx->nocc;
  const int64_t nstr = string_count(nact, nsig);
  if (ndet_arg != nstr * nstr)
    throw MbeError{MBE_EINVAL, "vector length does not match the active space"};
  const NoallocLayout L = noalloc_layout(nact, nsig, nstr);
  if (std::max(L.limit, L.total) > (size_t)MBE_NOALLOC_SCRATCH_BYTES)
    throw MbeError{MBE_EINVAL, "active space too large for the no-allocation scratch"};
  unsigned char* base = scratch_base(ctx->device);
  uint32_t* masks = (uint32_t*)(base + L.masks);
  double* ecore = (double*)(base + L.ecore);
  double* gp = (double*)(base + L.gp);
  double* hv = (double*)(base + L.hv);
  double* wt = (double*)(base + L.wt);
  uint32_t* olnk = (uint32_t*)(base + L.olnk);
  uint16_t* hidx = (uint16_t*)(base + L.hidx);
  ActList al = {};
  for (int i = 0; i < nact; i++) al.v[i] = a[i];
  launch_effints_raw(ctx, nullptr, &al, 1, nact, 2 * nsig, ecore, (double*)(base + L.heff),
                     (double*)(base + L.hp), gp, (double*)(base + L.jk));
  launch_direct_tables(ctx, nact, nsig, (int)nstr, masks, hidx, olnk);
  launch_direct_values(ctx, nact, nsig, (int)nstr, masks, 1, gp, hv, wt);
  const int64_t ndet = nstr * nstr;
  // the sigma kernel's CTAs read rows of c that others would overwrite
  const uintptr_t c0 = (uintptr_t)c_dev, s0 = (uintptr_t)sigma_dev;
  if (c0 < s0 + sizeof(double) * ndet && s0 < c0 + sizeof(double) * ndet) {
    CU_CHECK(cudaMemcpyAsync(base + L.c, c_dev, sizeof(double) * ndet, cudaMemcpyDeviceToDevice,
                             ctx->stream));
    c_dev = (const double*)(base + L.c);
  }
  const DirectSide side = {nsig, (int)nstr, masks, olnk, hidx, hv};
  sigma_direct_raw(ctx, nact, side, side, wt, gp, c_dev, ndet, sigma_dev, ndet, nullptr, 1,
                   ctx->opt.spin_shift, false);
  if (e_core) {
    CU_CHECK(cudaMemcpyAsync(e_core, ecore, sizeof(double), cudaMemcpyDeviceToHost, ctx->stream));
    CU_CHECK(cudaStreamSynchronize(ctx->stream));
  }
  return MBE_OK;
}
