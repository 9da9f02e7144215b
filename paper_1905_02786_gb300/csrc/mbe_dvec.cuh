// Streaming kernels of the Davidson iteration, shared by the FP64 solver
// (T = double) and the mixed one (T = float).
//
// Vectors.  A closed-shell vector is alpha-beta symmetric and kept packed
// (sym_index): nd = sym_nd diagonal elements, then the strictly upper
// triangle, L = sym_len in all; its dot products weigh the elements from nd
// on by 2.  An open-shell vector is the full one (nd = L, no weights).  L is
// a multiple of 4, the padding zero and every vector on a 16-byte boundary,
// so the kernels move 16 bytes per load.
//
// Reductions.  A CTA takes one chunk of `ch` elements; the partial sums of
// the chunks are combined in a fixed order by the last CTA of a tuple to
// finish (a counter per tuple, which it resets), which also does the small
// work that needs the sums -- the subspace matrix and its Ritz step, the
// convergence test, the norm -- so that none of it is a launch of its own:
// an iteration of a small batch is bound by its chain of dependent launches.
#pragma once
#include "mbe_internal.cuh"
#include "mbe_ritz.cuh"

namespace dvec {

constexpr int RT = RITZ_THREADS;   // threads of the reduction kernels

template <typename T>
struct Pack;
template <>
struct Pack<float> {
  using type = float4;
  static constexpr int E = 4;
  static __device__ __forceinline__ void get(const float* p, int64_t q, float (&x)[4]) {
    const float4 v = reinterpret_cast<const float4*>(p)[q];
    x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w;
  }
  static __device__ __forceinline__ void put(float* p, int64_t q, const float (&x)[4]) {
    reinterpret_cast<float4*>(p)[q] = make_float4(x[0], x[1], x[2], x[3]);
  }
};
template <>
struct Pack<double> {
  using type = double2;
  static constexpr int E = 2;
  static __device__ __forceinline__ void get(const double* p, int64_t q, double (&x)[2]) {
    const double2 v = reinterpret_cast<const double2*>(p)[q];
    x[0] = v.x; x[1] = v.y;
  }
  static __device__ __forceinline__ void put(double* p, int64_t q, const double (&x)[2]) {
    reinterpret_cast<double2*>(p)[q] = make_double2(x[0], x[1]);
  }
};

template <typename T, int E>
__device__ __forceinline__ T dotE(const T (&a)[E], const T (&b)[E], T acc) {
#pragma unroll
  for (int e = 0; e < E; e++) acc = fma(a[e], b[e], acc);
  return acc;
}

__device__ __forceinline__ double block_sum(double v, double* red) {
  for (int off = 16; off; off >>= 1) v += __shfl_down_sync(0xffffffffu, v, off);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  double s = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) s += red[w];
  return s;
}

// true in the last of n CTAs to arrive at *cnt (which it resets to 0); what
// the others wrote before is visible to it (read it with __ldcg)
__device__ __forceinline__ bool last_cta(int32_t* cnt, int n) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(cnt, 1) == n - 1;
  __syncthreads();
  if (!s_last) return false;
  __threadfence();
  if (threadIdx.x == 0) *cnt = 0;
  return true;
}

// sum of a row of chunk partials by one warp, in every lane
__device__ __forceinline__ double row_sum(const double* __restrict__ p, int nchunks) {
  double s = 0.0;
  for (int c = threadIdx.x & 31; c < nchunks; c += 32) s += __ldcg(p + c);
  return ritz_warp_sum(s);
}

// block sums of the per-thread accumulators sD[i][thread], i < rows, in FP64:
// row i to part[i * nchunks] (a warp per row: 13 FP64 additions where a
// shuffle tree in every warp takes 40, and FP64 is what these tails wait for)
template <typename T>
__device__ __forceinline__ void sums_to_partial(const T* sD, int rows, double* __restrict__ part,
                                                int nchunks) {
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  for (int i = warp; i < rows; i += RT / 32) {
    double v = 0.0;
#pragma unroll
    for (int j = 0; j < RT / 32; j++) v += (double)sD[i * RT + lane + 32 * j];
    v = ritz_warp_sum(v);
    if (lane == 0) part[(int64_t)i * nchunks] = v;
  }
}

// per-thread dots of the m vectors X_i with w Y over one chunk, into sD
template <typename T>
__device__ __forceinline__ void chunk_dots(const T* __restrict__ x, int64_t xv,
                                           const T* __restrict__ y, int m, int64_t q0, int64_t q1,
                                           int64_t ndq, T* sD) {
  constexpr int E = Pack<T>::E, GR = sizeof(T) == 4 ? 16 : 8;
  for (int i0 = 0; i0 < m; i0 += GR) {
    const int ni = min(GR, m - i0);
    T acc[GR];
#pragma unroll
    for (int i = 0; i < GR; i++) acc[i] = T(0);
    for (int64_t q = q0 + threadIdx.x; q < q1; q += RT) {
      T yv[E];
      Pack<T>::get(y, q, yv);
      const T w = q < ndq ? T(1) : T(2);   // exact scaling
#pragma unroll
      for (int e = 0; e < E; e++) yv[e] *= w;
#pragma unroll
      for (int i = 0; i < GR; i++)
        if (i < ni) {
          T xi[E];
          Pack<T>::get(x + (int64_t)(i0 + i) * xv, q, xi);
          acc[i] = dotE(xi, yv, acc[i]);
        }
    }
#pragma unroll
    for (int i = 0; i < GR; i++)
      if (i < ni) sD[(i0 + i) * RT + threadIdx.x] = acc[i];
  }
}

// out[b M + i] = X[b][i] . Y[b], i < m
template <typename T>
__global__ void __launch_bounds__(RT)
k_dots(const T* __restrict__ X, int64_t xb, int64_t xv, const T* __restrict__ Y, int64_t yb, int m,
       int M, int64_t L, int64_t nd, int ch, int nchunks, const int32_t* __restrict__ active,
       double* __restrict__ partial, int32_t* __restrict__ cnt, double* __restrict__ out) {
  const int b = blockIdx.y;
  if (active && !active[b]) return;
  extern __shared__ __align__(16) unsigned char dsm[];
  T* sD = reinterpret_cast<T*>(dsm);
  constexpr int E = Pack<T>::E;
  const int64_t q0 = (int64_t)blockIdx.x * (ch / E), q1 = min(L / E, q0 + ch / E);
  chunk_dots<T>(X + (int64_t)b * xb, xv, Y + (int64_t)b * yb, m, q0, q1, nd / E, sD);
  double* pb = partial + (int64_t)b * M * nchunks;
  sums_to_partial<T>(sD, m, pb + blockIdx.x, nchunks);
  if (!last_cta(cnt + b, nchunks)) return;
  for (int i = threadIdx.x >> 5; i < m; i += RT / 32) {
    const double s = row_sum(pb + (int64_t)i * nchunks, nchunks);
    if ((threadIdx.x & 31) == 0) out[(int64_t)b * M + i] = s;
  }
}

// The subspace step of a new vector V[m-1] with A V[m-1] in AV[m-1]: row m-1
// of G from the dots V_i . A V_{m-1}, then the Ritz step (theta, y).
// exact0 (T = float): V_0 carries an exact A V_0; its coupling is taken as
// theta_x (x.t) + r_x.t from the exact theta_x and residual RX, with x.t an
// error-free dot (two-product + compensated sum), no reduced-precision sigma.
// Z (32 x 32 per tuple): the Ritz step's eigenvectors, kept for the next
// call; warm: the last call was on the leading m - 1 vectors.
// Also clears *nact, the count of tuples still iterating (k_residual adds).
template <typename T>
__global__ void __launch_bounds__(RT)
k_subspace(const T* __restrict__ V, const T* __restrict__ AV, int64_t L, int64_t nd, int m, int M,
           int ch, int nchunks, const int32_t* __restrict__ active, double* __restrict__ partial,
           int32_t* __restrict__ cnt, int exact0, const T* __restrict__ RX,
           const double* __restrict__ thx, double* __restrict__ G, float* __restrict__ Z, int warm,
           double* __restrict__ theta, double* __restrict__ y, int32_t* __restrict__ nact) {
  const int b = blockIdx.y;
  if (blockIdx.x == 0 && b == 0 && threadIdx.x == 0) *nact = 0;
  if (!active[b]) return;
  extern __shared__ __align__(16) unsigned char dsm[];
  __shared__ double red[32], sdot[34];
  T* sD = reinterpret_cast<T*>(dsm);
  constexpr int E = Pack<T>::E;
  const int64_t q0 = (int64_t)blockIdx.x * (ch / E), q1 = min(L / E, q0 + ch / E);
  const T* Vb = V + (int64_t)b * M * L;
  chunk_dots<T>(Vb, L, AV + ((int64_t)b * M + m - 1) * L, m, q0, q1, nd / E, sD);
  double* pb = partial + (int64_t)b * (M + 2) * nchunks;
  const bool ex = exact0 && m > 1;
  if constexpr (sizeof(T) == 4) {
    if (ex) {
      // (s, lo): s + lo carries the running sum to ~2^-48 relative; every
      // product is split exactly (p + e = a b, fma) and every addition of p
      // to s exactly (TwoSum: s + p = t + err)
      const T* tv = Vb + (int64_t)(m - 1) * L;
      const T* rx = RX + (int64_t)b * L;
      float s = 0.f, lo = 0.f, r = 0.f;
      for (int64_t q = q0 + threadIdx.x; q < q1; q += RT) {
        float x[E], t[E], rr[E];
        Pack<T>::get(Vb, q, x);
        Pack<T>::get(tv, q, t);
        Pack<T>::get(rx, q, rr);
        const float w = q < nd / E ? 1.f : 2.f;
#pragma unroll
        for (int e = 0; e < E; e++) {
          const float a = x[e] * w;   // exact
          const float p = a * t[e];
          const float pe = fmaf(a, t[e], -p);
          const float u = s + p;
          const float bp = u - s;
          const float err = (s - (u - bp)) + (p - bp);
          s = u;
          lo += err + pe;
          r = fmaf(rr[e] * w, t[e], r);
        }
      }
      sD[m * RT + threadIdx.x] = r;
      const double tot = block_sum((double)s + (double)lo, red);
      if (threadIdx.x == 0) pb[(int64_t)(M + 1) * nchunks + blockIdx.x] = tot;
    }
  }
  sums_to_partial<T>(sD, m, pb + blockIdx.x, nchunks);
  if (ex) sums_to_partial<T>(sD + m * RT, 1, pb + (int64_t)M * nchunks + blockIdx.x, nchunks);
  if (!last_cta(cnt + b, nchunks)) return;
  for (int i = threadIdx.x >> 5; i < m + (ex ? 2 : 0); i += RT / 32) {
    const int row = i < m ? i : M + i - m;
    const double s = row_sum(pb + (int64_t)row * nchunks, nchunks);
    if ((threadIdx.x & 31) == 0) sdot[i] = s;
  }
  __syncthreads();
  double* Gb = G + (int64_t)b * M * M;
  if (threadIdx.x < m) {
    const int i = threadIdx.x;
    const double v = ex && i == 0 ? thx[b] * sdot[m + 1] + sdot[m] : sdot[i];
    Gb[(int64_t)(m - 1) * M + i] = v;
    Gb[(int64_t)i * M + m - 1] = v;
  }
  __syncthreads();
  ritz_lowest(Gb, m, M, *reinterpret_cast<RitzShared*>(dsm), Z + (int64_t)b * 1024, warm != 0,
              theta + b, y + (int64_t)b * M);
}
// dynamic shared memory of k_subspace
template <typename T>
inline size_t subspace_smem(int m) {
  const size_t d = (size_t)(m + 1) * RT * sizeof(T);
  return d > sizeof(RitzShared) ? d : sizeof(RitzShared);
}

// what the convergence test of an iteration needs
struct Converge {
  const double* tol_r;   // per tuple; relative to max(1, |theta|) with rel
  double tol_e;          // |theta - theta_old| (infinity: not tested)
  int rel, first;        // first: no test (nothing to compare with)
  double *theta_old, *rnorm;
  int32_t *active, *iters, *nact;
};

// The residual step with the preconditioner and the first orthogonalisation
// pass's dot products folded in:
//   x = V y,  r = AV y - theta x, or with exact0 (T = float)
//   r = y_0 (r_x + (theta_x - theta) V_0) + sum_{i>=1} y_i (AV_i - theta V_i),
//   |r|^2 partials, t = r / (theta - H_II) with |denominator| >= dmin,
//   partials of V_i . t, i < m
// and with olsen (T = float) u = x / (theta - H_II), its dots V_i . u and the
// sums x.t, x.u.  The second read of V_i[k] follows the first within the same
// thread and is served by the caches, so V streams from HBM once.  The
// per-thread dot accumulators live in shared memory (registers stay few and
// occupancy high: the FP32 kernel is bound by HBM).
// The last CTA of a tuple tests its convergence; without olsen it also
// leaves the coefficients V_i . t in coef and (yp != NULL) y in yp.
template <typename T>
__global__ void __launch_bounds__(RT)
k_residual(const T* __restrict__ V, const T* __restrict__ AV, const T* __restrict__ RX, int exact0,
           int m, int M, int64_t L, int64_t nd, const double* __restrict__ y,
           const double* __restrict__ theta, const double* __restrict__ thx,
           const T* __restrict__ hd, T* __restrict__ X, T* __restrict__ Tv, int ch, int nchunks,
           double* __restrict__ rpart, double* __restrict__ dpart, int olsen, T* __restrict__ Uo,
           double* __restrict__ upart, double* __restrict__ xpart, T dmin,
           int32_t* __restrict__ cnt, Converge cv, double* __restrict__ coef,
           double* __restrict__ yp) {
  const int b = blockIdx.y;
  if (!cv.active[b]) return;
  constexpr int E = Pack<T>::E;
  extern __shared__ __align__(16) unsigned char dsm[];
  T* sD = reinterpret_cast<T*>(dsm);            // V_i . t
  T* sU = sD + (int64_t)m * RT;                 // V_i . u (olsen)
  __shared__ T sy[32];
  __shared__ double red[32];
  const int tid = threadIdx.x;
  if (tid < m) sy[tid] = (T)y[(int64_t)b * M + tid];
  for (int i = 0; i < (olsen ? 2 * m : m); i++) sD[i * RT + tid] = T(0);
  __syncthreads();
  const T th = (T)theta[b];
  const T dth = exact0 ? (T)(thx[b] - theta[b]) : T(0);
  const int i0 = exact0 ? 1 : 0;
  const int64_t q0 = (int64_t)blockIdx.x * (ch / E), q1 = min(L / E, q0 + ch / E), ndq = nd / E;
  const T* Vb = V + (int64_t)b * M * L;
  const T* AVb = AV + (int64_t)b * M * L;
  T acc = T(0), xt = T(0), xu = T(0);
  for (int64_t q = q0 + tid; q < q1; q += RT) {
    T xs[E], rs[E];
#pragma unroll
    for (int e = 0; e < E; e++) xs[e] = rs[e] = T(0);
    if (exact0) {
      T v[E], r0[E];
      Pack<T>::get(Vb, q, v);
      Pack<T>::get(RX + (int64_t)b * L, q, r0);
#pragma unroll
      for (int e = 0; e < E; e++) {
        xs[e] = sy[0] * v[e];
        rs[e] = sy[0] * (r0[e] + dth * v[e]);
      }
    }
#pragma unroll 4
    for (int i = i0; i < m; i++) {
      T v[E], a[E];
      Pack<T>::get(Vb + (int64_t)i * L, q, v);
      Pack<T>::get(AVb + (int64_t)i * L, q, a);
#pragma unroll
      for (int e = 0; e < E; e++) {
        xs[e] = fma(sy[i], v[e], xs[e]);
        // FP64: two FMAs per element (the FP64 rate is what bounds it)
        if constexpr (sizeof(T) == 4) rs[e] = fma(sy[i], a[e] - th * v[e], rs[e]);
        else rs[e] = fma(sy[i], a[e], rs[e]);
      }
    }
    if constexpr (sizeof(T) == 8) {
#pragma unroll
      for (int e = 0; e < E; e++) rs[e] = rs[e] - th * xs[e];
    }
    Pack<T>::put(X + (int64_t)b * L, q, xs);
    T hv[E], ts[E], us[E], tw[E];
    Pack<T>::get(hd + (int64_t)b * L, q, hv);
    const T w = q < ndq ? T(1) : T(2);          // weight of the packed elements
#pragma unroll
    for (int e = 0; e < E; e++) {
      acc = fma(w * rs[e], rs[e], acc);
      T d = th - hv[e];
      if (fabs(d) < dmin) d = d < T(0) ? -dmin : dmin;
      ts[e] = rs[e] / d;
      tw[e] = w * ts[e];
      if constexpr (sizeof(T) == 4) us[e] = xs[e] / d;
    }
    Pack<T>::put(Tv + (int64_t)b * L, q, ts);
    if constexpr (sizeof(T) == 4) {
      if (olsen) {
        T uw[E];
        Pack<T>::put(Uo + (int64_t)b * L, q, us);
#pragma unroll
        for (int e = 0; e < E; e++) {
          uw[e] = w * us[e];
          xt = fma(w * xs[e], ts[e], xt);
          xu = fma(w * xs[e], us[e], xu);
        }
#pragma unroll 4
        for (int i = 0; i < m; i++) {
          T v[E];
          Pack<T>::get(Vb + (int64_t)i * L, q, v);
          sD[i * RT + tid] = dotE(v, tw, sD[i * RT + tid]);
          sU[i * RT + tid] = dotE(v, uw, sU[i * RT + tid]);
        }
        continue;
      }
    }
#pragma unroll 4
    for (int i = 0; i < m; i++) {
      T v[E];
      Pack<T>::get(Vb + (int64_t)i * L, q, v);
      sD[i * RT + tid] = dotE(v, tw, sD[i * RT + tid]);
    }
  }
  double* rb = rpart + (int64_t)b * nchunks;
  double* db = dpart + (int64_t)b * M * nchunks;
  const double tot = block_sum((double)acc, red);
  if (tid == 0) rb[blockIdx.x] = tot;
  sums_to_partial<T>(sD, m, db + blockIdx.x, nchunks);
  if (olsen) {
    sums_to_partial<T>(sU, m, upart + (int64_t)b * M * nchunks + blockIdx.x, nchunks);
    const double s_xt = block_sum((double)xt, red);
    if (tid == 0) xpart[((int64_t)b * 2) * nchunks + blockIdx.x] = s_xt;
    const double s_xu = block_sum((double)xu, red);
    if (tid == 0) xpart[((int64_t)b * 2 + 1) * nchunks + blockIdx.x] = s_xu;
  }
  if (!last_cta(cnt + b, nchunks)) return;
  if (!olsen)
    for (int i = tid >> 5; i < m; i += RT / 32) {
      const double s = row_sum(db + (int64_t)i * nchunks, nchunks);
      if ((tid & 31) == 0) coef[(int64_t)b * M + i] = s;
    }
  if (yp && tid < M) yp[(int64_t)b * M + tid] = tid < m ? y[(int64_t)b * M + tid] : 0.0;
  if (tid < 32) {
    const double rn = sqrt(row_sum(rb, nchunks));
    if (tid == 0) {
      const double t = theta[b];
      cv.rnorm[b] = rn;
      cv.iters[b] += 1;
      const double tr = cv.rel ? cv.tol_r[b] * fmax(1.0, fabs(t)) : cv.tol_r[b];
      const bool conv = !cv.first && fabs(t - cv.theta_old[b]) < cv.tol_e && rn < tr;
      cv.theta_old[b] = t;
      if (conv) cv.active[b] = 0;
      else atomicAdd(cv.nact, 1);
    }
  }
}

// One classical Gram-Schmidt update T <- T - sum_{i<m} c_i V_i (first T <- T -
// eps U with Uo), with the dot products the next step needs taken in the same
// pass (V_i[k] read twice by one thread, the second time from the caches):
//   norm == 0: V_i . T into coef (the second pass's coefficients),
//   norm == 1: T . T: 1 / |T| into inv, or the tuple is frozen where the
//              correction vanished (|T|^2 <= tiny).
template <typename T>
__global__ void __launch_bounds__(RT)
k_orth(T* __restrict__ Tv, const T* __restrict__ V, int m, int M, int64_t L, int64_t nd,
       double* __restrict__ coef, int32_t* __restrict__ active, int norm, int ch, int nchunks,
       double* __restrict__ partial, const T* __restrict__ Uo, const float* __restrict__ eps,
       int32_t* __restrict__ cnt, double* __restrict__ inv, double tiny) {
  const int b = blockIdx.y;
  if (!active[b]) return;
  constexpr int E = Pack<T>::E;
  extern __shared__ __align__(16) unsigned char dsm[];
  T* sD = reinterpret_cast<T*>(dsm);
  __shared__ T sc[32];
  __shared__ double red[32];
  const int tid = threadIdx.x;
  if (tid < m) sc[tid] = (T)coef[(int64_t)b * M + tid];
  if (!norm)
    for (int i = 0; i < m; i++) sD[i * RT + tid] = T(0);
  __syncthreads();
  const int64_t q0 = (int64_t)blockIdx.x * (ch / E), q1 = min(L / E, q0 + ch / E), ndq = nd / E;
  const T* Vb = V + (int64_t)b * M * L;
  T nacc = T(0);
  const T ee = Uo ? (T)eps[b] : T(0);
  for (int64_t q = q0 + tid; q < q1; q += RT) {
    T t[E], tw[E];
    Pack<T>::get(Tv + (int64_t)b * L, q, t);
    if (Uo) {
      T u[E];
      Pack<T>::get(Uo + (int64_t)b * L, q, u);
#pragma unroll
      for (int e = 0; e < E; e++) t[e] = fma(-ee, u[e], t[e]);
    }
#pragma unroll 4
    for (int i = 0; i < m; i++) {
      T v[E];
      Pack<T>::get(Vb + (int64_t)i * L, q, v);
#pragma unroll
      for (int e = 0; e < E; e++) t[e] = fma(-sc[i], v[e], t[e]);
    }
    Pack<T>::put(Tv + (int64_t)b * L, q, t);
    const T w = q < ndq ? T(1) : T(2);
#pragma unroll
    for (int e = 0; e < E; e++) tw[e] = w * t[e];
    if (norm) {
      nacc = dotE(t, tw, nacc);
    } else {
#pragma unroll 4
      for (int i = 0; i < m; i++) {
        T v[E];
        Pack<T>::get(Vb + (int64_t)i * L, q, v);
        sD[i * RT + tid] = dotE(v, tw, sD[i * RT + tid]);
      }
    }
  }
  double* pb = partial + (int64_t)b * M * nchunks;
  if (norm) {
    const double tot = block_sum((double)nacc, red);
    if (tid == 0) pb[blockIdx.x] = tot;
  } else {
    sums_to_partial<T>(sD, m, pb + blockIdx.x, nchunks);
  }
  if (!last_cta(cnt + b, nchunks)) return;
  if (norm) {
    if (tid < 32) {
      const double n2 = row_sum(pb, nchunks);
      if (tid == 0) {
        if (n2 > tiny) inv[b] = 1.0 / sqrt(n2);
        else active[b] = 0;
      }
    }
    return;
  }
  for (int i = tid >> 5; i < m; i += RT / 32) {
    const double s = row_sum(pb + (int64_t)i * nchunks, nchunks);
    if ((tid & 31) == 0) coef[(int64_t)b * M + i] = s;
  }
}

// Restart keeping two vectors: the current Ritz vector x = V y and the
// previous one, orthonormalised against x in coefficient space
// (q = y_prev - (y.y_prev) y, twice, normalised; V is orthonormal, so this
// avoids the cancellation of subtracting two nearly parallel long vectors).
// The new 2x2 projected matrix is [y q]^T G [y q].  One warp per tuple.
static __global__ void k_restart_coef(const double* __restrict__ y, double* __restrict__ yp, int m,
                                      int M, const int32_t* __restrict__ active,
                                      double* __restrict__ G) {
  const int b = blockIdx.x;
  if (!active[b]) return;
  __shared__ double sy[32], sq[32], sG[32][33];
  const int r = threadIdx.x;
  sy[r] = r < m ? y[(int64_t)b * M + r] : 0.0;
  sq[r] = r < m ? yp[(int64_t)b * M + r] : 0.0;
  for (int i = 0; i < m; i++)
    if (r < m) sG[i][r] = G[(int64_t)b * M * M + (int64_t)i * M + r];
  __syncwarp();
  for (int pass = 0; pass < 2; pass++) {
    const double d = ritz_warp_sum(sy[r] * sq[r]);
    sq[r] -= d * sy[r];
    __syncwarp();
  }
  double nq = sqrt(ritz_warp_sum(sq[r] * sq[r]));
  if (!(nq > 1e-14)) {
    // x did not move: take the unit vector on which x has least weight
    double a = r < m ? fabs(sy[r]) : 1e300;
    int idx = r;
    for (int off = 16; off; off >>= 1) {
      const double oa = __shfl_xor_sync(0xffffffffu, a, off);
      const int oi = __shfl_xor_sync(0xffffffffu, idx, off);
      if (oa < a || (oa == a && oi < idx)) { a = oa; idx = oi; }
    }
    sq[r] = (r == idx) ? 1.0 : 0.0;
    __syncwarp();
    const double d = ritz_warp_sum(sy[r] * sq[r]);
    sq[r] -= d * sy[r];
    __syncwarp();
    nq = sqrt(ritz_warp_sum(sq[r] * sq[r]));
  }
  sq[r] /= nq;
  __syncwarp();
  double gy = 0.0, gq = 0.0;   // (G y)_r, (G q)_r
  if (r < m)
    for (int j = 0; j < m; j++) {
      gy = fma(sG[r][j], sy[j], gy);
      gq = fma(sG[r][j], sq[j], gq);
    }
  const double g00 = ritz_warp_sum(sy[r] * gy), g01 = ritz_warp_sum(sy[r] * gq);
  const double g11 = ritz_warp_sum(sq[r] * gq), g10 = ritz_warp_sum(sq[r] * gy);
  if (r < m) yp[(int64_t)b * M + r] = sq[r];
  if (r == 0) {
    double* Gb = G + (int64_t)b * M * M;
    const double off = 0.5 * (g01 + g10);
    Gb[0] = g00;
    Gb[1] = off;
    Gb[M] = off;
    Gb[M + 1] = g11;
  }
}

// In place: V_0 = V y, V_1 = V q, AV_0 = AV y, AV_1 = AV q (q in yp)
template <typename T>
__global__ void k_restart_vec(T* __restrict__ V, T* __restrict__ AV, int m, int M, int64_t L,
                              const double* __restrict__ y, const double* __restrict__ q,
                              const int32_t* __restrict__ active) {
  const int b = blockIdx.y;
  if (!active[b]) return;
  __shared__ T sy[32], sq[32];
  if (threadIdx.x < m) {
    sy[threadIdx.x] = (T)y[(int64_t)b * M + threadIdx.x];
    sq[threadIdx.x] = (T)q[(int64_t)b * M + threadIdx.x];
  }
  __syncthreads();
  T* Vb = V + (int64_t)b * M * L;
  T* AVb = AV + (int64_t)b * M * L;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < L;
       k += (int64_t)gridDim.x * blockDim.x) {
    T x = T(0), xp = T(0), ax = T(0), axp = T(0);
    for (int i = 0; i < m; i++) {
      const T v = Vb[(int64_t)i * L + k], av = AVb[(int64_t)i * L + k];
      x = fma(sy[i], v, x);
      xp = fma(sq[i], v, xp);
      ax = fma(sy[i], av, ax);
      axp = fma(sq[i], av, axp);
    }
    Vb[k] = x;
    Vb[L + k] = xp;
    AVb[k] = ax;
    AVb[L + k] = axp;
  }
}

// y_prev right after a restart: the first unit vector
static __global__ void k_restart_yprev(double* __restrict__ yp, int M,
                                       const int32_t* __restrict__ active) {
  const int b = blockIdx.x;
  if (!active[b]) return;
  for (int i = threadIdx.x; i < M; i += blockDim.x) yp[(int64_t)b * M + i] = i == 0 ? 1.0 : 0.0;
}

// partial sums of x . y (full vectors, FP64) and their total
static __global__ void k_dot64(const double* __restrict__ X, const double* __restrict__ Y,
                               int64_t N, int ch, int nchunks, const int32_t* __restrict__ active,
                               double* __restrict__ partial, int32_t* __restrict__ cnt,
                               double* __restrict__ out) {
  const int b = blockIdx.y;
  if (active && !active[b]) return;
  __shared__ double red[32];
  const int64_t k0 = (int64_t)blockIdx.x * ch, k1 = min(N, k0 + ch);
  double acc = 0.0;
  for (int64_t k = k0 + threadIdx.x; k < k1; k += blockDim.x)
    acc = fma(X[(int64_t)b * N + k], Y[(int64_t)b * N + k], acc);
  const double tot = block_sum(acc, red);
  double* pb = partial + (int64_t)b * nchunks;
  if (threadIdx.x == 0) pb[blockIdx.x] = tot;
  if (!last_cta(cnt + b, nchunks)) return;
  if (threadIdx.x < 32) {
    const double s = row_sum(pb, nchunks);
    if (threadIdx.x == 0) out[b] = s;
  }
}

static __global__ void k_fill_i(int32_t* __restrict__ v, int n, int32_t x) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) v[i] = x;
}
static __global__ void k_fill_d(double* __restrict__ v, int n, double x) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) v[i] = x;
}

// reduction chunk: about `per_sm` CTAs per SM over the batch, 1024..16384
// elements (a multiple of 1024)
inline int chunk_of(int64_t L, int B, int nsm, int per_sm) {
  int ch = 16384;
  while (ch > 1024 && (int64_t)B * ((L + ch - 1) / ch) < (int64_t)per_sm * nsm) ch >>= 1;
  return ch;
}

// the kernels with up to 33 accumulator rows take more than 48 KB of dynamic
// shared memory: their attributes, once per device
template <typename T>
inline void set_attributes(int device) {
  static bool done[MBE_MAX_DEVICES] = {false};
  once_per_device(done, device, [] {
    const int one = 33 * RT * (int)sizeof(T);
    CU_CHECK(cudaFuncSetAttribute(k_dots<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, one));
    CU_CHECK(cudaFuncSetAttribute(k_subspace<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, one));
    CU_CHECK(cudaFuncSetAttribute(k_residual<T>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                  sizeof(T) == 4 ? 2 * one : one));
    CU_CHECK(cudaFuncSetAttribute(k_orth<T>, cudaFuncAttributeMaxDynamicSharedMemorySize, one));
  });
}

}  // namespace dvec
