// bs_cgvec.cuh -- the vector passes of a CG iteration inside the solvers.
//
// Algorithm 1 updates x and r together (BS5) and then the direction (BS2), 72
// bytes a node in FP64: p is read by both passes.  Here the pass that waits
// for alpha updates r alone (its r.r is all that beta needs) and the pass that
// waits for beta updates x with the old direction and then the direction, 64
// bytes a node; every value is the one the two separate operations give.
// The x pass belongs to an iteration whose r pass ran, also when that one set
// the stop flag, so it goes by its own flag (CgState::xdue), which the r
// pass of an iteration that is skipped takes back.  64 iterations at N = 7 on
// 32^3 (N_G = 11.4M): 22.7 -> 22.2 ms.  Running the r pass from the vectors'
// ends to their starts, so that it begins on what the gather has just left in
// L2, made no difference there and cost 2% on vectors of 19 MB.
#pragma once

#include "bs_stream.cuh"

namespace bs {

// r = fma(-alpha, Ap, r), ep(sum r^2).
template <typename T, int U, class Ep>
__global__ void __launch_bounds__(kReduceBlock)
    k_cg_r(Split sp, const T *alpha_p, const T *__restrict__ Ap, T *__restrict__ r,
           double *partials, unsigned int *counter, Ep ep, CgState *st) {
  using V = typename VecOf<T>::type;
  constexpr int W = VecOf<T>::W;
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * blockDim.x;
  if (cg_halted(st)) {
    if (tid == 0) st->xdue = 0;
    return;
  }
  const T nalpha = -*alpha_p;
  const V *Apv = reinterpret_cast<const V *>(Ap + sp.head);
  V *rv = reinterpret_cast<V *>(r + sp.head);
  Acc<T> acc[U];
  int64_t i = tid;
  for (; i + (U - 1) * nth < sp.nvec; i += U * nth) {
    V b[U], d[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      b[u] = Apv[i + u * nth];
      d[u] = rv[i + u * nth];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int k = 0; k < W; ++k) {
        vel(d[u], k) = fmaT(nalpha, vel(b[u], k), vel(d[u], k));
        acc[u].add(vel(d[u], k), vel(d[u], k));
      }
      rv[i + u * nth] = d[u];
    }
  }
  for (; i < sp.nvec; i += nth) {
    V b = Apv[i], d = rv[i];
#pragma unroll
    for (int k = 0; k < W; ++k) {
      vel(d, k) = fmaT(nalpha, vel(b, k), vel(d, k));
      acc[0].add(vel(d, k), vel(d, k));
    }
    rv[i] = d;
  }
  auto scalar = [&](int64_t j) {
    const T rj = fmaT(nalpha, Ap[j], r[j]);
    r[j] = rj;
    acc[0].add(rj, rj);
  };
  for (int64_t j = tid; j < sp.head; j += nth) scalar(j);
  for (int64_t j = sp.tail0 + tid; j < sp.n; j += nth) scalar(j);
#pragma unroll
  for (int u = 1; u < U; ++u) acc[0].merge(acc[u]);
  const double part = block_sum<kReduceBlock>(acc[0].value());
  double total;
  if (grid_combine<kReduceBlock>(part, partials, counter, &total) && threadIdx.x == 0) {
    ep(total);
    st->xdue = 1;
  }
}

template <typename T, class Ep>
int launch_cg_r(int64_t n, const T *alpha, const T *Ap, T *r, double *partials,
                unsigned int *counter, Ep ep, CgState *st, cudaStream_t s) {
  constexpr int U = 4;
  const void *ptrs[2] = {Ap, r};
  Split sp = make_split<T>(n, ptrs, 2);
  auto kern = k_cg_r<T, U, Ep>;
  const int64_t work = sp.nvec > 0 ? sp.nvec : n;
  int grid = reduce_grid(work, U, blocks_per_sm(kern, kReduceBlock), kOneBlockDot);
  if (grid < 1) return fail(BS_ERR_CUDA, "no device");
  if (grid > kMaxPartials) grid = kMaxPartials;
  kern<<<grid, kReduceBlock, 0, s>>>(sp, alpha, Ap, r, partials, counter, ep, st);
  BS_LAUNCH_CHECK();
  return BS_OK;
}

// x = fma(alpha, p, x); p = fma(1, z, beta p), when the r pass of this
// iteration ran.
template <typename T, int U>
__global__ void __launch_bounds__(kStreamBlock)
    k_cg_xp(Split sp, const T *alpha_p, const T *beta_p, const T *__restrict__ z,
            T *__restrict__ x, T *__restrict__ p, const CgState *st) {
  using V = typename VecOf<T>::type;
  constexpr int W = VecOf<T>::W;
  if (*((volatile const int *)&st->xdue) == 0) return;
  const T alpha = *alpha_p, beta = *beta_p;
  auto f = [&](T zv, T &xv, T &pv) {
    xv = fmaT(alpha, pv, xv);
    pv = fmaT(T(1), zv, beta * pv);
  };
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * blockDim.x;
  const V *zv = reinterpret_cast<const V *>(z + sp.head);
  V *xv = reinterpret_cast<V *>(x + sp.head), *pv = reinterpret_cast<V *>(p + sp.head);
  int64_t i = tid;
  for (; i + (U - 1) * nth < sp.nvec; i += U * nth) {
    V a[U], b[U], c[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      a[u] = zv[i + u * nth];
      b[u] = ld_stream(xv + i + u * nth);
      c[u] = pv[i + u * nth];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
#pragma unroll
      for (int k = 0; k < W; ++k) f(vel(a[u], k), vel(b[u], k), vel(c[u], k));
      st_stream(xv + i + u * nth, b[u]);
      pv[i + u * nth] = c[u];
    }
  }
  for (; i < sp.nvec; i += nth) {
    V a = zv[i], b = ld_stream(xv + i), c = pv[i];
#pragma unroll
    for (int k = 0; k < W; ++k) f(vel(a, k), vel(b, k), vel(c, k));
    st_stream(xv + i, b);
    pv[i] = c;
  }
  for (int64_t j = tid; j < sp.head; j += nth) f(z[j], x[j], p[j]);
  for (int64_t j = sp.tail0 + tid; j < sp.n; j += nth) f(z[j], x[j], p[j]);
}

template <typename T>
int launch_cg_xp(int64_t n, const T *alpha, const T *beta, const T *z, T *x, T *p,
                 const CgState *st, cudaStream_t s) {
  constexpr int U = 2;
  const void *ptrs[3] = {z, x, p};
  Split sp = make_split<T>(n, ptrs, 3);
  auto kern = k_cg_xp<T, U>;
  const int64_t work = sp.nvec > 0 ? sp.nvec : n;
  const int grid = stream_grid(work, U, kStreamBlock, blocks_per_sm(kern, kStreamBlock));
  if (grid < 1) return fail(BS_ERR_CUDA, "no device");
  kern<<<grid, kStreamBlock, 0, s>>>(sp, alpha, beta, z, x, p, st);
  BS_LAUNCH_CHECK();
  return BS_OK;
}

}  // namespace bs
