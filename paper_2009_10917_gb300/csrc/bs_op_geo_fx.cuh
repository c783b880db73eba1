// bs_op_geo_fx.cuh -- the general-hexahedron operator of bs_op_geo.cuh with its
// contractions in the exact fixed-point form of bs_op_fx.cuh, degrees 5..7.
//
// The FP64 kernel does 6 (N+1) + 12 FP64 operations a node and is bound by
// that pipe.  Here the gradient's three contractions (with D) and the flux's
// three (with D^T) are digit products on the tensor cores; what is left in
// FP64 is the flux G grad u (nine operations a node), the mass term and the
// result (four), plus 56 bytes of factors.  The same mapping as bs_op_fx.cuh:
// warps with their own layers, nodes (2t, g), (2t + 1, g); the digit planes are
// reused for u and then for each flux component (r and s need only a warp's
// own layers, t all of them).  The three components share one exponent, the
// element's largest flux.
//
// Elements that the digits do not serve, by u or by the fluxes (see
// kFxRange), take the FP64 sums of fxg_direct.
#pragma once

#include "bs_op_geo.cuh"

namespace bs {

// Three or four warps of two layers per element: 19683 elements at Nq = 6, 7, 8
// in 229, 268 and 284 us (FP64 kernel 434, 800, 1020); warps of four layers, or
// one warp per element, take 320 us and more (their registers spill or leave
// too few warps).  Nq = 5 stays with the FP64 kernel: 225 us against 196, the
// 5 x 5 layers fill 39% of the tiles.
template <int NQ>
constexpr bool use_fx_geo() {
  return NQ >= 6 && NQ <= kFxMaxNq;
}
template <int NQ>
struct FxGeoShape {
  static constexpr int NP = NQ * NQ * NQ;
  static constexpr int L = 2;                        // layers per warp
  static constexpr int WPE = (NQ + L - 1) / L;
  static constexpr int THREADS = 32 * WPE;           // one element per block
  static constexpr int BLOCKS = NQ == 8 ? 5 : (NQ == 7 ? 6 : 8);
  static constexpr int BASE = FxShape<NQ>::DIG + FxShape<NQ>::XCH;
  static constexpr int FX = BASE + WPE * 256;        // + columns' maxima
  static constexpr int DIRECT = 4 * NP * 8;          // u and the three fluxes
  static constexpr int SMEM = FX > DIRECT ? FX : DIRECT;
};

// A sum's order values without their start values, joined.
__device__ __forceinline__ uint64_t fx_join0(const uint32_t *s) {
  constexpr uint64_t m = kFxMagicBits;
  constexpr uint64_t start = m + kFxMagic2Bits / 512 + (m << 10) + (m << 20) + (m << 30) + (m << 40);
  return fx_join(s) - start;
}

// One element by FP64 sums, all threads of the block: x holds its values and
// room for three flux components.
template <int NQ>
__device__ __noinline__ void fxg_direct(double *x, double *__restrict__ out,
                                        const OpTab<double> *tab, const double *__restrict__ geo,
                                        int64_t NL, int64_t base, double ce, double lambda) {
  constexpr int NQ2 = NQ * NQ, NP = NQ * NQ2;
  const double *D = tab->D;
  double *fr = x + NP, *fs = fr + NP, *ft = fs + NP;
  for (int n = threadIdx.x; n < NP; n += blockDim.x) {
    const int i = n % NQ, j = n / NQ % NQ, k = n / NQ2;
    double ur = 0.0, us = 0.0, ut = 0.0;
    for (int m = 0; m < NQ; ++m) {
      ur = fma(D[i * NQ + m], x[m + NQ * j + NQ2 * k], ur);
      us = fma(D[j * NQ + m], x[i + NQ * m + NQ2 * k], us);
      ut = fma(D[k * NQ + m], x[i + NQ * j + NQ2 * m], ut);
    }
    const double *G = geo + base + n;
    const double g1 = G[NL], g2 = G[2 * NL], g4 = G[4 * NL];
    fr[n] = fma(G[0], ur, fma(g1, us, g2 * ut));
    fs[n] = fma(g1, ur, fma(G[3 * NL], us, g4 * ut));
    ft[n] = fma(g2, ur, fma(g4, us, G[5 * NL] * ut));
  }
  __syncthreads();
  for (int n = threadIdx.x; n < NP; n += blockDim.x) {
    const int i = n % NQ, j = n / NQ % NQ, k = n / NQ2;
    double s = 0.0;
    for (int m = 0; m < NQ; ++m) {
      s = fma(D[m * NQ + i], fr[m + NQ * j + NQ2 * k], s);
      s = fma(D[m * NQ + j], fs[i + NQ * m + NQ2 * k], s);
      s = fma(D[m * NQ + k], ft[i + NQ * j + NQ2 * m], s);
    }
    out[base + n] = fma(ce, s, lambda * (geo[6 * NL + base + n] * x[n]));
  }
}

template <int NQ, bool GATHER_IN>
__global__ void __launch_bounds__(FxGeoShape<NQ>::THREADS, FxGeoShape<NQ>::BLOCKS)
    k_ax_geo_fx(int64_t E, int64_t NL, const int32_t *__restrict__ order,
                const int32_t *__restrict__ ids, const double *__restrict__ in,
                double *__restrict__ out, const OpTab<double> *__restrict__ tab,
                const double *__restrict__ coef, const double *__restrict__ geo, double lambda,
                const CgState *st) {
  using S = FxGeoShape<NQ>;
  constexpr int NQ2 = NQ * NQ, NP = S::NP, D = kFxDigits, L = S::L, WPE = S::WPE;
  constexpr bool EVEN = NQ % 2 == 0;
  extern __shared__ __align__(128) unsigned char fxg_smem[];
  if (cg_halted(st)) return;
  const int64_t slot = blockIdx.x;
  const int64_t e = order ? (int64_t)order[slot] : slot;
  if (!chk(bs_pred_index(e, tab->ne), BS_CHK_OP_ENTRY)) return;  // block-uniform
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, warp = threadIdx.x >> 5;
  const int k0 = warp * L;
  unsigned char *dig = fxg_smem, *xch = dig + FxShape<NQ>::DIG;
  uint32_t *col = reinterpret_cast<uint32_t *>(fxg_smem + S::BASE);
  const uint32_t dig_s = (uint32_t)__cvta_generic_to_shared(dig);
  auto sync = [] {
    if (WPE == 1)
      __syncwarp();
    else
      __syncthreads();
  };
  auto layer = [&](int l) { return NQ % L == 0 || k0 + l < NQ; };
  const bool on0 = g < NQ && 2 * t < NQ, on1 = g < NQ && 2 * t + 1 < NQ;
  const int64_t base = e * NP, own = base + (int64_t)k0 * NQ2 + g * NQ + 2 * t;
  // a pair of values of this lane's layer l from an N_L-sized array
  auto pair = [&](const double *p, int l) {
    double2 v = make_double2(0.0, 0.0);
    if (EVEN) {
      if (on0 && layer(l)) v = __ldcs(reinterpret_cast<const double2 *>(p + own + l * NQ2));
    } else {
      if (on0 && layer(l)) v.x = __ldcs(p + own + l * NQ2);
      if (on1 && layer(l)) v.y = __ldcs(p + own + l * NQ2 + 1);
    }
    return v;
  };
  double u0[L], u1[L];
#pragma unroll
  for (int l = 0; l < L; ++l) {
    if (GATHER_IN) {
      int32_t a = on0 && layer(l) ? __ldcs(ids + own + l * NQ2) : -1;
      int32_t b = on1 && layer(l) ? __ldcs(ids + own + l * NQ2 + 1) : -1;
      if (!chk(bs_pred_map_entry(a, tab->ng), BS_CHK_OP_ENTRY)) a = -1;
      if (!chk(bs_pred_map_entry(b, tab->ng), BS_CHK_OP_ENTRY)) b = -1;
      u0[l] = a >= 0 ? in[a] : 0.0;
      u1[l] = b >= 0 ? in[b] : 0.0;
    } else {  // a caller's vector may be 8-byte aligned only
      u0[l] = on0 && layer(l) ? __ldcs(in + own + l * NQ2) : 0.0;
      u1[l] = on1 && layer(l) ? __ldcs(in + own + l * NQ2 + 1) : 0.0;
    }
  }
  const double ce = coef ? coef[e] : 1.0;
  uint32_t big0 = 0, big1 = 0;
#pragma unroll
  for (int l = 0; l < L; ++l) {
    big0 = max(big0, fx_size(u0[l]));
    big1 = max(big1, fx_size(u1[l]));
  }
  bool direct;
  int emax = fx_range<WPE>(big0, big1, col, warp, lane, sync, &direct);
  double r0[L], r1[L], s0[L], s1[L], t0[L], t1[L];  // grad u, then the flux
  if (!direct) {
#pragma unroll
    for (int l = 0; l < L; ++l) {
      if (!layer(l)) break;
      fx_store_digits<NQ>(dig, k0 + l, g, t, u0[l], u1[l], emax);
    }
    FxMul<NQ> mul(tab->fxg.d, lane);
    sync();
    // ---- the gradient
#pragma unroll
    for (int l = 0; l < L; ++l) {
      if (!layer(l)) break;
      uint32_t a[D], b[D];
      mul.along_t(dig_s, k0 + l, a, b);
      if (NQ == 8 || g < NQ)
        *fx_xch<NQ>(xch, k0 + l, g, t) = make_ulonglong2(fx_join0(a), fx_join0(b));
    }
    int p2 = emax - 1020 - tab->fxg.qd;
#pragma unroll
    for (int l = 0; l < L; l += 2) {
      if (!layer(l)) break;
      const int l0 = k0 + l, l1 = l0 + 1 < NQ ? l0 + 1 : l0;
      uint32_t s[4][D];
      mul.along_r(dig_s, l0, l1, s);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        r0[l + h] = fx_double((int64_t)fx_join0(s[2 * h]), p2);
        r1[l + h] = fx_double((int64_t)fx_join0(s[2 * h + 1]), p2);
        uint32_t a[D], b[D];
        mul.along_s(dig_s, h ? l1 : l0, a, b);
        s0[l + h] = fx_double((int64_t)fx_join0(a), p2);
        s1[l + h] = fx_double((int64_t)fx_join0(b), p2);
      }
    }
    sync();
    // ---- the flux; u becomes lambda M u
    big0 = big1 = 0;
#pragma unroll
    for (int l = 0; l < L; ++l) {
      if (!layer(l)) break;
      ulonglong2 v = make_ulonglong2(0, 0);
      if (NQ == 8 || g < NQ) v = *fx_xch<NQ>(xch, g, k0 + l, t);
      const double ut0 = fx_double((int64_t)v.x, p2), ut1 = fx_double((int64_t)v.y, p2);
      const double2 g0 = pair(geo, l), g1 = pair(geo + NL, l), g2 = pair(geo + 2 * NL, l);
      const double2 g3 = pair(geo + 3 * NL, l), g4 = pair(geo + 4 * NL, l);
      const double2 g5 = pair(geo + 5 * NL, l), M = pair(geo + 6 * NL, l);
      const double a0 = fma(g0.x, r0[l], fma(g1.x, s0[l], g2.x * ut0));
      const double b0 = fma(g1.x, r0[l], fma(g3.x, s0[l], g4.x * ut0));
      t0[l] = fma(g2.x, r0[l], fma(g4.x, s0[l], g5.x * ut0));
      const double a1 = fma(g0.y, r1[l], fma(g1.y, s1[l], g2.y * ut1));
      const double b1 = fma(g1.y, r1[l], fma(g3.y, s1[l], g4.y * ut1));
      t1[l] = fma(g2.y, r1[l], fma(g4.y, s1[l], g5.y * ut1));
      r0[l] = a0;
      r1[l] = a1;
      s0[l] = b0;
      s1[l] = b1;
      u0[l] = lambda * (M.x * u0[l]);
      u1[l] = lambda * (M.y * u1[l]);
      big0 = max(big0, max(fx_size(a0), max(fx_size(b0), fx_size(t0[l]))));
      big1 = max(big1, max(fx_size(a1), max(fx_size(b1), fx_size(t1[l]))));
    }
    emax = fx_range<WPE>(big0, big1, col, warp, lane, sync, &direct);
    if (WPE == 1) __syncwarp();  // every lane has read its exchanged sums
    if (!direct) {
      mul.set(tab->fxg.dt, lane);
      uint64_t T0[L], T1[L];
      // ---- D^T along r and s: a warp's own layers
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        fx_store_digits<NQ>(dig, k0 + l, g, t, r0[l], r1[l], emax);
      }
      __syncwarp();
#pragma unroll
      for (int l = 0; l < L; l += 2) {
        if (!layer(l)) break;
        const int l0 = k0 + l, l1 = l0 + 1 < NQ ? l0 + 1 : l0;
        uint32_t s[4][D];
        mul.along_r(dig_s, l0, l1, s);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          T0[l + h] = fx_join0(s[2 * h]);
          T1[l + h] = fx_join0(s[2 * h + 1]);
        }
      }
      __syncwarp();
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        fx_store_digits<NQ>(dig, k0 + l, g, t, s0[l], s1[l], emax);
      }
      __syncwarp();
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        uint32_t a[D], b[D];
        mul.along_s(dig_s, k0 + l, a, b);
        T0[l] += fx_join0(a);
        T1[l] += fx_join0(b);
      }
      __syncwarp();
      // ---- and along t
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        fx_store_digits<NQ>(dig, k0 + l, g, t, t0[l], t1[l], emax);
      }
      sync();
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        uint32_t a[D], b[D];
        mul.along_t(dig_s, k0 + l, a, b);
        if (NQ == 8 || g < NQ)
          *fx_xch<NQ>(xch, k0 + l, g, t) = make_ulonglong2(fx_join0(a), fx_join0(b));
      }
      sync();
      p2 = emax - 1020 - tab->fxg.qdt;
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        ulonglong2 v = make_ulonglong2(0, 0);
        if (NQ == 8 || g < NQ) v = *fx_xch<NQ>(xch, g, k0 + l, t);
        const double d0 = fx_double((int64_t)(T0[l] + v.x), p2);
        const double d1 = fx_double((int64_t)(T1[l] + v.y), p2);
        if (on0) __stcs(out + own + l * NQ2, fma(ce, d0, u0[l]));
        if (on1) __stcs(out + own + l * NQ2 + 1, fma(ce, d1, u1[l]));
      }
      return;
    }
  }
  // ---- the FP64 sums (block-uniform), on the element's values read again
  __syncthreads();
  double *x = reinterpret_cast<double *>(fxg_smem);
  for (int n = threadIdx.x; n < NP; n += S::THREADS) {
    if (GATHER_IN) {
      int32_t id = ids[base + n];
      if (!chk(bs_pred_map_entry(id, tab->ng), BS_CHK_OP_ENTRY)) id = -1;
      x[n] = id >= 0 ? in[id] : 0.0;
    } else {
      x[n] = in[base + n];
    }
  }
  __syncthreads();
  fxg_direct<NQ>(x, out, tab, geo, NL, base, ce, lambda);
}

}  // namespace bs
