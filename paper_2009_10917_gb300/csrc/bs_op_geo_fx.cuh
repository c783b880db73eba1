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
// The fluxes carry the quadrature weights, which differ by 1500 inside an element at
// N = 7: the digits are those of the fluxes times the weights' inverse powers of two,
// which the matrix then takes up exactly (P^-1 D^T P, P = diag(2^-p)).
// As in bs_op_fx.cuh the digits serve a gradient component, and then an entry, only where
// the sum of the sizes of its own terms is large enough (FxGeoTab::lowd, lowdt; a component
// by its line, along t from a plane of |u| in halves; an entry by its lines along r and
// s); the others take FP64 sums of the lines.  Elements beyond 2^+-900 or not finite, by u
// or by the fluxes, and those in which a quarter of the components do not, take the FP64 sums of
// fxg_direct.
#pragma once

#include "bs_op_geo.cuh"

namespace bs {

// Three or four warps of two layers per element: 13824, 13824 and 19683 elements at Nq =
// 6, 7, 8 in 186, 225 and 312 us on uniform values (FP64 kernel 295, 566, 1020; without the
// second look at small entries 159, 191, 296), 275, 470 and 1059 where all elements take
// FP64 sums after all; warps of four layers, or one warp per element, take longer (their
// registers spill or leave too few warps).  Nq = 5 stays with the FP64 kernel: 225 us against 196, the
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
  static constexpr int SIZES = FxShape<NQ>::DIG + FxShape<NQ>::XCH;  // a plane of |u|
  static constexpr int COL = SIZES + FxShape<NQ>::PLANE;             // words of the warps
  static constexpr int X = COL + 128;                                // u in FP64
  static constexpr int SMEM_FX = X + NP * 8;
  static constexpr int DIRECT = 4 * NP * 8;          // u and the three fluxes
  static constexpr int SMEM = SMEM_FX > DIRECT ? SMEM_FX : DIRECT;
  // (the fluxes of the nodes that take FP64 sums lie over all of it)
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
  const double *D = tab->fxg.D;
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

template <int NQ>
__device__ __noinline__ double fxg_line(const double *__restrict__ row, const double *x, int d) {
  double v = 0.0;
#pragma unroll
  for (int m = 0; m < NQ; ++m) v = fma(row[m], x[m * d], v);
  return v;
}

template <int NQ, bool GATHER_IN>
__global__ void __launch_bounds__(FxGeoShape<NQ>::THREADS, FxGeoShape<NQ>::BLOCKS)
    k_ax_geo_fx(int64_t E, int64_t NL, const int32_t *__restrict__ order,
                const int32_t *__restrict__ ids, const double *__restrict__ in,
                double *__restrict__ out, const OpTab<double> *__restrict__ tab,
                const double *__restrict__ coef, const double *__restrict__ geo, double lambda,
                const CgState *st, float slack) {
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
  uint32_t *col = reinterpret_cast<uint32_t *>(fxg_smem + S::COL);
  double *x = reinterpret_cast<double *>(fxg_smem + S::X);
  const uint32_t dig_s = (uint32_t)__cvta_generic_to_shared(dig);
  auto sync = [] { __syncthreads(); };
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
  uint32_t live = 0;  // bit 2l + h: outputs that are used
#pragma unroll
  for (int l = 0; l < L; ++l) {
    const bool a_on = on0 && layer(l), b_on = on1 && layer(l);
    if (GATHER_IN) {
      int32_t a = a_on ? __ldcs(ids + own + l * NQ2) : -1;
      int32_t b = b_on ? __ldcs(ids + own + l * NQ2 + 1) : -1;
      if (!chk(bs_pred_map_entry(a, tab->ng), BS_CHK_OP_ENTRY)) a = -1;
      if (!chk(bs_pred_map_entry(b, tab->ng), BS_CHK_OP_ENTRY)) b = -1;
      u0[l] = a >= 0 ? in[a] : 0.0;
      u1[l] = b >= 0 ? in[b] : 0.0;
      live |= (a >= 0 ? 1u : 0u) << 2 * l | (b >= 0 ? 2u : 0u) << 2 * l;
    } else {  // a caller's vector may be 8-byte aligned only
      u0[l] = a_on ? __ldcs(in + own + l * NQ2) : 0.0;
      u1[l] = b_on ? __ldcs(in + own + l * NQ2 + 1) : 0.0;
      live |= (a_on ? 1u : 0u) << 2 * l | (b_on ? 2u : 0u) << 2 * l;
    }
    if (a_on) x[(k0 + l) * NQ2 + g * NQ + 2 * t] = u0[l];
    if (b_on) x[(k0 + l) * NQ2 + g * NQ + 2 * t + 1] = u1[l];
  }
  const double ce = coef ? coef[e] : 1.0;
  uint32_t big = 0;
#pragma unroll
  for (int l = 0; l < L; ++l) big = max(big, max(fx_size(u0[l]), fx_size(u1[l])));
  bool zero;
  int emax = fx_emax<WPE>(
      big,
      [&] {
        uint32_t r = 0;
#pragma unroll
        for (int l = 0; l < L; ++l) r |= (uint32_t)(__double2loint(u0[l]) | __double2loint(u1[l]));
        return r;
      },
      col, warp, lane, sync, &zero);
  // a component's FP64 sum: row r of D on the line from node n, nodes d apart
  auto line = [&](int r, int n, int d) { return fxg_line<NQ>(tab->fxg.sD + r * NQ, x + n, d); };
  double r0[L], r1[L], s0[L], s1[L], t0[L], t1[L];  // sd grad u, then the flux
  bool sums = fx_far(emax);  // all of the element by FP64 sums
  const uint32_t da = __ldg(&tab->fxg.da[lane]);
  const float lowd = zero ? 0.f : slack * tab->fxg.lowd;  // zeros: the digits are exact
  float cr[2 * L], cs[2 * L];  // the sizes of the terms along r and s
  float least = INFINITY;
  if (!sums) {
#pragma unroll
    for (int l = 0; l < L; l += 2) {
      const uint32_t h0 = fx_sizes2(u0[l], u1[l], emax), h1 = fx_sizes2(u0[l + 1], u1[l + 1], emax);
      fx_terms_r(cr + 2 * l, da, h0, h1);
#pragma unroll
      for (int n = 0; n < 4; ++n) cs[2 * l + n] = 0.f;
      fx_terms_s(cs + 2 * l, da, h0, h1);
      uint32_t *hp = reinterpret_cast<uint32_t *>(fxg_smem + S::SIZES);
      const int k = k0 + l;
      if (layer(l)) hp[(k * 8 + (g ^ k)) * 4 + t] = h0;
      if (layer(l + 1)) hp[((k + 1) * 8 + (g ^ (k + 1))) * 4 + t] = h1;
    }
#pragma unroll
    for (int l = 0; l < L; ++l) {
      if (!layer(l)) break;
      fx_store_digits<NQ>(dig, k0 + l, g, t, u0[l], u1[l], emax);
    }
#pragma unroll
    for (int n = 0; n < 2 * L; ++n)
      if ((n & 1 ? on1 : on0) && layer(n / 2)) least = fminf(least, fminf(cr[n], cs[n]));
    // where a quarter of these components are for FP64 sums, the digits would come on top
    // of sums for most of the element (487, 642 and 1112 us for a field of such elements)
    uint32_t few = 0;
    if (__any_sync(0xffffffffu, least < lowd))
#pragma unroll
      for (int n = 0; n < 2 * L; ++n) {
        const bool use = (n & 1 ? on1 : on0) && layer(n / 2);
        few += __popc(__ballot_sync(0xffffffffu, use && cr[n] < lowd)) +
               __popc(__ballot_sync(0xffffffffu, use && cs[n] < lowd));
      }
    if (lane == 0) col[5 * WPE + warp] = few;
    sync();
    few = 0;
#pragma unroll
    for (int w = 0; w < WPE; ++w) few += col[5 * WPE + w];
    sums = few > NP / 2;
  }
  if (!sums) {
    FxMul<NQ> mul(tab->fxg.d, lane);
    // ---- the gradient; along t in the exchange's layout: nodes (2t, k0 + l, g)
    int p2 = emax - 1020 - tab->fxg.qd;
#pragma unroll
    for (int l = 0; l < L; ++l) {
      if (!layer(l)) break;
      const int j = k0 + l, krow = mul.mrow < NQ ? mul.mrow : NQ - 1;
      uint32_t a[D], b[D], h;
      mul.along_t(dig_s, j, a, b);
      fx_ldsm1t(&h, dig_s + S::SIZES + (krow * 8 + (j ^ krow)) * 16);
      float c[4] = {0.f, 0.f, 0.f, 0.f};
      fx_mma8(c, da, 0u, h);
      double v0 = fx_double((int64_t)fx_join0(a), p2), v1 = fx_double((int64_t)fx_join0(b), p2);
      if (__any_sync(0xffffffffu, fminf(c[0], c[1]) < lowd)) {
        if (on0 && c[0] < lowd) v0 = line(g, j * NQ + 2 * t, NQ2);
        if (on1 && c[1] < lowd) v1 = line(g, j * NQ + 2 * t + 1, NQ2);
      }
      if (NQ == 8 || g < NQ)
        *reinterpret_cast<double2 *>(fx_xch<NQ>(xch, j, g, t)) = make_double2(v0, v1);
    }
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
    if (__any_sync(0xffffffffu, least < lowd)) {
#pragma unroll
      for (int n = 0; n < 2 * L; ++n) {
        if (!((n & 1 ? on1 : on0) && layer(n / 2))) continue;
        const int i = 2 * t + (n & 1), k = (k0 + n / 2) * NQ2;
        double &r = n & 1 ? r1[n / 2] : r0[n / 2], &s = n & 1 ? s1[n / 2] : s0[n / 2];
        if (cr[n] < lowd) r = line(i, k + g * NQ, 1);
        if (cs[n] < lowd) s = line(g, k + i, NQ);
      }
    }
    sync();
    // ---- the flux; u becomes lambda M u.  The fluxes carry the quadrature weights, whose
    // range is 1500 at N = 7: their digits are those of 2^p times them, p = p_i + p_j + p_k
    const int q0 = on0 ? tab->fxg.p[2 * t] + tab->fxg.p[g] : 0;
    const int q1 = on1 ? tab->fxg.p[2 * t + 1] + tab->fxg.p[g] : 0;
    int w0[L], w1[L];
#pragma unroll
    for (int l = 0; l < L; ++l) {
      const int q = layer(l) ? tab->fxg.p[k0 + l] : 0;
      w0[l] = q0 + q;
      w1[l] = q1 + q;
    }
    auto size = [](double v, int p) {
      const uint32_t z = fx_size(v);
      return z ? z + ((uint32_t)p << 20) : 0u;
    };
    big = 0;
#pragma unroll
    for (int l = 0; l < L; ++l) {
      t0[l] = t1[l] = 0.0;
      if (!layer(l)) {
        r0[l] = r1[l] = s0[l] = s1[l] = 0.0;
        break;
      }
      double2 v = make_double2(0.0, 0.0);
      if (NQ == 8 || g < NQ) v = *reinterpret_cast<double2 *>(fx_xch<NQ>(xch, g, k0 + l, t));
      const double2 g0 = pair(geo, l), g1 = pair(geo + NL, l), g2 = pair(geo + 2 * NL, l);
      const double2 g3 = pair(geo + 3 * NL, l), g4 = pair(geo + 4 * NL, l);
      const double2 g5 = pair(geo + 5 * NL, l), M = pair(geo + 6 * NL, l);
      const double a0 = fma(g0.x, r0[l], fma(g1.x, s0[l], g2.x * v.x));
      const double b0 = fma(g1.x, r0[l], fma(g3.x, s0[l], g4.x * v.x));
      t0[l] = fma(g2.x, r0[l], fma(g4.x, s0[l], g5.x * v.x));
      const double a1 = fma(g0.y, r1[l], fma(g1.y, s1[l], g2.y * v.y));
      const double b1 = fma(g1.y, r1[l], fma(g3.y, s1[l], g4.y * v.y));
      t1[l] = fma(g2.y, r1[l], fma(g4.y, s1[l], g5.y * v.y));
      r0[l] = a0;
      r1[l] = a1;
      s0[l] = b0;
      s1[l] = b1;
      u0[l] = lambda * (M.x * u0[l]);
      u1[l] = lambda * (M.y * u1[l]);
      big = max(big, max(size(a0, w0[l]), max(size(b0, w0[l]), size(t0[l], w0[l]))));
      big = max(big, max(size(a1, w1[l]), max(size(b1, w1[l]), size(t1[l], w1[l]))));
    }
    // (the low words of the fluxes: those that are zero in the high word count as far)
    emax = fx_emax<WPE>(
        big,
        [&] {
          uint32_t r = 0;
#pragma unroll
          for (int l = 0; l < L; ++l)
            r |= (uint32_t)(__double2loint(r0[l]) | __double2loint(r1[l]) |
                            __double2loint(s0[l]) | __double2loint(s1[l]) |
                            __double2loint(t0[l]) | __double2loint(t1[l]));
          return r;
        },
        col + 2 * WPE, warp, lane, sync, &zero);
    if (!fx_far(emax)) {
      // the entries that the fluxes' digits do not serve: bit 2l + h
      uint32_t low = 0;
      if (!zero) {
        const uint32_t dta = __ldg(&tab->fxg.dta[lane]);
        const float lowdt = slack * tab->fxg.lowdt;
#pragma unroll
        for (int l = 0; l < L; l += 2) {
          auto sizes = [&](const double *a, const double *b, int m) {
            return fx_sizes2(a[m], b[m], emax, w0[m], w1[m]);
          };
          float c[4];
          fx_terms_r(c, dta, sizes(r0, r1, l), sizes(r0, r1, l + 1));
          fx_terms_s(c, dta, sizes(s0, s1, l), sizes(s0, s1, l + 1));
#pragma unroll
          for (int n = 0; n < 4; ++n) low |= c[n] < lowdt ? 1u << (2 * l + n) : 0u;
        }
        low &= live;
      }
      bool some = __any_sync(0xffffffffu, low);
      if (lane == 0) col[4 * WPE + warp] = some;
      mul.set(tab->fxg.dt, lane);
      uint64_t T0[L], T1[L];
      // ---- D^T along r and s: a warp's own layers
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        fx_store_digits<NQ>(dig, k0 + l, g, t, r0[l], r1[l], emax, w0[l], w1[l]);
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
        fx_store_digits<NQ>(dig, k0 + l, g, t, s0[l], s1[l], emax, w0[l], w1[l]);
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
        fx_store_digits<NQ>(dig, k0 + l, g, t, t0[l], t1[l], emax, w0[l], w1[l]);
      }
      sync();
#pragma unroll
      for (int w = 0; w < WPE; ++w) some = some || col[4 * WPE + w];
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
      const double c = ce * tab->fxg.inv;
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        ulonglong2 v = make_ulonglong2(0, 0);
        if (NQ == 8 || g < NQ) v = *fx_xch<NQ>(xch, g, k0 + l, t);
        const double d0 = fx_double((int64_t)(T0[l] + v.x), p2 - w0[l]);
        const double d1 = fx_double((int64_t)(T1[l] + v.y), p2 - w1[l]);
        if (on0) __stcs(out + own + l * NQ2, fma(c, d0, u0[l]));
        if (on1) __stcs(out + own + l * NQ2 + 1, fma(c, d1, u1[l]));
      }
      if (!some) return;
      // ---- the FP64 sums of the nodes in `low`, each by its own lane
      sync();  // the exchanged sums have been read
      double *f = reinterpret_cast<double *>(fxg_smem);
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        const int n = (k0 + l) * NQ2 + g * NQ + 2 * t;
        if (on0) f[n] = r0[l], f[NP + n] = s0[l], f[2 * NP + n] = t0[l];
        if (on1) f[n + 1] = r1[l], f[NP + n + 1] = s1[l], f[2 * NP + n + 1] = t1[l];
      }
      sync();
      const double cd = ce * tab->fxg.invd, *DT = tab->fxg.D;
#pragma unroll
      for (int b = 0; b < 2 * L; ++b) {
        if (!(low >> b & 1u)) continue;
        const int i = 2 * t + (b & 1), k = k0 + (b >> 1);
        double v = 0.0;
#pragma unroll 4
        for (int m = 0; m < NQ; ++m) {
          v = fma(DT[m * NQ + i], f[m + NQ * g + NQ2 * k], v);
          v = fma(DT[m * NQ + g], f[NP + i + NQ * m + NQ2 * k], v);
          v = fma(DT[m * NQ + k], f[2 * NP + i + NQ * g + NQ2 * m], v);
        }
        __stcs(out + own + (b >> 1) * NQ2 + (b & 1),
               fma(cd, v, (b & 1) ? u1[b >> 1] : u0[b >> 1]));
      }
      return;
    }
  }
  // ---- the FP64 sums (block-uniform), on the element's values read again
  __syncthreads();
  x = reinterpret_cast<double *>(fxg_smem);
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
