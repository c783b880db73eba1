// bs_op_fx4.cuh -- the fixed-point element operator of bs_op_fx.cuh for degrees
// 2 and 3, dense in the mma.sync tiles.
//
// An element of degree 3 is 16 lines of 4 nodes: in the 8 x 8 tiles of
// bs_op_fx.cuh it would fill a quarter.  Here the 16 products of an mma.sync
// m16n8k16 are four digits of four nodes, and its free side holds several
// orders at once:
//  - along r, A = the 16 lines (rows) with digits 0..3 (or 4, 5: k8), B = Kh^T for
//    two orders side by side (columns 4 od + i');
//  - along s and t, A = Kh for four orders (rows 4 od + j'), B = the digits of
//    (s', j) against (k, i), by ldmatrix.trans from the digits in shared memory.
// Either way a lane ends up with the even orders or the odd ones of its
// nodes, joins those and adds its partner's half: 16 mma.sync per element.
// With g = lane / 4, t = lane % 4 a lane owns the nodes i = 2 (t % 2), + 1, j = g % 4,
// k = 2 (g / 4) + t / 2.  One warp takes kFx4Epw elements, their values loaded
// together.  Degree 2 runs in the same tiles with zero digits (27 of 64 nodes, and
// still ahead).  With four nodes a line every order fits its start value of
// 1.5 * 2^23: no second start value.  Nodes whose terms are too small for the digits take
// FP64 sums, each on its own lane.
//
// What bounds it: integer and issue slots, as bs_op_fx.cuh.  A_L u on 16M (12.8M) local
// nodes: 606 -> 171 us at degree 3 (direct FP64 kernel before), 435 -> 324 at degree 2;
// where all nodes take FP64 sums 478 and 754.  Degree 1, 8 of 64 nodes, stays with the FP64 kernel.
#pragma once

#include "bs_op_fx16.cuh"

namespace bs {

// Elements per warp, warps per block, resident blocks per SM (96 registers): 390 us
// for 592704 elements at Nq = 4, A_L Z p alone; 2 elements a warp 387 with spills,
// 3 393, 6 404, 1 417; 124 registers (four blocks) 430.
constexpr int kFx4Epw = 4, kFx4Warps = 4, kFx4Blocks = 5;
constexpr int kFx4Epb = kFx4Epw * kFx4Warps;

template <int NQ>
constexpr bool use_fx4() {
  return NQ == 3 || NQ == 4;
}

constexpr int kFx4Digit = 36;                      // words of a digit: 32, and 4 of padding
constexpr int kFx4Words = 2 * kFxDigits * kFx4Digit;  // both layouts of an element

// A lane's half of the orders (x0, x1, x2: orders par, par + 2, par + 4, start
// values included) in the units of fx_join.
__device__ __forceinline__ uint64_t fx4_join(uint32_t x0, uint32_t x1, uint32_t x2, int par) {
  return ((uint64_t)x0 << (par ? 30 : 40)) + ((uint64_t)x1 << (par ? 10 : 20)) +
         (par ? (x2 + 512u) >> 10 : x2);
}
constexpr uint64_t kFx4Start =  // of both halves
    ((uint64_t)kFxMagicBits << 40) + ((uint64_t)kFxMagicBits << 20) + kFxMagicBits +
    ((uint64_t)kFxMagicBits << 30) + ((uint64_t)kFxMagicBits << 10) + (kFxMagicBits >> 10);

// out = A_L in; arguments as k_ax_fx.
template <int NQ, bool GATHER_IN, bool FUSED>
__global__ void __launch_bounds__(32 * kFx4Warps, kFx4Blocks)
    k_ax_fx4(int64_t E, const int32_t *__restrict__ order, const int32_t *__restrict__ ids,
             const double *__restrict__ in, double *__restrict__ out,
             const OpTab<double> *__restrict__ tab, const double *__restrict__ coef,
             const CgState *st, double *__restrict__ outG, double *__restrict__ partials,
             int vec, float slack) {
  static_assert(!FUSED || GATHER_IN, "the fused operator reads its input through the map");
  constexpr int NQ2 = NQ * NQ, NP = NQ * NQ2, D = kFxDigits, EPW = kFx4Epw;
  constexpr bool EVEN = NQ % 2 == 0;
  __shared__ __align__(16) uint32_t s_dig[kFx4Warps][kFx4Words];
  if (cg_halted(st)) return;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, warp = threadIdx.x >> 5;
  const int od = g >> 2, j = g & 3, kk = 2 * od + (t >> 1), i0 = 2 * (t & 1);
  uint32_t *P = s_dig[warp], *Q = P + D * kFx4Digit;
  const bool on0 = j < NQ && kk < NQ && i0 < NQ, on1 = j < NQ && kk < NQ && i0 + 1 < NQ;
  const int own = (kk * NQ + j) * NQ + i0;
  Acc<double> acc;
  const int64_t first = ((int64_t)blockIdx.x * kFx4Warps + warp) * EPW;
  // ---- the elements' values
  int64_t e[EPW];
  int32_t id0[EPW], id1[EPW];
  double u0[EPW], u1[EPW];
#pragma unroll
  for (int q = 0; q < EPW; ++q) {
    const int64_t slot = first + q;
    e[q] = slot < E ? (order ? (int64_t)order[slot] : slot) : -1;
    if (e[q] >= 0 && !chk(bs_pred_index(e[q], tab->ne), BS_CHK_OP_ENTRY)) e[q] = -1;
  }
#pragma unroll
  for (int q = 0; q < EPW; ++q) {
    id0[q] = id1[q] = -1;
    if (!GATHER_IN || e[q] < 0) continue;
    const int32_t *p = ids + e[q] * NP + own;
    if (EVEN) {
      if (on0) {
        const int2 v = __ldcs(reinterpret_cast<const int2 *>(p));
        id0[q] = v.x;
        id1[q] = v.y;
      }
    } else {
      if (on0) id0[q] = __ldcs(p);
      if (on1) id1[q] = __ldcs(p + 1);
    }
    if (!chk(FUSED ? bs_pred_fused_entry(id0[q], tab->ng) : bs_pred_map_entry(id0[q], tab->ng),
             BS_CHK_OP_ENTRY))
      id0[q] = -1;
    if (!chk(FUSED ? bs_pred_fused_entry(id1[q], tab->ng) : bs_pred_map_entry(id1[q], tab->ng),
             BS_CHK_OP_ENTRY))
      id1[q] = -1;
  }
#pragma unroll
  for (int q = 0; q < EPW; ++q) {
    u0[q] = u1[q] = 0.0;
    if (GATHER_IN) {
      if (FUSED ? id0[q] != -1 : id0[q] >= 0)
        u0[q] = in[FUSED && id0[q] < 0 ? -2 - id0[q] : id0[q]];
      if (FUSED ? id1[q] != -1 : id1[q] >= 0)
        u1[q] = in[FUSED && id1[q] < 0 ? -2 - id1[q] : id1[q]];
    } else if (e[q] >= 0) {
      const double *p = in + e[q] * NP + own;
      if (EVEN && vec) {
        if (on0) {
          const double2 v = __ldcs(reinterpret_cast<const double2 *>(p));
          u0[q] = v.x;
          u1[q] = v.y;
        }
      } else {
        if (on0) u0[q] = __ldcs(p);
        if (on1) u1[q] = __ldcs(p + 1);
      }
    }
  }
  // digits of Kh: v[x] = digit 2x + od - t / 2 of Kh[g % 4][2 (t % 2) ..]
  const uint32_t v0 = __ldg(&tab->fx4.w[0][lane]), v2 = __ldg(&tab->fx4.w[1][lane]);
  const uint32_t v4 = __ldg(&tab->fx4.w[2][lane]);
  const double2 wg = __ldg(reinterpret_cast<const double2 *>(tab->fx4.wg) + lane);
  const double2 wm = __ldg(reinterpret_cast<const double2 *>(tab->fx4.wm) + lane);
  const FxStart start(kFxMagicBits, kFxMagicBits);
  const uint32_t P_s = (uint32_t)__cvta_generic_to_shared(P);
  const uint32_t Q_s = (uint32_t)__cvta_generic_to_shared(Q);
  // ldmatrix: row (s', j) of digit pair x, half c; matrices (x, c) = (0, 0), (1, 0),
  // (0, 1), (1, 1), then (2, 0), (2, 1)
  const int mrow = lane & 7, mm = lane >> 3;
  const uint32_t row4 = (((2 * (mm & 1) + (mrow >> 2)) * kFx4Digit + (mrow & 3) * 8 + (mm >> 1) * 4) * 4);
  const uint32_t row2 = (((4 + (mrow >> 2)) * kFx4Digit + (mrow & 3) * 8 + (mm & 1) * 4) * 4);
  const bool hiT = t >= 2;
  // where the sums along t of this lane's nodes arrive
  const int src = (kk | ((j >> 1) << 2)) * 4 + (((j & 1) << 1) | (t & 1));
  const uint32_t ka = __ldg(&tab->fx4.a[lane]);  // |Kh[g % 4][2 (t % 2) ..]|
  const float least = slack * tab->fx4.low;
  auto element = [&](int64_t e, double a, double b, int32_t m0, int32_t m1) {
    bool zero;
    const int emax = fx_emax<1>(
        max(fx_size(a), fx_size(b)),
        [&] { return (uint32_t)(__double2loint(a) | __double2loint(b)); }, nullptr, 0, lane,
        [] {}, &zero);
    const bool far = fx_far(emax);
    const bool live0 = on0 && (!GATHER_IN || (FUSED ? m0 != -1 : m0 >= 0));
    const bool live1 = on1 && (!GATHER_IN || (FUSED ? m1 != -1 : m1 >= 0));
    bool low0 = far && live0, low1 = far && live1;  // nodes the digits do not serve
    if (!far && !zero) {
      // their terms' sizes: along r the lines with even k in columns 0-3 of rows
      // 0-7, those with odd k in columns 4-7 of rows 8-15; along s the matrix once per od
      const uint32_t h = fx_sizes2(a, b, emax);
      float r[4] = {0.f, 0.f, 0.f, 0.f};
      fx_mma8(r, hiT ? 0u : h, hiT ? h : 0u, ka);
      const float r0 = hiT ? r[2] : r[0], r1 = hiT ? r[3] : r[1];
      if (__any_sync(0xffffffffu, (live0 && r0 < least) || (live1 && r1 < least))) {
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        fx_mma8(s, od == (t >> 1) ? ka : 0u, 0u, fx_trans(h));
        low0 = live0 && r0 + s[0] < least;
        low1 = live1 && r1 + s[1] < least;
      }
    }
    const double ce = coef ? coef[e] : 1.0;
    double r0 = 0.0, r1 = 0.0;
    __syncwarp();  // the last element's digits have been read
    if (!far) {
      const uint64_t x = fx_fixed(a, emax), y = fx_fixed(b, emax);
      const uint32_t d[D] = {fx_digit2<0>(x, y), fx_digit2<1>(x, y), fx_digit2<2>(x, y),
                             fx_digit2<3>(x, y), fx_digit2<4>(x, y), fx_digit2<5>(x, y)};
#pragma unroll
      for (int s = 0; s < D; ++s) {
        P[s * kFx4Digit + j * 8 + kk * 2 + (t & 1)] = d[s];
        Q[s * kFx4Digit + kk * 8 + j * 2 + (t & 1)] = d[s];
      }
      // ---- along r: rows g (k even) and g + 8 (k odd), digits of a pair in lanes t, t ^ 2
      uint32_t f[D];  // A fragments of the digit pairs: rows g, rows g + 8
#pragma unroll
      for (int s = 0; s < D; s += 2) {
        const uint32_t o = __shfl_xor_sync(0xffffffffu, hiT ? d[s] : d[s + 1], 2);
        f[s] = hiT ? o : d[s];
        f[s + 1] = hiT ? d[s + 1] : o;
      }
      uint64_t T0, T1;
      {
        float c0[4], c2[4], c4[4];
        fx_mma0(c0, f[0], f[1], f[2], f[3], v0, 0u, start);
        fx_mma0(c2, f[0], f[1], f[2], f[3], v2, v0, start);
        fx_mma0(c4, f[0], f[1], f[2], f[3], v4, v2, start);
        fx_mma8(c4, f[4], f[5], v0);
        uint64_t s[4];
#pragma unroll
        for (int n = 0; n < 4; ++n)
          s[n] = fx4_join(__float_as_uint(c0[n]), __float_as_uint(c2[n]), __float_as_uint(c4[n]),
                          t >> 1);
        // rows g belong to t < 2, rows g + 8 to t >= 2
        T0 = (hiT ? s[2] : s[0]) + __shfl_xor_sync(0xffffffffu, hiT ? s[0] : s[2], 2);
        T1 = (hiT ? s[3] : s[1]) + __shfl_xor_sync(0xffffffffu, hiT ? s[1] : s[3], 2);
      }
      __syncwarp();
      // ---- along s (P) and t (Q): tiles c of eight columns; c = od is this lane's
      auto columns = [&](uint32_t base, uint64_t &S0, uint64_t &S1) {
        uint32_t b4[4], b2[2];
        fx_ldsm4t(b4, base + row4);
        fx_ldsm2t(b2, base + row2);
        uint64_t s[2][2];
#pragma unroll
        for (int c = 0; c < 2; ++c) {
          float lo[4], hi[4];
          fx_mma0(lo, v0, v2, 0u, v0, b4[2 * c], b4[2 * c + 1], start);
          fx_mma0(hi, v4, 0u, v2, 0u, b4[2 * c], b4[2 * c + 1], start);
          fx_mma8(hi, v0, 0u, b2[c]);
#pragma unroll
          for (int n = 0; n < 2; ++n)
            s[c][n] = fx4_join(__float_as_uint(lo[n]), __float_as_uint(lo[2 + n]),
                               __float_as_uint(hi[n]), od);
        }
        S0 = (od ? s[1][0] : s[0][0]) + __shfl_xor_sync(0xffffffffu, od ? s[0][0] : s[1][0], 16);
        S1 = (od ? s[1][1] : s[0][1]) + __shfl_xor_sync(0xffffffffu, od ? s[0][1] : s[1][1], 16);
      };
      uint64_t S0, S1;
      columns(P_s, S0, S1);
      T0 += S0;
      T1 += S1;
      columns(Q_s, S0, S1);
      T0 += __shfl_sync(0xffffffffu, S0, src) - 3u * kFx4Start;
      T1 += __shfl_sync(0xffffffffu, S1, src) - 3u * kFx4Start;
      const int p2 = emax - 1020 - tab->fx4.q;
      r0 = fx_double((int64_t)T0, p2);
      r1 = fx_double((int64_t)T1, p2);
    }
    if (__any_sync(0xffffffffu, low0 || low1)) {  // their FP64 sums
      __syncwarp();  // the digits have been read
      double *x = reinterpret_cast<double *>(P);
      if (on0) x[own] = a;
      if (on1) x[own + 1] = b;
      __syncwarp();
      if (NQ == 3) {  // 27 nodes: one a lane instead of two on every other (one pass)
        const int n = lane < NP ? lane : 0, i = n % NQ, jn = n / NQ % NQ, k = n / NQ2;
        const int owner = ((k >> 1) * 4 + jn) * 4 + (i >> 1) + 2 * (k & 1);
        const uint32_t m0 = __ballot_sync(0xffffffffu, low0), m1 = __ballot_sync(0xffffffffu, low1);
        double v = 0.0;
        if (lane < NP && ((i & 1 ? m1 : m0) >> owner & 1u)) v = fx_direct<NQ>(x, tab->kh, i, jn, k);
        const double v0 = __shfl_sync(0xffffffffu, v, own & 31);
        const double v1 = __shfl_sync(0xffffffffu, v, (own + 1) & 31);
        if (low0) r0 = v0;
        if (low1) r1 = v1;
      } else {
        if (low0) r0 = fx_direct<NQ>(x, tab->kh, i0, j, kk);
        if (low1) r1 = fx_direct<NQ>(x, tab->kh, i0 + 1, j, kk);
      }
    }
    if (coef) {
      r0 = ce * r0;
      r1 = ce * r1;
    }
    r0 = fma(wg.x, r0, wm.x * a);
    r1 = fma(wg.y, r1, wm.y * b);
    double *o = out + e * NP + own;
    if (FUSED) {
      auto one = [&](double r, int32_t id, double u, int h) {
        if (id >= 0) {
          __stcs(o + h, r);
        } else if (id != -1) {
          const double v = plus_zero(r);
          __stcs(outG + (-2 - id), v);
          acc.add(u, v);
        }
      };
      if (on0) one(r0, m0, a, 0);
      if (on1) one(r1, m1, b, 1);
    } else if (EVEN && vec) {
      if (on0) __stcs(reinterpret_cast<double2 *>(o), make_double2(r0, r1));
    } else {
      if (on0) __stcs(o, r0);
      if (on1) __stcs(o + 1, r1);
    }
  };
#pragma unroll 1
  for (int q = 0; q < EPW; ++q) {  // the elements not yet done are shifted down
    if (e[0] >= 0) element(e[0], u0[0], u1[0], id0[0], id1[0]);
#pragma unroll
    for (int n = 0; n + 1 < EPW; ++n) {
      e[n] = e[n + 1];
      u0[n] = u0[n + 1];
      u1[n] = u1[n + 1];
      id0[n] = id0[n + 1];
      id1[n] = id1[n + 1];
    }
    e[EPW - 1] = -1;
  }
  if (FUSED && partials) {
    const double part = block_sum<32 * kFx4Warps>(acc.value());
    if (threadIdx.x == 0) partials[blockIdx.x] = part;
  }
}

}  // namespace bs
