// bs_op_fx16.cuh -- the fixed-point element operator of bs_op_fx.cuh for
// degrees 8..15, in 16 x 16 tiles.
//
// The same digits, orders and joins; here a digit's contraction fills the 16
// products of an mma.sync by itself.  A lane owns, of every layer k of its
// warp, the nodes j = g, g + 8, i = 2t, 2t + 1, 2t + 8, 2t + 9 (g = lane / 4,
// t = lane % 4): its digit words are the A fragment along r (rows j, Kh^T as B, two
// tiles of eight columns), the transposed layer is the B fragment along s and
// the transposed (k, i) plane the one along t, with Kh as A.  Orders 3..5 take
// two accumulators, products of digits 2 and 3 in the second (Kh's scale is the
// largest for which both hold; checked where the table is made).
// Every warp has L layers (and planes j) of one element.  Nodes whose terms along r and s
// are too small for the digits take FP64 sums, as in bs_op_fx.cuh.
//
#pragma once

#include "bs_op_fx.cuh"

namespace bs {

template <int NQ>
constexpr bool use_fx16() {
  return NQ > kFxMaxNq && NQ <= kMaxNq;
}

// Two layers a warp, as many elements an SM as leave a thread 80 to 128
// registers: A_L u in ps a node 31, 28, 26, 21, 21, 16, 15, 12 at Nq = 9 .. 16
// (one layer a warp 38, 34, .., 29, .., 19; FP64 kernels 66, 63, 86 and 99 at Nq = 9,
// 10, 12 and 16).  The tiles' filling, (Nq / 16)^2, sets most of the difference.
template <int NQ>
struct FxShape16 {
  static constexpr int L = 2;                              // layers per warp
  static constexpr int WPE = (NQ + L - 1) / L;             // warps of an element
  static constexpr int THREADS = 32 * WPE;                 // one element per block
  static constexpr int PLANE = NQ * 512;                   // bytes of one digit plane
  static constexpr int DIG = kFxDigits * PLANE;
  static constexpr int XCH = NQ * NQ * 128;                // [j][k][16 i] uint64
  static constexpr int SMEM = DIG + XCH;
  static constexpr int BLOCKS = NQ == 9 ? 4 : (NQ <= 13 ? 3 : 2);  // resident per SM
};

// Shared address of row j, half c (i = 8c ..) of layer k in a digit plane: the
// 16-byte chunks of a layer permuted so that eight rows j of one layer and
// eight layers k of one row j lie in different banks.
__device__ __forceinline__ uint32_t fx16_chunk(int k, int j, int c) {
  return (uint32_t)(k * 512 + ((j * 2 + c) ^ (k & 7) ^ ((j >> 2) & 1)) * 16);
}

template <int NQ>
struct FxMul16 {
  static constexpr int D = kFxDigits, PLANE = FxShape16<NQ>::PLANE;
  uint32_t kw[D][4];  // digit b of Kh: (g, 2t), (g + 8, 2t), (g, 2t + 8), (g + 8, 2t + 8)
  FxStart start1, start2;
  int mrow, mmat;
  __device__ __forceinline__ FxMul16(const uint32_t (*w)[32][4], int lane)
      : start1(kFxMagicBits, kFxMagicBits),
        start2(kFxMagic2Bits, kFxMagic2Bits),
        mrow(lane & 7),
        mmat(lane >> 3) {
#pragma unroll
    for (int b = 0; b < D; ++b) {
      const uint4 v = __ldg(reinterpret_cast<const uint4 *>(&w[b][lane][0]));
      kw[b][0] = v.x;
      kw[b][1] = v.y;
      kw[b][2] = v.z;
      kw[b][3] = v.w;
    }
  }
  // s[n][o] (with one start value each) of one tile of eight columns; KA: Kh is
  // the A operand and f[a][2h], f[a][2h + 1] the B fragment, else f[a] is A.
  template <bool KA>
  __device__ __forceinline__ void tile(const uint32_t (*f)[4], int h, uint32_t (*s)[D]) const {
#pragma unroll
    for (int o = 0; o < D; ++o) {
      const FxStart &st = o == D - 1 ? start2 : start1;
      float c0[4], c1[4];
#pragma unroll
      for (int a = 0; a <= o; ++a) {
        const bool second = o >= 3 && (a == 2 || a == 3), first = a == 0 || (second && a == 2);
        float *c = second ? c1 : c0;
        const uint32_t *k = kw[o - a];
        if (KA) {
          if (first)
            fx_mma0(c, k[0], k[1], k[2], k[3], f[a][2 * h], f[a][2 * h + 1], st);
          else
            fx_mma(c, k[0], k[1], k[2], k[3], f[a][2 * h], f[a][2 * h + 1]);
        } else {
          if (first)
            fx_mma0(c, f[a][0], f[a][1], f[a][2], f[a][3], k[h], k[2 + h], st);
          else
            fx_mma(c, f[a][0], f[a][1], f[a][2], f[a][3], k[h], k[2 + h]);
        }
      }
#pragma unroll
      for (int n = 0; n < 4; ++n) {
        s[n][o] = __float_as_uint(c0[n]);
        if (o >= 3)
          s[n][o] += __float_as_uint(c1[n]) - (o == D - 1 ? kFxMagic2Bits : kFxMagicBits);
      }
    }
  }
  __device__ __forceinline__ void load(uint32_t (*f)[4], uint32_t addr, bool trans) const {
#pragma unroll
    for (int a = 0; a < D; ++a) {
      if (trans)
        fx_ldsm4t(f[a], addr + a * PLANE);
      else
        fx_ldsm4(f[a], addr + a * PLANE);
    }
  }
};

// out = A_L in; arguments as k_ax_fx.
template <int NQ, bool GATHER_IN, bool FUSED>
__global__ void __launch_bounds__(FxShape16<NQ>::THREADS, FxShape16<NQ>::BLOCKS)
    k_ax_fx16(int64_t E, const int32_t *__restrict__ order, const int32_t *__restrict__ ids,
              const double *__restrict__ in, double *__restrict__ out,
              const OpTab<double> *__restrict__ tab, const double *__restrict__ coef,
              const CgState *st, double *__restrict__ outG, double *__restrict__ partials,
              float slack) {
  static_assert(!FUSED || GATHER_IN, "the fused operator reads its input through the map");
  using S = FxShape16<NQ>;
  constexpr int NQ2 = NQ * NQ, NP = NQ * NQ2, D = kFxDigits, L = S::L, WPE = S::WPE;
  extern __shared__ __align__(128) unsigned char fx16_smem[];
  __shared__ uint32_t s_col[3 * WPE];
  if (cg_halted(st)) return;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3, warp = threadIdx.x >> 5;
  const int k0 = warp * L;
  unsigned char *dig = fx16_smem, *xch = dig + S::DIG;
  const uint32_t dig_s = (uint32_t)__cvta_generic_to_shared(dig);
  Acc<double> acc;
  const int64_t slot = blockIdx.x;
  int64_t e = order ? (int64_t)order[slot] : slot;
  if (!chk(bs_pred_index(e, tab->ne), BS_CHK_OP_ENTRY)) e = -1;  // block-uniform
  if (e >= 0) {
    const int64_t base = e * NP + (int64_t)k0 * NQ2;
    auto layer = [&](int l) { return NQ % L == 0 || k0 + l < NQ; };
    // a lane's eight nodes of a layer: q = 4 jj + 2 h + p, j = g + 8 jj, i = 2t + 8h + p
    auto node_j = [&](int q) { return g + 8 * (q >> 2); };
    auto node_i = [&](int q) { return 2 * t + 8 * ((q >> 1) & 1) + (q & 1); };
    auto on = [&](int q) { return node_j(q) < NQ && node_i(q) < NQ; };
    auto at = [&](int q) { return node_j(q) * NQ + node_i(q); };
    double u[L][8];
    int32_t id[GATHER_IN ? L : 1][8];
    if (GATHER_IN) {
#pragma unroll
      for (int l = 0; l < L; ++l)
#pragma unroll
        for (int q = 0; q < 8; ++q) {
          int32_t v = on(q) && layer(l) ? __ldcs(ids + base + l * NQ2 + at(q)) : -1;
          if (!chk(FUSED ? bs_pred_fused_entry(v, tab->ng) : bs_pred_map_entry(v, tab->ng),
                   BS_CHK_OP_ENTRY))
            v = -1;
          id[GATHER_IN ? l : 0][q] = v;
        }
    }
#pragma unroll
    for (int l = 0; l < L; ++l)
#pragma unroll
      for (int q = 0; q < 8; ++q) {
        if (GATHER_IN) {
          const int32_t v = id[GATHER_IN ? l : 0][q];
          u[l][q] = (FUSED ? v != -1 : v >= 0) ? in[FUSED && v < 0 ? -2 - v : v] : 0.0;
        } else {
          u[l][q] = on(q) && layer(l) ? __ldcs(in + base + l * NQ2 + at(q)) : 0.0;
        }
      }
    // ---- the largest exponent, and the nodes the digits do not serve: bit 8l + q
    uint32_t big = 0, low = 0;
#pragma unroll
    for (int l = 0; l < L; ++l)
#pragma unroll
      for (int q = 0; q < 8; ++q) big = max(big, fx_size(u[l][q]));
    auto rest = [&] {
      uint32_t r = 0;
#pragma unroll
      for (int l = 0; l < L; ++l)
#pragma unroll
        for (int q = 0; q < 8; ++q) r |= (uint32_t)__double2loint(u[l][q]);
      return r;
    };
    bool zero;
    const int emax =
        fx_emax<WPE>(big, rest, s_col, warp, lane, [] { __syncthreads(); }, &zero);
    const bool far = fx_far(emax);
    const float least = zero ? 0.f : slack * tab->fx16.low;  // zeros: the digits are exact
    // the sums of the sizes of layer l's terms along r and s: each(q, sum)
    auto terms = [&](int l, auto each) {
      const uint4 ka = __ldg(reinterpret_cast<const uint4 *>(&tab->fx16.a[lane][0]));
      uint32_t h[4];  // rows g, g + 8 of columns 2t, then of 2t + 8
#pragma unroll
      for (int q = 0; q < 8; q += 2) h[(q >> 2) + (q & 2)] = fx_sizes2(u[l][q], u[l][q + 1], emax);
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        float s[4] = {0.f, 0.f, 0.f, 0.f};
        fx_mma(s, h[0], h[1], h[2], h[3], c ? ka.y : ka.x, c ? ka.w : ka.z);            // along r
        fx_mma(s, ka.x, ka.y, ka.z, ka.w, fx_trans(h[2 * c]), fx_trans(h[2 * c + 1]));  // along s
#pragma unroll
        for (int n = 0; n < 4; ++n) each(4 * (n >> 1) + 2 * c + (n & 1), s[n]);
      }
    };
    bool some = far;  // of the element's nodes
    if (far) {
      low = (1u << 8 * L) - 1u;
    } else {
#pragma unroll
      for (int l = 0; l < L; ++l)
        terms(l, [&](int q, float s) {
          low |= on(q) && layer(l) && s < least ? 1u << (8 * l + q) : 0u;
        });
    }
    if (__any_sync(0xffffffffu, low)) {
#pragma unroll
      for (int b = 0; b < 8 * L; ++b) {  // those whose results are used
        const int l = b >> 3, q = b & 7;
        bool use = on(q) && layer(l);
        if (GATHER_IN && use && (low >> b & 1u) && u[l][q] == 0.0) {
          const int32_t v = __ldg(ids + base + l * NQ2 + at(q));
          use = FUSED ? v != -1 : v >= 0;
        }
        if (!use) low &= ~(1u << b);
      }
      some = far || __any_sync(0xffffffffu, low);
    }
    const double ce = coef ? coef[e] : 1.0;
    auto store = [&](int l, int q, double r, int32_t i, double v) {
      if (!on(q)) return;
      if (!FUSED || i >= 0) {
        __stcs(out + base + l * NQ2 + at(q), r);
      } else if (i != -1) {
        const double p = plus_zero(r);
        __stcs(outG + (-2 - i), p);
        if (!(low >> (8 * l + q) & 1u)) acc.add(v, p);
      }
    };
    // the element's values in memory order, over the digits once those are done with
    double *x = reinterpret_cast<double *>(dig);
    auto keep = [&] {
#pragma unroll
      for (int l = 0; l < L; ++l)
#pragma unroll
        for (int q = 0; q < 8; ++q)
          if (on(q) && layer(l)) x[(k0 + l) * NQ2 + at(q)] = u[l][q];
    };
    if (!far) {
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
#pragma unroll
        for (int q = 0; q < 8; q += 2) {
          const uint64_t x = fx_fixed(u[l][q], emax), y = fx_fixed(u[l][q + 1], emax);
          uint32_t *p = reinterpret_cast<uint32_t *>(dig + fx16_chunk(k0 + l, node_j(q), (q >> 1) & 1)) + t;
          constexpr int PW = S::PLANE / 4;
          p[0 * PW] = fx_digit2<0>(x, y);
          p[1 * PW] = fx_digit2<1>(x, y);
          p[2 * PW] = fx_digit2<2>(x, y);
          p[3 * PW] = fx_digit2<3>(x, y);
          p[4 * PW] = fx_digit2<4>(x, y);
          p[5 * PW] = fx_digit2<5>(x, y);
        }
      }
      const FxMul16<NQ> mul(tab->fx16.w, lane);
      __syncthreads();
      auto slot16 = [&](int j, int k, int c) {  // 16-byte slot c of row (j, k)
        return reinterpret_cast<ulonglong2 *>(xch) + (j * NQ + k) * 8 + (c ^ ((k ^ j) & 7));
      };
      const int mr = (mul.mmat & 1) * 8 + mul.mrow, mc = mul.mmat >> 1;  // ldmatrix row, half
      // ---- along t, planes j = k0 + l (layers past Nq repeat the last: zero digits of Kh)
      const int mk = mr < NQ ? mr : NQ - 1;
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        const int j = k0 + l;
        uint32_t f[D][4];
        mul.load(f, dig_s + fx16_chunk(mk, j, mc), true);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t s[4][D];
          mul.template tile<true>(f, h, s);
          *slot16(j, g, t + 4 * h) = make_ulonglong2(fx_join(s[0]), fx_join(s[1]));
          if (g + 8 < NQ)
            *slot16(j, g + 8, t + 4 * h) = make_ulonglong2(fx_join(s[2]), fx_join(s[3]));
        }
      }
      // ---- along r and s; the start values of all three directions come off
      uint64_t T[L][8];
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        const uint32_t a = dig_s + fx16_chunk(k0 + l, mr, mc);
        uint32_t f[D][4];
        mul.load(f, a, false);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t s[4][D];
          mul.template tile<false>(f, h, s);
#pragma unroll
          for (int n = 0; n < 4; ++n) T[l][4 * (n >> 1) + 2 * h + (n & 1)] = fx_join(s[n]);
        }
        mul.load(f, a, true);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          uint32_t s[4][D];
          mul.template tile<true>(f, h, s);
#pragma unroll
          for (int n = 0; n < 4; ++n) {
            constexpr uint64_t m = kFxMagicBits;
            constexpr uint64_t start =
                m + kFxMagic2Bits / 512 + (m << 10) + (m << 20) + (m << 30) + (m << 40);
            T[l][4 * (n >> 1) + 2 * h + (n & 1)] += fx_join(s[n]) - 3u * start;
          }
        }
      }
      if (lane == 0) s_col[2 * WPE + warp] = some;
      __syncthreads();
#pragma unroll
      for (int w = 0; w < WPE; ++w) some = some || s_col[2 * WPE + w];
      if (some) keep();
      // ---- results: w_k (c (h/2) w_i w_j sum + lambda (h/2)^3 w_i w_j u)
      const int p2 = emax - 1020 - tab->fx16.q;
      auto results = [&](auto with_coef) {
#pragma unroll
        for (int l = 0; l < L; ++l) {
          if (!layer(l)) break;
          const int k = k0 + l;
          const double wk = tab->fx16.w1[k];
#pragma unroll
          for (int q = 0; q < 8; q += 2) {
            ulonglong2 v = make_ulonglong2(0, 0);
            if (node_j(q) < NQ) v = *slot16(node_j(q), k, t + 4 * ((q >> 1) & 1));
            double d0 = fx_double((int64_t)(T[l][q] + v.x), p2);
            double d1 = fx_double((int64_t)(T[l][q + 1] + v.y), p2);
            const double2 wg =
                __ldg(reinterpret_cast<const double2 *>(tab->fx16.wg) + lane * 4 + q / 2);
            const double2 wm =
                __ldg(reinterpret_cast<const double2 *>(tab->fx16.wm) + lane * 4 + q / 2);
            if (decltype(with_coef)::value) {
              d0 = ce * d0;
              d1 = ce * d1;
            }
            store(l, q, wk * fma(wg.x, d0, wm.x * u[l][q]), id[GATHER_IN ? l : 0][q], u[l][q]);
            store(l, q + 1, wk * fma(wg.y, d1, wm.y * u[l][q + 1]),
                  id[GATHER_IN ? l : 0][q + 1], u[l][q + 1]);
          }
        }
      };
      if (coef)
        results(std::true_type{});
      else
        results(std::false_type{});
    } else {
      keep();
    }
    if (some) {  // ---- the FP64 sums of the nodes in `low`, as in fx_element
      __syncthreads();
      uint16_t *list = reinterpret_cast<uint16_t *>(xch) + k0 * NQ2;
      const int count = fx_list(low, 8 * L, lane, list, [&](int b) {
        return (k0 + (b >> 3)) * NQ2 + node_j(b & 7) * NQ + node_i(b & 7);
      });
      __syncthreads();
      fx_direct_list<NQ>(x, tab->kh, list, count, lane, [&](int n, double d) {
        const int i = n % NQ, j = n / NQ % NQ, k = n / NQ2;
        // the owner's table entry: lane (j % 8, i / 2 % 4), q
        const int own = ((j & 7) * 4 + (i & 7) / 2) * 8 + 4 * (j >> 3) + 2 * (i >> 3) + (i & 1);
        const double v = x[n];
        const double r = tab->fx16.w1[k] *
                         fma(tab->fx16.wg[own], coef ? ce * d : d, tab->fx16.wm[own] * v);
        int32_t to = 0;
        if (FUSED) {
          to = ids[e * NP + n];
          if (!chk(bs_pred_fused_entry(to, tab->ng), BS_CHK_OP_ENTRY)) to = -1;
        }
        if (to >= 0) {
          __stcs(out + e * NP + n, r);
        } else if (to != -1) {
          const double y = plus_zero(r);
          __stcs(outG + (-2 - to), y);
          acc.add(v, y);
        }
      });
    }
  }
  if (FUSED && partials) {
    const double part = block_sum<S::THREADS>(acc.value());
    if (threadIdx.x == 0) partials[blockIdx.x] = part;
  }
}

}  // namespace bs
