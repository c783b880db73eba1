// bs_op_fx.cuh -- the FP64 element operator of bs_op.cuh with its 1-D
// contractions on the tensor cores, in exact fixed-point pieces.
//
// GB300 executes FP64 at 1/64 of its FP32 rate (about 2 DFMA per clock and
// SM, tensor-core FP64 included), so the element operator, 24 FP64
// operations per node even in its even-odd form, ran at 88% of that pipe
// while HBM idled.  Here the contractions sum_m Kh_im u_m (Kh = W^-1 D^T W D)
// are integer arithmetic (an error-free splitting of the kind of Ozaki,
// Ogita, Oishi & Rump, Numer. Algorithms 59, 2012):
//  - an element's values are taken as 58-bit integers relative to its largest
//    exponent and cut into six signed 10-bit digits; so is Kh times a scale
//    that puts its largest entry near 511 2^50, on the host (FxTab);
//  - a digit fits a half exactly, and mma.sync m16n8k16 sums the products of
//    equal weight (order o = a + b, 48 at most) into an FP32 accumulator that
//    starts at 1.5 * 2^23: with the actual digits of Kh every partial sum is
//    an integer in [2^23, 2^24) (the host takes the largest scale for which
//    that holds), so nothing rounds and the accumulator's bits ARE the
//    integer: no conversion instructions, which share the FP64 pipe.  Order 5,
//    the last, would reach 1.3 times the range and starts at 1.5 * 2^24
//    instead, counting by two; its low ten bits are dropped anyway;
//  - orders 0..5 are joined into one 64-bit integer per node, the three
//    directions summed there, and only then is there a double, put together
//    by integer operations: two FP64 operations per node (the weighted sum
//    and the mass term), three with a coefficient.
// Dropped: u below 2^-58 of the element's largest power of two U, orders >= 6
// and the last ten bits, together about 2^-57.7 of U times Kh's largest power
// of two per node (standard deviation, N = 7), wherever the node is.  FP64
// sums are off by up to (2 Nq + 4) 2^-53 of the sum T of the sizes of the
// node's own terms, so the digits serve a node only where T is large enough
// that four deviations stay within that (FxTab::low).  T is bounded from below
// by its part along r, and where that is not enough by those along r and s,
// from |u| and |Kh| in half precision on the tensor cores (2% of the kernel's
// time: the halves are the lane's own fragments).  The other nodes, and all of
// an element whose largest value is not finite or outside [2^-900, 2^900], take
// FP64 sums from shared memory, compacted to full warps.  Inside the solvers,
// where A p goes on into sums and updates of the vectors' size, four
// deviations may be N - 1 times as large: the FP64 sums with tables made in
// double are themselves off by N - 1 times the bound and more at small entries
// (6.6 at N = 7, 53 at N = 15, the even-odd form 57 at N = 7).  CG's search
// directions have a few per cent of nodes below the line without that (N = 7:
// half of the elements, 8% of an iteration), almost none with it.
//
// One or two warps per element, each with its own layers k (and planes j of
// the t direction).  With g = lane / 4 and t = lane % 4, a lane owns the nodes
// i = 2t, 2t + 1, j = g of its layers; its digit pairs are at once the A fragment of the contraction
// along r (rows j of two layers, columns m; Kh^T as B), the transposed 8 x 8
// layers the B fragment along s and the transposed (k, i) planes the one along
// t, both by ldmatrix.trans from the digit planes in shared memory (row chunks
// XOR-swizzled by k: stores and loads without bank conflicts).  Results along
// r and s arrive in the owner's layout; those along t go through shared
// memory.  Nq < 8 runs in the same 8 x 8 tiles, padded with zero digits.
// The small tiles (K = 8 per digit) are why this is mma.sync and not tcgen05:
// the tensor pipe is not what bounds it, and the accumulators are wanted in
// registers at once.
//
// Measured (N = 7 on 36^3, 23.9M local nodes): A_L Z p 180 us, the even-odd
// FP64 kernel 1047 us; HBM alone would allow 60 us.  What bounds it now is
// spread out: issue slots 65%, integer pipe 57%, FP64 pipe 46%, L1 66%, HBM 26%.
// Conversions by two FP64 additions per node (instead of fx_double) and the
// weights multiplied node by node took 312 us with the FP64 pipe at 82%.
// Where every node takes FP64 sums (36^3, A_L u): 1177 us, the direct FP64
// kernel 1352; where a third to two thirds do (a layer exp(-12 t), values spread
// over e^+-9), digits and sums both, 1190 to 1310 us.
// Error against extended precision on uniform inputs 6e-17 normwise (the
// even-odd kernel 8.3e-16), entry by entry at most 0.1 of the bound.
#pragma once

#include <type_traits>

#include "bs_gather.cuh"

namespace bs {

constexpr uint32_t kFxMagicBits = 0x4B400000u;   // 1.5 * 2^23: counts by one
constexpr uint32_t kFxMagic2Bits = 0x4BC00000u;  // 1.5 * 2^24: counts by two

template <int NQ>
constexpr bool use_fx() {
  return NQ >= kFxMinNq && NQ <= kFxMaxNq;
}

// Two warps of four layers per element at Nq = 8 (72 registers, 14 elements per
// SM: 176 us for 46656 elements, A_L Z p without the look at each node's terms, against
// 180 with 80 registers,
// 190 for one warp of eight layers, 196 for four of two), one warp below (the
// last warp would idle: Nq = 5, 112 us against 147 for two layers per warp,
// Nq = 6 139 against 150).
template <int NQ>
struct FxShape {
  static constexpr int L = NQ == 8 ? 4 : (NQ + 1) / 2 * 2;  // layers per warp
  static constexpr int WPE = (NQ + L - 1) / L;              // warps per element
  static constexpr int THREADS = 32 * WPE;                  // one element per block
  static constexpr int BLOCKS = NQ == 8 ? 14 : (NQ == 7 ? 20 : 24);  // resident per SM
  static constexpr int PLANE = NQ * 8 * 16;       // bytes of one digit plane
  static constexpr int DIG = kFxDigits * PLANE;
  static constexpr int XCH = NQ * NQ * 64;        // [j][k][8 i] uint64
  static constexpr int WARP = DIG + XCH;          // bytes an element takes on one warp
  static constexpr int SMEM = WARP + (WPE > 1 ? WPE * 256 : 0);  // + columns' maxima
};

// c += A B on a 16 x 8 tile, 16 digit products per entry, all exact.
__device__ __forceinline__ void fx_mma(float *c, uint32_t a0, uint32_t a1, uint32_t a2,
                                       uint32_t a3, uint32_t b0, uint32_t b1) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
// Start values of a tile's four sums (rows 0-7 twice, rows 8-15 twice) in
// registers of their own, opaque to the compiler, which otherwise moves the
// constants into place for every sum (3% of all instructions).
struct FxStart {
  float v[4];
  __device__ __forceinline__ FxStart(uint32_t lo, uint32_t hi) {
    asm volatile("mov.b32 %0, %1;\n" : "=f"(v[0]) : "r"(lo));
    asm volatile("mov.b32 %0, %1;\n" : "=f"(v[1]) : "r"(lo));
    asm volatile("mov.b32 %0, %1;\n" : "=f"(v[2]) : "r"(hi));
    asm volatile("mov.b32 %0, %1;\n" : "=f"(v[3]) : "r"(hi));
  }
};
// The first product of a sum: c = A B + start.
__device__ __forceinline__ void fx_mma0(float *c, uint32_t a0, uint32_t a1, uint32_t a2,
                                        uint32_t a3, uint32_t b0, uint32_t b1,
                                        const FxStart &s) {
  asm("mma.sync.aligned.m16n8k16.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%10,%11,%12,%13};\n"
      : "=f"(c[0]), "=f"(c[1]), "=f"(c[2]), "=f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1), "f"(s.v[0]), "f"(s.v[1]),
        "f"(s.v[2]), "f"(s.v[3]));
}
__device__ __forceinline__ void fx_ldsm4(uint32_t *r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void fx_ldsm4t(uint32_t *r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void fx_ldsm2t(uint32_t *r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];\n"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(addr)
               : "memory");
}

__device__ __forceinline__ void fx_ldsm1t(uint32_t *r, uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x1.trans.shared.b16 {%0}, [%1];\n"
               : "=r"(r[0])
               : "r"(addr)
               : "memory");
}
__device__ __forceinline__ void fx_mma8(float *c, uint32_t a0, uint32_t a1, uint32_t b0) {
  asm("mma.sync.aligned.m16n8k8.row.col.f32.f16.f16.f32 {%0,%1,%2,%3}, {%4,%5}, {%6}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(b0));
}
// The transpose of an 8 x 8 matrix of halves held as a fragment.
__device__ __forceinline__ uint32_t fx_trans(uint32_t a) {
  uint32_t d;
  asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(d) : "r"(a));
  return d;
}

// High word of |x|: zero below 2^-1042 too.
__device__ __forceinline__ uint32_t fx_size(double x) {
  return (uint32_t)__double2hiint(x) & 0x7fffffffu;
}
// |a|, |b| as a pair of halves over 2^emax's power of two (the largest value in [1, 2)),
// cut off, never rounded up; nothing below 2^-14.
// pa, pb: powers of two the values count times.
__device__ __forceinline__ uint32_t fx_sizes2(double a, double b, int emax, int pa = 0,
                                              int pb = 0) {
  const uint32_t x = (uint32_t)__viaddmax_s32((int)fx_size(a), (15 - emax + pa) << 20, 0);
  const uint32_t y = (uint32_t)__viaddmax_s32((int)fx_size(b), (15 - emax + pb) << 20, 0);
  return x >> 10 | (y << 6 & 0xffff0000u);
}

// x as an integer of 58 bits in units of 2^(emax - 1080), rounded to nearest,
// plus 512 in every 10-bit digit (each digit of the result, less 512, is x's),
// shifted left by one: the significand << 6, shifted down to emax with one
// more bit, and for rounding 1 added (x >= 0) or its ones' complement taken.
// Values whose exponent field is 0 (zero, subnormal) shift out entirely.
__device__ __forceinline__ uint64_t fx_fixed(double x, int emax) {
  const uint32_t hw = (uint32_t)__double2hiint(x), lw = (uint32_t)__double2loint(x);
  const int d = min(emax - (int)((hw >> 20) & 0x7ffu), 63);
  const uint64_t m = ((uint64_t)((hw & 0xfffffu) | 0x100000u) << 32 | lw) << 6;
  const uint32_t sg = (uint32_t)((int32_t)hw >> 31);
  constexpr uint64_t bias = 1024ull * (1ull + (1ull << 10) + (1ull << 20) + (1ull << 30) +
                                       (1ull << 40) + (1ull << 50));
  return ((m >> d) ^ ((uint64_t)sg << 32 | sg)) + (bias + 1ull);
}

// Digit A (0 = most significant) of two values of fx_fixed as a pair of halves.
template <int A>
__device__ __forceinline__ uint32_t fx_digit2(uint64_t x, uint64_t y) {
  constexpr int S = 10 * (kFxDigits - 1 - A) + 1;
  const uint32_t h =
      (__byte_perm((uint32_t)(x >> S), (uint32_t)(y >> S), 0x5410) & 0x03ff03ffu) | 0x64006400u;
  uint32_t r;  // halves 1024 + digit + 512, less 1536
  asm("sub.f16x2 %0, %1, %2;\n" : "=r"(r) : "r"(h), "r"(0x66006600u));
  return r;
}

// The orders' integer sums as one 64-bit integer in units of 2^10 of order 5
// (whose accumulators count by two), rounded to nearest: a floor would bias
// every node the same way.
// Unsigned: the start values' bits may still be in the sums, modulo 2^64.
__device__ __forceinline__ uint64_t fx_join(const uint32_t *s) {
  uint64_t v = (uint64_t)(int64_t)((int)s[4] + ((int)(s[5] + 256u) >> 9));
  v += (uint64_t)((int64_t)(int)s[3] * 1024);
  v += (uint64_t)((int64_t)(int)s[2] * (1 << 20));
  v += (uint64_t)((int64_t)(int)s[1] * (1 << 30));
  v += (uint64_t)s[0] << 40;
  return v;
}

// v 2^p as a double, rounded once (|v| < 2^62, the result normal or zero), by
// integer operations alone: conversions and additions of doubles share the
// FP64 pipe.  The significand's implicit bit adds one to the exponent field,
// and so does a carry out of its rounding.
__device__ __forceinline__ double fx_double(int64_t v, int p) {
  const uint64_t a = (uint64_t)(v < 0 ? -v : v);
  const uint32_t hi = (uint32_t)(a >> 32), lo = (uint32_t)a;
  const int lz = __clz((int)(hi ? hi : lo)) + (hi ? 0 : 32);
  const uint64_t m = ((a << ((lz - 1) & 63)) + 512u) >> 10;  // leading bit at 52
  uint64_t b = m + ((uint64_t)(uint32_t)(p + 1085 - lz) << 52);
  b = a ? b : 0;
  return __longlong_as_double((int64_t)(b | ((uint64_t)v & 0x8000000000000000ull)));
}

// The matrix's digit words of a lane and the sums' start values, and the three
// contractions of digit planes (dig_s: shared address; plane a, layer k, row
// g ^ k, word t) with it.  The sums still hold their start values' bits.
template <int NQ>
struct FxMul {
  static constexpr int D = kFxDigits, PLANE = FxShape<NQ>::PLANE;
  uint32_t kw[D];
  FxStart start1, start2, start12;
  int mrow, mmat;  // ldmatrix: row, matrix of this lane
  __device__ __forceinline__ FxMul(const uint32_t (*w)[32], int lane)
      : start1(kFxMagicBits, kFxMagicBits),
        start2(kFxMagic2Bits, kFxMagic2Bits),
        start12(kFxMagicBits, kFxMagic2Bits),
        mrow(lane & 7),
        mmat(lane >> 3) {
    set(w, lane);
  }
  __device__ __forceinline__ void set(const uint32_t (*w)[32], int lane) {
#pragma unroll
    for (int b = 0; b < D; ++b) kw[b] = __ldg(&w[b][lane]);
  }
  __device__ __forceinline__ uint32_t kd(int b) const { return b >= 0 ? kw[b < D ? b : 0] : 0u; }
  // A = the matrix for the orders o (rows 0-7) and o + 1 (rows 8-15) against
  // digits a, a + 1, B = f; nodes (2t, row g), (2t + 1, row g)
  __device__ __forceinline__ void rows(const uint32_t *f, uint32_t *s0, uint32_t *s1) const {
#pragma unroll
    for (int o = 0; o < D; o += 2) {
      float c[4];
      fx_mma0(c, kd(o), kd(o + 1), kd(o - 1), kd(o), f[0], f[1], o + 2 == D ? start12 : start1);
#pragma unroll
      for (int a = 2; a <= o; a += 2)
        fx_mma(c, kd(o - a), kd(o + 1 - a), kd(o - a - 1), kd(o - a), f[a], f[a + 1]);
      s0[o] = __float_as_uint(c[0]);
      s1[o] = __float_as_uint(c[1]);
      s0[o + 1] = __float_as_uint(c[2]);
      s1[o + 1] = __float_as_uint(c[3]);
    }
  }
  // along t, plane j: rows k of the digit planes, transposed (rows past Nq
  // repeat the last one; the matrix's digits are zero there).  Nodes k = g.
  __device__ __forceinline__ void along_t(uint32_t dig_s, int j, uint32_t *s0,
                                          uint32_t *s1) const {
    const int krow = mrow < NQ ? mrow : NQ - 1;
    uint32_t f[D];
    const uint32_t row = dig_s + (krow * 8 + (j ^ krow)) * 16;
    fx_ldsm4t(f, row + mmat * PLANE);
    fx_ldsm2t(f + 4, row + (4 + (mmat & 1)) * PLANE);
    rows(f, s0, s1);
  }
  // along s, layer k: the transposed layer.  Nodes j = g.
  __device__ __forceinline__ void along_s(uint32_t dig_s, int k, uint32_t *s0,
                                          uint32_t *s1) const {
    uint32_t f[D];
    const uint32_t row = dig_s + (k * 8 + (mrow ^ k)) * 16;
    fx_ldsm4t(f, row + mmat * PLANE);
    fx_ldsm2t(f + 4, row + (4 + (mmat & 1)) * PLANE);
    rows(f, s0, s1);
  }
  // along r, layers l0 and l1: A = digits a, a + 1 of l0 (rows 0-7) and l1, B =
  // the matrix transposed.  s: (l0, 2t), (l0, 2t + 1), (l1, 2t), (l1, 2t + 1).
  __device__ __forceinline__ void along_r(uint32_t dig_s, int l0, int l1,
                                          uint32_t (*s)[D]) const {
    uint32_t f[D / 2][4];
    const int kk = (mmat & 1) ? l1 : l0;
#pragma unroll
    for (int a = 0; a < D; a += 2)
      fx_ldsm4(f[a / 2], dig_s + (a + (mmat >> 1)) * PLANE + (kk * 8 + (mrow ^ kk)) * 16);
#pragma unroll
    for (int o = 0; o < D; ++o) {
      float c[4];
      fx_mma0(c, f[0][0], f[0][1], f[0][2], f[0][3], kd(o), kd(o - 1),
              o + 1 == D ? start2 : start1);
#pragma unroll
      for (int a = 2; a <= o; a += 2)
        fx_mma(c, f[a / 2][0], f[a / 2][1], f[a / 2][2], f[a / 2][3], kd(o - a), kd(o - a - 1));
#pragma unroll
      for (int n = 0; n < 4; ++n) s[n][o] = __float_as_uint(c[n]);
    }
  }
};

// The digits of a lane's values of layer k (times 2^pa, 2^pb) into the planes.
template <int NQ>
__device__ __forceinline__ void fx_store_digits(unsigned char *dig, int k, int g, int t, double a,
                                                double b, int emax, int pa = 0, int pb = 0) {
  const uint64_t x = fx_fixed(a, emax - pa), y = fx_fixed(b, emax - pb);
  uint32_t *p = reinterpret_cast<uint32_t *>(dig) + (k * 8 + (g ^ k)) * 4 + t;
  constexpr int PW = FxShape<NQ>::PLANE / 4;
  p[0 * PW] = fx_digit2<0>(x, y);
  p[1 * PW] = fx_digit2<1>(x, y);
  p[2 * PW] = fx_digit2<2>(x, y);
  p[3 * PW] = fx_digit2<3>(x, y);
  p[4 * PW] = fx_digit2<4>(x, y);
  p[5 * PW] = fx_digit2<5>(x, y);
}

// Exchange of the sums along t between the layout they arrive in (plane j,
// node k = g) and the owner's (j = g, layer k): 64-byte rows (j, k), in an
// order that lets writes (fixed j, all k) and reads (fixed k, all j) miss no
// bank.
template <int NQ>
__device__ __forceinline__ ulonglong2 *fx_xch(unsigned char *xch, int j, int k, int t) {
  const int kk = NQ == 8 ? (k ^ j) : k;
  return reinterpret_cast<ulonglong2 *>(xch + (j * NQ + kk) * 64 + t * 16);
}

// The element's largest exponent from the largest value of a lane (a high word of
// fx_size) and the low words of its values or'ed (`rest`: asked for only where all high
// words are zero); *zero: all values are.  col: a word per warp, and WPE further on
// another for that rare case.
template <int WPE, class Sync, class Rest>
__device__ __forceinline__ int fx_emax(uint32_t big, Rest rest, uint32_t *col, int warp, int lane,
                                       Sync sync, bool *zero) {
  big = __reduce_max_sync(0xffffffffu, big);
  if (WPE > 1) {
    if (lane == 0) col[warp] = big;
    sync();
#pragma unroll
    for (int w = 0; w < WPE; ++w) big = max(big, col[w]);
  }
  *zero = false;
  if (big == 0) {  // the same for all warps of the element
    bool some = __any_sync(0xffffffffu, rest() != 0);
    if (WPE > 1) {
      if (lane == 0) col[WPE + warp] = some;
      sync();
#pragma unroll
      for (int w = 0; w < WPE; ++w) some = some || col[WPE + w];
    }
    *zero = !some;
    return some ? 0 : 1023;
  }
  return (int)(big >> 20);
}
// Beyond the digits: not finite, or outside [2^-900, 2^900].
__device__ __forceinline__ bool fx_far(int emax) { return emax < 123 || emax > 1923; }

// The sums of the sizes of the terms at the nodes (2t, g), (2t + 1, g) of two layers (h0,
// h1: their sizes as of fx_sizes2; a: the matrix's), s[0], s[1] of the first layer, s[2],
// s[3] of the second: those along r, and added to them those along s.
__device__ __forceinline__ void fx_terms_r(float *s, uint32_t a, uint32_t h0, uint32_t h1) {
#pragma unroll
  for (int n = 0; n < 4; ++n) s[n] = 0.f;
  fx_mma8(s, h0, h1, a);  // layers x matrix
}
__device__ __forceinline__ void fx_terms_s(float *s, uint32_t a, uint32_t h0, uint32_t h1) {
  fx_mma(s, a, 0u, 0u, a, fx_trans(h0), fx_trans(h1));  // matrix x layers
}

// The FP64 sums of one node (i, j, k) of an element with values x[] in memory order:
// the scaled W^-1 D^T W D (OpTab::kh) along r, s and t.
template <int NQ>
__device__ __noinline__ double fx_direct(const double *x, const double *__restrict__ kh, int i,
                                         int j, int k) {
  double ar = 0.0, as = 0.0, at = 0.0;
#pragma unroll(NQ <= 8 ? NQ : 4)
  for (int m = 0; m < NQ; ++m) {
    ar = fma(kh[i * NQ + m], x[m + NQ * (j + NQ * k)], ar);
    as = fma(kh[j * NQ + m], x[i + NQ * (m + NQ * k)], as);
    at = fma(kh[k * NQ + m], x[i + NQ * (j + NQ * m)], at);
  }
  return (ar + as) + at;
}
// The same of a warp's list of `count` nodes, result(n, sum) on one lane each.  An FP64
// instruction takes the pipe 16 clocks however few lanes it serves, and a list is mostly
// short: up to 16 nodes go eight at a time, a lane for each of their three lines (at N = 7
// ten instructions for eight nodes instead of 26 for 32).
template <int NQ, class Result>
__device__ __forceinline__ void fx_direct_list(const double *x, const double *__restrict__ kh,
                                               const uint16_t *list, int count, int lane,
                                               Result result) {
  if (count > 16) {
    for (int q = lane; q < count; q += 32) {
      const int n = list[q];
      result(n, fx_direct<NQ>(x, kh, n % NQ, n / NQ % NQ, n / (NQ * NQ)));
    }
    return;
  }
  for (int q0 = 0; q0 < count; q0 += 8) {
    const int q = q0 + (lane >> 2), d = lane & 3;
    const int n = list[q < count ? q : q0], i = n % NQ, j = n / NQ % NQ, k = n / (NQ * NQ);
    const int row = d == 0 ? i : (d == 1 ? j : k);
    const int step = d == 0 ? 1 : (d == 1 ? NQ : NQ * NQ);
    const double *line = x + (n - row * step), *c = kh + row * NQ;
    double v = 0.0;
#pragma unroll(NQ <= 8 ? NQ : 4)
    for (int m = 0; m < NQ; ++m) v = fma(c[m], line[m * step], v);
    const double v1 = __shfl_down_sync(0xffffffffu, v, 1), v2 = __shfl_down_sync(0xffffffffu, v, 2);
    if (d == 0 && q < count) result(n, (v + v1) + v2);
  }
}

// The nodes whose bit b of `low` is set (b < n; node(b): the index in the element), one
// lane after the other, into a warp's list; how many.
template <class Node>
__device__ __forceinline__ int fx_list(uint32_t low, int n, int lane, uint16_t *list, Node node) {
  int count = 0;
  for (int b = 0; b < n; ++b) {
    const uint32_t m = __ballot_sync(0xffffffffu, (low >> b) & 1u);
    if ((low >> b) & 1u) list[count + __popc(m & ((1u << lane) - 1u))] = (uint16_t)node(b);
    count += __popc(m);
  }
  return count;
}

// out = A_L in on one element e, by the WPE warps that call it with their own
// first layer k0 (of L) and the same shared memory (dig; see FxShape); sync()
// is a barrier of these warps.  Other arguments as k_ax_local (FUSED
// likewise); vec: out (and, without GATHER_IN, in) is 16-byte aligned; slack: what
// FxTab::low is multiplied by (fx_slack).
template <int NQ, int L, bool GATHER_IN, bool FUSED, class Sync>
__device__ __forceinline__ void fx_element(int64_t e, int k0, const int32_t *__restrict__ ids,
                                           const double *__restrict__ in,
                                           double *__restrict__ out,
                                           const OpTab<double> *__restrict__ tab,
                                           const double *__restrict__ coef,
                                           double *__restrict__ outG, Acc<double> &acc, int vec,
                                           float slack, unsigned char *dig, Sync sync) {
  static_assert(!FUSED || GATHER_IN, "the fused operator reads its input through the map");
  using S = FxShape<NQ>;
  constexpr int NQ2 = NQ * NQ, NP = NQ * NQ2, D = kFxDigits, WPE = (NQ + L - 1) / L;
  constexpr bool EVEN = NQ % 2 == 0;
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  unsigned char *xch = dig + S::DIG;
  uint32_t *col = reinterpret_cast<uint32_t *>(xch + S::XCH);
  const uint32_t dig_s = (uint32_t)__cvta_generic_to_shared(dig);
  const bool on0 = g < NQ && 2 * t < NQ, on1 = g < NQ && 2 * t + 1 < NQ;
  const int64_t base = e * NP + (int64_t)k0 * NQ2 + g * NQ + 2 * t;
  auto layer = [&](int l) { return NQ % L == 0 || k0 + l < NQ; };
  // ---- the values of nodes (2t, g, k0 + l), (2t + 1, g, k0 + l), l < L
  double u0[L], u1[L];
  int32_t id0[GATHER_IN ? L : 1], id1[GATHER_IN ? L : 1];
  if (GATHER_IN) {
#pragma unroll
    for (int l = 0; l < L; ++l) {
      id0[l] = id1[l] = -1;
      if (EVEN) {
        if (on0 && layer(l)) {
          const int2 q = __ldcs(reinterpret_cast<const int2 *>(ids + base + l * NQ2));
          id0[l] = q.x;
          id1[l] = q.y;
        }
      } else {
        if (on0 && layer(l)) id0[l] = __ldcs(ids + base + l * NQ2);
        if (on1 && layer(l)) id1[l] = __ldcs(ids + base + l * NQ2 + 1);
      }
      if (!chk(FUSED ? bs_pred_fused_entry(id0[l], tab->ng) : bs_pred_map_entry(id0[l], tab->ng),
               BS_CHK_OP_ENTRY))
        id0[l] = -1;
      if (!chk(FUSED ? bs_pred_fused_entry(id1[l], tab->ng) : bs_pred_map_entry(id1[l], tab->ng),
               BS_CHK_OP_ENTRY))
        id1[l] = -1;
    }
#pragma unroll
    for (int l = 0; l < L; ++l) {
      if (FUSED) {
        u0[l] = id0[l] != -1 ? in[id0[l] >= 0 ? id0[l] : -2 - id0[l]] : 0.0;
        u1[l] = id1[l] != -1 ? in[id1[l] >= 0 ? id1[l] : -2 - id1[l]] : 0.0;
      } else {
        u0[l] = id0[l] >= 0 ? in[id0[l]] : 0.0;
        u1[l] = id1[l] >= 0 ? in[id1[l]] : 0.0;
      }
    }
  } else {
#pragma unroll
    for (int l = 0; l < L; ++l) {
      u0[l] = u1[l] = 0.0;
      if (EVEN && vec) {
        if (on0 && layer(l)) {
          const double2 q = __ldcs(reinterpret_cast<const double2 *>(in + base + l * NQ2));
          u0[l] = q.x;
          u1[l] = q.y;
        }
      } else {
        if (on0 && layer(l)) u0[l] = __ldcs(in + base + l * NQ2);
        if (on1 && layer(l)) u1[l] = __ldcs(in + base + l * NQ2 + 1);
      }
    }
  }
  // ---- the largest exponent, and the nodes the digits do not serve: bit 2l + h
  uint32_t big = 0, low = 0;
#pragma unroll
  for (int l = 0; l < L; ++l) big = max(big, max(fx_size(u0[l]), fx_size(u1[l])));
  auto rest = [&] {
    uint32_t r = 0;
#pragma unroll
    for (int l = 0; l < L; ++l) r |= (uint32_t)(__double2loint(u0[l]) | __double2loint(u1[l]));
    return r;
  };
  const int warp = k0 / L;
  bool zero;
  const int emax = fx_emax<WPE>(big, rest, col, warp, lane, sync, &zero);
  const bool far = fx_far(emax);
  bool some = far;  // of the element's nodes
  auto used = [&] {  // of the bits set in `low`, those of nodes whose results are used
#pragma unroll
    for (int n = 0; n < 2 * L; ++n) {
      bool use = (n & 1 ? on1 : on0) && layer(n / 2);
      if (GATHER_IN && use && (low >> n & 1u) && (n & 1 ? u1[n / 2] : u0[n / 2]) == 0.0) {
        const int32_t id = __ldg(ids + base + n / 2 * NQ2 + (n & 1));
        use = FUSED ? id != -1 : id >= 0;
      }
      if (!use) low &= ~(1u << n);
    }
  };
  if (far) {
    low = (1u << 2 * L) - 1u;
    used();
  } else {
    const uint32_t ka = __ldg(&tab->fx.a[lane]);
    const float least = zero ? 0.f : slack * tab->fx.low;  // zeros: the digits are exact
    // the terms along r mostly suffice (they are the lane's own fragments)
    float s[2 * L], m = INFINITY;
    uint32_t h[L];
#pragma unroll
    for (int l = 0; l < L; ++l) h[l] = fx_sizes2(u0[l], u1[l], emax);
#pragma unroll
    for (int l = 0; l < L; l += 2) fx_terms_r(s + 2 * l, ka, h[l], h[l + 1]);
#pragma unroll
    for (int n = 0; n < 2 * L; ++n)
      if ((n & 1 ? on1 : on0) && layer(n / 2)) m = fminf(m, s[n]);
    if (__any_sync(0xffffffffu, m < least)) {
#pragma unroll
      for (int l = 0; l < L; l += 2) fx_terms_s(s + 2 * l, ka, h[l], h[l + 1]);
#pragma unroll
      for (int n = 0; n < 2 * L; ++n) low |= s[n] < least ? 1u << n : 0u;
      used();
      some = __any_sync(0xffffffffu, low);
    }
  }
  const double ce = coef ? coef[e] : 1.0;
  auto store = [&](int l, double r0, double r1, int32_t i0, int32_t i1, double v0, double v1) {
    if (FUSED) {
      auto one = [&](double r, int32_t id, double u, int h) {
        if (id >= 0) {
          __stcs(out + base + l * NQ2 + h, r);
        } else if (id != -1) {
          const double v = plus_zero(r);
          __stcs(outG + (-2 - id), v);
          if (!(low >> (2 * l + h) & 1u)) acc.add(u, v);
        }
      };
      if (on0) one(r0, i0, v0, 0);
      if (on1) one(r1, i1, v1, 1);
    } else if (EVEN && vec) {
      if (on0) __stcs(reinterpret_cast<double2 *>(out + base + l * NQ2), make_double2(r0, r1));
    } else {
      if (on0) __stcs(out + base + l * NQ2, r0);
      if (on1) __stcs(out + base + l * NQ2 + 1, r1);
    }
  };
  // the element's values in memory order, over the digits once those are done with
  double *x = reinterpret_cast<double *>(dig);
  auto keep = [&](int l) {
    const int n = 2 * t + NQ * (g + NQ * (k0 + l));
    if (on0) x[n] = u0[l];
    if (on1) x[n + 1] = u1[l];
  };
  if (!far) {
#pragma unroll
    for (int l = 0; l < L; ++l) {
      if (!layer(l)) break;
      fx_store_digits<NQ>(dig, k0 + l, g, t, u0[l], u1[l], emax);
    }
    const FxMul<NQ> mul(tab->fx.w, lane);
    sync();
    // ---- along t, planes j = k0 + l (the start values come off along r and s)
#pragma unroll
    for (int l = 0; l < L; ++l) {
      if (!layer(l)) break;
      uint32_t s0[D], s1[D];
      mul.along_t(dig_s, k0 + l, s0, s1);
      if (NQ == 8 || g < NQ)
        *fx_xch<NQ>(xch, k0 + l, g, t) = make_ulonglong2(fx_join(s0), fx_join(s1));
    }
    // ---- along r and s, two layers at a time
    uint64_t T0[L], T1[L];
#pragma unroll
    for (int l = 0; l < L; l += 2) {
      if (!layer(l)) break;
      const int l0 = k0 + l, l1 = l0 + 1 < NQ ? l0 + 1 : l0;  // odd Nq: the last layer twice
      uint32_t s[4][D];
      mul.along_r(dig_s, l0, l1, s);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        uint32_t s0[D], s1[D];
        mul.along_s(dig_s, h ? l1 : l0, s0, s1);
#pragma unroll
        for (int o = 0; o < D; ++o) {
          const uint32_t off = 3u * (o == D - 1 ? kFxMagic2Bits : kFxMagicBits);
          s[2 * h][o] += s0[o] - off;
          s[2 * h + 1][o] += s1[o] - off;
        }
        T0[l + h] = fx_join(s[2 * h]);
        T1[l + h] = fx_join(s[2 * h + 1]);
      }
    }
    if (WPE > 1 && lane == 0) col[2 * WPE + warp] = some;
    sync();
    if (WPE > 1)
#pragma unroll
      for (int w = 0; w < WPE; ++w) some = some || col[2 * WPE + w];
    // (ahead of the results with two warps an element, along with them with one: 2 us of
    // 273 at Nq = 8, 4 of 279 at Nq = 5 the other way round)
    if (WPE > 1 && some)
#pragma unroll
      for (int l = 0; l < L; ++l)
        if (layer(l)) keep(l);
    // ---- results: w_i w_j w_k (c h/2 sum + lambda (h/2)^3 u), the weights'
    // products from tables; sum = T 2^60 2^-q 2^(emax - 1080)
    const int p2 = emax - 1020 - tab->fx.q;
    // (two loops, not a select per node: a product by 1 costs the FP64 pipe
    // as much as any)
    auto results = [&](auto with_coef) {
#pragma unroll
      for (int l = 0; l < L; ++l) {
        if (!layer(l)) break;
        const int k = k0 + l;
        ulonglong2 v = make_ulonglong2(0, 0);
        if (NQ == 8 || g < NQ) v = *fx_xch<NQ>(xch, g, k, t);
        double d0 = fx_double((int64_t)(T0[l] + v.x), p2);
        double d1 = fx_double((int64_t)(T1[l] + v.y), p2);
        const double2 wg = __ldg(reinterpret_cast<const double2 *>(tab->fx.wg) + k * 32 + lane);
        const double2 wm = __ldg(reinterpret_cast<const double2 *>(tab->fx.wm) + k * 32 + lane);
        if (decltype(with_coef)::value) {
          d0 = ce * d0;
          d1 = ce * d1;
        }
        if (WPE == 1 && some) keep(l);
        store(l, fma(wg.x, d0, wm.x * u0[l]), fma(wg.y, d1, wm.y * u1[l]),
              id0[GATHER_IN ? l : 0], id1[GATHER_IN ? l : 0], u0[l], u1[l]);
      }
    };
    if (coef)
      results(std::true_type{});
    else
      results(std::false_type{});
  } else {
#pragma unroll
    for (int l = 0; l < L; ++l)
      if (layer(l)) keep(l);
  }
  if (!some) return;
  // ---- the FP64 sums of the nodes in `low`, over what the digits gave, 32 nodes of
  // the warp's at a time
  sync();  // the exchanged sums have been read
  uint16_t *list = reinterpret_cast<uint16_t *>(xch) + k0 * NQ2;
  const int count = fx_list(low, 2 * L, lane, list, [&](int b) {
    return 2 * t + (b & 1) + NQ * (g + NQ * (k0 + (b >> 1)));
  });
  sync();
  fx_direct_list<NQ>(x, tab->kh, list, count, lane, [&](int n, double d) {
    const int i = n % NQ, j = n / NQ % NQ, k = n / NQ2;
    const int own = (k * 32 + j * 4 + (i >> 1)) * 2 + (i & 1);  // the owner's table entry
    const double u = x[n];
    const double r = fma(tab->fx.wg[own], coef ? ce * d : d, tab->fx.wm[own] * u);
    int32_t id = 0;
    if (FUSED) {
      id = ids[e * NP + n];
      if (!chk(bs_pred_fused_entry(id, tab->ng), BS_CHK_OP_ENTRY)) id = -1;
    }
    if (id >= 0) {
      __stcs(out + e * NP + n, r);
    } else if (id != -1) {
      const double v = plus_zero(r);
      __stcs(outG + (-2 - id), v);
      acc.add(u, v);
    }
  });
}

template <int NQ, bool GATHER_IN, bool FUSED>
__global__ void __launch_bounds__(FxShape<NQ>::THREADS, FxShape<NQ>::BLOCKS)
    k_ax_fx(int64_t E, const int32_t *__restrict__ order, const int32_t *__restrict__ ids,
            const double *__restrict__ in, double *__restrict__ out,
            const OpTab<double> *__restrict__ tab, const double *__restrict__ coef,
            const CgState *st, double *__restrict__ outG, double *__restrict__ partials,
            int vec, float slack) {
  using S = FxShape<NQ>;
  extern __shared__ __align__(128) unsigned char fx_smem[];
  if (cg_halted(st)) return;
  Acc<double> acc;
  const int64_t slot = blockIdx.x;
  int64_t e = slot < E ? (order ? (int64_t)order[slot] : slot) : -1;
  if (e >= 0 && !chk(bs_pred_index(e, tab->ne), BS_CHK_OP_ENTRY)) e = -1;
  if (e >= 0)
    fx_element<NQ, S::L, GATHER_IN, FUSED>(e, (int)(threadIdx.x / 32) * S::L, ids, in, out, tab,
                                           coef, outG, acc, vec, slack, fx_smem, [] {
                                             if (S::WPE == 1)
                                               __syncwarp();
                                             else
                                               __syncthreads();
                                           });
  if (FUSED && partials) {
    const double part = block_sum<S::THREADS>(acc.value());
    if (threadIdx.x == 0) partials[blockIdx.x] = part;
  }
}

}  // namespace bs
