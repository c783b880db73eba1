// bs_gemm_s.cuh -- the network's GEMMs at the sizes of one training batch:
// C[M x N] = A[M x K] B[N x K]^T as in bs_mlp.cu, on small tiles, with either
// operand also readable as stored transposed ([K x M], [K x N]).
//
// A batch of 256 rows of a degree-5 element (D = 216, H = 256) is four 128 x 128
// tiles: four SMs, each waiting 21 times in turn for a 32-wide K step (35 us
// for the hidden layer, 136 us for a training step of 14 launches).  Here a
// block of four warps takes a 32 x 32 tile (64 x 64 where those fill the chip
// twice over), K in 64-wide chunks through a ring of cp.async stages deep
// enough that a batch's whole K is in flight after the first wait.  Transposed
// operands are read by ldmatrix.trans, which takes out the transposes; the
// loss and Adam with the refreshed bf16 operands are epilogues (their operands
// loaded ahead of the products), and the two weight gradients share a launch.
// A training step is five launches.  Products are summed over the same 16-wide K
// blocks in the same order as in the large kernel, so activations and gradients
// are bitwise the same; the loss is summed tile by tile and differs from k_mse's
// in its last bits.
#pragma once

#include "bs_mlp.cuh"

namespace bs {

enum {
  EPI_MSE = 10,  // e = acc - target: dY = bf16(2 e / (B D)), loss = mean e^2
  EPI_ADAM = 11  // acc = dL/dW[m][n]: Adam on W and its bf16 operand
};

struct TrainArgs {
  const float *target;          // EPI_MSE: [M x D]
  int D;
  double *partials, *loss;
  unsigned int *counter;
  float *w, *m1, *m2;           // EPI_ADAM: master and moments [M x N]
  __nv_bfloat16 *wb;            // operand rows [hi] or [hi | lo | hi]
  int split;
  float lr, b1, b2, eps, c1, c2;
};

// Adam (Kingma & Ba 2015) on one weight; c1 = 1 - b1^t, c2 = 1 - b2^t.
__device__ __forceinline__ float adam_step(float w, float g, float &m, float &v,
                                           const TrainArgs &a) {
  m = a.b1 * m + (1.0f - a.b1) * g;
  v = a.b2 * v + (1.0f - a.b2) * g * g;
  return w - a.lr * (m / a.c1) / (sqrtf(v / a.c2) + a.eps);
}

// One or two products of a launch (blockIdx.z).
struct GsArgs {
  GemmArgs g[2];
  TrainArgs t[2];
};

// A weight's entry in its operand: row of `n` columns, [hi] or [hi | lo | hi].
__device__ __forceinline__ void store_weight(__nv_bfloat16 *wb, int64_t row, int col, int n,
                                             int split, float w) {
  __nv_bfloat16 hi, lo;
  bf16_split(w, hi, lo);
  __nv_bfloat16 *p = wb + row * (split ? 3 * n : n) + col;
  p[0] = hi;
  if (split) {
    p[n] = lo;
    p[2 * n] = hi;
  }
}

constexpr int kGsThreads = 128, kGsK = 64;
template <int WT>
struct GsShape {
  static constexpr int BT = 2 * WT;                        // block tile (both ways)
  static constexpr int STAGES = WT == 16 ? 6 : 4;
  static constexpr int LDN = kGsK + 8, LDT = BT + 8;       // row lengths: as is, transposed
  static constexpr int OP = BT * LDN > kGsK * LDT ? BT * LDN : kGsK * LDT;  // values
  static constexpr int SMEM = STAGES * 2 * OP * 2;
};

__device__ __forceinline__ void gs_cp16(void *smem, const void *gmem, int bytes) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(s), "l"(gmem), "r"(bytes)
               : "memory");
}
template <bool T>
__device__ __forceinline__ void gs_ldsm4(uint32_t *r, const void *smem) {
  const unsigned s = (unsigned)__cvta_generic_to_shared(smem);
  if (T)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(s)
                 : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(s)
                 : "memory");
}
__device__ __forceinline__ void gs_mma(float *c, const uint32_t *a, const uint32_t *b) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
      "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// AT / BT: the operand is stored [K x M] / [K x N] (row length lda / ldb).
// M and N are multiples of 8 where transposed, K a multiple of 8.
template <int EPI, bool AT, bool BT, int WT>
__global__ void __launch_bounds__(kGsThreads) k_gemm_s(const __grid_constant__ GsArgs args) {
  using S = GsShape<WT>;
  const GemmArgs &g = args.g[blockIdx.z];
  const TrainArgs &ta = args.t[blockIdx.z];
  constexpr int MT = WT / 16, NT = WT / 8;
  extern __shared__ __align__(16) unsigned char gs_smem[];
  __nv_bfloat16 *sm = reinterpret_cast<__nv_bfloat16 *>(gs_smem);
  if (cg_halted(g.st)) return;
  const int64_t m0 = (int64_t)blockIdx.y * S::BT;
  const int n0 = blockIdx.x * S::BT;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int wm = (warp >> 1) * WT, wn = (warp & 1) * WT;
  if (m0 >= g.M || n0 >= g.N) return;  // the smaller of two products
  // one operand's chunk: rows r0.. of `rows`, columns k0.. of K
  auto load_op = [&](auto trans, __nv_bfloat16 *dst, const __nv_bfloat16 *src, int ld, int64_t r0,
                     int64_t rows, int k0) {
    if (decltype(trans)::value) {
      constexpr int CH = S::BT / 8;
#pragma unroll
      for (int c = tid; c < kGsK * CH; c += kGsThreads) {
        const int k = c / CH, q = (c % CH) * 8;
        const bool ok = k0 + k < g.K && r0 + q < rows;
        gs_cp16(dst + k * S::LDT + q, src + (ok ? (int64_t)(k0 + k) * ld + r0 + q : 0),
                ok ? 16 : 0);
      }
    } else {
      constexpr int CH = kGsK / 8;
#pragma unroll
      for (int c = tid; c < S::BT * CH; c += kGsThreads) {
        const int r = c / CH, q = (c % CH) * 8;
        const bool ok = r0 + r < rows && k0 + q < g.K;
        gs_cp16(dst + r * S::LDN + q, src + (ok ? (r0 + r) * ld + k0 + q : 0), ok ? 16 : 0);
      }
    }
  };
  auto load = [&](int chunk) {
    __nv_bfloat16 *a = sm + (chunk % S::STAGES) * 2 * S::OP, *b = a + S::OP;
    load_op(std::integral_constant<bool, AT>{}, a, g.A, g.lda, m0, g.M, chunk * kGsK);
    load_op(std::integral_constant<bool, BT>{}, b, g.B, g.ldb, n0, g.N, chunk * kGsK);
  };
  float acc[MT][NT][4];
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[i][j][k] = 0.f;
  const int nk = (g.K + kGsK - 1) / kGsK;
#pragma unroll
  for (int c = 0; c < S::STAGES - 1; ++c) {
    if (c < nk) load(c);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
  }
  // what the training epilogues read, a pair of columns at a time, ahead of the
  // products (the small tile; columns n, n + 1 are both inside: N is even)
  const int gq = lane >> 2, tq = lane & 3;
  constexpr bool PRE = WT == 16 && (EPI == EPI_MSE || EPI == EPI_ADAM);
  float2 pw[PRE ? MT * 2 * NT : 1], p1[PRE && EPI == EPI_ADAM ? MT * 2 * NT : 1],
      p2[PRE && EPI == EPI_ADAM ? MT * 2 * NT : 1];
  auto fetch = [&](int64_t m, int n, float2 &w, float2 &a, float2 &b) {
    if constexpr (EPI == EPI_MSE) {
      w.x = n < ta.D ? ta.target[m * ta.D + n] : 0.f;
      w.y = n + 1 < ta.D ? ta.target[m * ta.D + n + 1] : 0.f;
    } else if constexpr (EPI == EPI_ADAM) {
      const int64_t o = m * g.ldc + n;
      w = *reinterpret_cast<const float2 *>(ta.w + o);
      a = *reinterpret_cast<const float2 *>(ta.m1 + o);
      b = *reinterpret_cast<const float2 *>(ta.m2 + o);
    }
  };
  if constexpr (PRE) {
#pragma unroll
    for (int i = 0; i < MT * 2 * NT; ++i) {
      const int64_t m = m0 + wm + (i / (2 * NT)) * 16 + gq + 8 * (i / NT % 2);
      const int n = n0 + wn + (i % NT) * 8 + 2 * tq;
      if (m < g.M && n < g.N)
        fetch(m, n, pw[i], p1[EPI == EPI_ADAM ? i : 0], p2[EPI == EPI_ADAM ? i : 0]);
    }
  }
  for (int kt = 0; kt < nk; ++kt) {
    asm volatile("cp.async.wait_group %0;\n" ::"n"(S::STAGES - 2) : "memory");
    __syncthreads();  // chunk kt has landed; everyone is done with chunk kt - 1
    if (kt + S::STAGES - 1 < nk) load(kt + S::STAGES - 1);
    asm volatile("cp.async.commit_group;\n" ::: "memory");
    const __nv_bfloat16 *sa = sm + (kt % S::STAGES) * 2 * S::OP, *sb = sa + S::OP;
#pragma unroll
    for (int kk = 0; kk < kGsK; kk += 16) {
      if (kt * kGsK + kk >= g.K) break;  // as the large kernel: no products of padding
      uint32_t af[MT][4], bf[NT][2];
#pragma unroll
      for (int i = 0; i < MT; ++i)
        gs_ldsm4<AT>(af[i], AT ? sa + (kk + (lane & 7) + ((lane >> 4) & 1) * 8) * S::LDT + wm +
                                     i * 16 + ((lane >> 3) & 1) * 8
                               : sa + (wm + i * 16 + (lane & 15)) * S::LDN + kk + (lane >> 4) * 8);
#pragma unroll
      for (int j = 0; j < NT / 2; ++j) {
        uint32_t r[4];
        gs_ldsm4<BT>(r, BT ? sb + (kk + (lane & 7) + ((lane >> 3) & 1) * 8) * S::LDT + wn + j * 16 +
                                 ((lane >> 4) & 1) * 8
                           : sb + (wn + j * 16 + (lane & 7) + ((lane >> 4) << 3)) * S::LDN + kk +
                                 ((lane >> 3) & 1) * 8);
        bf[2 * j][0] = r[0];
        bf[2 * j][1] = r[1];
        bf[2 * j + 1][0] = r[2];
        bf[2 * j + 1][1] = r[3];
      }
#pragma unroll
      for (int i = 0; i < MT; ++i)
#pragma unroll
        for (int j = 0; j < NT; ++j) gs_mma(acc[i][j], af[i], bf[j]);
    }
  }
  asm volatile("cp.async.wait_group 0;\n" ::: "memory");
  double loss = 0.0;
  const float sc = EPI == EPI_MSE ? (float)(2.0 / ((double)g.M * ta.D)) : 0.f;
#pragma unroll
  for (int i = 0; i < MT; ++i)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t m = m0 + wm + i * 16 + gq + 8 * h;
      if (m >= g.M) continue;
      const int32_t *idrow = nullptr;
      if (EPI == EPI_SCATTER_F64) {
        const int64_t em = g.order ? g.order[m] : m;
        idrow = chk(bs_pred_index(em, g.M), BS_CHK_PREC_ENTRY) ? g.ids + em * g.np : nullptr;
      }
#pragma unroll
      for (int j = 0; j < NT; ++j) {
        const int n = n0 + wn + j * 8 + 2 * tq, pi = (i * 2 + h) * NT + j;
        const float v0 = acc[i][j][2 * h], v1 = acc[i][j][2 * h + 1];
        if constexpr (EPI == EPI_MSE || EPI == EPI_ADAM) {
          if (n >= g.N) continue;
          float2 w, a, b;
          if constexpr (PRE) {
            w = pw[pi];
            a = p1[EPI == EPI_ADAM ? pi : 0];
            b = p2[EPI == EPI_ADAM ? pi : 0];
          } else {
            fetch(m, n, w, a, b);
          }
          if constexpr (EPI == EPI_MSE) {
            __nv_bfloat162 d = __floats2bfloat162_rn(0.f, 0.f);
            if (n < ta.D) {
              const float e = v0 - w.x;
              loss = fma((double)e, (double)e, loss);
              d.x = __float2bfloat16_rn(sc * e);
            }
            if (n + 1 < ta.D) {
              const float e = v1 - w.y;
              loss = fma((double)e, (double)e, loss);
              d.y = __float2bfloat16_rn(sc * e);
            }
            *reinterpret_cast<__nv_bfloat162 *>(g.out_b16 + m * g.ldc + n) = d;
          } else {
            const int64_t o = m * g.ldc + n;
            w.x = adam_step(w.x, v0, a.x, b.x, ta);
            w.y = adam_step(w.y, v1, a.y, b.y, ta);
            *reinterpret_cast<float2 *>(ta.m1 + o) = a;
            *reinterpret_cast<float2 *>(ta.m2 + o) = b;
            *reinterpret_cast<float2 *>(ta.w + o) = w;
            store_weight(ta.wb, m, n, g.N, ta.split, w.x);
            store_weight(ta.wb, m, n + 1, g.N, ta.split, w.y);
          }
        } else {
          if (n < g.N) gemm_store<EPI>(g, m, n, v0, idrow);
          if (n + 1 < g.N) gemm_store<EPI>(g, m, n + 1, v1, idrow);
        }
      }
    }
  if constexpr (EPI == EPI_MSE) {
    const double part = block_sum<kGsThreads>(loss);
    const unsigned nb = gridDim.x * gridDim.y;
    __shared__ bool s_last;
    if (tid == 0) {
      ta.partials[blockIdx.y * gridDim.x + blockIdx.x] = part;
      __threadfence();
      s_last = atomicAdd(ta.counter, 1u) == nb - 1;
    }
    __syncthreads();
    if (!s_last) return;
    __threadfence();
    double v = 0.0;
    for (unsigned b = tid; b < nb; b += kGsThreads) v = v + __ldcg(ta.partials + b);
    v = block_sum<kGsThreads>(v);
    if (tid == 0) {
      *ta.loss = v / ((double)g.M * ta.D);
      *ta.counter = 0u;
    }
  }
}

// Blocks of the 32 x 32 (or 64 x 64) form.
inline int64_t gs_blocks(int64_t M, int N, int bt) {
  return ((M + bt - 1) / bt) * ((N + bt - 1) / bt);
}

// The tile of a launch: 64 x 64 tiles read half as much per product, once
// there are enough of them.
inline int gs_tile(int64_t M, int N, int sms) { return gs_blocks(M, N, 64) >= 2 * sms ? 64 : 32; }

// args.g[0], and args.g[1] when two (of about the same size).
template <int EPI, bool AT, bool BT>
int launch_gemm_s(const GsArgs &args, int two, cudaStream_t s) {
  DeviceInfo di;
  if (int rc = device_info(&di)) return rc;
  int64_t M = args.g[0].M;
  int N = args.g[0].N;
  if (two) {
    M = M > args.g[1].M ? M : args.g[1].M;
    N = N > args.g[1].N ? N : args.g[1].N;
  }
  auto run = [&](auto kern, int bt, int smem) -> int {
    if (occupancy_blocks_smem((const void *)kern, kGsThreads, smem) < 1)
      return fail(BS_ERR_CUDA, "gemm: %d B of shared memory refused", smem);
    const int64_t gy = (M + bt - 1) / bt;
    if (gy > 65535) return fail(BS_ERR_ARG, "gemm: M too large");
    kern<<<dim3((unsigned)((N + bt - 1) / bt), (unsigned)gy, two ? 2 : 1), kGsThreads, smem, s>>>(
        args);
    BS_LAUNCH_CHECK();
    return BS_OK;
  };
  if (gs_tile(M, N, di.sms) == 64)
    return run(k_gemm_s<EPI, AT, BT, 32>, GsShape<32>::BT, GsShape<32>::SMEM);
  return run(k_gemm_s<EPI, AT, BT, 16>, GsShape<16>::BT, GsShape<16>::SMEM);
}
template <int EPI, bool AT, bool BT>
int launch_gemm_s(const GemmArgs &a, const TrainArgs &t, cudaStream_t s) {
  GsArgs args{};
  args.g[0] = a;
  args.t[0] = t;
  return launch_gemm_s<EPI, AT, BT>(args, 0, s);
}

}  // namespace bs
