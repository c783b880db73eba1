// bs_op.cu -- GLL tables (host), problem objects and the C ABI of the
// operator A = Z^T (c S_L + lambda M_L) Z (eqs. global_system,
// assembled_stiff, assembled_mass).
#include <cmath>
#include <cstdlib>
#include <cstring>
#include <algorithm>
#include <thread>
#include <vector>

#include "bs_op_ff.cuh"

namespace bs {

int g_op_fusion = 0;
int g_op_evenodd = 1;

// GLL nodes on [-1, 1] (Sec. 2, eq. basis): the N+1 zeros of (1 - x^2) P_N'(x).
// Newton on the Legendre-Vandermonde recurrence
//   x <- x - (x P_N(x) - P_{N-1}(x)) / ((N + 1) P_N(x)),
// started from the Chebyshev-Lobatto points cos(pi i / N), converges to all
// N+1 nodes, endpoints included.  Weights 2 / (N (N+1) P_N(x_i)^2).  The
// derivative matrix D[a][i] = l_i'(x_a) comes from barycentric weights
// b_j = 1 / prod_{k != j} (x_j - x_k):
//   D[a][i] = (b_i / b_a) / (x_a - x_i)  (a != i),  D[a][a] = -sum_{i != a} D[a][i].
static void gll_tables(int N, double *x, double *w, double *D) {
  const int Nq = N + 1;
  const double pi = 3.141592653589793238462643383279502884;
  std::vector<double> P((size_t)Nq * Nq);
  for (int i = 0; i <= N; ++i) x[i] = std::cos(pi * (N - i) / N);  // ascending
  for (int it = 0; it < 200; ++it) {
    double change = 0.0;
    for (int i = 0; i <= N; ++i) {
      double p0 = 1.0, p1 = x[i];
      for (int k = 2; k <= N; ++k) {
        const double p2 = ((2.0 * k - 1.0) * x[i] * p1 - (k - 1.0) * p0) / k;
        p0 = p1;
        p1 = p2;
      }
      // p1 = P_N, p0 = P_{N-1}
      const double dx = (x[i] * p1 - p0) / (Nq * p1);
      x[i] -= dx;
      change = std::fmax(change, std::fabs(dx));
    }
    if (change < 1e-16) break;
  }
  for (int i = 0; i <= N / 2; ++i) {  // exact symmetry
    const double s = 0.5 * (x[N - i] - x[i]);
    x[i] = -s;
    x[N - i] = s;
  }
  if (N % 2 == 0) x[N / 2] = 0.0;
  for (int i = 0; i <= N; ++i) {
    double p0 = 1.0, p1 = x[i];
    for (int k = 2; k <= N; ++k) {
      const double p2 = ((2.0 * k - 1.0) * x[i] * p1 - (k - 1.0) * p0) / k;
      p0 = p1;
      p1 = p2;
    }
    w[i] = 2.0 / (N * (N + 1.0) * p1 * p1);
  }
  std::vector<double> b(Nq, 1.0);
  for (int j = 0; j <= N; ++j) {
    for (int k = 0; k <= N; ++k)
      if (k != j) b[j] *= (x[j] - x[k]);
    b[j] = 1.0 / b[j];
  }
  for (int a = 0; a <= N; ++a) {
    double diag = 0.0;
    for (int i = 0; i <= N; ++i) {
      if (i == a) continue;
      const double v = (b[i] / b[a]) / (x[a] - x[i]);
      D[a * Nq + i] = v;
      diag -= v;
    }
    D[a * Nq + a] = diag;
  }
}

// K = D^T W D, the 1-D stiffness on [-1, 1].
static void stiffness_1d(int N, const double *w, const double *D, double *K) {
  const int Nq = N + 1;
  for (int i = 0; i < Nq; ++i)
    for (int m = 0; m < Nq; ++m) {
      double s = 0.0;
      for (int a = 0; a < Nq; ++a) s = std::fma(D[a * Nq + i] * w[a], D[a * Nq + m], s);
      K[i * Nq + m] = s;
    }
}

// A double-double value (hi + lo), for the tables that need more than 53 bits
// (Dekker's and Knuth's error-free transformations, std::fma for products).
struct DD {
  double h, l;
  DD(double a = 0.0, double b = 0.0) : h(a), l(b) {}
};
static DD dd_fast(double a, double b) {
  const double s = a + b;
  return DD(s, b - (s - a));
}
static DD operator+(DD a, DD b) {
  const double s = a.h + b.h, t = s - a.h;
  const double e = (a.h - (s - t)) + (b.h - t);
  return dd_fast(s, e + (a.l + b.l));
}
static DD operator-(DD a) { return DD(-a.h, -a.l); }
static DD operator-(DD a, DD b) { return a + (-b); }
static DD operator*(DD a, DD b) {
  const double p = a.h * b.h;
  return dd_fast(p, std::fma(a.h, b.h, -p) + (a.h * b.l + a.l * b.h));
}
static DD operator/(DD a, DD b) {
  const double q = a.h / b.h;
  const DD r = a - b * DD(q);
  return dd_fast(q, (r.h + r.l) / b.h);
}

// v (|v| < 2^15) as the bits of a half, rounded to nearest.
static uint32_t half_bits(double v) {
  const uint32_t sign = v < 0 ? 0x8000u : 0u;
  const double a = std::fabs(v);
  int e = 0;
  std::frexp(a, &e);  // a in [2^(e-1), 2^e)
  if (a == 0.0 || e < -13) return sign | (uint32_t)std::rint(std::ldexp(a, 24));  // subnormal
  return sign | (((uint32_t)(e + 13) << 10) + (uint32_t)std::rint(std::ldexp(a, 11 - e)));
}

// A matrix in digits (bs_op_fx.cuh): each entry times a scale s 2^q, the largest near
// 511 2^50 (the first digit then uses its range, and what the digit products leave out
// is smallest against the entries), as an integer, the diagonal minus the rest of its
// row where the rows sum to zero, then signed 10-bit digits by the bias of 512 per
// digit that the kernels use for their values, as the bits of a half.  The scale is the
// largest, in steps, for which no sum of products can leave its accumulator; false
// where there is none (there is, for the matrices of degrees 2..15).
// word(b, i, m, bits): the digits b of entries (i, m), (i, m + 1), m even; b =
// kFxDigits: the entries' sizes, over 2^*e.
// *low: with the digits that fall off taken as independent and uniform, an entry of
// `dirs` such sums is off by 4 standard deviations at most (1 in 16000; the joins'
// rounding and that of the values included).  Where the sum of the sizes of its terms,
// in units of 2^*e and the power of two of the element's largest value, is *low, that
// is `allow` 2^-53 of it.
template <class M, class W>
static bool fx_digits(int Nq, M mat, bool zero_rows, int dirs, double allow, W word, double *s,
                      int *q, float *low) {
  double big = 0.0;
  for (int i = 0; i < Nq; ++i)
    for (int m = 0; m < Nq; ++m) big = std::fmax(big, std::fabs(mat(i, m).h));
  int64_t Ki[kMaxNq][kMaxNq] = {};
  int64_t bias = 0;
  for (int d = 0; d < kFxDigits; ++d) bias += (int64_t)512 << (10 * d);
  auto digit = [&](int i, int m, int d) {
    return (int)(((bias + Ki[i][m]) >> (10 * (kFxDigits - 1 - d))) & 0x3ff) - 512;
  };
  // the largest sum an accumulator can meet: digits of a value up to 257
  // (the first) or 512 in magnitude, products a + b = o of one row; beyond
  // kFxMaxNq those of digits 2 and 3 have an accumulator of their own (o >= 3)
  auto fits = [&] {
    for (int o = 0; o < kFxDigits; ++o)
      for (int i = 0; i < Nq; ++i) {
        int64_t t[2] = {0, 0};
        for (int a = 0; a <= o; ++a)
          for (int m = 0; m < Nq; ++m)
            t[Nq > kFxMaxNq && o >= 3 && (a == 2 || a == 3)] +=
                (a ? 512 : 257) * std::abs(digit(i, m, o - a));
        // the last order counts by two, but for degrees 2 and 3
        const int64_t most = o == kFxDigits - 1 && Nq >= kFxMinNq ? 1 << 23 : 1 << 22;
        if (t[0] > most || t[1] > most) return false;
      }
    return true;
  };
  double scale = 0.0;
  bool ok = false;
  for (int step = 0; step < 96 && !ok; ++step) {
    scale = std::ldexp(511.0 * (1.0 - step / 128.0), 50) / big;
    for (int i = 0; i < Nq; ++i) {
      int64_t rest = 0;
      for (int m = 0; m < Nq; ++m) {
        const DD v = mat(i, m) * DD(scale);
        const double n = std::rint(v.h);
        Ki[i][m] = (int64_t)n + (int64_t)std::rint((v.h - n) + v.l);
        if (m != i) rest += Ki[i][m];
      }
      if (zero_rows) Ki[i][i] = -rest;
    }
    ok = fits();
  }
  if (!ok) return false;
  *q = std::ilogb(scale);
  *s = std::ldexp(scale, -*q);
  // variance of one sum in units of 2^60 of the integer products: the products a + b = 6
  // (digits uniform in +-512: 2^18 / 3) at 2^-20 each, the last places of the value and
  // of the matrix, the join (1/12)
  double var = 0.0;
  for (int i = 0; i < Nq; ++i) {
    double d = 0.0, v = 0.0;
    for (int m = 0; m < Nq; ++m) {
      for (int b = 1; b < kFxDigits; ++b) d += (double)digit(i, m, b) * digit(i, m, b);
      v += std::ldexp((double)Ki[i][m], -60) * std::ldexp((double)Ki[i][m], -60);
    }
    var = std::fmax(var, d * std::ldexp(1.0, 18 - 40) / 3 + v / 12);
  }
  const double sigma = std::sqrt(dirs * (var + 1.0 / 12 + 0.01 * Nq));
  int e = 0;
  std::frexp(big, &e);  // big < 2^e
  // 4 sigma 2^60 / scale in units of the value's 2^-57, against allow 2^-53 low 2^e
  *low = (float)(4.0 * sigma * std::ldexp(1.0, 60 - 57 + 53 - e) / (allow * scale));
  for (int d = 0; d <= kFxDigits; ++d)
    for (int i = 0; i < Nq; ++i)
      for (int m = 0; m < Nq; m += 2) {
        auto bits = [&](int mm) -> uint32_t {
          if (mm >= Nq) return 0;
          return half_bits(d < kFxDigits ? (double)digit(i, mm, d)
                                         : std::ldexp(std::fabs(mat(i, mm).h), -e));
        };
        word(d, i, m, bits(m) | bits(m + 1) << 16);
      }
  return true;
}

// The digits of Kh = W^-1 K and, up to degree 7, D and D^T (bs_op_fx.cuh,
// bs_op_fx16.cuh, bs_op_fx4.cuh, bs_op_geo_fx.cuh), from GLL nodes, weights and derivative matrix redone in double-double (Newton on the
// nodes x, as gll_tables): a 58-bit entry holds more than a double, and an
// error common to every element would shift the operator's low modes
// coherently.  Also the weights' products of the affine kernel.
static bool fx_table(int N, const double *x0, double h, double lambda, OpTab<double> *tab) {
  FxTab *t = &tab->fx;
  FxGeoTab *tg = &tab->fxg;
  FxTab16 *t16 = &tab->fx16;
  FxTab4 *t4 = &tab->fx4;
  const int Nq = N + 1;
  DD x[kMaxNq], w[kMaxNq], D[kMaxNq][kMaxNq], Kh[kMaxNq][kMaxNq];
  auto legendre = [&](DD z, DD *pn, DD *pm) {  // P_N, P_{N-1}
    DD p0(1.0), p1 = z;
    for (int k = 2; k <= N; ++k) {
      const DD p2 = (DD(2.0 * k - 1.0) * z * p1 - DD(k - 1.0) * p0) / DD(k);
      p0 = p1;
      p1 = p2;
    }
    *pn = p1;
    *pm = p0;
  };
  for (int i = 0; i < Nq; ++i) {
    DD pn, pm;
    x[i] = DD(x0[i]);
    for (int it = 0; it < 3; ++it) {
      legendre(x[i], &pn, &pm);
      x[i] = x[i] - (x[i] * pn - pm) / (DD(Nq) * pn);
    }
    legendre(x[i], &pn, &pm);
    w[i] = DD(2.0) / (DD((double)N * Nq) * pn * pn);
  }
  DD b[kMaxNq];
  for (int j = 0; j < Nq; ++j) {
    DD p(1.0);
    for (int k = 0; k < Nq; ++k)
      if (k != j) p = p * (x[j] - x[k]);
    b[j] = DD(1.0) / p;
  }
  for (int a = 0; a < Nq; ++a) {
    DD diag;
    for (int i = 0; i < Nq; ++i)
      if (i != a) {
        D[a][i] = (b[i] / b[a]) / (x[a] - x[i]);
        diag = diag - D[a][i];
      }
    D[a][a] = diag;
  }
  for (int i = 0; i < Nq; ++i)
    for (int m = 0; m < Nq; ++m) {
      DD s;
      for (int a = 0; a < Nq; ++a) s = s + D[a][i] * w[a] * D[a][m];
      Kh[i][m] = s / w[i];
    }
  const DD g(0.5 * h), ml = DD(lambda) * g * g * g;
  // (2 Nq + 4) 2^-53 of the sum of an entry's terms: the bound of the FP64 sums
  const double allow = 2.0 * Nq + 4.0;
  auto kh = [&](int i, int m) { return Kh[i][m]; };
  double s = 1.0;
  auto scaled_kh = [&] {
    for (int i = 0; i < Nq; ++i)
      for (int m = 0; m < Nq; ++m) tab->kh[i * Nq + m] = (Kh[i][m] * DD(s)).h;
  };
  if (Nq > kFxMaxNq) {
    auto word = [&](int b, int i, int m, uint32_t bits) {
      (b < kFxDigits ? t16->w[b] : t16->a)[(i % 8) * 4 + m % 8 / 2][i / 8 + 2 * (m / 8)] = bits;
    };
    if (!fx_digits(Nq, kh, true, 3, allow, word, &s, &t16->q, &t16->low)) return false;
    scaled_kh();
    for (int k = 0; k < Nq; ++k) t16->w1[k] = w[k].h;
    for (int lane = 0; lane < 32; ++lane)
      for (int q = 0; q < 8; ++q) {
        const int j = (lane >> 2) + 8 * (q >> 2), i = 2 * (lane & 3) + 8 * ((q >> 1) & 1) + (q & 1);
        if (i >= Nq || j >= Nq) continue;
        t16->wg[lane * 8 + q] = (w[i] * w[j] * g / DD(s)).h;
        t16->wm[lane * 8 + q] = (w[i] * w[j] * ml).h;
      }
    return true;
  }
  if (Nq < kFxMinNq) {
    auto word = [&](int b, int i, int m, uint32_t bits) {
      if (b == kFxDigits)
        for (int g4 = 0; g4 < 2; ++g4)
          for (int th = 0; th < 2; ++th) t4->a[(4 * g4 + i) * 4 + 2 * th + m / 2] = bits;
      for (int x = 0; x < kFxDigits / 2; ++x)
        for (int od = 0; od < 2; ++od)
          for (int th = 0; th < 2; ++th)
            if (2 * x + od - th == b) t4->w[x][(4 * od + i) * 4 + 2 * th + m / 2] = bits;
    };
    if (!fx_digits(Nq, kh, true, 3, allow, word, &s, &t4->q, &t4->low)) return false;
    scaled_kh();
    for (int lane = 0; lane < 32; ++lane)
      for (int hf = 0; hf < 2; ++hf) {
        const int g4 = lane >> 2, t = lane & 3;
        const int i = 2 * (t & 1) + hf, j = g4 & 3, k = 2 * (g4 >> 2) + (t >> 1);
        if (i >= Nq || j >= Nq || k >= Nq) continue;
        const DD w3 = w[i] * w[j] * w[k];
        t4->wg[lane * 2 + hf] = (w3 * g / DD(s)).h;
        t4->wm[lane * 2 + hf] = (w3 * ml).h;
      }
    return true;
  }
  auto words = [](uint32_t (*to)[32], uint32_t *sizes) {
    return [to, sizes](int b, int i, int m, uint32_t bits) {
      (b < kFxDigits ? to[b] : sizes)[i * 4 + m / 2] = bits;
    };
  };
  auto M = [&](int i, int m) { return D[m][i] * DD(std::ldexp(1.0, tg->p[i] - tg->p[m])); };
  // the weights' powers of two, by rounding down or to the nearest, whichever leaves
  // P^-1 D^T P the smaller largest entry (7.5, 10.5, 14 at degrees 5, 6, 7; else 14, 20, 26)
  auto powers = [&](double up) {
    double big = 0.0;
    for (int i = 0; i < Nq; ++i) tg->p[i] = -(int)std::floor(std::log2(w[i].h) + up);
    for (int i = 0; i < Nq; ++i)
      for (int m = 0; m < Nq; ++m) big = std::fmax(big, std::fabs(M(i, m).h));
    return big;
  };
  powers(powers(0.5) < powers(0.0) ? 0.5 : 0.0);
  // on general hexahedra (2 Nq + 8) 2^-53 of B = the sum of |D|^T |G| |D| |u|: the components
  // within Nq + 2 of their lines' terms, the entries within Nq + 6 of the fluxes' (the
  // sizes of the fluxes' own terms, not of the fluxes, make up B)
  double sd, sdt;
  if (!fx_digits(Nq, kh, true, 3, allow, words(t->w, t->a), &s, &t->q, &t->low) ||
      !fx_digits(Nq, [&](int i, int m) { return D[i][m]; }, true, 1, Nq + 2.0,
                 words(tg->d, tg->da), &sd, &tg->qd, &tg->lowd) ||
      !fx_digits(Nq, M, false, 3, Nq + 6.0,
                 words(tg->dt, tg->dta), &sdt, &tg->qdt, &tg->lowdt))
    return false;
  scaled_kh();
  for (int i = 0; i < Nq; ++i)
    for (int m = 0; m < Nq; ++m) {
      tg->sD[i * Nq + m] = (D[i][m] * DD(sd)).h;
      tg->D[i * Nq + m] = D[i][m].h;
    }
  tg->invd = 1.0 / sd;
  tg->inv = (DD(1.0) / (DD(sd) * DD(sdt))).h;
  for (int k = 0; k < Nq; ++k)
    for (int lane = 0; lane < 32; ++lane)
      for (int hf = 0; hf < 2; ++hf) {
        const int i = 2 * (lane & 3) + hf, j = lane >> 2;
        if (i >= Nq || j >= Nq) continue;
        const DD w3 = w[i] * w[j] * w[k];
        t->wg[(k * 32 + lane) * 2 + hf] = (w3 * g / DD(s)).h;
        t->wm[(k * 32 + lane) * 2 + hf] = (w3 * ml).h;
      }
  return true;
}

// diag(A_L) per local node: c_e (h/2) (K_ii w_j w_k + w_i K_jj w_k + w_i w_j K_kk)
// + lambda (h/2)^3 w_i w_j w_k.
template <typename T>
__global__ void k_diag_local(int64_t NL, int Nq, const OpTab<T> *__restrict__ tab,
                             const double *__restrict__ coef, T g, T mlam,
                             T *__restrict__ out) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * blockDim.x;
  const int64_t Np = (int64_t)Nq * Nq * Nq;
  for (int64_t l = tid; l < NL; l += nth) {
    const int64_t e = l / Np;
    const int r = (int)(l - e * Np);
    const int i = r % Nq, j = (r / Nq) % Nq, k = r / (Nq * Nq);
    const T wi = tab->w[i], wj = tab->w[j], wk = tab->w[k];
    T s = tab->K[i * Nq + i] * wj * wk;
    s = s + wi * tab->K[j * Nq + j] * wk;
    s = s + wi * wj * tab->K[k * Nq + k];
    const T c = coef ? T(coef[e]) : T(1);
    out[l] = fmaT(c * g, s, mlam * (wi * wj * wk));
  }
}

static int check_prob(const bs_problem *p, const char *fn) {
  if (!p) return fail(BS_ERR_ARG, "%s: problem is NULL", fn);
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev != p->device)
    return fail(BS_ERR_ARG, "%s: problem belongs to device %d, current is %d", fn, p->device,
                dev);
  return BS_OK;
}

static void free_problem(bs_problem *p) {
  if (!p) return;
  if (p->graph) cudaGraphExecDestroy(p->graph);
  if (p->cap_stream) cudaStreamDestroy(p->cap_stream);
  cudaFree(p->d_coef);
  cudaFree(p->d_geo);
  cudaFree(p->d_tab);
  cudaFree(p->d_tabf);
  cudaFree(p->d_tabff);
  cudaFree(p->d_ApL);
  cudaFree(p->d_vec);
  cudaFree(p->d_state);
  cudaFree(p->d_partials);
  cudaFree(p->d_op_partials);
  cudaFree(p->d_f32);
  cudaFree(p->d_Lvec);
  cudaFree(p->d_owner);
  cudaFree(p->d_bj);
  if (p->h_state) cudaFreeHost(p->h_state);
  free(p);
}

// diag(A_L) per local node n = (i, j, k): the unit vector's quadratic form,
//   c_e [sum_m D_mi^2 G_rr(m,j,k) + sum_m D_mj^2 G_ss(i,m,k) + sum_m D_mk^2 G_tt(i,j,m)
//        + 2 (D_ii D_jj G_rs + D_ii D_kk G_rt + D_jj D_kk G_st)(n)] + lambda M_n
// (grad_r l_n is nonzero only on the three lines through n, and two of its
// components only at n itself).
static __global__ void k_diag_geo(int64_t NL, int Nq, const OpTab<double> *__restrict__ tab,
                           const double *__restrict__ coef, const double *__restrict__ geo,
                           double lambda, double *__restrict__ out) {
  const int64_t tid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t nth = (int64_t)gridDim.x * blockDim.x;
  const int Nq2 = Nq * Nq, Np = Nq2 * Nq;
  const double *D = tab->D;
  for (int64_t l = tid; l < NL; l += nth) {
    const int64_t e = l / Np;
    const int n = (int)(l - e * Np);
    const int i = n % Nq, j = (n / Nq) % Nq, k = n / Nq2;
    const int64_t b = e * Np;
    double s = 0.0;
    for (int m = 0; m < Nq; ++m) {
      const double di = D[m * Nq + i], dj = D[m * Nq + j], dk = D[m * Nq + k];
      s = fma(di * di, geo[b + m + Nq * j + Nq2 * k], s);
      s = fma(dj * dj, geo[3 * NL + b + i + Nq * m + Nq2 * k], s);
      s = fma(dk * dk, geo[5 * NL + b + i + Nq * j + Nq2 * m], s);
    }
    const double dii = D[i * Nq + i], djj = D[j * Nq + j], dkk = D[k * Nq + k];
    s = fma(2.0 * dii * djj, geo[NL + l], s);
    s = fma(2.0 * dii * dkk, geo[2 * NL + l], s);
    s = fma(2.0 * djj * dkk, geo[4 * NL + l], s);
    out[l] = fma(coef ? coef[e] : 1.0, s, lambda * geo[6 * NL + l]);
  }
}

}  // namespace bs

using namespace bs;

extern "C" {

int bs_problem_create(const bs_map *map, double h, double lambda, const double *h_coef,
                      bs_problem **out) {
  BS_ARG(out != nullptr, "bs_problem_create: out is NULL");
  *out = nullptr;
  BS_ARG(map != nullptr, "bs_problem_create: map is NULL");
  BS_ARG(h > 0.0 && std::isfinite(h), "bs_problem_create: h must be positive");
  BS_ARG(lambda >= 0.0 && std::isfinite(lambda), "bs_problem_create: lambda must be >= 0");
  const int N = map->N, Nq = N + 1;
  BS_ARG(Nq <= kMaxNq, "bs_problem_create: degree %d unsupported", N);
  if (h_coef)
    for (int64_t e = 0; e < map->E; ++e)
      BS_ARG(h_coef[e] > 0.0 && std::isfinite(h_coef[e]),
             "bs_problem_create: coef[%lld] must be positive", (long long)e);
  bs_problem *p = (bs_problem *)calloc(1, sizeof(bs_problem));
  if (!p) return fail(BS_ERR_ALLOC, "bs_problem_create: host allocation");
  p->map = map;
  p->N = N;
  p->h = h;
  p->lambda = lambda;
  double x[kMaxNq], w[kMaxNq], D[kMaxNq * kMaxNq], K[kMaxNq * kMaxNq];
  gll_tables(N, x, w, D);
  stiffness_1d(N, w, D, K);
  OpTab<double> tab{};
  OpTab<float> tabf{};
  OpTabFF tabff{};
  // float pairs v = hi + lo (hi = v rounded to float, lo = the rest rounded)
  auto split = [](double v, float &hi, float &lo) {
    hi = (float)v;
    lo = (float)(v - (double)hi);
  };
  if (Nq % 2 == 0) {  // even-odd halves of W^-1 K, centrosymmetrised
    const int hq = Nq / 2;
    auto kh = [&](int a, int m) {
      return 0.5 * (K[a * Nq + m] / w[a] + K[(Nq - 1 - a) * Nq + (Nq - 1 - m)] / w[Nq - 1 - a]);
    };
    for (int a = 0; a < hq; ++a)
      for (int m = 0; m < hq; ++m) {
        const double e = 0.5 * (kh(a, m) + kh(a, Nq - 1 - m));
        const double o = 0.5 * (kh(a, m) - kh(a, Nq - 1 - m));
        tab.Ee[a * hq + m] = e;
        tab.Eo[a * hq + m] = o;
        tabf.Ee[a * hq + m] = (float)e;
        tabf.Eo[a * hq + m] = (float)o;
        split(e, tabff.Eeh[a * hq + m], tabff.Eel[a * hq + m]);
        split(o, tabff.Eoh[a * hq + m], tabff.Eol[a * hq + m]);
      }
  }
  if (Nq > 2 && !fx_table(N, x, h, lambda, &tab)) {
    free(p);
    return fail(BS_ERR_ARG, "bs_problem_create: digit tables of degree %d out of range", N);
  }
  for (int i = 0; i < Nq; ++i) {
    tab.w[i] = w[i];
    tabf.w[i] = (float)w[i];
    split(w[i], tabff.wh[i], tabff.wl[i]);
    for (int m = 0; m < Nq; ++m) {
      tab.K[i * Nq + m] = K[i * Nq + m];
      tab.D[i * Nq + m] = D[i * Nq + m];
      tabf.D[i * Nq + m] = (float)D[i * Nq + m];
      split(D[i * Nq + m], tabff.Dh[i * Nq + m], tabff.Dl[i * Nq + m]);
      tabf.K[i * Nq + m] = (float)K[i * Nq + m];
      split(K[i * Nq + m], tabff.Kh[i * Nq + m], tabff.Kl[i * Nq + m]);
      split(w[i] * w[m], tabff.Wh[i * Nq + m], tabff.Wl[i * Nq + m]);
    }
  }
  const int64_t NL = map->NL, NG = map->NG;
  tab.ne = tabf.ne = tabff.ne = map->E;
  tab.ng = tabf.ng = tabff.ng = NG;
  cudaError_t e = cudaGetDevice(&p->device);
  if (e == cudaSuccess && h_coef) e = cudaMalloc(&p->d_coef, sizeof(double) * (map->E + 1));
  if (e == cudaSuccess && h_coef)
    e = cudaMemcpy(p->d_coef, h_coef, sizeof(double) * map->E, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(&p->d_tab, sizeof(tab));
  if (e == cudaSuccess) e = cudaMalloc(&p->d_tabf, sizeof(tabf));
  if (e == cudaSuccess) e = cudaMemcpy(p->d_tab, &tab, sizeof(tab), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(p->d_tabf, &tabf, sizeof(tabf), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(&p->d_tabff, sizeof(tabff));
  if (e == cudaSuccess) e = cudaMemcpy(p->d_tabff, &tabff, sizeof(tabff), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMalloc(&p->d_ApL, sizeof(double) * (NL + 2));
  if (e == cudaSuccess) e = cudaMalloc(&p->d_vec, sizeof(double) * 6 * vec_stride(NG));
  if (e == cudaSuccess) e = cudaMalloc(&p->d_state, sizeof(CgState));
  if (e == cudaSuccess) e = cudaMemset(p->d_state, 0, sizeof(CgState));
  if (e == cudaSuccess) e = cudaMalloc(&p->d_partials, sizeof(double) * kMaxPartials + 256);
  if (e == cudaSuccess) e = cudaMemset(p->d_partials, 0, sizeof(double) * kMaxPartials + 256);
  // one partial per element-kernel block: at most one block per element,
  // whichever kernel form (direct, even-odd) a later call selects
  if (e == cudaSuccess) e = cudaMalloc(&p->d_op_partials, sizeof(double) * (map->E + 1));
  if (e == cudaSuccess) e = cudaMallocHost(&p->h_state, sizeof(CgState));
  if (e == cudaSuccess) e = cudaStreamCreateWithFlags(&p->cap_stream, cudaStreamNonBlocking);
  if (e != cudaSuccess) {
    free_problem(p);
    return fail(BS_ERR_CUDA, "bs_problem_create: %s", cudaGetErrorString(e));
  }
  p->d_counter = (unsigned int *)(p->d_partials + kMaxPartials);
  *out = p;
  return BS_OK;
}

int bs_problem_create_geo(const bs_map *map, double lambda, const double *h_coef,
                          const double *h_verts, bs_problem **out) {
  BS_ARG(out != nullptr, "bs_problem_create_geo: out is NULL");
  *out = nullptr;
  BS_ARG(map != nullptr, "bs_problem_create_geo: map is NULL");
  BS_ARG(map->N + 1 <= kGeoMaxNq, "bs_problem_create_geo: degree %d > %d", map->N,
         kGeoMaxNq - 1);
  BS_ARG(map->E == 0 || h_verts != nullptr, "bs_problem_create_geo: verts is NULL");
  const int N = map->N, Nq = N + 1, Np = Nq * Nq * Nq;
  const int64_t E = map->E, NL = map->NL;
  double x[kMaxNq], w[kMaxNq], D[kMaxNq * kMaxNq];
  gll_tables(N, x, w, D);
  // G = w det J J^-1 J^-T (upper triangle) and M = w det J at every node,
  // J = dx/dr of the trilinear map of the element's eight corners
  std::vector<double> fac((size_t)kGeoFactors * (size_t)NL);
  // elements split over host threads; bad[t] is the first degenerate
  // element thread t met (or -1)
  const int nth = (int)std::max(1u, std::min(32u, std::thread::hardware_concurrency()));
  std::vector<int64_t> bad((size_t)nth, -1);
  auto work = [&](int t) {
  for (int64_t e = t; e < E; e += nth) {
    const double *X = h_verts + 24 * e;
    for (int n = 0; n < Np; ++n) {
      const int i = n % Nq, j = (n / Nq) % Nq, k = n / (Nq * Nq);
      const double r = x[i], s = x[j], t = x[k];
      double J[3][3] = {{0, 0, 0}, {0, 0, 0}, {0, 0, 0}};
      for (int v = 0; v < 8; ++v) {
        const double sx = (v & 1) ? 1.0 : -1.0, sy = (v & 2) ? 1.0 : -1.0,
                     sz = (v & 4) ? 1.0 : -1.0;
        const double dr = 0.125 * sx * (1.0 + sy * s) * (1.0 + sz * t);
        const double ds = 0.125 * (1.0 + sx * r) * sy * (1.0 + sz * t);
        const double dt = 0.125 * (1.0 + sx * r) * (1.0 + sy * s) * sz;
        for (int d = 0; d < 3; ++d) {
          J[d][0] += X[3 * v + d] * dr;
          J[d][1] += X[3 * v + d] * ds;
          J[d][2] += X[3 * v + d] * dt;
        }
      }
      // adjugate: C[p][d] = cofactor, J^-1 = C / det (rows: reference p)
      double C[3][3];
      C[0][0] = J[1][1] * J[2][2] - J[1][2] * J[2][1];
      C[0][1] = J[0][2] * J[2][1] - J[0][1] * J[2][2];
      C[0][2] = J[0][1] * J[1][2] - J[0][2] * J[1][1];
      C[1][0] = J[1][2] * J[2][0] - J[1][0] * J[2][2];
      C[1][1] = J[0][0] * J[2][2] - J[0][2] * J[2][0];
      C[1][2] = J[0][2] * J[1][0] - J[0][0] * J[1][2];
      C[2][0] = J[1][0] * J[2][1] - J[1][1] * J[2][0];
      C[2][1] = J[0][1] * J[2][0] - J[0][0] * J[2][1];
      C[2][2] = J[0][0] * J[1][1] - J[0][1] * J[1][0];
      const double det = J[0][0] * C[0][0] + J[0][1] * C[1][0] + J[0][2] * C[2][0];
      if (!(det > 0.0) || !std::isfinite(det)) {
        if (bad[(size_t)t] < 0) bad[(size_t)t] = e;
        continue;
      }
      const double wq = w[i] * w[j] * w[k];
      // w det J (C/det)(C/det)^T = (w / det) C C^T
      const double sc = wq / det;
      auto cc = [&](int p, int q) {
        return C[p][0] * C[q][0] + C[p][1] * C[q][1] + C[p][2] * C[q][2];
      };
      const size_t l = (size_t)(e * Np + n);
      fac[0 * (size_t)NL + l] = sc * cc(0, 0);
      fac[1 * (size_t)NL + l] = sc * cc(0, 1);
      fac[2 * (size_t)NL + l] = sc * cc(0, 2);
      fac[3 * (size_t)NL + l] = sc * cc(1, 1);
      fac[4 * (size_t)NL + l] = sc * cc(1, 2);
      fac[5 * (size_t)NL + l] = sc * cc(2, 2);
      fac[6 * (size_t)NL + l] = wq * det;
    }
  }
  };
  {
    std::vector<std::thread> pool;
    for (int t = 1; t < nth; ++t) pool.emplace_back(work, t);
    work(0);
    for (auto &th : pool) th.join();
  }
  for (int64_t b : bad)
    if (b >= 0)
      return fail(BS_ERR_ARG, "bs_problem_create_geo: element %lld is inverted or degenerate",
                  (long long)b);
  bs_problem *p = nullptr;
  if (int rc = bs_problem_create(map, 1.0, lambda, h_coef, &p)) return rc;
  cudaError_t err = cudaMalloc(&p->d_geo, sizeof(double) * (fac.size() + 1));
  if (err == cudaSuccess && !fac.empty())
    err = cudaMemcpy(p->d_geo, fac.data(), sizeof(double) * fac.size(), cudaMemcpyHostToDevice);
  if (err != cudaSuccess) {
    free_problem(p);
    return fail(BS_ERR_CUDA, "bs_problem_create_geo: %s", cudaGetErrorString(err));
  }
  *out = p;
  return BS_OK;
}

int bs_problem_destroy(bs_problem *p) {
  free_problem(p);
  return BS_OK;
}

int bs_apply_local(const bs_problem *p, const double *uL, double *AuL, void *stream) {
  if (int rc = check_prob(p, "bs_apply_local")) return rc;
  if (p->map->NL == 0) return BS_OK;
  BS_ARG(uL && AuL, "bs_apply_local: NULL vector");
  const double g = 0.5 * p->h, mlam = p->lambda * g * g * g;
  if (p->d_geo)
    return launch_ax_geo<false>(p->N, p->map->E, p->map->NL, nullptr, nullptr, uL, AuL,
                                p->d_tab, p->d_coef, p->d_geo, p->lambda, nullptr,
                                as_stream(stream));
  return launch_ax_local<double, false>(p->N, p->map->E, nullptr, nullptr, uL, AuL, p->d_tab,
                                        p->d_coef, g, mlam, nullptr, as_stream(stream));
}

int bs_apply_A(const bs_problem *p, const double *x, double *Ax, void *stream) {
  if (int rc = check_prob(p, "bs_apply_A")) return rc;
  if (p->map->NG == 0) return BS_OK;
  BS_ARG(x && Ax, "bs_apply_A: NULL vector");
  const double g = 0.5 * p->h, mlam = p->lambda * g * g * g;
  return apply_A_global<double, false, EpNone>(p, false, p->d_tab, x, Ax, p->d_ApL, g, mlam,
                                               EpNone{}, nullptr, as_stream(stream));
}

int bs_apply_A_ff(const bs_problem *p, const double *x, double *Ax, void *stream) {
  if (int rc = check_prob(p, "bs_apply_A_ff")) return rc;
  if (p->map->NG == 0) return BS_OK;
  BS_ARG(x && Ax, "bs_apply_A_ff: NULL vector");
  const double g = 0.5 * p->h, mlam = p->lambda * g * g * g;
  return apply_A_global<double, false, EpNone>(p, true, p->d_tab, x, Ax, p->d_ApL, g, mlam,
                                               EpNone{}, nullptr, as_stream(stream));
}

int bs_diag_A(const bs_problem *p, double *d_diag, void *stream) {
  if (int rc = check_prob(p, "bs_diag_A")) return rc;
  if (p->map->NG == 0) return BS_OK;
  BS_ARG(d_diag != nullptr, "bs_diag_A: NULL output");
  const double g = 0.5 * p->h, mlam = p->lambda * g * g * g;
  cudaStream_t s = as_stream(stream);
  if (p->map->NL > 0) {
    const int grid = stream_grid(p->map->NL, 1, kStreamBlock, 8);
    if (p->d_geo)
      k_diag_geo<<<grid, kStreamBlock, 0, s>>>(p->map->NL, p->N + 1, p->d_tab, p->d_coef,
                                               p->d_geo, p->lambda, p->d_ApL);
    else
      k_diag_local<double><<<grid, kStreamBlock, 0, s>>>(p->map->NL, p->N + 1, p->d_tab,
                                                        p->d_coef, g, mlam, p->d_ApL);
    BS_LAUNCH_CHECK();
  }
  return launch_gather<double, false, EpNone>(p->map, p->d_ApL, d_diag, nullptr, nullptr,
                                              nullptr, EpNone{}, nullptr, s);
}

int bs_operator_mode(int32_t mode) {
  const int prev = (g_op_fusion ? BS_OP_FUSED : 0) | (g_op_evenodd ? 0 : BS_OP_DIRECT);
  if (mode >= 0) {
    g_op_fusion = (mode & BS_OP_FUSED) ? 1 : 0;
    g_op_evenodd = (mode & BS_OP_DIRECT) ? 0 : 1;
  }
  return prev;
}

}  // extern "C"
