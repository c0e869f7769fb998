// Learning stage on the GPU for CNF formulas: loopy belief propagation on the surrogate
// Hamiltonian (Sec. "4-SAT Problems Near Computational Phase Transitions"; App. "Loopy Belief
// propagation for k-local Hamiltonians over conjugate normal form"), connected backbone growth
// (Sec. "Generating backbones of rigid variables") and the two-chain schedule of Algorithm 1.
//
// Messages live on the edges e = a * kmax + q of the clause slots (literal id 2v + neg, padding
// literal 2n) for S seeds at once, seed-fastest ([e][S]), so the threads of a warp handle the
// same edge of 32 seeds and every load is coalesced. One LBP iteration = a variable pass (the
// cavity fields h_{i->a} of every edge of a variable from its total field) then a clause pass
// (u_{a->i} of every literal of a clause from the other literals' h). Double precision.
//
// Frames: spin r = 2x - 1; literal i of clause a is satisfied by sigma_ai (+1 positive, -1
// negated). h_{i->a} = sigma_ai (lambda eps_i s*_i + sum_{b != a} sigma_bi u_{b->i});
// u_{a->i} = -1/2 ln[1 - (1 - e^{-2 beta}) prod_{j != i} (1 - tanh h_{j->a}) / 2].
//
// Two forms of the same iteration. The product form keeps m = 1 - e^{-2u} and E = e^{2h} instead of
// u and h: sums of u become products of 1 - m, (1 - tanh h) / 2 is 1 / (1 + E), and an iteration
// needs neither exponentials nor logarithms (13 double-precision instructions per message instead of
// 82; the log form was bound by them, 85% of the pipe). It is used whenever no e^{2 field} can leave
// the range of a double and the tolerance is above the resolution of m; the log form runs otherwise.
//
// Its error stays that of the log form: a small u has a small m, E near 1 is kept as E - 1, and the
// products are carried with the sum of their rounding errors (ProductSum, clause_messages). Largest
// error of a converged call against 80 bits, product form over log form, mean of 84 4-SAT inputs of 300
// to 5,000 variables at beta = 1: 0.90 marginals, 0.99 correlations (root mean square 0.84, 0.86); 36
// sparser inputs at beta = 4: 0.85, 0.97; without a bias at beta = 1e-3: 0.46, 0.92. With 1 - m, E and
// plain products kept instead: 1.08, 1.11 at beta = 1 and 440 without a bias at beta = 1e-3.
//
// 4-SAT, 5,000 variables, 64 seeds: clause pass 1,920 -> 149 us, variable pass 120 -> 141, a call with
// its backbones 122 -> 26.4 ms (22.8 with the plain products); 500 variables, 5 seeds: 5.6 -> 2.8 ms.
#include <math.h>

#include "nmc_internal.h"

namespace nmc {

namespace {

constexpr int kLbpBlock = 256;
enum : int { kRunning = 0, kWaiting = 1, kFinished = 2 };

__device__ __forceinline__ double lit_sigma(int l) { return (l & 1) ? -1.0 : 1.0; }

// h of every edge at the first lambda: sigma lambda eps s*.
__global__ void lbp_init_h_kernel(const int32_t *__restrict__ clits, long long n_edges, int32_t n,
                                  int32_t S, const double *__restrict__ bias, double *h) {
  const long long total = n_edges * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long e = i / S;
    const int s = (int)(i % S);
    const int l = clits[e];
    h[i] = l >= 2 * n ? 0.0 : lit_sigma(l) * bias[(size_t)(l >> 1) * S + s];
  }
}

// bias[v][s] = lambda eps_v s*_{v,s} (eps and x_star in new variable order).
__global__ void lbp_bias_kernel(const double *__restrict__ eps, const uint8_t *__restrict__ xs,
                                int32_t n, int32_t S, double lambda, double *bias) {
  const long long total = (long long)n * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(i / S);
    bias[i] = lambda * eps[v] * (2.0 * (double)xs[i] - 1.0);
  }
}

// Clause pass: u of every literal of clause a for seed s; the largest change per seed goes to
// dmax (non-negative doubles order like their bit patterns).
__global__ void lbp_clause_kernel(const int32_t *__restrict__ clits, int32_t m, int32_t kmax,
                                  int32_t n, int32_t S, const double *__restrict__ h, double *u,
                                  double c, const int32_t *__restrict__ status,
                                  unsigned long long *dmax, int track) {
  const long long total = (long long)m * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long a = i / S;
    const int s = (int)(i % S);
    if (status && status[s] != kRunning) continue;
    double f[8];
    int k = 0;
    for (int q = 0; q < kmax; ++q) {
      const long long e = a * kmax + q;
      f[q] = 1.0;
      if (clits[e] < 2 * n) {
        f[q] = 1.0 / (1.0 + exp(2.0 * h[e * S + s]));  // (1 - tanh h) / 2, one exp
        ++k;
      }
    }
    double dm = 0.0;
    for (int q = 0; q < kmax; ++q) {
      const long long e = a * kmax + q;
      if (clits[e] >= 2 * n) continue;
      double prod = 1.0;
      for (int j = 0; j < kmax; ++j)
        if (j != q) prod *= f[j];  // padding slots hold 1.0
      const double un = -0.5 * log1p(-c * prod);
      const double d = fabs(un - u[e * S + s]);
      if (d > dm) dm = d;
      u[e * S + s] = un;
    }
    (void)k;
    if (track && dm > 0.0) atomicMax(&dmax[s], (unsigned long long)__double_as_longlong(dm));
  }
}

// Variable pass: total field of v for seed s, then the cavity field of each of its edges.
__global__ void lbp_var_kernel(const int32_t *__restrict__ vptr, const int32_t *__restrict__ vedge,
                               const int32_t *__restrict__ clits, int32_t n, int32_t S,
                               const double *__restrict__ bias, const double *__restrict__ u,
                               double *h, const int32_t *__restrict__ status) {
  const long long total = (long long)n * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(i / S), s = (int)(i % S);
    if (status[s] != kRunning) continue;
    double field = bias[i];
    const int p0 = vptr[v], p1 = vptr[v + 1];
    for (int p = p0; p < p1; ++p) {
      const long long e = vedge[p];
      field += lit_sigma(clits[e]) * u[e * S + s];
    }
    for (int p = p0; p < p1; ++p) {
      const long long e = vedge[p];
      const double sg = lit_sigma(clits[e]);
      h[e * S + s] = sg * (field - sg * u[e * S + s]);
    }
  }
}

// ---- product form -----------------------------------------------------------------------------

// E of an edge as one double v: E - 1 where the variable's e^{+-2 field} is at least a half, so that
// fields near zero keep their relative precision, else -2^1000 E, at most -2^19 as long as |field| <
// 340. E - 1 is above -1, so the two do not meet.
constexpr double kEdgeScale = 0x1p1000;
__device__ __forceinline__ bool edge_scaled(double v) {  // v <= -1
  return (unsigned)__double2hiint(v) >= 0xBFF00000u;
}
__device__ __forceinline__ double edge_plus_one(double v) {  // 1 + E
  const bool sc = edge_scaled(v);
  return fma(v, sc ? -1.0 / kEdgeScale : 1.0, sc ? 1.0 : 2.0);
}

// Largest 1 + E a clause product takes: with it the K factors of a clause stay below 2^1000. A
// larger one (a literal false with probability below 2^-125) leaves every other m below 2^-125.
template <int K>
__device__ __forceinline__ double cut_factor(double d) {
  constexpr int kHi = (1023 + 1000 / K) << 20;  // high word of 2^(1000 / K)
  return __double2hiint(d) >= kHi ? __hiloint2double(kHi, 0) : d;
}

// |x| and x cut off to 24 bits as a float, for |x| < 2^128 (0 below 2^-126), with integer operations
// only (a conversion takes the double-precision pipe).
__device__ __forceinline__ float approx_abs(double x) {
  const int h = (__double2hiint(x) & 0x7FFFFFFF) - (896 << 20);
  return h <= 0 ? 0.0f : __int_as_float((int)__funnelshift_l((unsigned)__double2loint(x), (unsigned)h, 3));
}
__device__ __forceinline__ float approx(double x) {
  return __int_as_float(__float_as_int(approx_abs(x)) | (__double2hiint(x) & (int)0x80000000));
}

// g[v][s] = expm1(2 |lambda eps_v|) with the sign of the bias lambda eps_v s*_{v,s}.
__global__ void lbp_gain_kernel(const double *__restrict__ eps, const uint8_t *__restrict__ xs,
                                int32_t n, int32_t S, double lambda, double *g) {
  const long long total = (long long)n * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const double b = 2.0 * lambda * eps[i / S] * (2.0 * (double)xs[i] - 1.0);
    g[i] = copysign(expm1(fabs(b)), b);
  }
}

// Edges at the first lambda: E = e^{+-2 bias}.
__global__ void lbp_init_prod_kernel(const int32_t *__restrict__ clits, long long n_edges, int32_t n,
                                     int32_t S, const double *__restrict__ g, double *E) {
  const long long total = n_edges * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int l = clits[i / S];
    if (l >= 2 * n) continue;
    const double b = g[(size_t)(l >> 1) * S + i % S], a = fabs(b);
    if ((b < 0.0) == ((l & 1) != 0)) E[i] = a;  // the literal is the bias's: e^{|2 bias|}
    else E[i] = a <= 1.0 ? -a / (1.0 + a) : -kEdgeScale / (1.0 + a);
  }
}

// |ln(w / w_old)| of w = 1 - m, from the change of m and the smaller of the two w: the series where
// it is short enough, else log1p.
__device__ __forceinline__ double log_change(double chg, double m_max) {
  const double r = fabs(chg) / (1.0 - m_max);
  if (r < 1e-4) return r * fma(r, fma(r, fma(r, -0.25, 1.0 / 3.0), -0.5), 1.0);
  return log1p(r);
}

// m = c prod_{j != i} 1 / (1 + E_j) of the K literals of a clause from their d = 1 + E: one
// reciprocal of the product of all, by two Newton steps r (2 - x r) from the hardware's approximation,
// with the rounding errors of that product in the second (first order: err is what the exact product
// is above `all`). Without them the roundings of the product, larger than those of a product of
// 1 / (1 + E) < 1, are amplified by e^{2 beta} in u. 1 <= all <= 2^1000, so nothing leaves the range.
template <int K>
__device__ __forceinline__ void clause_messages(const double (&d)[K], double c, double (&m)[K]) {
  double all = d[0], err = 0.0;
#pragma unroll
  for (int q = 1; q < K; ++q) {
    const double p = all * d[q];
    const double e = fma(all, d[q], -p);
    err = q > 1 ? fma(err, d[q], e) : e;
    all = p;
  }
  double r;
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(r) : "d"(all));
  r = fma(r, fma(-all, r, 1.0), r);
  r = c * fma(r, fma(-err, r, fma(-all, r, 1.0)), r);
#pragma unroll
  for (int q = 0; q < K; ++q) m[q] = __dmul_rn(d[q], r);  // not one operation with m - m_old
}

// Clause pass. The largest change of u per seed, |ln(w / w_old)| / 2, is found in two steps: single
// precision picks the edges that can hold the maximum, and only those are evaluated in double
// precision, usually one per thread. The single-precision value is log1p(|m - m_old| / w), w the
// smaller of the two 1 - m, whose relative error e^{2 beta} 2^-23 (m cut off to 24 bits, w >= e^{-2
// beta}) outweighs all others; `slack` is four times its bound, so an edge is passed over only when
// a larger value is already recorded, and the recorded maximum does not depend on which thread comes
// first.
// Bound by the double-precision pipe (2 lanes per cycle and SM).
template <int K>
__global__ void lbp_clause_prod_kernel(const int32_t *__restrict__ clits, int32_t m, int32_t n,
                                       int32_t S, const double *__restrict__ E, double *msg, double c,
                                       const int32_t *__restrict__ status, unsigned long long *dmax,
                                       int track, float slack) {
  const long long total = (long long)m * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long a = i / S;
    const int s = (int)(i - a * S);
    if (status && status[s] != kRunning) continue;
    const size_t e0 = (size_t)(a * K) * S + s;
    double d[K], old[K], now[K];
    bool used[K];
#pragma unroll
    for (int q = 0; q < K; ++q) {
      used[q] = clits[a * K + q] < 2 * n;
      d[q] = used[q] ? cut_factor<K>(edge_plus_one(E[e0 + (size_t)q * S])) : 1.0;
      old[q] = used[q] && track ? msg[e0 + (size_t)q * S] : 0.0;
    }
    clause_messages<K>(d, c, now);
    double chg[K], big[K], chg_top = 0.0, big_top = 0.0;
    float est[K], top = 0.0f;
#pragma unroll
    for (int q = 0; q < K; ++q) {
      if (used[q]) msg[e0 + (size_t)q * S] = now[q];
      chg[q] = used[q] ? now[q] - old[q] : 0.0;
      big[q] = __double2hiint(chg[q]) < 0 ? old[q] : now[q];
      est[q] = 0.0f;
      if (track) {
        est[q] = log1pf(__fdividef(approx_abs(chg[q]), 1.0f - approx_abs(big[q])));
        if (est[q] > top) {
          top = est[q];
          chg_top = chg[q];
          big_top = big[q];
        }
      }
    }
    if (!track || top == 0.0f) continue;
    const float seen = approx_abs(__longlong_as_double((long long)*(volatile unsigned long long *)&dmax[s]));
    if (0.5f * top * (1.0f + slack) < seen) continue;
    double dm = log_change(chg_top, big_top);
    const float tie = top * (1.0f - slack);
    int ties = 0;
#pragma unroll
    for (int q = 0; q < K; ++q) ties += est[q] >= tie;
    if (ties > 1) {  // another edge may hold the larger change
#pragma unroll
      for (int q = 0; q < K; ++q)
        if (est[q] >= tie) dm = fmax(dm, log_change(chg[q], big[q]));
    }
    if (dm > 0.0) atomicMax(&dmax[s], (unsigned long long)__double_as_longlong(0.5 * dm));
  }
}

// A product of factors 1 - m as p + r, r the sum of p's rounding errors (first order; single precision
// holds it well enough, and off the double-precision pipe. It counts errors as zero once p is below
// 2^-73, a sum of u beyond 25).
struct ProductSum {
  double p;
  float r;
  __device__ __forceinline__ void factor(double m) {
    const double q = fma(-p, m, p);
    // the error of q: p - q is exact up to m = 1/2, beyond it as good as m itself
    const double e = fma(-p, m, p - q);
    r = fmaf(-r, approx_abs(m), r + approx(e));
    p = q;
  }
};
__device__ __forceinline__ ProductSum times(const ProductSum &a, const ProductSum &b) {
  const double q = a.p * b.p;
  return ProductSum{q, fmaf(approx_abs(a.p), b.r, fmaf(a.r, approx_abs(b.p), approx(fma(a.p, b.p, -q))))};
}

// e^{2 field} = top / den of a variable, with num = top - den.
struct FieldRatio {
  double num, top, den;
};
// From the products of 1 - m over the positive and the negated edges and the bias's g. The bias
// multiplies the side that it makes larger, so nothing is taken from 1.
__device__ __forceinline__ FieldRatio field_ratio(const ProductSum &pos, const ProductSum &neg, double g) {
  const bool up = !(g < 0.0);
  const double a = fabs(g);
  const double ps = up ? neg.p : pos.p, pw = up ? pos.p : neg.p;
  const double rs = (double)(up ? neg.r : pos.r), rw = (double)(up ? pos.r : neg.r);
  const double num = fma(a, ps, ps - pw) + fma(a, rs, rs - rw);
  const double big = fma(a, ps, ps) + fma(a, rs, rs), other = pw + rw;
  return up ? FieldRatio{num, big, other} : FieldRatio{-num, other, big};
}

// Edges a lane of the variable pass requests together (with one lane a variable other warps hide the
// latency: eight at a time 143 us a pass instead of 141, 64 seeds of 5,000 variables).
__host__ __device__ constexpr int edge_batch(int lanes) { return lanes == 1 ? 4 : 8; }

// Products over the positive and the negated edges of variable v for seed s, always in the same
// order, whatever the launch: four of each, over every fourth edge, then (0 2)(1 3). LANES = 4: one of
// the four in each of four consecutive lanes (all get the result); LANES = 1: all in one.
template <int LANES>
__device__ __forceinline__ void edge_products(const int32_t *vedge, const int32_t *clits, int p0,
                                              int p1, int S, int s, const double *msg,
                                              ProductSum &pos, ProductSum &neg) {
  constexpr int PER = 4 / LANES, BATCH = edge_batch(LANES);
  const int sub = LANES == 1 ? 0 : (int)threadIdx.x % LANES;
  ProductSum f[2][PER];
#pragma unroll
  for (int j = 0; j < PER; ++j) f[0][j] = f[1][j] = ProductSum{1.0, 0.0f};
#pragma unroll (LANES == 1 ? 2 : 1)
  for (int p = p0 + sub; p < p1; p += BATCH * LANES) {
    double m[BATCH];
    int sign[BATCH];
#pragma unroll
    for (int j = 0; j < BATCH; ++j) {
      m[j] = 0.0;
      sign[j] = 0;
      if (p + j * LANES < p1) {
        const long long e = vedge[p + j * LANES];
        m[j] = msg[e * S + s];
        sign[j] = clits[e] & 1;
      }
    }
#pragma unroll
    for (int j = 0; j < BATCH; ++j) {  // a factor of m = 0 changes nothing
      ProductSum x = sign[j] ? f[1][j % PER] : f[0][j % PER];
      x.factor(m[j]);
      f[0][j % PER] = sign[j] ? f[0][j % PER] : x;
      f[1][j % PER] = sign[j] ? x : f[1][j % PER];
    }
  }
  if constexpr (LANES == 1) {
    pos = times(times(f[0][0], f[0][2]), times(f[0][1], f[0][3]));
    neg = times(times(f[1][0], f[1][2]), times(f[1][1], f[1][3]));
  } else {
    const unsigned team = 0xFu << ((threadIdx.x & 31) - sub);
#pragma unroll
    for (int z = 0; z < 2; ++z)
#pragma unroll
      for (int o = 2; o > 0; o >>= 1) {
        const ProductSum &mine = f[z][0];
        const ProductSum other{__shfl_xor_sync(team, mine.p, o), __shfl_xor_sync(team, mine.r, o)};
        f[z][0] = sub & o ? times(other, mine) : times(mine, other);
      }
    pos = f[0][0];
    neg = f[1][0];
  }
}

// Variable pass: the field of v for seed s, and E = e^{+-2 field} (1 - m) of each edge (the cavity
// takes the edge's own message out again). LANES = 1 where there are enough variables and seeds to
// fill the GPU (coalesced over seeds), 4 where a single lane's chain of loads and products would be
// the time (5 seeds of a 500-variable formula).
template <int LANES>
__global__ void lbp_var_prod_kernel(const int32_t *__restrict__ vptr, const int32_t *__restrict__ vedge,
                                    const int32_t *__restrict__ clits, int32_t n, int32_t S,
                                    const double *__restrict__ g, const double *__restrict__ msg,
                                    double *E, const int32_t *__restrict__ status) {
  const long long total = (long long)n * S;
  const int sub = threadIdx.x % LANES;
  // whole teams run the same iterations (blockDim is a multiple of LANES)
  for (long long i = (blockIdx.x * (long long)blockDim.x + threadIdx.x) / LANES; i < total;
       i += (long long)gridDim.x * blockDim.x / LANES) {
    const int v = (int)(i / S), s = (int)(i - (long long)v * S);
    if (status[s] != kRunning) continue;
    const int p0 = vptr[v], p1 = vptr[v + 1];
    ProductSum pos, neg;
    edge_products<LANES>(vedge, clits, p0, p1, S, s, msg, pos, neg);
    const FieldRatio f = field_ratio(pos, neg, g[i]);
    // an edge's v as a m + b, for each sign (see edge_scaled)
    const auto line = [](double top, double den, double num, double &a, double &b) {
      const double y = num / den;
      b = y < -0.5 ? -kEdgeScale * (top / den) : y;
      a = y < -0.5 ? -b : -(1.0 + y);
    };
    double ap, bp, an, bn;
    line(f.top, f.den, f.num, ap, bp);
    line(f.den, f.top, -f.num, an, bn);
    constexpr int BATCH = edge_batch(LANES);
#pragma unroll 1
    for (int p = p0 + sub; p < p1; p += BATCH * LANES) {
      long long at[BATCH];
      double m[BATCH];
      bool sign[BATCH];
#pragma unroll
      for (int j = 0; j < BATCH; ++j) {
        at[j] = -1;
        m[j] = 0.0;
        sign[j] = false;
        if (p + j * LANES < p1) {
          const long long e = vedge[p + j * LANES];
          sign[j] = clits[e] & 1;
          at[j] = e * S + s;
          m[j] = msg[at[j]];
        }
      }
#pragma unroll
      for (int j = 0; j < BATCH; ++j)
        if (at[j] >= 0) E[at[j]] = fma(sign[j] ? an : ap, m[j], sign[j] ? bn : bp);
    }
  }
}

// Marginals <r_v> = tanh field = num / (top + den), each seed at its own lambda; away from zero as
// 1 - 2 den / (top + den) or its mirror image, whichever term is the small one.
__global__ void lbp_marg_prod_kernel(const int32_t *__restrict__ vptr, const int32_t *__restrict__ vedge,
                                     const int32_t *__restrict__ clits,
                                     const int32_t *__restrict__ orig, int32_t n, int32_t S,
                                     const double *__restrict__ eps, const uint8_t *__restrict__ xs,
                                     const double *__restrict__ lambdas,
                                     const int32_t *__restrict__ lam_idx,
                                     const double *__restrict__ msg, double *marg) {
  const long long total = (long long)n * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(i / S), s = (int)(i - (long long)v * S);
    ProductSum pos, neg;
    edge_products<1>(vedge, clits, vptr[v], vptr[v + 1], S, s, msg, pos, neg);
    const double b = 2.0 * lambdas[lam_idx[s]] * eps[v] * (2.0 * (double)xs[i] - 1.0);
    const FieldRatio f = field_ratio(pos, neg, copysign(expm1(fabs(b)), b));
    const double sum = f.top + f.den;
    marg[(size_t)s * n + orig[v]] = 4.0 * fabs(f.num) < sum ? f.num / sum
                                    : f.num > 0.0           ? fma(-2.0, f.den / sum, 1.0)
                                                            : fma(2.0, f.top / sum, -1.0);
  }
}

// (p, q1) of one seed per block, in a fixed summation order.
__global__ void lbp_overlap_kernel(const int32_t *__restrict__ orig, int32_t n, int32_t S,
                                   const uint8_t *__restrict__ xs, const double *__restrict__ marg,
                                   double *overlap) {
  const int s = blockIdx.x;
  __shared__ double sp[kLbpBlock], sq[kLbpBlock];
  double p = 0.0, q = 0.0;
  for (int v = threadIdx.x; v < n; v += blockDim.x) {
    const double mv = marg[(size_t)s * n + orig[v]];
    p += (2.0 * (double)xs[(size_t)v * S + s] - 1.0) * mv;
    q += mv * mv;
  }
  sp[threadIdx.x] = p;
  sq[threadIdx.x] = q;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sp[threadIdx.x] += sp[threadIdx.x + o];
      sq[threadIdx.x] += sq[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    overlap[2 * s] = sp[0] / n;
    overlap[2 * s + 1] = sq[0] / n;
  }
}

// Clause correlations as lbp_corr_kernel, from f = 1 / (1 + E) = (1 - t) / 2 and t = tanh h, each from
// whichever of E - 1, E and 1 / E is the small one.
__global__ void lbp_corr_prod_kernel(const int32_t *__restrict__ clits, int32_t m, int32_t kmax,
                                     int32_t n, int32_t S, const double *__restrict__ E, double c,
                                     double *corr) {
  const long long total = (long long)m * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long a = i / S;
    const int s = (int)(i - a * S);
    double free_prod = 1.0, viol_prod = 1.0, sign = 1.0;
    int k = 0;
    for (int q = 0; q < kmax; ++q) {
      const long long e = a * kmax + q;
      const int l = clits[e];
      if (l >= 2 * n) continue;
      const double sg = lit_sigma(l), v = E[e * S + s];
      double f = 1.0 / edge_plus_one(v), t;
      if (v >= 1.0) {  // E >= 2
        t = fma(-2.0, f, 1.0);
      } else if (v > -0.5) {
        t = v * f;
        f = fma(-0.5, t, 0.5);
      } else {
        const double x = edge_scaled(v) ? v * (-1.0 / kEdgeScale) : 1.0 + v;
        t = fma(2.0 * x, f, -1.0);
        f = fma(-x, f, 1.0);
      }
      free_prod *= sg * t;
      viol_prod *= f;
      sign *= -sg;
      ++k;
    }
    corr[(size_t)s * m + a] = k > 0 ? fma(-c * sign, viol_prod, free_prod) / fma(-c, viol_prod, 1.0) : 0.0;
  }
}

template <int K>
void clause_prod(const int32_t *clits, int32_t m, int32_t n, int32_t S, const double *E, double *msg,
                 double c, const int32_t *status, unsigned long long *dmax, int track, float slack,
                 unsigned grid, cudaStream_t st) {
  lbp_clause_prod_kernel<K><<<grid, kLbpBlock, 0, st>>>(clits, m, n, S, E, msg, c, status, dmax, track,
                                                      slack);
}

// Per seed after an iteration at lambda index k: count, convergence, failure, bookkeeping.
__global__ void lbp_control_kernel(int32_t S, int32_t k, int32_t n_lambda, double tol,
                                   int32_t max_iter, int32_t *status, int32_t *iters,
                                   double *deltas, int32_t *n_done, int32_t *lam_idx,
                                   int32_t *copy_flag, unsigned long long *dmax, int32_t *running) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s >= S || status[s] != kRunning) return;
  const double d = __longlong_as_double((long long)dmax[s]);
  dmax[s] = 0ull;
  const int it = ++iters[(size_t)s * n_lambda + k];
  deltas[(size_t)s * n_lambda + k] = d;
  if (d < tol) {
    n_done[s] = k + 1;
    lam_idx[s] = k;
    copy_flag[s] = 1;  // work -> good
    status[s] = kWaiting;
  } else if (it >= max_iter) {
    if (n_done[s] > 0) copy_flag[s] = 2;  // good -> work (fall back)
    else lam_idx[s] = k;
    status[s] = kFinished;
  } else {
    atomicAdd(running, 1);
  }
}

__global__ void lbp_copy_kernel(long long n_edges, int32_t S, int32_t *copy_flag, double *h,
                                double *u, double *hg, double *ug) {
  const long long total = n_edges * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int f = copy_flag[i % S];
    if (f == 1) {
      hg[i] = h[i];
      ug[i] = u[i];
    } else if (f == 2) {
      h[i] = hg[i];
      u[i] = ug[i];
    }
  }
}

__global__ void lbp_clear_flags_kernel(int32_t S, int32_t *copy_flag) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < S) copy_flag[s] = 0;
}

// Start of lambda index k: waiting seeds run again (k < n_lambda) or finish.
__global__ void lbp_advance_kernel(int32_t S, int32_t k, int32_t n_lambda, int32_t *status) {
  const int s = blockIdx.x * blockDim.x + threadIdx.x;
  if (s < S && status[s] == kWaiting) status[s] = k < n_lambda ? kRunning : kFinished;
}

// Marginals <r_v> (new order -> original order) with each seed's own lambda, and (p, q1) per
// seed in a fixed summation order (one block per seed).
__global__ void lbp_marg_kernel(const int32_t *__restrict__ vptr, const int32_t *__restrict__ vedge,
                                const int32_t *__restrict__ clits, const int32_t *__restrict__ orig,
                                int32_t n, int32_t S, const double *__restrict__ eps,
                                const uint8_t *__restrict__ xs, const double *__restrict__ lambdas,
                                const int32_t *__restrict__ lam_idx, const double *__restrict__ u,
                                double *marg, double *overlap) {
  const int s = blockIdx.x;
  const double lam = lambdas[lam_idx[s]];
  __shared__ double sp[kLbpBlock], sq[kLbpBlock];
  double p = 0.0, q = 0.0;
  for (int v = threadIdx.x; v < n; v += blockDim.x) {
    const double sv = 2.0 * (double)xs[(size_t)v * S + s] - 1.0;
    double field = lam * eps[v] * sv;
    for (int k = vptr[v]; k < vptr[v + 1]; ++k) {
      const long long e = vedge[k];
      field += lit_sigma(clits[e]) * u[e * S + s];
    }
    const double mv = tanh(field);
    marg[(size_t)s * n + orig[v]] = mv;
    p += sv * mv;
    q += mv * mv;
  }
  sp[threadIdx.x] = p;
  sq[threadIdx.x] = q;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      sp[threadIdx.x] += sp[threadIdx.x + o];
      sq[threadIdx.x] += sq[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    overlap[2 * s] = sp[0] / n;
    overlap[2 * s + 1] = sq[0] / n;
  }
}

// <prod_{i in a} r_i> = [prod_i sigma_i t_i - c prod_i (-sigma_i) (1 - t_i)/2] / z_a,
// z_a = 1 - c prod_i (1 - t_i)/2, t_i = tanh h_{i->a} (the clause's configurations summed in
// closed form: the violating configuration r_i = -sigma_i carries weight e^{-2 beta}).
__global__ void lbp_corr_kernel(const int32_t *__restrict__ clits, int32_t m, int32_t kmax,
                                int32_t n, int32_t S, const double *__restrict__ h, double c,
                                double *corr) {
  const long long total = (long long)m * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const long long a = i / S;
    const int s = (int)(i % S);
    double free_prod = 1.0, viol_prod = 1.0, sign = 1.0;
    int k = 0;
    for (int q = 0; q < kmax; ++q) {
      const long long e = a * kmax + q;
      const int l = clits[e];
      if (l >= 2 * n) continue;
      const double sg = lit_sigma(l), t = tanh(h[e * S + s]);
      free_prod *= sg * t;
      viol_prod *= (1.0 - t) / 2.0;
      sign *= -sg;
      ++k;
    }
    const double z = 1.0 - c * viol_prod;
    corr[(size_t)s * m + a] = k > 0 ? (free_prod - c * sign * viol_prod) / z : 0.0;
  }
}

unsigned blocks_for(long long work) {
  long long g = (work + kLbpBlock - 1) / kLbpBlock;
  if (g > 152 * 32) g = 152 * 32;
  return (unsigned)(g < 1 ? 1 : g);
}

}  // namespace

// xs[v][s] = x_in[s][orig v] (0/1), eps[v] = eps_in[orig v] or, without eps_in, the number of
// clauses of v.
static __global__ void lbp_prepare_kernel(const uint8_t *__restrict__ x_in, const double *__restrict__ eps_in,
                                   const int32_t *__restrict__ orig, const int32_t *__restrict__ vptr,
                                   int32_t n, int32_t S, uint8_t *xs, double *eps) {
  const long long total = (long long)n * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int v = (int)(i / S), s = (int)(i % S);
    xs[i] = x_in[(size_t)s * n + orig[v]];
    if (s == 0) eps[v] = eps_in ? eps_in[orig[v]] : (double)(vptr[v + 1] - vptr[v]);
  }
}

size_t lbp_scratch_bytes(int32_t n, int32_t m, int32_t kmax, int32_t S, int32_t n_lambda) {
  auto up = [](size_t b) { return (b + 255) & ~static_cast<size_t>(255); };
  const size_t E = (size_t)m * kmax;
  return 4 * up(sizeof(double) * E * S) + up(sizeof(double) * (size_t)n * S) +
         up(sizeof(unsigned long long) * S) + 3 * up(sizeof(int32_t) * S) + up(sizeof(int32_t)) +
         up(sizeof(double) * n_lambda);
}

cudaError_t lbp_prepare(const uint8_t *x_in, const double *eps_in, const int32_t *orig,
                        const int32_t *vptr, int32_t n, int32_t S, uint8_t *xs, double *eps,
                        cudaStream_t st) {
  lbp_prepare_kernel<<<blocks_for((long long)n * S), kLbpBlock, 0, st>>>(x_in, eps_in, orig, vptr, n,
                                                                      S, xs, eps);
  return cudaGetLastError();
}

int lbp_run(const LbpArgs &A, cudaStream_t st) {
  auto up = [](size_t b) { return (b + 255) & ~static_cast<size_t>(255); };
  const int32_t S = A.S, n = A.n, m = A.m, kmax = A.kmax, L = A.n_lambda;
  const long long E = (long long)m * kmax;
  char *p = static_cast<char *>(A.scratch);
  double *h = reinterpret_cast<double *>(p); p += up(sizeof(double) * E * S);
  double *u = reinterpret_cast<double *>(p); p += up(sizeof(double) * E * S);
  double *hg = reinterpret_cast<double *>(p); p += up(sizeof(double) * E * S);
  double *ug = reinterpret_cast<double *>(p); p += up(sizeof(double) * E * S);
  double *bias = reinterpret_cast<double *>(p); p += up(sizeof(double) * (size_t)n * S);
  unsigned long long *dmax = reinterpret_cast<unsigned long long *>(p); p += up(sizeof(unsigned long long) * S);
  int32_t *status = reinterpret_cast<int32_t *>(p); p += up(sizeof(int32_t) * S);
  int32_t *lam_idx = reinterpret_cast<int32_t *>(p); p += up(sizeof(int32_t) * S);
  int32_t *copy_flag = reinterpret_cast<int32_t *>(p); p += up(sizeof(int32_t) * S);
  int32_t *running = reinterpret_cast<int32_t *>(p); p += up(sizeof(int32_t));
  double *lam_dev = reinterpret_cast<double *>(p);
  const double c = -expm1(-2.0 * A.beta);
  cudaError_t e;
#define LBP_CHECK(x)                 \
  do {                               \
    if ((e = (x)) != cudaSuccess) return (int)e; \
  } while (0)
  LBP_CHECK(cudaMemsetAsync(dmax, 0, sizeof(unsigned long long) * S, st));
  LBP_CHECK(cudaMemsetAsync(status, 0, sizeof(int32_t) * S, st));  // kRunning
  LBP_CHECK(cudaMemsetAsync(lam_idx, 0, sizeof(int32_t) * S, st));
  LBP_CHECK(cudaMemsetAsync(copy_flag, 0, sizeof(int32_t) * S, st));
  LBP_CHECK(cudaMemsetAsync(A.iters, 0, sizeof(int32_t) * S * L, st));
  LBP_CHECK(cudaMemsetAsync(A.deltas, 0, sizeof(double) * S * L, st));
  LBP_CHECK(cudaMemsetAsync(A.n_done, 0, sizeof(int32_t) * S, st));
  LBP_CHECK(cudaMemsetAsync(u, 0, sizeof(double) * E * S, st));
  LBP_CHECK(cudaMemcpyAsync(lam_dev, A.lambdas, sizeof(double) * L, cudaMemcpyHostToDevice, st));
  const unsigned gS = (unsigned)((S + kLbpBlock - 1) / kLbpBlock);
  const unsigned gVS = blocks_for((long long)n * S), gMS = blocks_for((long long)m * S),
                 gES = blocks_for(E * S);
  // the product form needs every product of 1 - m and every e^{2 field} inside the range of a double:
  // u lies in [0, beta], so |field| <= beta deg + |lambda eps|. m near c is resolved to about 1e-16, a
  // change of u to 1e-16 e^{2 beta} / 2: smaller tolerances take the log form, which has settled as
  // far as it can there
  const bool prod = A.beta <= 4.0 && A.beta * A.max_deg + A.max_bias < 340.0 &&
                    A.tol >= 2e-15 * exp(2.0 * A.beta);
  // four lanes a variable where there would be fewer than eight warps an SM otherwise, in blocks small
  // enough to reach every SM (5 seeds of 500 variables: 40 blocks of 256 threads, 157 of 64)
  constexpr int kSplitBlock = 64;
  const bool split = (long long)n * S < 152 * 256;
  const unsigned gSplit = (unsigned)((4LL * n * S + kSplitBlock - 1) / kSplitBlock);
  const float slack = (float)((exp(2.0 * A.beta) + 8.0) * 0x1p-21);
  const auto clause = [&](const int32_t *seeds, int track) {
    if (!prod) {
      lbp_clause_kernel<<<gMS, kLbpBlock, 0, st>>>(A.clits, m, kmax, n, S, h, u, c, seeds, dmax, track);
      return;
    }
    switch (kmax) {
#define LBP_CASE(k) \
  case k: clause_prod<k>(A.clits, m, n, S, h, u, c, seeds, dmax, track, slack, gMS, st); break;
      LBP_CASE(1) LBP_CASE(2) LBP_CASE(3) LBP_CASE(4)
      LBP_CASE(5) LBP_CASE(6) LBP_CASE(7) LBP_CASE(8)
#undef LBP_CASE
    }
  };
  const auto bias_at = [&](double lambda) {
    if (prod) lbp_gain_kernel<<<gVS, kLbpBlock, 0, st>>>(A.eps, A.xs, n, S, lambda, bias);
    else lbp_bias_kernel<<<gVS, kLbpBlock, 0, st>>>(A.eps, A.xs, n, S, lambda, bias);
  };
  // initial messages at lambda_0: h from the bias, u from those h
  bias_at(A.lambdas[0]);
  if (prod) lbp_init_prod_kernel<<<gES, kLbpBlock, 0, st>>>(A.clits, E, n, S, bias, h);
  else lbp_init_h_kernel<<<gES, kLbpBlock, 0, st>>>(A.clits, E, n, S, bias, h);
  clause(nullptr, 0);
  LBP_CHECK(cudaGetLastError());
  for (int32_t k = 0; k < L; ++k) {
    if (k > 0) {
      lbp_advance_kernel<<<gS, kLbpBlock, 0, st>>>(S, k, L, status);
      bias_at(A.lambdas[k]);
    }
    // One iteration is always queued behind the one whose outcome the host reads: once no seed is
    // running the queued one changes nothing (every kernel leaves seeds that are not running
    // alone), and the GPU does not wait for the host in between.
    for (int32_t it = 0; it < A.max_iter; ++it) {
      if (prod && split)
        lbp_var_prod_kernel<4><<<gSplit, kSplitBlock, 0, st>>>(A.vptr, A.vedge, A.clits, n, S, bias, u, h,
                                                             status);
      else if (prod)
        lbp_var_prod_kernel<1><<<gVS, kLbpBlock, 0, st>>>(A.vptr, A.vedge, A.clits, n, S, bias, u, h,
                                                          status);
      else
        lbp_var_kernel<<<gVS, kLbpBlock, 0, st>>>(A.vptr, A.vedge, A.clits, n, S, bias, u, h, status);
      clause(status, 1);
      LBP_CHECK(cudaMemsetAsync(running, 0, sizeof(int32_t), st));
      lbp_control_kernel<<<gS, kLbpBlock, 0, st>>>(S, k, L, A.tol, A.max_iter, status, A.iters,
                                                   A.deltas, A.n_done, lam_idx, copy_flag, dmax,
                                                   running);
      LBP_CHECK(cudaGetLastError());
      LBP_CHECK(cudaMemcpyAsync(A.seen + (it & 1), running, sizeof(int32_t), cudaMemcpyDeviceToHost, st));
      LBP_CHECK(cudaEventRecord(A.ev[it & 1], st));
      if (it == 0) continue;
      LBP_CHECK(cudaEventSynchronize(A.ev[(it - 1) & 1]));
      if (A.seen[(it - 1) & 1] == 0) break;
    }
    // seeds that converged or gave up at this lambda stopped changing: snapshots once, at its end
    lbp_copy_kernel<<<gES, kLbpBlock, 0, st>>>(E, S, copy_flag, h, u, hg, ug);
    lbp_clear_flags_kernel<<<gS, kLbpBlock, 0, st>>>(S, copy_flag);
    LBP_CHECK(cudaGetLastError());
  }
  lbp_advance_kernel<<<gS, kLbpBlock, 0, st>>>(S, L, L, status);
  if (prod) {
    lbp_marg_prod_kernel<<<gVS, kLbpBlock, 0, st>>>(A.vptr, A.vedge, A.clits, A.orig, n, S, A.eps,
                                                    A.xs, lam_dev, lam_idx, u, A.marg);
    lbp_overlap_kernel<<<S, kLbpBlock, 0, st>>>(A.orig, n, S, A.xs, A.marg, A.overlap);
    lbp_corr_prod_kernel<<<gMS, kLbpBlock, 0, st>>>(A.clits, m, kmax, n, S, h, c, A.corr);
  } else {
    lbp_marg_kernel<<<S, kLbpBlock, 0, st>>>(A.vptr, A.vedge, A.clits, A.orig, n, S, A.eps, A.xs,
                                            lam_dev, lam_idx, u, A.marg, A.overlap);
    lbp_corr_kernel<<<gMS, kLbpBlock, 0, st>>>(A.clits, m, kmax, n, S, h, c, A.corr);
  }
  LBP_CHECK(cudaGetLastError());
#undef LBP_CHECK
  return 0;
}

// ---- backbones ------------------------------------------------------------------------------
//
// J~_a = atanh|<prod r>| / beta. Factors with J~ above the cutoff or the seed threshold link
// their variables; components under the linking factors are found by label propagation (min
// original id, with pointer jumping); a component is a backbone when it holds a seed factor
// (J~ above the seed threshold). Labels: the component's smallest original variable id, -1
// outside every backbone. S problems (seeds) side by side: labels [S][n] in new order.
namespace {

constexpr int32_t kNoLabel = 0x7FFFFFFF;

__global__ void bb_init_kernel(const int32_t *__restrict__ clits, int32_t m, int32_t kmax,
                               int32_t n, int32_t S, const double *__restrict__ corr, double beta,
                               double seed_thr, double cutoff, const int32_t *__restrict__ orig,
                               uint8_t *link, int32_t *label) {
  const long long total = (long long)m * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int s = (int)(i / m);
    const long long a = i % m;
    const double jt = atanh(fabs(corr[(size_t)s * m + a])) / beta;
    const uint8_t f = (uint8_t)((jt > cutoff || jt > seed_thr) ? 1 : 0) | (uint8_t)(jt > seed_thr ? 2 : 0);
    link[i] = f;
    if (f)
      for (int q = 0; q < kmax; ++q) {
        const int l = clits[a * kmax + q];
        if (l < 2 * n) label[(size_t)s * n + (l >> 1)] = orig[l >> 1];  // same value from every writer
      }
  }
}

__global__ void bb_fill_kernel(int32_t n, int32_t S, int32_t *label) {
  const long long total = (long long)n * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x)
    label[i] = kNoLabel;
}

__global__ void bb_propagate_kernel(const int32_t *__restrict__ clits, int32_t m, int32_t kmax,
                                    int32_t n, int32_t S, const uint8_t *__restrict__ link,
                                    int32_t *label, int32_t *changed) {
  const long long total = (long long)m * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    if (!link[i]) continue;
    const int s = (int)(i / m);
    const long long a = i % m;
    int32_t *ls = label + (size_t)s * n;
    int mn = kNoLabel;
    for (int q = 0; q < kmax; ++q) {
      const int l = clits[a * kmax + q];
      if (l < 2 * n) mn = min(mn, ls[l >> 1]);
    }
    for (int q = 0; q < kmax; ++q) {
      const int l = clits[a * kmax + q];
      if (l < 2 * n && atomicMin(&ls[l >> 1], mn) > mn) *changed = 1;
    }
  }
}

// Pointer jumping: a label is the original id of a variable whose own label may be smaller.
__global__ void bb_jump_kernel(int32_t n, int32_t S, const int32_t *__restrict__ newid,
                               int32_t *label, int32_t *changed) {
  const long long total = (long long)n * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int s = (int)(i / n);
    const int l = label[i];
    if (l == kNoLabel) continue;
    const int l2 = label[(size_t)s * n + newid[l]];
    if (l2 < l && atomicMin(&label[i], l2) > l2) *changed = 1;
  }
}

__global__ void bb_seed_kernel(const int32_t *__restrict__ clits, int32_t m, int32_t kmax,
                               int32_t n, int32_t S, const uint8_t *__restrict__ link,
                               const int32_t *__restrict__ label, const int32_t *__restrict__ newid,
                               uint8_t *seeded) {
  const long long total = (long long)m * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    if (!(link[i] & 2)) continue;
    const int s = (int)(i / m);
    const long long a = i % m;
    for (int q = 0; q < kmax; ++q) {
      const int l = clits[a * kmax + q];
      if (l < 2 * n) {
        seeded[(size_t)s * n + newid[label[(size_t)s * n + (l >> 1)]]] = 1;
        break;
      }
    }
  }
}

__global__ void bb_final_kernel(int32_t n, int32_t S, const int32_t *__restrict__ orig,
                                const int32_t *__restrict__ newid, const int32_t *__restrict__ label,
                                const uint8_t *__restrict__ seeded, int32_t *out, int32_t *n_clusters) {
  const long long total = (long long)n * S;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int s = (int)(i / n), v = (int)(i % n);
    const int l = label[i];
    int r = -1;
    if (l != kNoLabel && seeded[(size_t)s * n + newid[l]]) {
      r = l;
      if (orig[v] == l) atomicAdd(&n_clusters[s], 1);
    }
    out[(size_t)s * n + orig[v]] = r;
  }
}

// The two-chain schedule of Algorithm 1 in Q16, step-major: per cycle t_hot steps with the
// backbone at base / heat and the rest held, t_cold steps with the backbone held and the rest at
// base, t_unlearn steps with every variable at base.
__global__ void bb_schedule_kernel(const int32_t *__restrict__ lab, const int32_t *__restrict__ orig,
                                   int32_t n, int32_t n_steps,
                                   float base, float heat, int32_t t_hot, int32_t t_cold,
                                   int32_t t_unlearn, uint32_t *bq) {
  const long long total = (long long)n * n_steps;
  const uint32_t qb = __float2uint_rn(base * 65536.0f);
  const uint32_t qh = __float2uint_rn(__fdiv_rn(base, heat) * 65536.0f);
  const int cyc = t_hot + t_cold + t_unlearn;
  for (long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x; i < total;
       i += (long long)gridDim.x * blockDim.x) {
    const int t = (int)(i / n), v = (int)(i % n);
    const int pos = t % cyc;
    const bool bb = lab[orig[v]] >= 0;
    uint32_t q;
    if (pos < t_hot) q = bb ? qh : kFrozenQ16;
    else if (pos < t_hot + t_cold) q = bb ? kFrozenQ16 : qb;
    else q = qb;
    bq[i] = q;
  }
}

}  // namespace

size_t backbone_scratch_bytes(int32_t n, int32_t m, int32_t S) {
  auto up = [](size_t b) { return (b + 255) & ~static_cast<size_t>(255); };
  return up((size_t)m * S) + up(sizeof(int32_t) * (size_t)n * S) + up((size_t)n * S) +
         2 * up(sizeof(int32_t) * S) + up(sizeof(int32_t));
}

int backbone_run(const BackboneArgs &A, cudaStream_t st) {
  auto up = [](size_t b) { return (b + 255) & ~static_cast<size_t>(255); };
  const int32_t n = A.n, m = A.m, S = A.S;
  char *p = static_cast<char *>(A.scratch);
  uint8_t *link = reinterpret_cast<uint8_t *>(p); p += up((size_t)m * S);
  int32_t *label = reinterpret_cast<int32_t *>(p); p += up(sizeof(int32_t) * (size_t)n * S);
  uint8_t *seeded = reinterpret_cast<uint8_t *>(p); p += up((size_t)n * S);
  p += 2 * up(sizeof(int32_t) * S);
  int32_t *changed = reinterpret_cast<int32_t *>(p);
  cudaError_t e;
  if ((e = cudaMemsetAsync(seeded, 0, (size_t)n * S, st)) != cudaSuccess) return (int)e;
  if ((e = cudaMemsetAsync(A.n_clusters, 0, sizeof(int32_t) * S, st)) != cudaSuccess) return (int)e;
  bb_fill_kernel<<<blocks_for((long long)n * S), kLbpBlock, 0, st>>>(n, S, label);
  bb_init_kernel<<<blocks_for((long long)m * S), kLbpBlock, 0, st>>>(A.clits, m, A.kmax, n, S, A.corr,
                                                                  A.beta, A.seed_thr, A.cutoff,
                                                                  A.orig, link, label);
  if ((e = cudaGetLastError()) != cudaSuccess) return (int)e;
  // every round lowers some label or stops; n rounds bound any component's propagation
  for (int32_t round = 0; round <= n + 1; ++round) {
    if ((e = cudaMemsetAsync(changed, 0, sizeof(int32_t), st)) != cudaSuccess) return (int)e;
    bb_propagate_kernel<<<blocks_for((long long)m * S), kLbpBlock, 0, st>>>(A.clits, m, A.kmax, n, S,
                                                                         link, label, changed);
    bb_jump_kernel<<<blocks_for((long long)n * S), kLbpBlock, 0, st>>>(n, S, A.newid, label, changed);
    if ((e = cudaGetLastError()) != cudaSuccess) return (int)e;
    int32_t ch = 0;
    if ((e = cudaMemcpyAsync(&ch, changed, sizeof(int32_t), cudaMemcpyDeviceToHost, st)) != cudaSuccess ||
        (e = cudaStreamSynchronize(st)) != cudaSuccess)
      return (int)e;
    if (!ch) break;
  }
  bb_seed_kernel<<<blocks_for((long long)m * S), kLbpBlock, 0, st>>>(A.clits, m, A.kmax, n, S, link,
                                                                  label, A.newid, seeded);
  bb_final_kernel<<<blocks_for((long long)n * S), kLbpBlock, 0, st>>>(n, S, A.orig, A.newid, label,
                                                                   seeded, A.labels, A.n_clusters);
  return (int)cudaGetLastError();
}

cudaError_t backbone_schedule(const int32_t *lab, const int32_t *orig, int32_t n, int32_t n_steps,
                              float base, float heat, int32_t t_hot, int32_t t_cold,
                              int32_t t_unlearn, uint32_t *bq, cudaStream_t st) {
  bb_schedule_kernel<<<blocks_for((long long)n * n_steps), kLbpBlock, 0, st>>>(
      lab, orig, n, n_steps, base, heat, t_hot, t_cold, t_unlearn, bq);
  return cudaGetLastError();
}

}  // namespace nmc
