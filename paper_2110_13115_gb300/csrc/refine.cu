// Candidate refinement (step a8): J(theta) = |Z(theta)|^2 / sigma^2 of a non-spinning TaylorF2
// template at its own coalescence time, its adjoint with respect to theta = (mc, eta, t_c, phi_c),
// and an in-kernel gradient ascent. The matched filter is Eq. (1) of arXiv:2110.13115 evaluated at
// t_0 = t_c (Eq. 3-4); the paper stops at the triggers, so the ascent rule is this library's own
// (see include/rbmf.h). One CTA or a cluster per candidate recomputes the whitened template frequency by
// frequency in every pass.
//
// Arithmetic. The GPU does two FP64 operations per clock and SM against 128 in FP32, and a point took about 90 of
// them (four divisions among them). FP64 is left to the phase, which needs it (Psi reaches 1e5 rad and more and is
// rounded to FP32 only after its reduction modulo 2 pi), in 16 operations: 1 / v comes from a table of 1 / vf and one
// Newton step that rounds it correctly, 2 pi f from a table, the reduction multiplies by 1 / (2 pi). The rest runs in FP32
// with values in three parts (an unevaluated sum, 72 bits; the products and sums are the classical error-free ones): the
// term amp s_hat e^(i Psi), and its sums. The derivatives of Psi are linear in f, F5 = (pi f)^(-5/3), F3 = (pi f)^(-1) and
// F2 = (pi f)^(-2/3) with coefficients that are constant over the points, so a pass sums the terms and their moments
// with those four, and one thread forms the gradient.
// Precision. Against sums in 64-bit mantissas over the same sines and cosines, relative to the norm of what is summed
// (rms over candidates; mc, eta, t_c, phi_c): n = 2^14 3.5, 2.3, 1.6, 1.1 x 1e-16, where plain FP64 had 5.2, 23.9, 2.6,
// 2.9; n = 2^16, third order 7.2, 3.0, 2.7, 1.7 (8.6, 5.9, 5.2, 5.1); n = 2^19 7.6, 5.0, 2.9, 2.8 (10.3, 24.6, 6.6, 6.8). With
// pairs of values (48 bits) it was 20 to 40 throughout.
// Range. amp goes with the PSD and the units of the strain over hundreds of decades, s_hat over FP32's: the products
// amp s_hat are formed in FP64 and kept as values of order one with an exponent of their own, and a candidate takes them
// relative to the largest exponent of its own support. So neither a bin outside the support nor another candidate moves
// them, and what is lost is 2^-126 of the support's largest value and below.
// Measured (FP64 issue bounds it, 16 operations a point; the FP32 work beside it is twice that of pairs and nearly free):
// value and gradient of 500 candidates at n = 2^19 1.55 ms against 4.39 ms with every point in FP64 and 1.51 ms with
// pairs. A phase in pairs too would take 0.65 ms, but it rounds to another FP32 phase at one point in some thousands.
//
// The ascent stays in FP64 (k_refine_ascend): a last digit of the gradient is a last digit of theta, which moves the FP32
// phase of a few points, and so J by 1e-9, and now and then the choice of a step; with sums in FP32 parts, J came out up to
// 6e-9 (norm over the candidates) from what this library gave before. It does the same roundings in the same order (the FMAs
// are written out, so that no compiler regroups them) in 45 FP64 operations a point instead of about 90: quotients by
// reciprocals formed once per pass, 1 / v as above, tables, sine and cosine widened by their bits, no sums twice.
// 512 candidates x 20 steps at n = 2^17: 7.11 ms against 15.3 ms, bit for bit.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "common.cuh"
#include "internal.h"

namespace cg = cooperative_groups;

namespace {

constexpr double kMsunS = 4.925491025543576e-06;
constexpr double kPi = 3.14159265358979323846;
constexpr double kFref = 100.0;
constexpr double kEtaMin = 0.05;
constexpr int kThreads = 128;
constexpr int kMaxRanks = 8;  // CTAs (a cluster) that share a candidate's frequencies in value and adjoint, at most
// Value and adjoint sum a candidate's frequencies in `strands` of every strands-th block of kThreads, as many as CTAs may
// share a candidate at this n, each by one CTA from beginning to end, and the strands' sums in their order: a candidate's
// result has the same bits however many CTAs its company leaves it. One CTA with all the strands loses 1 to 3 % to a single
// sum (value and adjoint at n = 2^17, 456 candidates: 443 us before, 457 so; n = 2^19, 500: 1.70 and 1.72 ms).
constexpr int kAscThreads = 256;  // threads of a candidate in the ascent
// CTAs (a cluster) that these are spread over, in 20 steps of 512 candidates at n = 2^17 / of 64 at n = 2^15:
// one 7.07 / 0.89 ms (two resident per SM, so that 512 leave the second wave two thirds empty), two 6.38 / 0.67,
// four 6.81 / 0.66, eight 7.40 / 0.68.
constexpr int kAscRanks = 2;

enum { R_EVAL = 0, R_ADJOINT = 1 };

// Workspace header: flags, the first frequency above every candidate's support.
struct Header {
  unsigned flags, jmax;
};

struct RefArgs {
  const float2* shat;
  const double* psd;
  Header* head;
  float4* w;      // 2^-e amp s_hat in three parts: (re h, im h, re m, im m), amp = f^(-7/6) sqrt(4 df / S)
  float4* wl;     // (re l, im l, e as an integer: the exponent of the larger part)
  double2* v;     // (vf, 1 / vf), vf = (pi f)^(1/3)
  double* x;      // 2 pi f
  float4* g;      // (F5 h, F5 m, F3 h, F3 m) over their values at the band's first frequency
  float2* gl;     // (F5 l, F3 l)
  float4* g2;     // (F2 h, F2 m, F2 l)
  double* amp2;   // amp^2, zero below the band
  double* chunk;  // sums of amp2 over blocks of kThreads frequencies
  int* top;       // the largest e of these blocks
  // the ascent's tables, in the place of w and amp2: s_hat and f^(-7/6) sqrt(4 df / S) in FP64
  double2* sh;
  double* amp;
  int64_t half, jlo;
  int strands;  // 1, 2, 4 or 8
  double df;
  double amp0;                       // amp = amp0 j^(-7/6) / sqrt(S)
  double r53, r33, r23;              // jlo^(5/3), jlo, jlo^(2/3)
  double f5, f3, f2;                 // F5, F3, F2 at the band's first frequency
  int pn;
  const double* theta_in;
  double* theta_out;
  double* J;
  double* Z;
  const double* dJ;
  double* dtheta;
  int64_t n_cand;
  int steps;
  double alpha0, alpha_max;
};

// --- division -----------------------------------------------------------------------------------
// Quotients and reciprocals by the corrections with fused multiply-adds of Markstein (IBM J. Res. Dev. 34, 1990): the
// residual of a guess within a few units in the last place is exact, and its correction rounds once, so the result is the
// rounded quotient unless that lies within some 2^-50 units of a tie.
// x / d by the rounded r = 1 / d
__host__ __device__ __forceinline__ double quotient(double x, double d, double r) {
  const double q = x * r;
  return fma(fma(-d, q, x), r, q);
}
// 1 / v
__host__ __device__ __forceinline__ double reciprocal(double v, double guess) { return fma(guess, fma(-v, guess, 1.0), guess); }

// --- values in three parts ------------------------------------------------------------------------
// An unevaluated sum of three FP32 values, 72 bits: it holds an FP64 value exactly.
struct Three {
  float h, m, l;
};
__device__ __forceinline__ Three to_three(double x) {
  const float h = (float)x;
  if (!isfinite(h)) return {h, 0.f, 0.f};
  const double r = x - (double)h;
  const float m = (float)r;
  return {h, m, (float)(r - (double)m)};
}
// s + e = a + b exactly (Knuth)
__device__ __forceinline__ float two_sum(float a, float b, float& e) {
  const float s = __fadd_rn(a, b), t = __fsub_rn(s, a);
  e = __fadd_rn(__fsub_rn(a, __fsub_rn(s, t)), __fsub_rn(b, t));
  return s;
}
// p + e = a b exactly
__device__ __forceinline__ float two_prod(float a, float b, float& e) {
  const float p = __fmul_rn(a, b);
  e = __fmaf_rn(a, b, -p);
  return p;
}
__device__ __forceinline__ void add(Three& s, const Three& o) {
  float e1, e2, e3;
  s.h = two_sum(s.h, o.h, e1);
  const float x = two_sum(e1, o.m, e2);
  s.m = two_sum(s.m, x, e3);
  s.l = __fadd_rn(s.l, __fadd_rn(__fadd_rn(e2, e3), o.l));
}
__device__ __forceinline__ Three shuffle_xor(const Three& s, int off) {
  return {__shfl_xor_sync(0xffffffffu, s.h, off), __shfl_xor_sync(0xffffffffu, s.m, off), __shfl_xor_sync(0xffffffffu, s.l, off)};
}
__device__ __forceinline__ Three mul(const Three& a, float b) {
  float e1, e2, e3;
  const float p = two_prod(a.h, b, e1), q = two_prod(a.m, b, e2), m = two_sum(e1, q, e3);
  return {p, m, __fmaf_rn(a.l, b, __fadd_rn(e2, e3))};
}
__device__ __forceinline__ Three mul(const Three& a, const Three& b) {
  float e1, e2, e3, e4, e5;
  const float p = two_prod(a.h, b.h, e1), q = two_prod(a.h, b.m, e2), r = two_prod(a.m, b.h, e3);
  const float s = two_sum(q, r, e4), m = two_sum(s, e1, e5);
  return {p, m, __fmaf_rn(a.h, b.l, __fmaf_rn(a.m, b.m, __fmaf_rn(a.l, b.h, __fadd_rn(__fadd_rn(e2, e3), __fadd_rn(e4, e5)))))};
}
// a b + c d
__device__ __forceinline__ Three dot(const Three& a, float b, const Three& c, float d) {
  float e1, e2, e3, e4, e5, e6, e7, e8, e9;
  const float p = two_prod(a.h, b, e1), q = two_prod(c.h, d, e2), h = two_sum(p, q, e3);
  const float r = two_prod(a.m, b, e4), t = two_prod(c.m, d, e5);
  const float x = two_sum(e1, e2, e6), y = two_sum(r, t, e7), z = two_sum(x, y, e8), m = two_sum(z, e3, e9);
  const float l = __fadd_rn(__fadd_rn(e4, e5), __fadd_rn(__fadd_rn(e6, e7), __fadd_rn(e8, e9)));
  return {h, m, __fmaf_rn(a.l, b, __fmaf_rn(c.l, d, l))};
}

// The exponent e of a complex value: its larger part lies in [2^e, 2^(e + 1)) (zero and below FP64's normal range:
// -1023; not finite: 1024).
__device__ __forceinline__ int exponent(double re, double im) {
  return (int)(__double_as_longlong(fmax(fabs(re), fabs(im))) >> 52) - 1023;
}

// PSD check (0 < j < half), and the end of the candidates' supports (an FP32 estimate with a margin: it only bounds
// the tables).
__global__ void __launch_bounds__(kThreads) k_refine_check(RefArgs a) {
  const int64_t tid = blockIdx.x * (int64_t)blockDim.x + threadIdx.x, stride = (int64_t)gridDim.x * blockDim.x;
  bool bad = false;
  for (int64_t j = tid + 1; j < a.half; j += stride) {
    const double S = a.psd[j];
    if (!(S > 0.0) || isinf(S)) bad = true;
  }
  unsigned top = 0;
  for (int64_t c = tid; c < a.n_cand; c += stride) {
    const float mc = (float)a.theta_in[4 * c], eta = (float)a.theta_in[4 * c + 1];
    if (!(mc > 0.f) || !(eta > 0.f)) {  // (or below FP32: the whole band; an invalid candidate is refused later)
      top = (unsigned)a.half;
      continue;
    }
    const float fcut = 1.001f / (14.6969385f * (float)kPi * mc * powf(eta, -0.6f) * (float)kMsunS);
    top = max(top, (unsigned)fminf((float)a.half, fcut / (float)a.df + 4.f));
  }
  top = __reduce_max_sync(0xffffffffu, top);
  bad = __any_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0) {
    if (top) atomicMax(&a.head->jmax, top);
    if (bad) atomicOr(&a.head->flags, (unsigned)RB_FLAG_BAD_PSD);
  }
}

// Sum over the block of one double per thread (every thread calls; the result on thread 0 only).
__device__ __forceinline__ double block_sum(double v, double* red) {
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) v += __shfl_xor_sync(0xffffffffu, v, off);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0)
    for (int w = 1; w < kThreads / 32; ++w) v += red[w];
  return v;
}

// The largest of one int per thread over the block (every thread calls and receives it).
__device__ __forceinline__ int block_max(int v, int* red) {
  v = __reduce_max_sync(0xffffffffu, v);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = v;
  __syncthreads();
  v = red[0];
#pragma unroll
  for (int w = 1; w < kThreads / 32; ++w) v = max(v, red[w]);
  return v;
}

constexpr int kNoExponent = -(1 << 20);  // of frequencies outside the band

// The tables on [jlo, jmax): everything is a power of y = j^(-1/6) (an FP32 estimate and a Newton step in FP64, which
// takes its error from 1e-6 to 1e-11). The powers' roundings are kept (x2 .. x10) and so is what y itself is off by, d
// relative to it: with both the table values are rounded once or twice, where a seventh or a tenth power of a rounded y would
// be off by several units, as much as the sums.
__global__ void __launch_bounds__(kThreads) k_refine_tables(RefArgs a) {
  __shared__ double red[kThreads / 32];
  __shared__ int red_e[kThreads / 32];
  const int64_t jmax = min((int64_t)a.head->jmax, a.half);
  for (int64_t c = a.jlo / kThreads + blockIdx.x; c * kThreads < jmax; c += gridDim.x) {
    const int64_t j = c * kThreads + threadIdx.x;
    double a2 = 0.0;
    int e = kNoExponent;
    float4 lows = make_float4(0.f, 0.f, __int_as_float(kNoExponent), 0.f);
    if (j >= a.jlo && j < jmax) {
      const double f = j * a.df, x = (double)(int)j, S = a.psd[j];
      double y = (double)exp2f(log2f((float)(int)j) * (-1.f / 6.f));
      {
        const double y2 = y * y, y6 = y2 * y2 * y2;
        y = y * (fma(-x, y6, 7.0) * (1.0 / 6.0));
      }
      const double y2 = y * y, x2 = fma(y, y, -y2), y3 = y2 * y, x3 = fma(x2, y, fma(y2, y, -y3));
      const double y4 = y2 * y2, x4 = fma(2.0 * y2, x2, fma(y2, y2, -y4)), y6 = y3 * y3, x6 = fma(2.0 * y3, x3, fma(y3, y3, -y6));
      const double d = (fma(-x, y6, 1.0) - x * x6) * (1.0 / 6.0);
      const double y7 = y6 * y, x7 = fma(x6, y, fma(y6, y, -y7));
      const double y10 = y6 * y4, x10 = fma(x6, y4, fma(y6, x4, fma(y6, y4, -y10)));
      // 1 / sqrt(S) = s (1 + h)
      const double s = rsqrt(S), u = S * s, h = 0.5 * (fma(-u, s, 1.0) - fma(S, s, -u) * s);
      const double am = (a.amp0 * s) * (y7 + fma(fma(7.0, d, h), y7, x7));
      const float2 sh = a.shat[j];
      const double wr = am * (double)sh.x, wi = am * (double)sh.y;
      e = exponent(wr, wi);
      const Three re = to_three(scalbn(wr, -e)), im = to_three(scalbn(wi, -e));
      const Three f5 = to_three(a.r53 * (y10 + fma(10.0 * d, y10, x10))), f3 = to_three(a.r33 * (y6 + fma(6.0 * d, y6, x6))),
                  f2 = to_three(a.r23 * (y4 + fma(4.0 * d, y4, x4)));
      const double vf = cbrt(kPi * f);
      a.v[j] = make_double2(vf, 1.0 / vf);
      a.x[j] = 2.0 * kPi * f;
      a.w[j] = make_float4(re.h, im.h, re.m, im.m);
      a.g[j] = make_float4(f5.h, f5.m, f3.h, f3.m);
      a.gl[j] = make_float2(f5.l, f3.l);
      if (a.pn >= 3) a.g2[j] = make_float4(f2.h, f2.m, f2.l, 0.f);
      lows = make_float4(re.l, im.l, __int_as_float(e), 0.f);
      a2 = am * am;
    }
    if (j < a.half) {
      a.amp2[j] = a2;
      a.wl[j] = lows;
    }
    a2 = block_sum(a2, red);
    e = block_max(e, red_e);
    if (threadIdx.x == 0) {
      a.chunk[c] = a2;
      a.top[c] = e;
    }
  }
}

// The ascent's tables on [jlo, jmax).
__global__ void __launch_bounds__(kThreads) k_ascend_tables(RefArgs a) {
  const int64_t jmax = min((int64_t)a.head->jmax, a.half);
  for (int64_t j = a.jlo + blockIdx.x * (int64_t)kThreads + threadIdx.x; j < jmax; j += (int64_t)gridDim.x * kThreads) {
    const double f = j * a.df, vf = cbrt(kPi * f);
    const float2 sh = a.shat[j];
    a.v[j] = make_double2(vf, 1.0 / vf);
    a.x[j] = 2.0 * kPi * f;
    a.sh[j] = make_double2(sh.x, sh.y);
    a.amp[j] = pow(f, -7.0 / 6.0) * sqrt(4.0 * a.df / a.psd[j]);
  }
}

// --- one pass over the frequencies ---------------------------------------------------------------
// A candidate's constants (from one thread, by way of shared memory).
struct Point {
  double m13, r13, c0, c2, c3, tc, phic;  // v = m13 vf, r13 = 1 / m13; Psi's coefficients
  // coefficients of the moments in dPsi/dmc (F5, F3, F2) and dPsi/deta (F3, F2)
  double m5, m3, m2, e3, e2;
};

__device__ void make_point(const RefArgs& a, const double (&th)[4], Point& p) {
  const double mc = th[0], eta = th[1], tc = th[2], phic = th[3];
  const double c2 = a.pn >= 2 ? (20.0 / 9.0) * (743.0 / 336.0 + 11.0 * eta / 4.0) : 0.0;
  const double dc2 = a.pn >= 2 ? (20.0 / 9.0) * (11.0 / 4.0) : 0.0;
  const double c3 = a.pn >= 3 ? -16.0 * kPi : 0.0;
  const double mt = mc * pow(eta, -0.6) * kMsunS;
  p.m13 = cbrt(mt);
  p.r13 = 1.0 / p.m13;
  p.c0 = 3.0 / (128.0 * eta);
  p.c2 = c2;
  p.c3 = c3;
  p.tc = tc;
  p.phic = phic;
  // Psi = A5 F5 + A3 F3 + A2 F2, the F's over their values at the band's first frequency
  const double r2 = p.r13 * p.r13, a5 = p.c0 * (r2 * r2 * p.r13) * a.f5, a3 = p.c0 * c2 * (r2 * p.r13) * a.f3,
               a2 = p.c0 * c3 * r2 * a.f2;
  p.m5 = -5.0 / 3.0 * a5 / mc;
  p.m3 = -a3 / mc;
  p.m2 = -2.0 / 3.0 * a2 / mc;
  p.e3 = p.c0 * (r2 * p.r13) * a.f3 * (dc2 - 0.4 * c2 / eta);
  p.e2 = -0.6 * a2 / eta;
}

// The sums of a pass (thread 0 of the cluster's first CTA after evaluate): Z and the moments with j, F5, F3, F2.
struct Sums {
  double z[2], s1[2], m5[2], m3[2], m2[2];
};

// Sums of V values over a warp into out[V]: halves of the list are exchanged while there is more than one value left.
template <int V>
__device__ __forceinline__ void warp_sums(Three (&v)[V], double* out) {
  const int lane = threadIdx.x & 31;
  int first = 0;
#pragma unroll
  for (int step = 0, keep = V / 2; step < 5; ++step, keep /= 2) {
    const int off = 16 >> step;
    const bool up = (lane & off) != 0;
    if (keep > 0) {
      first += up ? keep : 0;
#pragma unroll
      for (int i = 0; i < keep; ++i) {
        const Three give = up ? v[i] : v[i + keep];
        v[i] = up ? v[i + keep] : v[i];
        add(v[i], shuffle_xor(give, off));
      }
    } else {
      add(v[0], shuffle_xor(v[0], off));
    }
  }
  constexpr int kCopies = 32 / V;  // lanes that hold the same value
  // (an infinite term leaves NaN in the parts below the first)
  if ((lane & (kCopies - 1)) == 0)
    out[first] = isfinite(v[0].h) ? (double)v[0].h + ((double)v[0].m + (double)v[0].l) : (double)v[0].h;
}

// `first` and `parts` lie in the shared memory of the cluster's first CTA: the constants, and the strands' sums. `red` holds
// those of a CTA's warps in each of its strands.
// The sums come divided by 2^top, top the largest exponent of the support.
template <bool GRAD, bool PN3>
__device__ void evaluate(const RefArgs& a, const cg::cluster_group& cluster, const Point* first, int64_t jhi, int top,
                         double* red, double* parts, Sums& out) {
  constexpr int V = GRAD ? 8 : 2;
  const int rank = (int)cluster.block_rank(), ranks = (int)cluster.num_blocks();
  const double m13 = first->m13, r13 = first->r13, c0 = first->c0, c2 = first->c2, c3 = first->c3, tc = first->tc,
               phic = first->phic;
  constexpr int NV = GRAD && PN3 ? V + 2 : V;
  const int own = a.strands / ranks;
  __syncthreads();  // (red may still be read)
#pragma unroll 1
  for (int q = 0; q < own; ++q) {
    Three v[V] = {}, v2[2] = {};
#pragma unroll 2
    for (int j = (int)a.jlo + (rank * own + q) * kThreads + (int)threadIdx.x; j < (int)jhi; j += a.strands * kThreads) {  // (< 2^20)
      Three wr, wi;
      {  // to the support's scale: 2^(e - top), nothing below 2^-126
        const float4 w = __ldg(a.w + j), l = __ldg(a.wl + j);
        const float unit = __int_as_float((max(__float_as_int(l.z) - top, -127) + 127) << 23);
        wr = {w.x * unit, w.z * unit, l.x * unit};
        wi = {w.y * unit, w.w * unit, l.y * unit};
      }
      const double2 vt = __ldg(a.v + j);
      const double vv = m13 * vt.x, guess = r13 * vt.y;  // 1 / vv within two units in the last place
      const double iv = reciprocal(vv, guess);
      const double iv2 = iv * iv, iv3 = iv2 * iv, iv5 = iv3 * iv2;
      double phase = __ldg(a.x + j) * tc - phic - 0.25 * kPi;
      if constexpr (GRAD) {  // (rounded as in the ascent)
        const double in = __fma_rn(c2, iv3, iv5);
        phase = __dadd_rn(phase, __dmul_rn(c0, PN3 ? __fma_rn(c3, iv2, in) : in));
      } else {
        phase += PN3 ? c0 * (iv5 + c2 * iv3 + c3 * iv2) : c0 * (iv5 + c2 * iv3);
      }
      // the nearest whole number of turns, by an addition that leaves no fraction bits (|turns| < 2^51)
      const double k = fma(phase, 1.0 / (2.0 * kPi), 6755399441055744.0) - 6755399441055744.0;
      phase -= 2.0 * kPi * k;
      const float psi = (float)phase;
      float sn, cs;
      sincosf(psi, &sn, &cs);
      // term = w exp(i Psi)
      const Three t[2] = {dot(wr, cs, wi, -sn), dot(wr, sn, wi, cs)};
      Three f5, f3, f2;
      if constexpr (GRAD) {
        const float4 g = __ldg(a.g + j);
        const float2 l = __ldg(a.gl + j);
        f5 = {g.x, g.y, l.x};
        f3 = {g.z, g.w, l.y};
      }
      if constexpr (GRAD && PN3) {
        const float4 g = __ldg(a.g2 + j);
        f2 = {g.x, g.y, g.z};
      }
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        add(v[c], t[c]);
        if constexpr (GRAD) {
          add(v[2 + c], mul(t[c], (float)j));  // (exact)
          add(v[4 + c], mul(t[c], f5));
          add(v[6 + c], mul(t[c], f3));
          if constexpr (PN3) add(v2[c], mul(t[c], f2));
        }
      }
    }
    // sums over a warp in parts, over the warps and the strands in FP64
    double* const sums = red + (q * (kThreads / 32) + (threadIdx.x >> 5)) * NV;
    warp_sums<V>(v, sums);
    if constexpr (GRAD && PN3) warp_sums<2>(v2, sums + V);
  }
  __syncthreads();
  if (threadIdx.x < own * NV) {
    const int q = threadIdx.x / NV, i = threadIdx.x % NV;
    double t = red[q * (kThreads / 32) * NV + i];
    for (int w = 1; w < kThreads / 32; ++w) t += red[(q * (kThreads / 32) + w) * NV + i];
    parts[(rank * own + q) * 10 + i] = t;
  }
  cluster.sync();
  if (rank != 0) return;
  if (threadIdx.x < NV) {
    double t = parts[threadIdx.x];
    for (int q = 1; q < a.strands; ++q) t += parts[q * 10 + threadIdx.x];
    red[threadIdx.x] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    out.z[0] = red[0];
    out.z[1] = red[1];
    if constexpr (GRAD) {
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        out.s1[c] = red[2 + c];
        out.m5[c] = red[4 + c];
        out.m3[c] = red[6 + c];
        out.m2[c] = PN3 ? red[8 + c] : 0.0;
      }
    }
  }
}

// Re(conj(zeta) dZ/dtheta_k) for zeta = (zr, zi), dZ/dtheta_k = i sum dPsi_k term (thread 0)
__device__ __forceinline__ void derivatives(const RefArgs& a, const Point& p, const Sums& s, int top, double zr, double zi,
                                            double (&d)[4]) {
  double t[3][2];
#pragma unroll
  for (int c = 0; c < 2; ++c) {
    t[0][c] = p.m5 * s.m5[c] + p.m3 * s.m3[c] + p.m2 * s.m2[c];
    t[1][c] = p.e3 * s.m3[c] + p.e2 * s.m2[c];
    t[2][c] = 2.0 * kPi * a.df * s.s1[c];
#pragma unroll
    for (int k = 0; k < 3; ++k) t[k][c] = scalbn(t[k][c], top);
  }
#pragma unroll
  for (int k = 0; k < 3; ++k) d[k] = zi * t[k][0] - zr * t[k][1];
  d[3] = zr * scalbn(s.z[1], top) - zi * scalbn(s.z[0], top);  // dPsi/dphi_c = -1
}

__device__ __forceinline__ int64_t support_end(const RefArgs& a, double mc0, double eta0) {
  const double mt0 = mc0 * pow(eta0, -0.6) * kMsunS;
  const double fcut = 1.0 / (pow(6.0, 1.5) * kPi * mt0);
  const double top = floor(fcut / a.df) + 2.0;  // (before the cast: a tiny mass puts it beyond 64 bits)
  int64_t jhi = top < (double)a.half ? (int64_t)top : a.half;
  while (jhi > a.jlo && (double)(jhi - 1) * a.df >= fcut) --jhi;
  return max(jhi, a.jlo);
}

template <int MODE, bool PN3>
__global__ void __launch_bounds__(kThreads, MODE == R_EVAL ? 6 : 5) k_refine(RefArgs a) {
  // (of the cluster's first CTA: point, parts, s_jhi)
  __shared__ double red[kMaxRanks * (kThreads / 32) * 10], parts[kMaxRanks * 10];
  __shared__ int red_e[kThreads / 32];
  __shared__ Point point;
  __shared__ int64_t s_jhi;
  const cg::cluster_group cluster = cg::this_cluster();
  const bool lead = cluster.block_rank() == 0;
  const int64_t c = blockIdx.x / cluster.num_blocks();
  const Point* const first = cluster.map_shared_rank(&point, 0);
  double* const sums = cluster.map_shared_rank(parts, 0);
  double th[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) th[i] = a.theta_in[4 * c + i];
  if (!(th[0] > 0.0) || !(th[1] > 0.0) || !(th[1] <= 0.25) || !isfinite(th[2]) || !isfinite(th[3])) {
    if (lead && threadIdx.x == 0) {
      atomicOr(&a.head->flags, (unsigned)RB_FLAG_BAD_STRAIN);
      if (a.J) a.J[c] = __longlong_as_double(0x7ff8000000000000ll);
    }
    return;  // (every CTA of the cluster)
  }
  if (lead && threadIdx.x == 0) s_jhi = support_end(a, th[0], th[1]);
  if (lead && threadIdx.x == 32) make_point(a, th, point);
  cluster.sync();
  const int64_t jhi = min(*cluster.map_shared_rank(&s_jhi, 0), (int64_t)a.head->jmax);
  // the support's largest exponent, and sigma^2, from the chunks' and the last chunk's part
  const int64_t whole = jhi / kThreads, part = whole * kThreads + threadIdx.x;
  int top = kNoExponent;
  for (int64_t k = a.jlo / kThreads + threadIdx.x; k < whole; k += kThreads) top = max(top, a.top[k]);
  if (part < jhi && part >= a.jlo) top = max(top, __float_as_int(a.wl[part].z));
  top = block_max(top, red_e);
  double sig2 = 0.0;  // (the lead's thread 0)
  if (lead) {
    for (int64_t k = a.jlo / kThreads + threadIdx.x; k < whole; k += kThreads) sig2 += a.chunk[k];
    if (part < jhi && part >= a.jlo) sig2 += a.amp2[part];
    sig2 = block_sum(sig2, red);
  }
  Sums s;
  if (MODE == R_EVAL) {
    evaluate<false, PN3>(a, cluster, first, jhi, top, red, sums, s);
    if (lead && threadIdx.x == 0) {
      const double zr = scalbn(s.z[0], top), zi = scalbn(s.z[1], top);
      a.J[c] = (zr * zr + zi * zi) / sig2;
      a.Z[2 * c] = zr;
      a.Z[2 * c + 1] = zi;
    }
  } else if (MODE == R_ADJOINT) {
    evaluate<true, PN3>(a, cluster, first, jhi, top, red, sums, s);
    if (lead && threadIdx.x == 0) {
      const double g = a.dJ[c];
      double d[4];
      derivatives(a, point, s, top, a.Z[2 * c], a.Z[2 * c + 1], d);
#pragma unroll
      for (int k = 0; k < 4; ++k) a.dtheta[4 * c + k] = g * 2.0 * d[k] / sig2;
    }
  }
}

// --- the ascent ------------------------------------------------------------------------------------
// a sine or cosine (zero, normal or NaN) in FP64 by its bits: conversions run at the FP64 rate
__device__ __forceinline__ double widen(float x) {
  const unsigned b = __float_as_uint(x), m = b & 0x7fffffffu;
  const unsigned hi = m == 0 ? 0u : m < 0x7f800000u ? (m >> 3) + 0x38000000u : 0x7ff80000u;
  return __hiloint2double((int)((b & 0x80000000u) | hi), (int)(b << 29));
}

// A candidate's constants in the ascent, and the reciprocals of what is divided by.
struct AscPoint {
  double m13, r13, c0, c2, c3, tc, phic;
  double k3, k2, c0d;  // 3 c2, 2 c3, c0 dc2
  double dm, rdm, mt, mc, rmc, eta, reta, de;  // 128 eta mt, mt, mc, eta, -0.6 mt / eta
};

__device__ void make_point(const RefArgs& a, const double (&th)[4], AscPoint& p) {
  const double mc = th[0], eta = th[1];
  const double mt = mc * pow(eta, -0.6) * kMsunS;
  const double dc2 = a.pn >= 2 ? (20.0 / 9.0) * (11.0 / 4.0) : 0.0;
  p.m13 = cbrt(mt);
  p.r13 = 1.0 / p.m13;
  p.c0 = 3.0 / (128.0 * eta);
  p.c2 = a.pn >= 2 ? (20.0 / 9.0) * (743.0 / 336.0 + 11.0 * eta / 4.0) : 0.0;
  p.c3 = a.pn >= 3 ? -16.0 * kPi : 0.0;
  p.tc = th[2];
  p.phic = th[3];
  p.k3 = 3.0 * p.c2;
  p.k2 = 2.0 * p.c3;
  p.c0d = p.c0 * dc2;
  p.dm = 128.0 * eta * mt;
  p.rdm = 1.0 / p.dm;
  p.mt = mt;
  p.mc = mc;
  p.rmc = 1.0 / mc;
  p.eta = eta;
  p.reta = 1.0 / eta;
  p.de = -0.6 * mt / eta;
}

// Z (v[0..1]) and dZ/dtheta_k (v[2 + 2k .. 3 + 2k]), on the cluster's first thread.
template <bool PN3>
__device__ void evaluate_fp64(const RefArgs& a, const cg::cluster_group& cluster, const AscPoint* first, int64_t jhi, double* sums,
                              double (&v)[10]) {
  const double m13 = first->m13, r13 = first->r13, c0 = first->c0, c2 = first->c2, c3 = first->c3, tc = first->tc, phic = first->phic;
  const double k3 = first->k3, k2 = first->k2, c0d = first->c0d, dm = first->dm, rdm = first->rdm, mt = first->mt, mc = first->mc,
               rmc = first->rmc, eta = first->eta, reta = first->reta, de = first->de;
  const int tid = (int)cluster.thread_rank();
#pragma unroll
  for (int i = 0; i < 10; ++i) v[i] = 0.0;
  for (int64_t j = a.jlo + tid; j < jhi; j += kAscThreads) {
    const double2 vt = __ldg(a.v + j), sh = __ldg(a.sh + j);
    const double x = __ldg(a.x + j), am = __ldg(a.amp + j);
    const double vv = __dmul_rn(m13, vt.x), guess = r13 * vt.y;  // 1 / vv within two units in the last place
    const double iv = reciprocal(vv, guess);
    const double iv2 = __dmul_rn(iv, iv), iv3 = __dmul_rn(iv2, iv), iv5 = __dmul_rn(iv3, iv2);
    double in = __fma_rn(c2, iv3, iv5);
    if (PN3) in = __fma_rn(c3, iv2, in);
    const double psi_pn = __dmul_rn(c0, in);
    double psi = __dadd_rn(__fma_rn(x, tc, -phic), -0.25 * kPi);
    psi = __dadd_rn(psi, psi_pn);
    const double k = __dadd_rn(__fma_rn(psi, 1.0 / (2.0 * kPi), 6755399441055744.0), -6755399441055744.0);
    psi = __fma_rn(-2.0 * kPi, k, psi);
    float snf, csf;
    sincosf((float)psi, &snf, &csf);
    const double sn = widen(snf), cs = widen(csf);
    const double ir = __fma_rn(sh.x, cs, -__dmul_rn(sh.y, sn)), ii = __fma_rn(sh.x, sn, __dmul_rn(sh.y, cs));
    const double tr = __dmul_rn(am, ir), ti = __dmul_rn(am, ii);
    v[0] = __dadd_rn(v[0], tr);
    v[1] = __dadd_rn(v[1], ti);
    double num = __fma_rn(-5.0, iv5, -__dmul_rn(k3, iv3));
    if (PN3) num = __fma_rn(-k2, iv2, num);
    const double dpsi = quotient(num, dm, rdm);
    const double d0 = quotient(__dmul_rn(dpsi, mt), mc, rmc);
    const double deta = __dadd_rn(__dmul_rn(c0d, iv3), quotient(-psi_pn, eta, reta));
    const double d1 = __fma_rn(dpsi, de, deta);
    v[2] = __fma_rn(-d0, ti, v[2]);
    v[3] = __fma_rn(d0, tr, v[3]);
    v[4] = __fma_rn(-d1, ti, v[4]);
    v[5] = __fma_rn(d1, tr, v[5]);
    v[6] = __fma_rn(-x, ti, v[6]);
    v[7] = __fma_rn(x, tr, v[7]);
  }
  constexpr int NV = 8;
#pragma unroll
  for (int i = 0; i < NV; ++i)
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) v[i] += __shfl_xor_sync(0xffffffffu, v[i], off);
  if ((tid & 31) == 0)
#pragma unroll
    for (int i = 0; i < NV; ++i) sums[(tid >> 5) * 10 + i] = v[i];
  cluster.sync();
  if (tid == 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      double s = 0.0;
      for (int w = 0; w < kAscThreads / 32; ++w) s += sums[w * 10 + i];
      v[i] = s;
    }
    v[8] = v[1];  // dPsi/dphi_c = -1
    v[9] = -v[0];
  }
}

template <bool PN3>
__global__ void __launch_bounds__(kAscThreads / kAscRanks, 2 * kAscRanks) k_refine_ascend(RefArgs a) {
  // (of the cluster's first CTA)
  __shared__ double red[(kAscThreads / 32) * 10];
  __shared__ AscPoint point;
  __shared__ int64_t s_jhi;
  __shared__ int s_go;
  const cg::cluster_group cluster = cg::this_cluster();
  const int tid = (int)cluster.thread_rank();
  const int64_t c = blockIdx.x / kAscRanks;
  const AscPoint* const first = cluster.map_shared_rank(&point, 0);
  double* const sums = cluster.map_shared_rank(red, 0);
  double th[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) th[i] = a.theta_in[4 * c + i];
  if (!(th[0] > 0.0) || !(th[1] > 0.0) || !(th[1] <= 0.25) || !isfinite(th[2]) || !isfinite(th[3])) {
    if (tid == 0) {
      atomicOr(&a.head->flags, (unsigned)RB_FLAG_BAD_STRAIN);
      a.J[c] = __longlong_as_double(0x7ff8000000000000ll);
    }
    return;  // (every CTA of the cluster)
  }
  if (tid == 0) {
    s_jhi = support_end(a, th[0], th[1]);
    make_point(a, th, point);
  }
  cluster.sync();
  const int64_t jhi = min(*cluster.map_shared_rank(&s_jhi, 0), (int64_t)a.head->jmax);
  double sig2 = 0.0;
  for (int64_t j = a.jlo + tid; j < jhi; j += kAscThreads) sig2 += a.amp[j] * a.amp[j];
#pragma unroll
  for (int off = 16; off > 0; off >>= 1) sig2 += __shfl_xor_sync(0xffffffffu, sig2, off);
  if ((tid & 31) == 0) sums[tid >> 5] = sig2;
  cluster.sync();
  if (tid == 0) {
    sig2 = 0.0;
    for (int w = 0; w < kAscThreads / 32; ++w) sig2 += red[w];
  }
  cluster.sync();  // (red is free again)
  const double scale[4] = {th[0], 1.0, 1.0 / kFref, 1.0};
  double v[10], u[4], ut[4], grad[4], J = 0.0, alpha = a.alpha0;
#pragma unroll
  for (int k = 0; k < 4; ++k) u[k] = th[k] / scale[k];
  for (int step = -1; step < a.steps; ++step) {  // step -1: the starting point
    if (step >= 0) {
      if (tid == 0) {
        double gu[4], nrm = 0.0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          gu[k] = grad[k] * scale[k];
          nrm += gu[k] * gu[k];
        }
        nrm = sqrt(nrm);
        s_go = nrm > 0.0;
        if (nrm > 0.0) {
#pragma unroll
          for (int k = 0; k < 4; ++k) ut[k] = u[k] + alpha * gu[k] / nrm;
          ut[1] = fmin(fmax(ut[1], kEtaMin), 0.25);
          double tt[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) tt[k] = ut[k] * scale[k];
          make_point(a, tt, point);
        }
      }
      cluster.sync();
      if (!*cluster.map_shared_rank(&s_go, 0)) break;  // (the gradient stays what it is)
    }
    evaluate_fp64<PN3>(a, cluster, first, jhi, sums, v);
    if (tid == 0) {
      const double Jt = (v[0] * v[0] + v[1] * v[1]) / sig2;
      if (step < 0 || Jt > J) {
        J = Jt;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          if (step >= 0) u[k] = ut[k];
          grad[k] = 2.0 * __fma_rn(v[0], v[2 + 2 * k], __dmul_rn(v[1], v[3 + 2 * k])) / sig2;
        }
        if (step >= 0) alpha = fmin(2.0 * alpha, a.alpha_max);
      } else {
        alpha *= 0.5;
      }
    }
  }
  if (tid == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) a.theta_out[4 * c + k] = u[k] * scale[k];
    a.J[c] = J;
  }
  cluster.sync();  // the first CTA's shared memory is read until here
}

size_t a256(size_t x) { return (x + 255) & ~size_t(255); }

// Workspace: header, then the tables over the frequencies (104 bytes each; the ascent uses 48 of them, value and adjoint 88
// below the phase's third order: the size is a matter of n alone). base == nullptr: only the size.
size_t carve(int64_t half, char* base, RefArgs* a) {
  size_t off = 0;
  auto take = [&](size_t bytes) {
    char* p = base ? base + off : nullptr;
    off += a256(bytes);
    return p;
  };
  a->head = (Header*)take(256);
  a->w = (float4*)take(sizeof(float4) * half);
  a->sh = (double2*)a->w;
  a->v = (double2*)take(sizeof(double2) * half);
  a->x = (double*)take(sizeof(double) * half);
  a->g = (float4*)take(sizeof(float4) * half);
  a->gl = (float2*)take(sizeof(float2) * half);
  a->g2 = (float4*)take(sizeof(float4) * half);
  a->amp2 = (double*)take(sizeof(double) * half);
  a->amp = a->amp2;
  a->chunk = (double*)take(sizeof(double) * ((half + kThreads - 1) / kThreads));
  a->wl = (float4*)take(sizeof(float4) * half);
  a->top = (int*)take(sizeof(int) * ((half + kThreads - 1) / kThreads));
  return off;
}

int prepare(const rb_refine_desc* d, const float* shat, const double* psd, const void* theta, int64_t n_cand,
            void* ws, size_t bytes, bool ascent, RefArgs& a, cudaStream_t st) {
  if (!d || !shat || !psd || !theta || n_cand < 0) {
    rb::set_detail("NULL argument or negative count");
    return RB_ERR_BAD_INPUT;
  }
  if (!rb_is_pow2(d->n) || d->n < (1 << 10) || d->n > (1 << 20) || !(d->fs > 0) || !(d->f_low > 0) ||
      !(d->pn_order == 0 || d->pn_order == 2 || d->pn_order == 3) || d->steps < 0 || !(d->alpha0 > 0) ||
      !(d->alpha_max >= d->alpha0)) {
    rb::set_detail("bad refine descriptor");
    return RB_ERR_BAD_INPUT;
  }
  const size_t need = rb_refine_workspace_bytes(d);
  if (!ws || bytes < need || ((uintptr_t)ws & 255)) {
    rb::set_detail("workspace too small: need %zu bytes", need);
    return RB_ERR_OOM;
  }
  const int64_t half = d->n / 2;
  carve(half, (char*)ws, &a);
  a.shat = (const float2*)shat;
  a.psd = psd;
  a.theta_in = (const double*)theta;
  a.half = half;
  a.df = d->fs / (double)d->n;
  // first frequency of the band: j >= 1, j df >= f_low
  const double low = std::floor(d->f_low / a.df) - 1.0;
  a.jlo = low < 1.0 ? 1 : low < (double)half ? (int64_t)low : half;
  while (a.jlo < half && (double)a.jlo * a.df < d->f_low) ++a.jlo;
  a.strands = 1;
  while (a.strands < kMaxRanks && half / (2 * a.strands * kThreads) >= 32) a.strands *= 2;
  a.amp0 = 2.0 * std::pow(a.df, -2.0 / 3.0);  // 2 sqrt(df) df^(-7/6)
  const double lo = (double)a.jlo, base = kPi * (lo * a.df);
  a.r53 = std::pow(lo, 5.0 / 3.0);
  a.r33 = lo;
  a.r23 = std::pow(lo, 2.0 / 3.0);
  a.f5 = std::pow(base, -5.0 / 3.0);
  a.f3 = 1.0 / base;
  a.f2 = std::pow(base, -2.0 / 3.0);
  a.pn = d->pn_order;
  a.n_cand = n_cand;
  a.steps = d->steps;
  a.alpha0 = d->alpha0;
  a.alpha_max = d->alpha_max;
  RB_CUDA_TRY(cudaMemsetAsync(a.head, 0, 256, st));
  k_refine_check<<<(int)std::min<int64_t>(304, (half + kThreads - 1) / kThreads), kThreads, 0, st>>>(a);
  RB_LAUNCH_CHECK();
  const int blocks = (int)std::min<int64_t>(1216, (half + kThreads - 1) / kThreads);
  if (ascent)
    k_ascend_tables<<<blocks, kThreads, 0, st>>>(a);
  else
    k_refine_tables<<<blocks, kThreads, 0, st>>>(a);
  RB_LAUNCH_CHECK();
  return RB_OK;
}

// The call's status, once its kernels are done.
int finish(const RefArgs& a, cudaStream_t st) {
  unsigned flags = 0;
  RB_CUDA_TRY(cudaMemcpyAsync(&flags, &a.head->flags, sizeof(flags), cudaMemcpyDeviceToHost, st));
  RB_CUDA_TRY(cudaStreamSynchronize(st));
  if (flags & RB_FLAG_BAD_PSD) {
    rb::set_detail("PSD not finite and positive on 0 < j < n/2");
    return RB_ERR_BAD_INPUT;
  }
  if (flags & RB_FLAG_BAD_STRAIN) {
    rb::set_detail("a candidate has mc <= 0, eta outside (0, 0.25] or a non-finite t_c / phi_c");
    return RB_ERR_BAD_INPUT;
  }
  return RB_OK;
}

template <int MODE>
int run(const RefArgs& a, cudaStream_t st) {
  if (a.n_cand > 0) {
    // CTAs per candidate: more while the chip (152 SMs, up to four of these CTAs each) has room for them and a thread
    // keeps 32 frequencies of the block. Value and adjoint with 1 / 2 / 4 / 8 CTAs, us: n = 2^19, 16 candidates
    // 786 / 465 / 318 / 271, 64: 775 / 466 / 382 / 379, 128: 771 / 591 / 566 / 611, 227: 971 / 761 / 923 / 882,
    // 456: 1318 / 1550 / 1508 / 1515; n = 2^17, 64: 303 / 224 / 207 / 220, 227: 358 / 301 / 391 / 386; n = 2^14, 64:
    // 157 / 150 / 150 / 174, 300: 168 / 184 / 230 / 284.
    int ranks = 1;
    while (ranks < a.strands && 2 * ranks * a.n_cand <= 512) ranks *= 2;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = (unsigned)ranks;
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(a.n_cand * ranks));
    cfg.blockDim = dim3(kThreads);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    RB_CUDA_TRY(a.pn >= 3 ? cudaLaunchKernelEx(&cfg, k_refine<MODE, true>, a) : cudaLaunchKernelEx(&cfg, k_refine<MODE, false>, a));
    RB_LAUNCH_CHECK();
  }
  return finish(a, st);
}

int ascend(const RefArgs& a, cudaStream_t st) {
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = kAscRanks;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  constexpr int64_t kMost = ((int64_t)1 << 30) / kAscRanks;  // candidates of a launch (a grid has less than 2^31 CTAs)
  for (int64_t c = 0; c < a.n_cand; c += kMost) {
    RefArgs part = a;
    part.n_cand = std::min(kMost, a.n_cand - c);
    part.theta_in += 4 * c;
    part.theta_out += 4 * c;
    part.J += c;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(part.n_cand * kAscRanks));
    cfg.blockDim = dim3(kAscThreads / kAscRanks);
    cfg.stream = st;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    RB_CUDA_TRY(part.pn >= 3 ? cudaLaunchKernelEx(&cfg, k_refine_ascend<true>, part)
                             : cudaLaunchKernelEx(&cfg, k_refine_ascend<false>, part));
    RB_LAUNCH_CHECK();
  }
  return finish(a, st);
}

}  // namespace

extern "C" {

size_t rb_refine_workspace_bytes(const rb_refine_desc* d) {
  if (!d || d->n < 2) return 0;
  RefArgs a{};
  return carve(d->n / 2, nullptr, &a);
}

int rb_refine_eval(const rb_refine_desc* d, const float* s_hat, const double* psd, const double* theta, double* J,
                   double* Z, int64_t n_cand, void* workspace, size_t workspace_bytes, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  RefArgs a{};
  int rc = prepare(d, s_hat, psd, theta, n_cand, workspace, workspace_bytes, false, a, st);
  if (rc) return rc;
  if (!J || !Z) {
    rb::set_detail("NULL output");
    return RB_ERR_BAD_INPUT;
  }
  a.J = J;
  a.Z = Z;
  return run<R_EVAL>(a, st);
}

int rb_refine_adjoint(const rb_refine_desc* d, const float* s_hat, const double* psd, const double* theta,
                      const double* Z, const double* dJ, double* dtheta, int64_t n_cand, void* workspace,
                      size_t workspace_bytes, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  RefArgs a{};
  int rc = prepare(d, s_hat, psd, theta, n_cand, workspace, workspace_bytes, false, a, st);
  if (rc) return rc;
  if (!Z || !dJ || !dtheta) {
    rb::set_detail("NULL argument");
    return RB_ERR_BAD_INPUT;
  }
  a.Z = (double*)Z;
  a.dJ = dJ;
  a.dtheta = dtheta;
  return run<R_ADJOINT>(a, st);
}

int rb_refine(const rb_refine_desc* d, const float* s_hat, const double* psd, double* theta, double* J,
              int64_t n_cand, void* workspace, size_t workspace_bytes, void* stream) {
  cudaStream_t st = (cudaStream_t)stream;
  RefArgs a{};
  int rc = prepare(d, s_hat, psd, theta, n_cand, workspace, workspace_bytes, true, a, st);
  if (rc) return rc;
  if (!J) {
    rb::set_detail("NULL output");
    return RB_ERR_BAD_INPUT;
  }
  a.theta_out = theta;
  a.J = J;
  return ascend(a, st);
}

}  // extern "C"

// Host-only test hook (not part of the C ABI): the quotients a / b and the reciprocals 1 / (a b) as the kernels form them.
extern "C" int rbx_refine_division(int64_t n, const double* a, const double* b, double* q, double* inv) {
  for (int64_t i = 0; i < n; ++i) {
    q[i] = quotient(a[i], b[i], 1.0 / b[i]);
    inv[i] = reciprocal(a[i] * b[i], (1.0 / a[i]) * (1.0 / b[i]));
  }
  return 0;
}
