// Model evaluation and error norms.
//
// u_hat(x) = (1/L) sum_l sum_j w_j(x) sum_k a_ljk phi_ljk(x)   (paper Eq.
// multilevel_solution): one warp per point.  Lane j forms the window of
// covering subdomain j in FP64, the lanes then share the features of each
// covering subdomain, in fixed point that is more accurate than FP64
// (fixed.cuh).  The covering subdomains of a point are those of its cell (the
// common refinement of all supports).
//
// Error norms (paper Eq. l1_error): e_L1 = sum |u_hat - u| / (M std(u)) with
// the population standard deviation, plus the relative L2 error and the max
// error; fixed-order two-stage reductions in FP64.
#include <algorithm>
#include <cmath>

#include "elmfb_internal.cuh"
#include "fixed.cuh"
#include "tanh_table.cuh"

namespace {

constexpr double kPiHi = 3.141592653589793116, kPiLo = 1.2246467991473532e-16;   // pi = hi + lo

__device__ __forceinline__ double warp_sum_d(double v) {
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 1-D window factor [1 + cos(pi dx / sigma)]^2 = 4 cos^4(pi dx / (2 sigma)) on the
// open support |dx| < sigma; near the edge cos(theta/2) = sin(pi u / 2) with
// u = (sigma - |dx|) / sigma.
__device__ __forceinline__ double factor(double dx, double sigma, double inv_sigma) {
  const double adx = fabs(dx);
  if (!(adx < sigma)) return 0.0;
  const double u = (sigma - adx) * inv_sigma;
  const double c = u < 0.5 ? sinpi(0.5 * u) : cospi(0.5 * dx * inv_sigma);
  const double c2 = c * c;
  return 4.0 * c2 * c2;
}

// the hard-constraint factor A(x) of paper §4.3 (1 without the ansatz)
__device__ __forceinline__ double ansatz_value(const Ansatz& an, const double* x, int dim) {
  if (!(an.w > 0.0)) return 1.0;
  double A, dA[2], ddA[2];
  ansatz_at(an, x, dim, A, dA, ddA);
  return A;
}

__global__ void __launch_bounds__(256) k_eval(const double* __restrict__ xs, int64_t n, int dim,
                                              int K, int L, const double* __restrict__ bnd,
                                              int nc0, int nc1, const SubGeom* __restrict__ sub,
                                              const int* __restrict__ cell_level_off,
                                              const int* __restrict__ cover_sub,
                                              const double* __restrict__ W,
                                              const double* __restrict__ B,
                                              const double* __restrict__ a,
                                              double* __restrict__ out, const Ansatz an) {
  const int lane = threadIdx.x & 31;
  const int64_t pt = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (pt >= n) return;
  double x[2] = {xs[pt * dim], dim == 2 ? xs[pt * dim + 1] : 0.0};
  // cell of the point
  int c[2] = {0, 0};
  const int ncs[2] = {nc0, nc1};
  const double* bb = bnd;
  for (int i = 0; i < dim; ++i) {
    int lo = 0, hi = ncs[i];
    while (hi - lo > 1) {
      int mid = (lo + hi) >> 1;
      if (bb[mid] <= x[i]) lo = mid;
      else hi = mid;
    }
    c[i] = lo;
    bb += ncs[i] + 1;
  }
  const int cell = c[1] * nc0 + c[0];
  const int e0 = cell_level_off[(int64_t)cell * (L + 1)];
  const int m = cell_level_off[(int64_t)cell * (L + 1) + L] - e0;
  if (m <= 32) {
    // lane j takes covering entry e0 + j: its window factor (FP64 sin/cos, so
    // once per entry instead of once per lane and entry) and scaled input
    double wj = 0.0, xj[2] = {0.0, 0.0};
    int lvl = -1, sj = 0;
    if (lane < m) {
      sj = cover_sub[e0 + lane];
      const SubGeom g = sub[sj];
      lvl = g.level;
      wj = 1.0;
      for (int i = 0; i < dim; ++i) {
        xj[i] = (x[i] - g.mu[i]) * g.inv_sigma_d[i];
        wj *= factor(x[i] - g.mu[i], g.sigma_d[i], g.inv_sigma_d[i]);
      }
    }
    // partition of unity per level: S_l = sum of the level's factors
    double Sj = 0.0;
    for (int l = 0; l < L; ++l) {
      const double S = warp_sum_d(lvl == l ? wj : 0.0);
      if (lvl == l) Sj = S;
    }
    const double cj = (Sj > 0.0 && wj != 0.0) ? wj / Sj : 0.0;
    // each lane sums its features over the entries; one reduction at the end
    double acc = 0.0;
    for (int j = 0; j < m; ++j) {
      const double cw = __shfl_sync(0xffffffffu, cj, j);
      if (cw == 0.0) continue;   // warp-uniform
      const int s = __shfl_sync(0xffffffffu, sj, j);
      const double x0 = __shfl_sync(0xffffffffu, xj[0], j);
      const double x1 = __shfl_sync(0xffffffffu, xj[1], j);
      for (int f = lane; f < K; f += 32) {
        const int64_t q = (int64_t)s * K + f;
        const double arg = W[q * dim] * x0 + (dim == 2 ? W[q * dim + 1] * x1 : 0.0) + B[q];
        acc += cw * (a[q] * tanh(arg));
      }
    }
    const double total = warp_sum_d(acc);
    if (lane == 0) out[pt] = total / L * ansatz_value(an, x, dim);
    return;
  }
  double total = 0.0;   // more than 32 covering subdomains: entry by entry
  for (int l = 0; l < L; ++l) {
    const int b = cell_level_off[(int64_t)cell * (L + 1) + l];
    const int e = cell_level_off[(int64_t)cell * (L + 1) + l + 1];
    double S = 0.0;
    for (int k = b; k < e; ++k) {
      const SubGeom g = sub[cover_sub[k]];
      double w = 1.0;
      for (int i = 0; i < dim; ++i) w *= factor(x[i] - g.mu[i], g.sigma_d[i], g.inv_sigma_d[i]);
      S += w;
    }
    if (!(S > 0.0)) continue;
    for (int k = b; k < e; ++k) {
      const int s = cover_sub[k];
      const SubGeom g = sub[s];
      double w = 1.0, xt[2] = {0.0, 0.0};
      for (int i = 0; i < dim; ++i) {
        xt[i] = (x[i] - g.mu[i]) * g.inv_sigma_d[i];
        w *= factor(x[i] - g.mu[i], g.sigma_d[i], g.inv_sigma_d[i]);
      }
      if (w == 0.0) continue;
      double part = 0.0;
      for (int f = lane; f < K; f += 32) {
        const int64_t q = (int64_t)s * K + f;
        double arg = W[q * dim] * xt[0] + (dim == 2 ? W[q * dim + 1] * xt[1] : 0.0) + B[q];
        part += a[q] * tanh(arg);
      }
      part = warp_sum_d(part);
      total += (w / S) * part;
    }
  }
  if (lane == 0) out[pt] = total / L * ansatz_value(an, x, dim);
}

// ---- the fixed-point form -------------------------------------------------
// One column as k_eval_fx reads it: weights, bias and coefficient in fixed
// point.  The coefficients of a subdomain share an exponent: a = a_fx
// 2^(ea - abits) with 2^ea above the largest, and the terms a_k phi_k are summed as
// 64-bit integers in units of 2^(ea - abits + 1), as fine as a lane's K / 32 terms
// leave room for (eval_bits).
struct __align__(16) EvalCol {
  int4 w;    // w0.hi, w0.lo, w1.hi, w1.lo
  int4 ba;   // bias (low, high word), a.hi, a.lo
};
constexpr int kWide = -100000;       // no shared exponent: the subdomain is evaluated in FP64
constexpr int kNone = kWide + 1;     // all coefficients zero

// v 2^k to the nearest integer (v finite, |v 2^k| <= 2^62), on the integer pipes
__device__ __forceinline__ int64_t to_fixed(double v, int k) {
  const int64_t bits = __double_as_longlong(v);
  const int e = (int)(bits >> 52) & 0x7ff;
  const int64_t m = (bits & 0xfffffffffffffll) | (e ? 0x10000000000000ll : 0ll);
  const int sh = max(e, 1) - 1075 + k;
  const int r = min(max(-sh, 0), 62);
  const int64_t n = sh >= 0 ? m << min(sh, 10) : (m + (((int64_t)1 << r) >> 1)) >> r;
  return bits < 0 ? -n : n;
}

// A warp per subdomain: its columns in fixed point and their exponent ea, or
// kWide where a coefficient is not finite or the exponent out of range, kNone
// where all are zero.  32 bytes written for every 24 or 32 read; a block per
// subdomain, with conversions in FP64, took 6 ns a subdomain whatever its K: one
// point of a model of 256^2 subdomains, K = 16, 412 us, 50 us with this kernel (33 us
// in FP64, which it is dispatched to), one of 7 levels to 64^2, K = 64, 85 us and 55.
__global__ void __launch_bounds__(128) k_eval_pack(const double* __restrict__ W,
                                                   const double* __restrict__ B,
                                                   const double* __restrict__ a, int dim, int K,
                                                   int n_sub, int wexp, int abits,
                                                   EvalCol* __restrict__ cols,
                                                   int* __restrict__ expo) {
  const int s = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), lane = threadIdx.x & 31;
  if (s >= n_sub) return;
  const int64_t q0 = (int64_t)s * K;
  int64_t mx = 0;   // |a| orders as its bits do, not finite values above the others
#pragma unroll 2
  for (int f = lane; f < K; f += 32)
    mx = max(mx, (int64_t)(__double_as_longlong(a[q0 + f]) & 0x7fffffffffffffffll));
  for (int o = 16; o > 0; o >>= 1) mx = max(mx, (int64_t)__shfl_xor_sync(0xffffffffu, mx, o));
  const int ea = (int)(mx >> 52) - 1022;
  const bool bad = mx != 0 && (ea < -900 || ea > 900);
  if (lane == 0) expo[s] = bad ? kWide : (mx != 0 ? ea : kNone);
#pragma unroll 2
  for (int f = lane; f < K; f += 32) {
    const int64_t q = q0 + f;
    const fx::Val w0 = fx::split(to_fixed(W[q * dim], 61 - wexp));
    const fx::Val w1 = fx::split(dim == 2 ? to_fixed(W[q * dim + 1], 61 - wexp) : 0ll);
    const int64_t b = to_fixed(B[q], 60 - wexp);
    const fx::Val av = fx::split(bad || mx == 0 ? 0ll : to_fixed(a[q], abits - ea));
    cols[q].w = make_int4(w0.hi, w0.lo, w1.hi, w1.lo);
    cols[q].ba = make_int4((int)(uint32_t)b, (int)(b >> 32), av.hi, av.lo);
  }
}

// 1-D window factor 4 cos^4(pi x / 2) at x = xh + xl, |x| < 1, to within a unit
// in the last place: the terms of u_hat are summed without rounding, so the
// windows are what its accuracy comes down to.  With u = 1 - |x|, cos(pi x / 2)
// is sin(pi u / 2) near the edge, else 1 - 2 sin^2(pi x / 4); the sine by its
// Taylor polynomial (|argument| <= pi / 4, next term below 2^-63), sine, cosine
// and its square as sums hi + lo.
__device__ __forceinline__ double window_factor64(double xh, double xl) {
  const double ax = fabs(xh);
  const double u = (1.0 - ax) - (xh < 0.0 ? -xl : xl);
  const bool edge = u < 0.5;
  const double v = edge ? 0.5 * u : 0.25 * ax;   // xl is below v's last place there
  const double x = v * kPiHi, z = x * x;
  double p = 2.8114572543455206e-15;          // 1 / 17!
  p = fma(p, z, -7.6471637318198164e-13);     // -1 / 15!
  p = fma(p, z, 1.6059043836821613e-10);      // 1 / 13!
  p = fma(p, z, -2.5052108385441720e-08);     // -1 / 11!
  p = fma(p, z, 2.7557319223985893e-06);      // 1 / 9!
  p = fma(p, z, -1.9841269841269841e-04);     // -1 / 7!
  p = fma(p, z, 8.3333333333333332e-03);      // 1 / 5!
  p = fma(p, z, -1.6666666666666666e-01);     // -1 / 3!
  // what x's rounding left out, pi's low part included
  const double t = fma(x * z, p, fma(v, kPiLo, fma(v, kPiHi, -x)));
  double ch = x + t, cl = t - (ch - x);
  if (!edge) {
    const double s = ch;
    ch = fma(-2.0 * s, s, 1.0);
    cl = fma(-2.0 * s, s, 1.0 - ch) - 4.0 * s * cl;
  }
  const double c2 = ch * ch, c2l = fma(ch, ch, -c2) + 2.0 * ch * cl;
  const double c4 = c2 * c2, c4l = fma(c2, c2, -c4) + 2.0 * c2 * c2l;
  return 4.0 * (c4 + c4l);
}

// a number that orders as the double does
__device__ __forceinline__ int64_t order_key(double v) {
  const int64_t b = __double_as_longlong(v);
  return b ^ ((b >> 63) & 0x7fffffffffffffffll);
}

// Warp per point, as k_eval's m <= 32 form (every cell's covering subdomains
// fit a warp).  Terms and their sums are integers; per point and lane about 100
// FP64 instructions remain (the windows, their partition of unity and the
// final sum), which the FP64 pipe issues in 6400 cycles of a sub-partition
// beside the integer pipes' work: 130 instructions a term, a third of them
// multiply-adds, and three 16-byte table loads.  The FP64 form spent 3200
// cycles of a sub-partition on a warp of terms, almost all in tanh: 262144
// points of a 7-level 2-D model with K = 64 took 31.2 ms and take 2.82 ms, 1000
// points of a 1-D model 45 us and 29 us (the whole call); the error against a
// 113-bit evaluation is 1.4e-16 to 2.8e-16 of the result in the mean square over
// eight models, its mean below 1e-16, where the FP64 form's was 1.8e-16 to 3.8e-16
// (what is left is the windows' part of it).
template <bool kTwo>
__global__ void __launch_bounds__(256) k_eval_fx(
    const double* __restrict__ xs, int64_t n, int K, int L, const double* __restrict__ bnd,
    int nc0, int nc1, const SubGeom* __restrict__ sub, const int* __restrict__ cell_level_off,
    const int* __restrict__ cover_sub, const EvalCol* __restrict__ cols,
    const int* __restrict__ expo, int shift, int rows, int abits, int room,
    const double* __restrict__ W,
    const double* __restrict__ B, const double* __restrict__ a, double* __restrict__ out,
    const Ansatz an) {
  constexpr int dim = kTwo ? 2 : 1;
  extern __shared__ __align__(16) int4 tab[];
  for (int i = threadIdx.x; i < 3 * rows; i += blockDim.x) tab[i] = kTanhTable[i];
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t pt = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (pt >= n) return;
  const double x[2] = {xs[pt * dim], kTwo ? xs[pt * dim + 1] : 0.0};
  int cell = 0;
  {
    const double* bb = bnd;
    int stride = 1;
#pragma unroll
    for (int i = 0; i < dim; ++i) {
      const int nc = i == 0 ? nc0 : nc1;
      const int64_t key = order_key(x[i]);   // integer comparisons: the FP64 pipe is the busy one
      int lo = 0, hi = nc;
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (order_key(bb[mid]) <= key) lo = mid;
        else hi = mid;
      }
      cell += lo * stride;
      stride = nc0;
      bb += nc + 1;
    }
  }
  const int* lo_l = cell_level_off + (int64_t)cell * (L + 1);
  const int e0 = lo_l[0], m = lo_l[L] - e0;
  // lane j: covering entry e0 + j, its window factor and scaled input
  double wj = 0.0, xd[2] = {0.0, 0.0}, xl[2] = {0.0, 0.0};
  int sj = 0, gb = 0, ge = 0, ea = 0;   // its level's entries gb .. ge - 1
  if (lane < m) {
    sj = cover_sub[e0 + lane];
    const SubGeom g = sub[sj];
    gb = lo_l[g.level] - e0;
    ge = lo_l[g.level + 1] - e0;
    ea = expo[sj];
    wj = 1.0;
#pragma unroll
    for (int i = 0; i < dim; ++i) {
      // dx / sigma = xd + xl
      const double dx = x[i] - g.mu[i];
      xd[i] = dx * g.inv_sigma_d[i];
      xl[i] = fma(-xd[i], g.sigma_d[i], dx) * g.inv_sigma_d[i];
      wj *= fabs(dx) < g.sigma_d[i] ? window_factor64(xd[i], xl[i]) : 0.0;
    }
  }
  // partition of unity: the sum over the level's entries, which are
  // neighbouring lanes (each lane reads its own level's)
  double S = 0.0;
  const int len = __reduce_max_sync(0xffffffffu, ge - gb);
  for (int k = 0; k < len; ++k) {
    const double v = __shfl_sync(0xffffffffu, wj, min(gb + k, 31));
    if (gb + k < ge) S += v;
  }
  const double cw = S > 0.0 && wj != 0.0 ? wj / (S * L) : 0.0;
  const fx::Val x0 = fx::split(__double2ll_rn(xd[0] * 0x1p61) + __double2ll_rn(xl[0] * 0x1p61));
  const fx::Val x1 =
      fx::split(kTwo ? __double2ll_rn(xd[1] * 0x1p61) + __double2ll_rn(xl[1] * 0x1p61) : 0ll);
  // cw = cm 2^(ec - 61), cm in [2^60, 2^61): an entry's sum times cm has the
  // exponent ea + ec, and all are aligned to the largest of the point, `room`
  // bits lower so that they cannot overflow
  const int64_t cb = __double_as_longlong(cw);
  const int ex = (int)(cb >> 52);
  const fx::Val cm = fx::split(((cb & 0xfffffffffffffll) | 0x10000000000000ll) << 8);
  const bool is_wide = cw != 0.0 && ea == kWide;
  const bool is_live = ex > 0 && ea > kNone;
  const int en = is_live ? ea + ex - 1022 : kWide;
  const int emax = __reduce_max_sync(0xffffffffu, en);
  const int down = min(emax - en + room, 62);
  const unsigned live = __ballot_sync(0xffffffffu, is_live);
  const unsigned wide = __ballot_sync(0xffffffffu, is_wide);
  int64_t acc = 0;
  for (int j = 0; j < m; ++j) {
    if (!((live >> j) & 1u)) continue;
    const int s = __shfl_sync(0xffffffffu, sj, j);
    const fx::Val y0 = {__shfl_sync(0xffffffffu, x0.hi, j), __shfl_sync(0xffffffffu, x0.lo, j)};
    fx::Val y1 = {0, 0};
    if (kTwo)
      y1 = {__shfl_sync(0xffffffffu, x1.hi, j), __shfl_sync(0xffffffffu, x1.lo, j)};
    const EvalCol* col = cols + (int64_t)s * K;
    int64_t sum = 0;
#pragma unroll 2
    for (int f = lane; f < K; f += 32) {
      const int4 w = col[f].w, ba = col[f].ba;
      const int64_t b = (int64_t)(((uint64_t)(uint32_t)ba.y << 32) | (uint32_t)ba.x);
      const int64_t arg = fx::argument({w.x, w.y}, y0, {w.z, w.w}, y1, b, kTwo);
      sum = fx::mul_add({ba.z, ba.w}, fx::split(fx::tanh61(arg, shift, tab, rows)), sum);
    }
    const fx::Val c = {__shfl_sync(0xffffffffu, cm.hi, j), __shfl_sync(0xffffffffu, cm.lo, j)};
    const int d = __shfl_sync(0xffffffffu, down, j);
    // to nearest, halves up in even lanes and down in odd ones
    const int64_t half = (((int64_t)1 << d) - (lane & 1)) >> 1;
    acc += (fx::mul_exact(fx::split(sum), c, lane & 1) + half) >> d;
  }
  double part = live ? (double)acc * scalbn(1.0, emax - abits + 2 + room) : 0.0;
  if (wide) {   // subdomains whose coefficients have no shared exponent
    for (int j = 0; j < m; ++j) {
      if (!((wide >> j) & 1u)) continue;
      const int s = __shfl_sync(0xffffffffu, sj, j);
      const double c = __shfl_sync(0xffffffffu, cw, j);
      const double y0 = __shfl_sync(0xffffffffu, xd[0], j);
      const double y1 = __shfl_sync(0xffffffffu, xd[1], j);
      for (int f = lane; f < K; f += 32) {
        const int64_t q = (int64_t)s * K + f;
        const double arg = W[q * dim] * y0 + (kTwo ? W[q * dim + 1] * y1 : 0.0) + B[q];
        part += c * (a[q] * tanh(arg));
      }
    }
  }
  const double total = warp_sum_d(part);
  if (lane == 0) out[pt] = total * ansatz_value(an, x, dim);
}

// Bits of the coefficients: 62 at most (two 31-bit halves), and a lane's ceil(K / 32)
// terms, each below 2^(abits - 1), stay below 2^62.
int eval_bits(int K) {
  int bits = 62;
  while (ceil_div(K, 32) > (int64_t)1 << (63 - bits)) --bits;
  return bits;
}
// Bits the aligned sums of a point's m entries, each below 2^61, are moved down by to
// stay below 2^63.
int eval_room(int m) {
  int room = 0;
  while ((4 << room) < m) ++room;
  return room;
}

// pass 1: sum u, sum |d|, sum d^2, sum u^2, max |d|  (per block)
__global__ void k_err_pass1(const double* __restrict__ uh, const double* __restrict__ ur,
                            int64_t n, double* __restrict__ part) {
  __shared__ double sh[5][32];
  double su = 0, sad = 0, sd2 = 0, su2 = 0, mx = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double d = uh[i] - ur[i];
    su += ur[i];
    sad += fabs(d);
    sd2 += d * d;
    su2 += ur[i] * ur[i];
    mx = fmax(mx, fabs(d));
  }
  double v[5] = {su, sad, sd2, su2, mx};
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  for (int k = 0; k < 5; ++k) {
    double t = v[k];
    for (int o = 16; o > 0; o >>= 1) {
      double y = __shfl_xor_sync(0xffffffffu, t, o);
      t = k == 4 ? fmax(t, y) : t + y;
    }
    if (lane == 0) sh[k][wid] = t;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < 5; ++k) {
      double t = 0.0;
      for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t = k == 4 ? fmax(t, sh[k][w]) : t + sh[k][w];
      part[blockIdx.x * 5 + k] = t;
    }
  }
}

// pass 2: sum (u - mean)^2 per block
__global__ void k_err_pass2(const double* __restrict__ ur, int64_t n,
                            const double* __restrict__ part1, int nb, double* __restrict__ part2) {
  __shared__ double sh[32];
  double su = 0.0;
  for (int b = 0; b < nb; ++b) su += part1[b * 5 + 0];
  const double mean = su / (double)n;
  double acc = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    double d = ur[i] - mean;
    acc += d * d;
  }
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += sh[w];
    part2[blockIdx.x] = t;
  }
}

}  // namespace

void eval_model(elmfb_ctx* h, const double* xs, int64_t n, double* out) {
  if (n == 0) return;
  cudaStream_t st = h->stream;
  stage_begin(h, 6);
  // points and results in device memory are used where they are (unless they
  // overlap), others staged
  const size_t xb = n * h->dim * sizeof(double), ob = n * sizeof(double);
  const char *x0 = (const char*)xs, *o0 = (const char*)out;
  const bool apart = x0 + xb <= o0 || o0 + ob <= x0;
  DevBuf dx, dout;
  const double* x = xs;
  double* o = out;
  if (!apart || !usable_in_place(h, xs, sizeof(double))) {
    dx.alloc(xb, st);
    CUDA_CHECK(cudaMemcpyAsync(dx.p, xs, xb, cudaMemcpyDefault, st));
    x = dx.as<double>();
  }
  if (!apart || !usable_in_place(h, out, sizeof(double))) {
    dout.alloc(ob, st);
    o = dout.as<double>();
  }
  // Fixed point wherever a point's covering subdomains fit a warp and the
  // weight scale is in its range (fixed.cuh); FP64 otherwise: below the range
  // FP64's error, relative to the small arguments, is the smaller one.
  // Few points of a model of many columns too: packing the columns takes 3 us and
  // 1.1e-5 us a column (measured), where FP64 takes 0.9 us more than fixed point for
  // every 32 features of the point's subdomains, or 2.4 us once a block of 8 points
  // shares an SM, for each wave of blocks.
  const double a = h->cfg.weight_scale;
  const int wexp = a > 0.0 ? fx::weight_exp(a) : fx::kMinExp - 1;
  const double slower = n <= 4 ? 0.9 : 2.4 * (double)ceil_div(n, 8 * 152);
  const bool few = slower * (double)(h->max_cover * ceil_div(h->K, 32)) < 3.0 + 1.1e-5 * h->NPhi;
  bool fixed = h->max_cover <= 32 && wexp >= fx::kMinExp && wexp <= fx::kMaxExp && !few;
  if (fixed) {
    // columns, then exponents: a workspace of the handle, rewritten on each call; FP64
    // needs none, so a device that is full does not fail the call
    try {
      h->d_eval.alloc((size_t)h->NPhi * sizeof(EvalCol) + (size_t)h->n_sub * sizeof(int), st);
    } catch (const elmfb_error& e) {
      if (e.code != ELMFB_ERR_OOM) throw;
      cudaGetLastError();
      fixed = false;
    }
  }
  if (fixed) {
    const int rows = fx::tanh_rows(h->dim, wexp), abits = eval_bits(h->K);
    const size_t smem = (size_t)rows * 3 * sizeof(int4);
    EvalCol* const cols = h->d_eval.as<EvalCol>();
    int* const expo = reinterpret_cast<int*>(cols + h->NPhi);
    k_eval_pack<<<(unsigned)ceil_div(h->n_sub, 4), 128, 0, st>>>(
        h->d_W64.as<double>(), h->d_b64.as<double>(), h->d_a.as<double>(), h->dim, h->K, h->n_sub,
        wexp, abits, cols, expo);
    // few points: half-size blocks, so that they spread over more SMs
    const int threads = n < 152 * 16 ? 128 : 256;
#define ELMFB_EVAL_FX(TWO)                                                                     \
  do {                                                                                         \
    ensure_dyn_smem((const void*)k_eval_fx<TWO>, smem);                                        \
    k_eval_fx<TWO><<<(unsigned)ceil_div(n * 32, threads), threads, smem, st>>>(                \
        x, n, h->K, h->L, h->d_bnd.as<double>(), h->nc[0], h->nc[1], h->d_sub.as<SubGeom>(),   \
        h->d_cell_level_off.as<int>(), h->d_cover_sub.as<int>(), cols, expo, 54 - wexp, rows,  \
        abits, eval_room(h->max_cover), h->d_W64.as<double>(), h->d_b64.as<double>(),           \
        h->d_a.as<double>(), o, make_ansatz(h->cfg));                                          \
  } while (0)
    if (h->dim == 2) ELMFB_EVAL_FX(true);
    else ELMFB_EVAL_FX(false);
#undef ELMFB_EVAL_FX
    check_launch("k_eval_fx");
    count_launch(h, 2);
  } else {
    const int64_t threads = n * 32;
    k_eval<<<(unsigned)ceil_div(threads, 256), 256, 0, st>>>(
        x, n, h->dim, h->K, h->L, h->d_bnd.as<double>(), h->nc[0], h->nc[1],
        h->d_sub.as<SubGeom>(), h->d_cell_level_off.as<int>(), h->d_cover_sub.as<int>(),
        h->d_W64.as<double>(), h->d_b64.as<double>(), h->d_a.as<double>(), o,
        make_ansatz(h->cfg));
    check_launch("k_eval");
    count_launch(h);
  }
  if (dout.p) CUDA_CHECK(cudaMemcpyAsync(out, dout.p, ob, cudaMemcpyDefault, st));
  stage_end(h, 6);
}

void error_norms(elmfb_ctx* h, const double* uh, const double* ur, int64_t n, double* out3) {
  cudaStream_t st = h->stream;
  const int nb = (int)std::min<int64_t>(ceil_div(n, 256), 256);
  DevBuf du, dr, p1, p2;
  du.alloc(n * sizeof(double), st);
  dr.alloc(n * sizeof(double), st);
  p1.alloc(nb * 5 * sizeof(double), st);
  p2.alloc(nb * sizeof(double), st);
  CUDA_CHECK(cudaMemcpyAsync(du.p, uh, n * sizeof(double), cudaMemcpyDefault, st));
  CUDA_CHECK(cudaMemcpyAsync(dr.p, ur, n * sizeof(double), cudaMemcpyDefault, st));
  k_err_pass1<<<nb, 256, 0, st>>>(du.as<double>(), dr.as<double>(), n, p1.as<double>());
  k_err_pass2<<<nb, 256, 0, st>>>(dr.as<double>(), n, p1.as<double>(), nb, p2.as<double>());
  check_launch("k_err");
  count_launch(h, 2);
  std::vector<double> a(nb * 5), b(nb);
  CUDA_CHECK(cudaMemcpyAsync(a.data(), p1.p, nb * 5 * sizeof(double), cudaMemcpyDeviceToHost, st));
  CUDA_CHECK(cudaMemcpyAsync(b.data(), p2.p, nb * sizeof(double), cudaMemcpyDeviceToHost, st));
  stream_sync(h);
  double sad = 0, sd2 = 0, su2 = 0, mx = 0, var = 0;
  for (int i = 0; i < nb; ++i) {
    sad += a[i * 5 + 1];
    sd2 += a[i * 5 + 2];
    su2 += a[i * 5 + 3];
    mx = std::max(mx, a[i * 5 + 4]);
    var += b[i];
  }
  const double sd = std::sqrt(var / (double)n);
  out3[0] = su2 > 0.0 ? std::sqrt(sd2 / su2) : NAN;
  out3[1] = sd > 0.0 ? sad / ((double)n * sd) : NAN;
  out3[2] = mx;
}
