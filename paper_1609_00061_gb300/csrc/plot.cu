// Plot kernels: the sample-in-center plot of Sec. 3.2 for polynomial relations.
//
// Pixel e is on when f(c_e) is finite and |f(c_e)| <= eps (PA_EQ; f <= eps for
// PA_LE, f < eps for PA_LT; strict makes every test "<").  The decision is
// defined by the IEEE double evaluation fixed in pa.h.  GB300 runs FP64 at a
// small fraction of its FP32 rate, so everything is first evaluated in FP32
// against a rigorous bound on |f32 - f64|.
//
// The FP32 filter.  With every port but the last fixed, f is a polynomial
// sum_j g_j y^j in the last port y.  The g_j are computed once per row in FP32
// (GB300 does 238 FP32 against 1.7 FP64 flops per SM and clock: with the row
// polynomials in FP64 the 90 plots of 512^3 in 38 random networks took 4.1 ms,
// most of it on the FP64 pipe).  Each 64-pixel word then expands its row's
// polynomial about its middle pixel,
//   f(y_c + t) = sum_k a_k t^k,   a_k by synthetic division,
// decides the whole word when |a_0| and S = sum_k |a_k| h^k (k >= 1, h >= the
// distance from y_c to any centre of the word) leave no doubt, and otherwise
// evaluates its pixels as polynomials in the integer offset s = (y - y_c) / delta
// (a_k scaled by delta^k, D fused multiply-adds per pixel).
//
// Units.  The filter holds coordinates in units of powers of two, x_p = 2^k_p z_p
// with 2^k_p >= X_p, and f in units of 2^q >= A (X and A below), folded into the
// coefficients on the host.  No rounding changes by that, but |z_p| <= 1 and
// |c_e| <= 2^D whatever the box and the coefficients are, so that nothing leaves
// FP32's range.
//
// Error bound.  u = 2^-24, X_p >= |x_p| on port p's range (widened by three
// pixels on the last port), and
//   A = sum_e |c_e| prod_p X_p^e_p   (all exponents, the last port's included).
// Every expansion is about the middle pixel (nb >> 1) of the nb pixels it serves,
// so y_c +- t stays within one pixel of them, and |y_c| + |t| <= X of the last port
// for every pixel that is decided.
// Every quantity the kernel computes is a sum of rounded products of the
// coefficients' monomials, so its error is at most (roundings on a monomial's
// path) u A.  A monomial of total degree at most D meets: the rounding of c_e
// (1); per factor x_p the error of the FP32 centre (2.2: two roundings of a
// value within X_p, see centre32) and one or two roundings of products; at
// most D + 1 roundings of sums per port, D + 1 in the synthetic division, one
// per factor in the scaling by delta^k and D + 1 in the final Horner sum.
// Together less than K = 7 D + n (D + 1) + 14 for n ports.  The FP64 value's own error
// (the same counts of 2^-53) is covered by the factor 1.05.
// Underflow: a product that underflows loses at most 2^-150.  Coordinates being at
// most 1, a loss before the expansion grows by no more than 2^D (coefficients) and
// 3^D (expansion and offsets), so the up to 2^22 of them stay below 2^-80.  One in
// delta^k is multiplied by a_k <= 2^D and, in the Horner sum, by s^k <= 33^k: below
// 2^-51 for D = 16.  With f in units of 2^q (A between 1/2 and 1) and
//   B = 1.05 K u A + 2^-21 eps + 2^-48
// (eps is rounded to FP32) the FP64 decision equals the sign of |f32| - eps
// (f32 - eps for PA_LE / PA_LT) whenever that value exceeds B in magnitude.
// The whole-word test keeps 3 B.  Pixels within B, some per cent of the band
// edges on a fine grid, are collected and decided by the FP64 evaluation of
// pa.h from scratch: the result is the FP64 decision, bit for bit.  A relation
// for which FP64 itself might overflow or underflow on the way takes FP64 at every
// pixel.
#include <float.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "expr_eval.cuh"
#include "pa_internal.h"

namespace pa {

// -------------------------------------------------------- nested evaluation
// nest(k, rem) = sum_{e_k = 0}^{rem} nest(k-1, rem - e_k) * x_k^{e_k}, with
// nest(-1, .) the next coefficient in nest order (read through cp).  No
// evaluation recurses at run time: a recursive device function runs on the
// 1 KB default call stack, which an 8-port relation (eight frames) overflows.
__device__ __forceinline__ double mul_rn(double a, double b) { return __dmul_rn(a, b); }
__device__ __forceinline__ double add_rn(double a, double b) { return __dadd_rn(a, b); }
__device__ __forceinline__ float mul_rn(float a, float b) { return __fmul_rn(a, b); }
__device__ __forceinline__ float add_rn(float a, float b) { return __fadd_rn(a, b); }

template <int K, class T>
__device__ __forceinline__ T nest_t(int rem, const T*& cp, const T* x) {
  if constexpr (K < 0) {
    return *cp++;
  } else {
    T s = 0, pw = 1;
    for (int e = 0; e <= rem; ++e) {
      const T term = mul_rn(nest_t<K - 1, T>(rem - e, cp, x), pw);
      s = (e == 0) ? term : add_rn(s, term);
      pw = mul_rn(pw, x[K]);
    }
    return s;
  }
}

template <class T>
struct NestOut {
  T v;
  const T* cp;  // past the coefficients read
};

// Any depth as a loop over an explicit per-depth state (partial sum, power of
// x_L, exponent, remaining degree): the same products and sums in the same
// order as nest_t, out of line and with few registers, for the deep cases.
template <class T>
__device__ __noinline__ NestOut<T> nest_deep(int k, int rem, const T* cp, const T* x) {
  if (k < 0) return {*cp, cp + 1};
  T s[kMaxDim], pw[kMaxDim];
  int e[kMaxDim], rm[kMaxDim];
  int L = k;
  rm[k] = rem;
  e[k] = 0;
  pw[k] = 1;
  s[k] = 0;
  for (;;) {
    // open the term e[L] of depth L down to depth 0
    while (L > 0) {
      rm[L - 1] = rm[L] - e[L];
      e[L - 1] = 0;
      pw[L - 1] = 1;
      s[L - 1] = 0;
      --L;
    }
    T v = *cp++;  // nest(-1, .): the next coefficient
    // close terms upward while depths complete
    for (;;) {
      const T term = mul_rn(v, pw[L]);
      s[L] = (e[L] == 0) ? term : add_rn(s[L], term);
      pw[L] = mul_rn(pw[L], x[L]);
      if (++e[L] <= rm[L]) break;
      if (L == k) return {s[k], cp};
      v = s[L];
      ++L;
    }
  }
}

template <class T>
__device__ __forceinline__ T nest_rows(int k, int rem, const T*& cp, const T* x) {
  switch (k) {
    case -1: return nest_t<-1, T>(rem, cp, x);
    case 0: return nest_t<0, T>(rem, cp, x);
    case 1: return nest_t<1, T>(rem, cp, x);
    case 2: return nest_t<2, T>(rem, cp, x);
    default: {
      const NestOut<T> o = nest_deep<T>(k, rem, cp, x);
      cp = o.cp;
      return o.v;
    }
  }
}

// The row polynomial g_0..g_DS of a 2- or 3-port relation at one row, FP32, for
// a degree fixed at compile time (Horner in the row ports, every index
// constant).  c: the coefficients in nest order.
template <int DS>
__device__ __forceinline__ void row_poly2(const float* __restrict__ c, float x0, float* g) {
  int at = 0;
#pragma unroll
  for (int j = 0; j <= DS; ++j) {
    float s = c[at + DS - j];
#pragma unroll
    for (int e = DS - j - 1; e >= 0; --e) s = __fmaf_rn(s, x0, c[at + e]);
    at += DS - j + 1;
    g[j] = s;
  }
}

template <int DS>
__device__ __forceinline__ void row_poly3(const float* __restrict__ c, float x0, float x1,
                                          float* g) {
  int at = 0;
#pragma unroll
  for (int j = 0; j <= DS; ++j) {
    // the sums over x0 of the blocks e1 = 0..DS - j, then Horner in x1
    float t[DS + 1];
#pragma unroll
    for (int e1 = 0; e1 <= DS - j; ++e1) {
      const int m = DS - j - e1;
      float s = c[at + m];
#pragma unroll
      for (int e = m - 1; e >= 0; --e) s = __fmaf_rn(s, x0, c[at + e]);
      at += m + 1;
      t[e1] = s;
    }
    float s1 = t[DS - j];
#pragma unroll
    for (int e1 = DS - j - 1; e1 >= 0; --e1) s1 = __fmaf_rn(s1, x1, t[e1]);
    g[j] = s1;
  }
}

__device__ __forceinline__ double centre(double lo, double delta, int64_t i) {
  return __dadd_rn(lo, __dmul_rn(__dadd_rn((double)i, 0.5), delta));
}

__device__ __forceinline__ bool decide64(double f, int kind, double eps, int strict) {
  if (!isfinite(f)) return false;
  if (kind == PA_EQ) {
    const double d = fabs(f);
    return strict ? (d < eps) : (d <= eps);
  }
  if (kind == PA_LE) return strict ? (f < eps) : (f <= eps);
  return f < eps;
}

// The nested FP64 sums of pa.h for 2 or 3 ports and a degree fixed at compile
// time: the products and sums of nest_t in the same order, with the powers of
// each port formed once and every sum unrolled, so that independent sums
// proceed side by side (the FP64 chain is what a pixel decided in FP64 costs).
template <int DS>
__device__ __forceinline__ double nest2(const double* __restrict__ cp, double x0, double x1) {
  double p0[DS + 1];
  p0[0] = 1.0;
#pragma unroll
  for (int e = 1; e <= DS; ++e) p0[e] = __dmul_rn(p0[e - 1], x0);
  double f = 0.0, p1 = 1.0;
#pragma unroll
  for (int j = 0; j <= DS; ++j) {
    double s = __dmul_rn(cp[0], p0[0]);
#pragma unroll
    for (int e = 1; e <= DS - j; ++e) s = __dadd_rn(s, __dmul_rn(cp[e], p0[e]));
    cp += DS - j + 1;
    const double term = __dmul_rn(s, p1);
    f = j == 0 ? term : __dadd_rn(f, term);
    p1 = __dmul_rn(p1, x1);
  }
  return f;
}

template <int DS>
__device__ __forceinline__ double nest3(const double* __restrict__ cp, double x0, double x1,
                                        double x2) {
  double p0[DS + 1], p1[DS + 1];
  p0[0] = 1.0;
  p1[0] = 1.0;
#pragma unroll
  for (int e = 1; e <= DS; ++e) {
    p0[e] = __dmul_rn(p0[e - 1], x0);
    p1[e] = __dmul_rn(p1[e - 1], x1);
  }
  double f = 0.0, p2 = 1.0;
#pragma unroll
  for (int j = 0; j <= DS; ++j) {
    double s1 = 0.0;
#pragma unroll
    for (int e1 = 0; e1 <= DS - j; ++e1) {
      double s = __dmul_rn(cp[0], p0[0]);
#pragma unroll
      for (int e = 1; e <= DS - j - e1; ++e) s = __dadd_rn(s, __dmul_rn(cp[e], p0[e]));
      cp += DS - j - e1 + 1;
      const double term = __dmul_rn(s, p1[e1]);
      s1 = (e1 == 0) ? term : __dadd_rn(s1, term);
    }
    const double term = __dmul_rn(s1, p2);
    f = j == 0 ? term : __dadd_rn(f, term);
    p2 = __dmul_rn(p2, x2);
  }
  return f;
}

// The FP64 decision of one pixel: the full nested evaluation of pa.h at its
// centre.
template <int DS>
__device__ __noinline__ bool decide_pixel64(const PlotJob* J, int64_t row, int64_t i) {
  const int ndim = J->ndim, arity = J->arity;
  if constexpr (DS >= 0) {
    if (J->filter && (arity == 2 || arity == 3) && row < (1ll << 31)) {
      // port p on axis p
      const double xl = centre(J->lo[arity - 1], J->delta[arity - 1], i);
      uint32_t r0 = (uint32_t)row, r1 = 0;
      if (arity == 3) {
        const uint32_t q = r0 / (uint32_t)J->res[1];
        r1 = r0 - q * (uint32_t)J->res[1];
        r0 = q;
      }
      const double x0 = centre(J->lo[0], J->delta[0], r0);
      const double f = arity == 2 ? nest2<DS>(J->coeffs, x0, xl)
                                  : nest3<DS>(J->coeffs, x0, centre(J->lo[1], J->delta[1], r1), xl);
      return decide64(f, J->kind, J->eps, J->strict);
    }
  }
  int64_t rest = row;
  int64_t idx[kMaxDim];
  idx[ndim - 1] = i;
  for (int a = ndim - 2; a >= 0; --a) {
    idx[a] = rest % J->res[a];
    rest /= J->res[a];
  }
  double x[kMaxDim];
  for (int p = 0; p < arity; ++p) x[p] = centre(J->lo[p], J->delta[p], idx[J->port_axis[p]]);
  const double* cp = J->coeffs;
  return decide64(nest_rows<double>(arity - 1, J->degree, cp, x), J->kind, J->eps, J->strict);
}

// The FP32 centre of pixel i of port p (fi = i + 1/2, exact below 2^23): lo and
// delta as sums of two floats, one rounding in each of the two larger steps,
// so |error| <= 2.2 u max(|lo|, |hi|).
__device__ __forceinline__ float centre32(const PlotJob* J, int p, float fi) {
  return __fadd_rn(__fmaf_rn(fi, J->d_hi[p], J->lo_hi[p]), __fmaf_rn(fi, J->d_lo[p], J->lo_lo[p]));
}

// --------------------------------------------------------------- plot kernel
// One block plots a tile of rows.  Set-up: each row's FP32 polynomial goes to
// shared memory (one thread per row).  Then, for up to kPass words of the tile
// at a time, in phases that each run with full warps on a list the phase
// before made:
//   1. every word is tested as a whole (neighbouring threads take neighbouring
//      words, so decided words are stored in full sectors);
//   2. an undecided word on which f is provably monotone has its band edges
//      solved for (Newton, then the two pixels on either side of each edge are
//      evaluated: by monotonicity they decide every other pixel), about 130
//      instructions against 450 for 64 pixel evaluations;
//   3. the others are evaluated pixel by pixel, one thread per word;
//   4. a word with a pixel within B of eps is evaluated again by a warp, which
//      collects those pixels;
//   5. the collected pixels are decided in FP64, a thread each.
// Phases 4 and 5 exist because one such pixel handled in place holds up its
// whole warp.  What bounds it: instruction issue (no pipe above 40 %; the
// output is 1/8 byte per pixel), and on small plots the chain of phases.
// Against FP64 row polynomials, FP32 centre tables from a launch of their own
// and 64 evaluations per undecided word (ncu, cold): 38 random networks, 12.7
// Gpixel, 4.14 -> 2.11 ms; 4096 chains, 4.9 Gpixel, 1.37 + 0.10 -> 0.70 ms;
// four 256^3 plots 55 + 3 -> 29 us; eight 2048^2 plots 19 + 3 -> 14 us.
constexpr int kPlotThreads = 256;
static_assert(sizeof(PlotJob) % 4 == 0, "plot descriptors are copied as 32-bit words");
constexpr int kPass = 2048;      // words per pass (the lists' entries are 16-bit)
constexpr int kPendCap = 512;    // collected FP64 pixels per pass; more are evaluated in place

// Clear the listed ranges with every thread of the grid, eight words per
// thread and step: chunk c covers words [8c, 8c + 8) of the ranges' flat
// index space and may cross from one range into the next.
__device__ __forceinline__ void clear_ranges(const ZeroRange* __restrict__ zr, int nzero,
                                             int64_t zero_words) {
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t gstride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t c = gid; c * 8 < zero_words; c += gstride) {
    int64_t w = c * 8;
    const int64_t wend = min(zero_words, w + 8);
    int lo = 0, hi = nzero - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (zr[mid].w0 <= w) lo = mid; else hi = mid - 1;
    }
    for (int r = lo; w < wend && r < nzero; ++r) {
      const int64_t end = min(wend, zr[r].w0 + zr[r].words);
      for (; w < end; ++w) zr[r].p[w - zr[r].w0] = 0ull;
    }
  }
}

// Taylor coefficients about yc of the polynomial in a (in place, synthetic
// division).
template <int DS, int N>
__device__ __forceinline__ void taylor_shift(float (&a)[N], int D, float yc) {
  if constexpr (DS >= 0) {
#pragma unroll
    for (int i = 0; i < DS; ++i)
#pragma unroll
      for (int j = DS - 1; j >= i; --j) a[j] = __fmaf_rn(yc, a[j + 1], a[j]);
  } else {
    for (int i = 0; i < D; ++i)
      for (int j = D - 1; j >= i; --j) a[j] = __fmaf_rn(yc, a[j + 1], a[j]);
  }
}

// The value compared with 0 at integer offset s from the expansion point:
// |f| - eps (PA_EQ) or f - eps.  a: scaled Taylor coefficients.
template <int DS, bool EQ, int N>
__device__ __forceinline__ float excess(const float (&a)[N], int D, float s, float eps) {
  float f;
  if constexpr (DS >= 0) {
    f = a[DS];
#pragma unroll
    for (int k = DS - 1; k >= 0; --k) f = __fmaf_rn(f, s, a[k]);
  } else {
    f = a[D];
    for (int k = D - 1; k >= 0; --k) f = __fmaf_rn(f, s, a[k]);
  }
  return __fsub_rn(EQ ? fabsf(f) : f, eps);
}

// The smaller of two values, NaN when either is.
__device__ __forceinline__ float min_nan(float a, float b) {
  float r;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(r) : "f"(a), "f"(b));
  return r;
}

// P pixels (8 or 32) at offsets s0, s0 + 1, ...: bit b of the result is the
// sign of pixel b's excess (1: on), *closest the smallest |excess|, or NaN (no
// pixel of the word is taken as decided then).
template <int DS, bool EQ, int P, int S0, int N>
__device__ __forceinline__ uint32_t eval_pixels(const float (&a)[N], int D, float eps,
                                                float* closest) {
  uint32_t m = 0;
  float c = *closest;
#pragma unroll
  for (int b = P - 1; b >= 0; --b) {
    const float e = excess<DS, EQ>(a, D, (float)(S0 + b), eps);
    m = __funnelshift_l(__float_as_uint(e), m, 1);
    c = min_nan(c, fabsf(e));
  }
  *closest = c;
  return m;
}

// The number of offsets in [lo, hi] (integers) at which the increasing
// polynomial a is below T, when the offsets on either side of the crossing are
// more than B from it; false when that is not established.
template <int DS, int N>
__device__ __forceinline__ bool count_below(const float (&a)[N], int D, float T, float r, float lo,
                                            float hi, float B, int* n) {
  float s = __fmul_rn(T - a[0], r);
#pragma unroll
  for (int it = 0; it < 2; ++it) {
    s = fminf(fmaxf(s, lo - 1.0f), hi + 1.0f);
    float f, d = 0.0f;
    if constexpr (DS >= 0) {
      f = a[DS];
#pragma unroll
      for (int k = DS - 1; k >= 0; --k) {
        d = __fmaf_rn(d, s, f);
        f = __fmaf_rn(f, s, a[k]);
      }
    } else {
      f = a[D];
      for (int k = D - 1; k >= 0; --k) {
        d = __fmaf_rn(d, s, f);
        f = __fmaf_rn(f, s, a[k]);
      }
    }
    s = __fmaf_rn(T - f, __frcp_rn(d), s);
  }
  s = floorf(fminf(fmaxf(s, lo - 1.0f), hi));
  const float e0 = excess<DS, false>(a, D, s, T), e1 = excess<DS, false>(a, D, s + 1.0f, T);
  *n = (int)(s + 1.0f - lo);
  return (s < lo || e0 < -B) && (s >= hi || e1 > B);
}

template <int DS>
__global__ void __launch_bounds__(kPlotThreads, 4)
plot_kernel(const PlotJob* __restrict__ jobs, int njobs, int gstride,
            const ZeroRange* __restrict__ zr, int nzero, int64_t zero_words) {
  extern __shared__ __align__(16) float g32s[];  // [rows][gstride] row polynomials
  // the launch before this one may be the upload of the descriptors; those after
  // it read theirs before they wait for this grid, so they may only start when
  // that upload is complete
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;");
  __shared__ PlotJob sJ;
  __shared__ uint16_t list[kPass], list_px[kPass], list_re[kPass];
  __shared__ uint32_t plist[kPendCap];
  __shared__ int s_n, s_npx, s_nre, s_np;
  {
    const int job = find_entry([&](int i) { return jobs[i].tile0; }, njobs, (int64_t)blockIdx.x);
    const uint32_t* src = reinterpret_cast<const uint32_t*>(jobs + job);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&sJ);
    for (int i = threadIdx.x; i < (int)(sizeof(PlotJob) / 4); i += blockDim.x) dst[i] = src[i];
  }
  if (threadIdx.x == 0) s_n = s_npx = s_nre = s_np = 0;
  __syncthreads();
  const PlotJob* J = &sJ;
  const int D = DS >= 0 ? DS : J->degree;
  constexpr int kG = DS >= 0 ? DS + 1 : kMaxDeg + 1;
  const int row_words = (int)J->row_words;
  const int last = J->ndim - 1;
  const int res_last = J->res[last];
  const int R = J->rows_per_tile;
  const int64_t row0 = ((int64_t)blockIdx.x - J->tile0) * R;
  const int nr = (int)min((int64_t)R, J->nrows - row0);
  const bool filter = J->filter != 0;
  const int arity = J->arity;
  if (filter) {
    for (int r = threadIdx.x; r < nr; r += blockDim.x) {
      float x[kMaxDim];
      const int64_t row = row0 + r;
      if (row < (1ll << 31)) {
        uint32_t rest = (uint32_t)row;
        for (int a = last - 1; a >= 0; --a) {
          const uint32_t q = a > 0 ? rest / (uint32_t)J->res[a] : 0u;
          x[a] = centre32(J, a, (float)(rest - q * (uint32_t)J->res[a]) + 0.5f);
          rest = q;
        }
      } else {
        int64_t rest = row;
        for (int a = last - 1; a >= 0; --a) {
          x[a] = centre32(J, a, (float)(rest % J->res[a]) + 0.5f);
          rest /= J->res[a];
        }
      }
      float* gr = g32s + r * gstride;
      const float* cp = J->c32;
      bool done = false;
      if constexpr (DS >= 0) {
        if (arity == 2 || arity == 3) {
          float gv[DS + 1];
          if (arity == 2) row_poly2<DS>(cp, x[0], gv);
          else row_poly3<DS>(cp, x[0], x[1], gv);
#pragma unroll
          for (int j = 0; j <= DS; ++j) gr[j] = gv[j];
          done = true;
        }
      }
      // filtered jobs have port p on axis p (every variable on one port)
      for (int j = 0; !done && j <= D; ++j) gr[j] = nest_rows<float>(arity - 2, D - j, cp, x);
    }
  }
  // the later contractions' result buffers that start at zero (each block a
  // share; a block's share is small next to its plot tile)
  if (zero_words > 0) clear_ranges(zr, nzero, zero_words);
  __syncthreads();
  const bool eq = J->kind == PA_EQ;
  uint64_t* __restrict__ out = J->out + row0 * row_words;  // the tile's words are consecutive
  // read once: the stores to `out` below could otherwise make the compiler
  // reload these from the job descriptor in every loop
  const float eps = J->eps32, B = J->bound;
  const float dl = J->d_hi[arity - 1], dabs = J->dabs;
  const float ylo_hi = J->lo_hi[arity - 1], ylo_lo = J->lo_lo[arity - 1], dl_lo = J->d_lo[arity - 1];
  const int nwords = nr * row_words;
  const float inv_rw = 1.0f / (float)row_words;
  // row of the tile's word t (exact: with several rows a tile has few words)
  auto row_of = [&](int t) { return nr == 1 ? 0 : (int)(((float)t + 0.5f) * inv_rw); };
  auto ycentre = [&](int i) {
    const float fi = (float)i + 0.5f;
    return __fadd_rn(__fmaf_rn(fi, dl, ylo_hi), __fmaf_rn(fi, dl_lo, ylo_lo));
  };
  auto load_g = [&](int r, float (&a)[kG]) {
    const float* gr = g32s + r * gstride;
#pragma unroll
    for (int j = 0; j < kG; ++j) a[j] = (DS >= 0 || j <= D) ? gr[j] : 0.0f;
  };
  const int lane = threadIdx.x & 31;
  const int nthr = (int)blockDim.x;
  // Taylor coefficients about pixel ic of row r, scaled to steps of one pixel
  auto expand = [&](int r, int ic, float (&a)[kG]) {
    load_g(r, a);
    taylor_shift<DS>(a, D, ycentre(ic));
    float pw = dl;
    if constexpr (DS >= 0) {
#pragma unroll
      for (int j = 1; j <= DS; ++j) {
        a[j] = __fmul_rn(a[j], pw);
        pw = __fmul_rn(pw, dl);
      }
    } else {
      for (int j = 1; j <= D; ++j) {
        a[j] = __fmul_rn(a[j], pw);
        pw = __fmul_rn(pw, dl);
      }
    }
  };
  auto full_mask = [](int nb) { return nb >= 64 ? ~0ull : (1ull << nb) - 1ull; };
  // warp-aggregated append of k to a shared list (every lane of the warp)
  auto append = [&](uint16_t* to, int* count, bool keep, int k) {
    const unsigned m = __ballot_sync(0xffffffffu, keep);
    if (!m) return;
    int off = 0;
    if (lane == 0) off = atomicAdd(count, __popc(m));
    off = __shfl_sync(0xffffffffu, off, 0);
    if (keep) to[off + __popc(m & ((1u << lane) - 1u))] = (uint16_t)k;
  };
  for (int t0 = 0; t0 < nwords; t0 += kPass) {
    const int np = min(kPass, nwords - t0);
    if (!filter) {
      // FP64 at every pixel, eight pixels per thread
      for (int e = threadIdx.x; e < 8 * np; e += nthr) {
        const int t = t0 + (e >> 3), c8 = e & 7, r = row_of(t), w = t - r * row_words;
        const int i0 = w * 64 + 8 * c8, nb = min(8, res_last - i0);
        uint32_t bits = 0;
        for (int b = 0; b < nb; ++b)
          if (decide_pixel64<DS>(J, row0 + r, i0 + b)) bits |= 1u << b;
        reinterpret_cast<uint8_t*>(out + t)[c8] = (uint8_t)bits;
      }
      continue;
    }
    // ---- phase 1: whole words
    for (int base = 0; base < np; base += nthr) {
      const int k = base + threadIdx.x;
      bool keep = k < np;
      if (keep) {
        const int t = t0 + k, r = row_of(t), w = t - r * row_words;
        const int nb = min(64, res_last - w * 64), c = nb >> 1;
        float a[kG];
        load_g(r, a);
        taylor_shift<DS>(a, D, ycentre(w * 64 + c));
        const float h = __fmul_rn((float)c, dabs);
        float S = fabsf(a[D]);
        if constexpr (DS >= 0) {
#pragma unroll
          for (int j = DS - 1; j >= 1; --j) S = __fmaf_rn(S, h, fabsf(a[j]));
        } else {
          for (int j = D - 1; j >= 1; --j) S = __fmaf_rn(S, h, fabsf(a[j]));
        }
        if (D >= 1) S = __fmul_rn(S, h);
        else S = 0.0f;
        const float v = eq ? fabsf(a[0]) : a[0], margin = __fmaf_rn(3.0f, B, S);
        const bool off = v - eps > margin, on = eps - v > margin;
        if (off || on) {
          out[t] = off ? 0ull : full_mask(nb);
          keep = false;
        }
      }
      append(list, &s_n, keep, k);
    }
    __syncthreads();
    // ---- phase 2: band edges of words on which f is monotone
    const int nlist = s_n;
    for (int base = 0; base < nlist; base += nthr) {
      const int e = base + threadIdx.x;
      bool hard = false;
      int k = 0;
      if (e < nlist) {
        k = list[e];
        const int t = t0 + k, r = row_of(t), w = t - r * row_words;
        const int nb = min(64, res_last - w * 64), ic = nb >> 1;
        float a[kG];
        expand(r, w * 64 + ic, a);
        // f' keeps a_1's sign when a_1 outweighs the other terms at the
        // word's ends by more than the coefficients' errors (D B / hs)
        const float hs = (float)ic;
        float Q = 0.0f;
        if constexpr (DS >= 2) {
          Q = (float)DS * fabsf(a[DS]);
#pragma unroll
          for (int j = DS - 1; j >= 2; --j) Q = __fmaf_rn(Q, hs, (float)j * fabsf(a[j]));
          Q = __fmul_rn(Q, hs);
        } else if constexpr (DS < 0) {
          for (int j = D; j >= 2; --j) Q = __fmaf_rn(Q, hs, (float)j * fabsf(a[j]));
          Q = __fmul_rn(Q, hs);
        }
        const float a1 = D >= 1 ? a[D >= 1 ? 1 : 0] : 0.0f;
        hard = !((fabsf(a1) * 0.999f - Q) * hs > (float)(2 * D) * B);
        if (!hard) {
          const bool up = a1 > 0.0f;
#pragma unroll
          for (int j = 0; j < kG; ++j)
            if (DS >= 0 || j <= D) a[j] = up ? a[j] : -a[j];
          const float rc = __frcp_rn(fabsf(a1));
          const float lo = -(float)ic, hi = (float)(nb - 1 - ic);
          uint64_t bits;
          if (eq) {
            int n0, n1;
            hard = !(count_below<DS>(a, D, -eps, rc, lo, hi, B, &n0) &
                     count_below<DS>(a, D, eps, rc, lo, hi, B, &n1));
            bits = full_mask(n1) & ~full_mask(n0);
          } else {
            int n;
            hard = !count_below<DS>(a, D, up ? eps : -eps, rc, lo, hi, B, &n);
            bits = up ? full_mask(n) : full_mask(nb) & ~full_mask(n);
          }
          if (!hard) out[t] = bits;
        }
      }
      append(list_px, &s_npx, hard, k);
    }
    __syncthreads();
    // ---- phase 3: pixels.  A block with few such words cuts each into eight
    // pieces of 8 pixels, so that they spread over its threads.
    const int npx = s_npx;
    const int C = 4 * npx <= nthr ? 8 : 1;
    for (int base = 0; base < npx * C; base += nthr) {
      const int e = base + threadIdx.x;
      bool close = false;
      int k = 0;
      if (e < npx * C) {
        k = list_px[C == 1 ? e : e >> 3];
        const int c8 = C == 1 ? 0 : e & 7;
        const int t = t0 + k, r = row_of(t), w = t - r * row_words;
        const int i0 = w * 64 + 8 * c8;                      // first pixel of the piece
        const int nb = min(C == 1 ? 64 : 8, res_last - i0);  // <= 0: padding past the row
        uint64_t bits = 0;
        if (nb > 0) {
          // expanded about the piece's own middle, as the bound assumes; the
          // offsets run past a piece that the row's end cuts, those bits dropped
          const int ic = nb >> 1;
          float a[kG];
          expand(r, i0 + ic, a);
          float closest = INFINITY;
          if (C == 1 && nb > 32) {
            uint32_t lo, hi;
            if (eq) {
              lo = eval_pixels<DS, true, 32, -32>(a, D, eps, &closest);
              hi = eval_pixels<DS, true, 32, 0>(a, D, eps, &closest);
            } else {
              lo = eval_pixels<DS, false, 32, -32>(a, D, eps, &closest);
              hi = eval_pixels<DS, false, 32, 0>(a, D, eps, &closest);
            }
            bits = (((uint64_t)hi << 32) | lo) >> (32 - ic);
          } else if (C == 1 && nb > 16) {
            bits = (eq ? eval_pixels<DS, true, 32, -16>(a, D, eps, &closest)
                       : eval_pixels<DS, false, 32, -16>(a, D, eps, &closest)) >> (16 - ic);
          } else if (C == 8 && nb > 4) {
            bits = (eq ? eval_pixels<DS, true, 8, -4>(a, D, eps, &closest)
                       : eval_pixels<DS, false, 8, -4>(a, D, eps, &closest)) >> (4 - ic);
          } else {
            closest = 0.0f;  // few pixels: left to phase 4
          }
          bits &= full_mask(nb);
          close = !(closest > B);
        }
        if (C == 1) out[t] = bits;
        else reinterpret_cast<uint8_t*>(out + t)[c8] = (uint8_t)bits;
      }
      append(list_re, &s_nre, close, k);  // (a word may be listed once per piece)
    }
    __syncthreads();
    // ---- phase 4: words with pixels FP32 cannot decide, a warp each
    const int nre = s_nre;
    for (int e = threadIdx.x >> 5; e < nre; e += nthr >> 5) {
      const int k = list_re[e];
      const int t = t0 + k, r = row_of(t), w = t - r * row_words;
      const int nb = min(64, res_last - w * 64), ic = nb >> 1;
      float a[kG];
      expand(r, w * 64 + ic, a);
      uint32_t half[2];
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int b = 32 * q + lane;
        const float s = (float)(b - ic);
        const float ex = eq ? excess<DS, true>(a, D, s, eps) : excess<DS, false>(a, D, s, eps);
        bool on = b < nb && ex < 0.0f;
        if (b < nb && !(fabsf(ex) > B)) {
          const int at = atomicAdd(&s_np, 1);
          on = false;
          if (at < kPendCap) plist[at] = (uint32_t)k * 64u + (uint32_t)b;
          else on = decide_pixel64<DS>(J, row0 + r, (int64_t)w * 64 + b);
        }
        half[q] = __ballot_sync(0xffffffffu, on);
      }
      if (lane == 0) out[t] = ((uint64_t)half[1] << 32) | half[0];
    }
    __syncthreads();
    // ---- phase 5: the collected pixels in FP64, into the words stored above
    const int npend = min(s_np, kPendCap);
    for (int q = threadIdx.x; q < npend; q += nthr) {
      const int k = (int)(plist[q] >> 6), b = (int)(plist[q] & 63u);
      const int t = t0 + k, r = row_of(t), w = t - r * row_words;
      if (decide_pixel64<DS>(J, row0 + r, (int64_t)w * 64 + b))
        atomicOr(reinterpret_cast<unsigned long long*>(out + t), 1ull << b);
    }
    if (t0 + kPass < nwords) {
      __syncthreads();
      if (threadIdx.x == 0) s_n = s_npx = s_nre = s_np = 0;
      __syncthreads();
    }
  }
}

// ------------------------------------------------------- corner-rule plots
// The corner rule of pa.h (pa_rule), one thread per output byte (8 pixels of
// the last axis).  For each of the 2^(d-1) corner choices on the leading axes,
// f is evaluated at the lattice points i0 .. i0 + nb of the last axis (9 for a
// full byte); bit j of the masks n / p / q records that lattice point j passes
// the comparison / has a finite value above 0 / below 0.  Pixel b has lattice
// points b and b + 1 on the last axis, so its bit in each pixel mask is
// m | m >> 1.  Bytes past the last pixel of a row are written as 0.  Off by
// default and evaluated in plain FP64 (no FP32 filter): every corner value
// costs one full evaluation, 9/8 per pixel and leading corner choice.
__device__ __forceinline__ double lattice_point(double lo, double delta, int64_t i) {
  return __dadd_rn(lo, __dmul_rn((double)i, delta));
}

__global__ void __launch_bounds__(256)
plot_corner_kernel(const CornerJob* __restrict__ jobs, int njobs, int64_t total_bytes) {
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total_bytes;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int64_t w = t >> 3;
    const int byte = (int)(t & 7);
    int lo = 0, hi = njobs - 1;
    while (lo < hi) {
      const int mid = (lo + hi + 1) >> 1;
      if (jobs[mid].word0 <= w) lo = mid; else hi = mid - 1;
    }
    const CornerJob& J = jobs[lo];
    const int64_t lw = w - J.word0;
    const int64_t row = lw / J.row_words;
    const int64_t wi = lw - row * J.row_words;
    const int last = J.ndim - 1;
    int64_t idx[kMaxDim];
    int64_t rest = row;
    for (int a = last - 1; a >= 0; --a) {
      idx[a] = rest % J.res[a];
      rest /= J.res[a];
    }
    const int i0 = (int)(wi * 64) + 8 * byte;
    const int nb = min(8, J.res[last] - i0);  // pixels of this byte (<= 0: padding)
    uint32_t near = 0, pos = 0, neg = 0;  // per pixel, OR over its corners
    for (int m = 0; nb > 0 && m < (1 << last); ++m) {
      double x[kMaxDim];
      for (int p = 0; p < J.arity; ++p) {
        const int a = J.port_axis[p];
        if (a != last) x[p] = lattice_point(J.lo[p], J.delta[p], idx[a] + ((m >> a) & 1));
      }
      uint32_t n = 0, pp = 0, q = 0;  // lattice points 0..nb
      for (int j = 0; j <= nb; ++j) {
        for (int p = 0; p < J.arity; ++p)
          if (J.port_axis[p] == last) x[p] = lattice_point(J.lo[p], J.delta[p], i0 + j);
        double f;
        if (J.prog) {
          f = run_expr(J.prog, J.nops, J.consts, x);
        } else {
          const double* cp = J.coeffs;
          f = nest_rows<double>(J.arity - 1, J.degree, cp, x);
        }
        n |= (decide64(f, J.kind, J.eps, J.strict) ? 1u : 0u) << j;
        pp |= ((isfinite(f) && f > 0.0) ? 1u : 0u) << j;
        q |= ((isfinite(f) && f < 0.0) ? 1u : 0u) << j;
      }
      near |= n | (n >> 1);
      pos |= pp | (pp >> 1);
      neg |= q | (q >> 1);
    }
    uint32_t bits = near | (J.kind == PA_EQ ? (pos & neg) : 0u);
    bits = nb > 0 ? bits & ((1u << nb) - 1u) : 0u;
    reinterpret_cast<uint8_t*>(J.out + lw)[byte] = (uint8_t)bits;
  }
}

void launch_plot_corner(const CornerJob* d_jobs, int njobs, int64_t total_words, cudaStream_t s) {
  if (njobs <= 0 || total_words <= 0) return;
  const int64_t bytes = 8 * total_words;
  int64_t blocks = (bytes + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  plot_corner_kernel<<<(unsigned)blocks, 256, 0, s>>>(d_jobs, njobs, bytes);
}

// Blocks of the plot kernel (of this degree) that the GPU holds at once:
// per SM as the occupancy calculator gives it for 256 threads and a typical
// 4 KB of row polynomials (registers are the limit), times the SMs.  Cached;
// 4 x 152 when the device cannot be asked.
int plot_resident_blocks(int common_degree) {
  static std::mutex mu;
  static std::map<std::pair<int, int>, int> cache;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) {
    cudaGetLastError();
    return 4 * 152;
  }
  const std::pair<int, int> key(dev, common_degree);
  {
    std::lock_guard<std::mutex> lk(mu);
    auto it = cache.find(key);
    if (it != cache.end()) return it->second;
  }
  const void* fn;
  switch (common_degree) {
    case 1: fn = reinterpret_cast<const void*>(plot_kernel<1>); break;
    case 2: fn = reinterpret_cast<const void*>(plot_kernel<2>); break;
    case 3: fn = reinterpret_cast<const void*>(plot_kernel<3>); break;
    case 4: fn = reinterpret_cast<const void*>(plot_kernel<4>); break;
    default: fn = reinterpret_cast<const void*>(plot_kernel<-1>); break;
  }
  int sms = 0, per = 0;
  int v = 4 * 152;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess &&
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, fn, kPlotThreads, 4 * 1024) ==
          cudaSuccess &&
      sms > 0 && per > 0)
    v = sms * per;
  else
    cudaGetLastError();
  std::lock_guard<std::mutex> lk(mu);
  cache[key] = v;
  return v;
}

cudaError_t probe_kernel_image() {
  cudaFuncAttributes attr;
  return cudaFuncGetAttributes(&attr, plot_kernel<-1>);
}

void launch_plot(const PlotJob* d_jobs, int njobs, int64_t total_tiles, int max_rows_per_tile,
                 int max_degree, int common_degree, const ZeroRange* d_zero, int nzero,
                 int64_t zero_words, cudaStream_t s) {
  if (total_tiles <= 0) return;
  const int gstride = max_degree + 1;
  const size_t smem = (size_t)max_rows_per_tile * gstride * sizeof(float);
  // programmatic dependent launch: the blocks are scheduled while the launch
  // before them (the upload of a kept program) runs
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)total_tiles);
  cfg.blockDim = dim3(kPlotThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
#define PA_PLOT(DD)                                                                          \
  do {                                                                                       \
    smem_limit(reinterpret_cast<const void*>(plot_kernel<DD>), smem);                        \
    cudaLaunchKernelEx(&cfg, plot_kernel<DD>, d_jobs, njobs, gstride, d_zero, nzero,         \
                       zero_words);                                                          \
  } while (0)
  switch (common_degree) {
    case 1: PA_PLOT(1); break;
    case 2: PA_PLOT(2); break;
    case 3: PA_PLOT(3); break;
    case 4: PA_PLOT(4); break;
    default: PA_PLOT(-1); break;
  }
#undef PA_PLOT
}

}  // namespace pa
