// Plots of expression relations (Sec. 3.2, sample-in-center plot, for
// relations built from the ports with arithmetic and elementary functions,
// as in the examples of Sec. 2.1 and Sec. 2.4).
//
// The program of a pixel costs hundreds of FP64 operations (GB300: 1.7 flops per
// SM and clock), and a plotted curve leaves most pixels far from eps, so runs of
// pixels are first decided as a whole by interval arithmetic in FP32: the
// program is run once on intervals that hold the coordinates of every pixel of
// the run, each operation returning an interval that holds every value the FP64
// program can take.  A run whose final interval lies outside the accepted set is
// off, one inside it on; the rest is evaluated in FP64, pixel by pixel, so the
// result is the FP64 decision in every case.
//   - + - * / sqrt: FP32 operations rounded outwards.  FP64 rounding is monotone
//     and the endpoints are FP64 numbers, so the rounded FP64 result stays inside.
//   - the elementary functions: CUDA's FP32 function at the ends (at the middle,
//     with the half width as the bound, for sin and cos), widened by 2^-19 of the
//     value: 16 units in the last place, four times the largest error CUDA
//     states for any of them, which also covers the FP64 functions' own.
//   - operations that may leave a function's domain return what the points inside
//     it give and set a flag; the others are NaN, which stays NaN through every
//     operation but pow (then: any value) and turns the pixel off.  A run is only
//     decided "on" without the flag.
// Blocks test whole words (64 pixels; not on small grids), then the 8-pixel pieces of
// the words left,
// then evaluate the pieces left with eight lanes each.  What bounds it: the FP64
// pipe on the pieces left, and the interpreter's instructions.  Whole solves against
// FP64 at every pixel: butterfly at 2048 px 1523 -> 113 us, 3-D arrays at 75 px
// 248 -> 55.
#include <float.h>
#include <math.h>

#include "expr_eval.cuh"
#include "pa_internal.h"

namespace pa {
namespace {

__device__ __forceinline__ double expr_centre(double lo, double delta, int64_t i) {
  return __dadd_rn(lo, __dmul_rn(__dadd_rn((double)i, 0.5), delta));
}

struct Iv {
  float lo, hi;
};

__device__ __forceinline__ Iv whole() { return {-INFINITY, INFINITY}; }

// Endpoints of a function's values, widened by 2^-19 and never further in than
// the largest finite number (an FP32 overflow of the lower end says only that
// the value is large).
__device__ __forceinline__ Iv widen(float lo, float hi) {
  lo = fminf(lo, FLT_MAX);
  hi = fmaxf(hi, -FLT_MAX);
  return {__fsub_rd(lo, __fmaf_ru(fabsf(lo), 0x1p-19f, 1e-37f)),
          __fadd_ru(hi, __fmaf_ru(fabsf(hi), 0x1p-19f, 1e-37f))};
}

// An interval with a NaN end (inf - inf, 0 * inf) holds any value.
__device__ __forceinline__ Iv checked(float lo, float hi, bool* bad) {
  if (isnan(lo) || isnan(hi)) {
    *bad = true;
    return whole();
  }
  return {lo, hi};
}

__device__ __forceinline__ Iv iv_mul(Iv a, Iv b, bool* bad) {
  const float p = __fmul_rd(a.lo, b.lo), q = __fmul_rd(a.lo, b.hi), r = __fmul_rd(a.hi, b.lo),
              s = __fmul_rd(a.hi, b.hi);
  const float P = __fmul_ru(a.lo, b.lo), Q = __fmul_ru(a.lo, b.hi), R = __fmul_ru(a.hi, b.lo),
              S = __fmul_ru(a.hi, b.hi);
  if (isnan(p) || isnan(q) || isnan(r) || isnan(s)) {
    *bad = true;
    return whole();
  }
  return {fminf(fminf(p, q), fminf(r, s)), fmaxf(fmaxf(P, Q), fmaxf(R, S))};
}

__device__ __forceinline__ Iv iv_div(Iv a, Iv b, bool* bad) {
  if (!(b.lo > 0.0f || b.hi < 0.0f)) {
    *bad = true;
    return whole();
  }
  const float p = __fdiv_rd(a.lo, b.lo), q = __fdiv_rd(a.lo, b.hi), r = __fdiv_rd(a.hi, b.lo),
              s = __fdiv_rd(a.hi, b.hi);
  const float P = __fdiv_ru(a.lo, b.lo), Q = __fdiv_ru(a.lo, b.hi), R = __fdiv_ru(a.hi, b.lo),
              S = __fdiv_ru(a.hi, b.hi);
  if (isnan(p) || isnan(q) || isnan(r) || isnan(s)) {
    *bad = true;
    return whole();
  }
  return {fminf(fminf(p, q), fminf(r, s)), fmaxf(fmaxf(P, Q), fmaxf(R, S))};
}

__device__ __forceinline__ Iv iv_abs(Iv a) {
  if (a.lo >= 0.0f) return a;
  if (a.hi <= 0.0f) return {-a.hi, -a.lo};
  return {0.0f, fmaxf(-a.lo, a.hi)};
}

__device__ __noinline__ Iv iv_exp(Iv a) {
  const Iv r = widen(expf(a.lo), expf(a.hi));
  return {fmaxf(r.lo, 0.0f), r.hi};
}

__device__ __noinline__ Iv iv_log(Iv a, bool* bad) {
  if (!(a.lo > 0.0f)) *bad = true;  // 0 and below: -inf and NaN
  if (!(a.hi > 0.0f)) return whole();
  const float hi = logf(a.hi);
  return a.lo > 0.0f ? widen(logf(a.lo), hi) : Iv{-INFINITY, widen(hi, hi).hi};
}

// sin (or cos) moves at most as far as its argument
__device__ __noinline__ Iv iv_sincos(Iv a, bool cosine, bool* bad) {
  const float mid = 0.5f * a.lo + 0.5f * a.hi;
  const float r = fmaxf(__fsub_ru(a.hi, mid), __fsub_ru(mid, a.lo));
  if (!(r < 4.0f) || !(fabsf(mid) < 1e6f)) {
    if (!(a.lo > -INFINITY && a.hi < INFINITY)) *bad = true;
    return {-1.0f, 1.0f};
  }
  const float v = cosine ? cosf(mid) : sinf(mid);
  const Iv w = widen(v, v);
  return {fmaxf(-1.0f, __fsub_rd(w.lo, r)), fminf(1.0f, __fadd_ru(w.hi, r))};
}

// tan rises between its poles; the ends have to lie on one branch, clear of the
// rounding of x / pi
__device__ __noinline__ Iv iv_tan(Iv a, bool* bad) {
  const float ql = a.lo * 0.318309886f + 0.5f, qh = a.hi * 0.318309886f + 0.5f;
  const float fl = floorf(ql), fh = floorf(qh);
  if (!(fabsf(a.lo) < 1e3f && fabsf(a.hi) < 1e3f) || fl != fh || !(ql - fl > 1e-3f) ||
      !(qh - fh < 1.0f - 1e-3f)) {
    *bad = true;
    return whole();
  }
  return widen(tanf(a.lo), tanf(a.hi));
}

__device__ __noinline__ Iv iv_powi(Iv a, int arg, bool* bad) {
  const int n = arg < 0 ? -arg : arg;
  if (n == 0) return {1.0f, 1.0f};
  Iv r;
  const bool mixed = a.lo < 0.0f && a.hi > 0.0f;
  if (n % 2 == 0 || !mixed) {
    // |a|^n by products rounded outwards, then the sign
    const Iv m = iv_abs(a);
    r = m;
    for (int j = 1; j < n; ++j) r = checked(__fmul_rd(r.lo, m.lo), __fmul_ru(r.hi, m.hi), bad);
    if (n % 2 && a.hi <= 0.0f) r = {-r.hi, -r.lo};
  } else {
    r = a;  // odd power over 0: each end by itself
    for (int j = 1; j < n; ++j)
      r = checked(-__fmul_ru(fabsf(r.lo), fabsf(a.lo)), __fmul_ru(r.hi, a.hi), bad);
  }
  return arg < 0 ? iv_div({1.0f, 1.0f}, r, bad) : r;
}

__device__ __noinline__ Iv iv_pow(Iv a, Iv b, bool* bad) {
  // (a NaN operand can give 1: pow(x, 0), pow(1, y))
  if (*bad || !(a.lo > 0.0f)) {
    *bad = true;
    return whole();
  }
  return iv_exp(iv_mul(b, iv_log(a, bad), bad));
}

// The program on intervals; *bad: some point may be NaN or infinite on the way.
__device__ Iv run_interval(const int32_t* __restrict__ prog, int nops,
                           const float2* __restrict__ c32, const Iv* x, bool* bad) {
  Iv st[PA_EXPR_MAX_STACK];
  int sp = 0;
  *bad = false;
  for (int k = 0; k < nops; ++k) {
    const int32_t ins = __ldg(prog + k);
    const int op = ins & 0xff, arg = ins >> 8;
    if (op == PA_X_CONST) {
      const float2 c = __ldg(c32 + arg);
      st[sp++] = {c.x, c.y};
      continue;
    }
    if (op == PA_X_VAR) {
      st[sp++] = x[arg];
      continue;
    }
    Iv r;
    if ((op >= PA_X_ADD && op <= PA_X_DIV) || op == PA_X_POW) {
      const Iv b = st[--sp], a = st[sp - 1];
      switch (op) {
        case PA_X_ADD: r = checked(__fadd_rd(a.lo, b.lo), __fadd_ru(a.hi, b.hi), bad); break;
        case PA_X_SUB: r = checked(__fsub_rd(a.lo, b.hi), __fsub_ru(a.hi, b.lo), bad); break;
        case PA_X_MUL: r = iv_mul(a, b, bad); break;
        case PA_X_DIV: r = iv_div(a, b, bad); break;
        default: r = iv_pow(a, b, bad); break;
      }
    } else {
      const Iv a = st[sp - 1];
      switch (op) {
        case PA_X_NEG: r = {-a.hi, -a.lo}; break;
        case PA_X_ABS: r = iv_abs(a); break;
        case PA_X_SQRT:
          if (a.lo < 0.0f) *bad = true;
          r = a.hi >= 0.0f ? Iv{__fsqrt_rd(fmaxf(a.lo, 0.0f)), __fsqrt_ru(a.hi)} : whole();
          break;
        case PA_X_EXP: r = iv_exp(a); break;
        case PA_X_LOG: r = iv_log(a, bad); break;
        case PA_X_SIN: r = iv_sincos(a, false, bad); break;
        case PA_X_COS: r = iv_sincos(a, true, bad); break;
        case PA_X_TAN: r = iv_tan(a, bad); break;
        case PA_X_SINH: r = widen(sinhf(a.lo), sinhf(a.hi)); break;
        case PA_X_COSH: {
          const Iv m = iv_abs(a);
          r = widen(coshf(m.lo), coshf(m.hi));
          break;
        }
        case PA_X_TANH: r = widen(tanhf(a.lo), tanhf(a.hi)); break;
        case PA_X_ATAN: r = widen(atanf(a.lo), atanf(a.hi)); break;
        case PA_X_POWI: r = iv_powi(a, arg, bad); break;
        default: r = whole(); break;
      }
    }
    // an infinite end means values FP64 may hold as infinities
    if (!(r.lo > -INFINITY && r.hi < INFINITY)) *bad = true;
    st[sp - 1] = r;
  }
  return sp == 1 ? st[0] : whole();
}

// The job, row and word of flat word w; idx: the row's axis indices.
struct Place {
  const ExprJob* J;
  int64_t word;   // within the job
  int wi;         // word of the row
  int idx[kMaxDim];
};
__device__ __forceinline__ void locate(const ExprJob* __restrict__ jobs, int njobs, int64_t w, Place& P) {
  int lo = 0, hi = njobs - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) >> 1;
    if (jobs[mid].word0 <= w) lo = mid; else hi = mid - 1;
  }
  P.J = jobs + lo;
  P.word = w - P.J->word0;
  int64_t rest = P.word / P.J->row_words;
  P.wi = (int)(P.word - rest * P.J->row_words);
  for (int a = P.J->ndim - 2; a >= 0; --a) {
    P.idx[a] = (int)(rest % P.J->res[a]);
    rest /= P.J->res[a];
  }
}

// Pixels [i0, i1] of a word's row as a whole: 1 all off, 2 all on, 0 undecided.
__device__ __forceinline__ int decide_run(const Place& P, int i0, int i1) {
  const ExprJob& J = *P.J;
  Iv x[kMaxDim];
  for (int p = 0; p < J.arity; ++p) {
    const int a = J.port_axis[p];
    const bool last = a == J.ndim - 1;
    // the centres rise with the index
    const double c0 = expr_centre(J.lo[p], J.delta[p], last ? i0 : P.idx[a]);
    const double c1 = last ? expr_centre(J.lo[p], J.delta[p], i1) : c0;
    x[p] = {__double2float_rd(c0), __double2float_ru(c1)};
  }
  bool bad;
  const Iv f = run_interval(J.prog, J.nops, J.c32, x, &bad);
  const double lo = f.lo, hi = f.hi;
  if (J.kind == PA_EQ) {
    if (lo > J.eps || hi < -J.eps) return 1;
    return (!bad && lo > -J.eps && hi < J.eps) ? 2 : 0;
  }
  if (lo > J.eps) return 1;
  return (!bad && hi < J.eps) ? 2 : 0;
}

// THREADS: the block, and the most words it takes.  FIRST: what the block starts with,
// whole words, the 8-pixel pieces of every word, or every pixel in FP64.
enum { kWords, kPieces, kPixels };
template <int THREADS, int FIRST>
__global__ void __launch_bounds__(THREADS)
plot_expr_kernel(const ExprJob* __restrict__ jobs, int njobs, int64_t total_words, int words) {
  __shared__ uint16_t wlist[THREADS], plist[8 * THREADS];
  __shared__ int s_w, s_p;
  const int tid = threadIdx.x;
  const int64_t w0 = (int64_t)blockIdx.x * words;
  const int mine = (int)min((int64_t)words, total_words - w0);  // words of this block
  if (tid == 0) {
    s_w = FIRST == kPieces ? mine : 0;
    s_p = FIRST == kPixels ? 8 * mine : 0;
  }
  __syncthreads();
  if (FIRST == kPixels)
    for (int e = tid; e < 8 * mine; e += THREADS) plist[e] = (uint16_t)e;
  if (tid < mine) {
    if constexpr (FIRST == kWords) {
      Place P;
      locate(jobs, njobs, w0 + tid, P);
      const int i0 = P.wi * 64, nb = min(64, P.J->res[P.J->ndim - 1] - i0);
      const int dec = decide_run(P, i0, i0 + nb - 1);
      if (dec) P.J->out[P.word] = dec == 1 ? 0ull : nb == 64 ? ~0ull : (1ull << nb) - 1ull;
      else wlist[atomicAdd(&s_w, 1)] = (uint16_t)tid;
    } else {
      wlist[tid] = (uint16_t)tid;
    }
  }
  __syncthreads();
  // the 8-pixel pieces of the words left (a byte of the word each)
  const int nw = s_w;
  for (int e = tid; e < 8 * nw; e += THREADS) {
    const int k = wlist[e >> 3], c = e & 7;
    Place P;
    locate(jobs, njobs, w0 + k, P);
    const int i0 = P.wi * 64 + 8 * c, nb = min(8, P.J->res[P.J->ndim - 1] - i0);
    const int dec = nb > 0 ? decide_run(P, i0, i0 + nb - 1) : 1;
    if (dec) reinterpret_cast<uint8_t*>(P.J->out + P.word)[c] = dec == 1 ? 0 : (uint8_t)((1u << nb) - 1u);
    else plist[atomicAdd(&s_p, 1)] = (uint16_t)(8 * k + c);
  }
  __syncthreads();
  // the pieces left, a lane per pixel
  const int np = s_p;
  const int lane = tid & 31;
  for (int base = 0; base < 8 * np; base += THREADS) {
    const int e = base + tid;
    bool on = false;
    Place P;
    int c = 0;
    if (e < 8 * np) {
      const int piece = plist[e >> 3];
      c = piece & 7;
      locate(jobs, njobs, w0 + (piece >> 3), P);
      const ExprJob& J = *P.J;
      const int i = P.wi * 64 + 8 * c + (e & 7);
      if (i < J.res[J.ndim - 1]) {
        double x[kMaxDim];
        for (int p = 0; p < J.arity; ++p) {
          const int a = J.port_axis[p];
          x[p] = expr_centre(J.lo[p], J.delta[p], a == J.ndim - 1 ? (int64_t)i : P.idx[a]);
        }
        const double f = run_expr(J.prog, J.nops, J.consts, x);
        if (isfinite(f)) {
          const double d = (J.kind == PA_EQ) ? fabs(f) : f;
          on = (J.strict || J.kind == PA_LT) ? (d < J.eps) : (d <= J.eps);
        }
      }
    }
    const uint32_t bits = __ballot_sync(0xffffffffu, on);
    if (e < 8 * np && (lane & 7) == 0)
      reinterpret_cast<uint8_t*>(P.J->out + P.word)[c] = (uint8_t)(bits >> (lane & 24));
  }
}

}  // namespace

void launch_plot_expr(const ExprJob* d_jobs, int njobs, int64_t total_words, cudaStream_t s) {
  if (njobs <= 0 || total_words <= 0) return;
  // A small grid is bound by a chain of programs and by FP64 on the SMs that its few
  // undecided words are on: small blocks of few words each, at least seven per SM, and
  // no test whose lanes would not fill half the GPU (words; a quarter for pieces,
  // whose test spares FP64), as it only lengthens the chain.  Butterfly, whole
  // solves, alone / among others, against the launch below: 40 px 104 / 58.7 -> 79 / 49.6,
  // 125 px 114 / 69.7 -> 81 / 47.5, 300 px 109 / 63.1 -> 91 / 47.6, 500 px 109 / 64.1 -> 99 / 53.0; FP64 at
  // every pixel in blocks of 256: 84 / 57, 89 / 55, 115 / 73 and 173 / 129.
  if (8 * total_words <= 152 * 1024) {
    int64_t words = 1;
    while (words < 128 && total_words / (2 * words) >= 152 * 7) words *= 2;
    const unsigned grid = (unsigned)((total_words + words - 1) / words);
    if (64 * total_words <= 152 * 512)
      plot_expr_kernel<128, kPixels><<<grid, 128, 0, s>>>(d_jobs, njobs, total_words, (int)words);
    else
      plot_expr_kernel<128, kPieces><<<grid, 128, 0, s>>>(d_jobs, njobs, total_words, (int)words);
    return;
  }
  // Others: up to one word per thread, fewer while the blocks do not fill the GPU four
  // times over (the undecided pieces of neighbouring words end up in one block).  At
  // 800 px and 75^3 this is as fast as the small blocks (70.5 against 72.8 us, 56.8
  // against 55.7), at 4096 px faster than any of them (209 against 212).
  int64_t words = 32;
  while (words < 256 && total_words / words > 152 * 16) words *= 2;
  plot_expr_kernel<256, kWords><<<(unsigned)((total_words + words - 1) / words), 256, 0, s>>>(
      d_jobs, njobs, total_words, (int)words);
}

}  // namespace pa
