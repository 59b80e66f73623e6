// Contraction kernels: Eq. (GAM) of Sec. 3.3 for one two-array cluster (Sec. 3.5)
// over the Boolean semiring, on bit-packed arrays.
//
// After the planner has brought both operands into matrix form
//   A[b][m][k]  (k packed along rows)   and   B[b][k][n]  (n packed along rows),
// the cluster is C[b][m][n] = OR_k A[b][m][k] AND B[b][k][n], computed row-wise:
// row (b, m) of C is the OR of the rows B[b][k][:] selected by the set bits of
// row (b, m) of A.  Curve plots are sparse and their set bits come in runs, so
// with ORs of aligned blocks of B rows the work is proportional to the number
// of maximal aligned all-ones blocks of A (at most its set bits) times the
// packed width of B, not to M*K*N.
#include <cuda.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <mutex>

#include "pa_internal.h"
#include "row_walk.h"

namespace pa {

// --------------------------------------------------------------- reshape
// Every reshape launch runs a table of descriptors: problem p owns blocks
// [cta0[p], cta0[p+1]) and its descriptor is copied into shared memory; the
// kernels' grid-stride loops run over the problem's own blocks.  (One launch
// per kind serves all reshapes of one tree level of every system of a batch.)
struct RsCtx {
  int64_t bid, nblk;
};
__device__ __forceinline__ RsCtx rs_pick(const ReshapeDesc* __restrict__ descs,
                                         const int64_t* __restrict__ cta0, int n, ReshapeDesc* sd) {
  const int lo = find_entry([&](int i) { return cta0[i]; }, n, (int64_t)blockIdx.x);
  const int64_t* src = reinterpret_cast<const int64_t*>(descs + lo);
  int64_t* dst = reinterpret_cast<int64_t*>(sd);
  for (int i = threadIdx.x; i < (int)(sizeof(ReshapeDesc) / 8); i += blockDim.x) dst[i] = src[i];
  __syncthreads();
  return RsCtx{(int64_t)blockIdx.x - cta0[lo], cta0[lo + 1] - cta0[lo]};
}

// Bit mode: one warp per output word, one lane per bit (two ballots pack the
// 64 bits).  Every bit is decoded and gathered on its own, OR-ed over the
// reduced axes with an early exit.  With row_any set, every packed input axis
// is reduced and red_* hold only the reduced row axes: a bit is then the OR of
// whole input rows, scanned by words (padding bits are zero).  When those rows
// are long together (kAnyScan words or more per bit) a block takes an output
// word and its warps one bit after another, a bit's words dealt over the lanes:
// a lane scanning them alone is a chain of as many loads.
constexpr int64_t kAnyScan = 64;
__device__ void any_rows(const ReshapeDesc& d, int64_t bid, int64_t nblk) {
  __shared__ uint32_t s_bits[2];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  const int64_t total = d.out_nrows * d.out_row_words;
  const int outer = d.out_ndim - d.out_inner;
  int64_t red_total = 1;
  for (int q = 0; q < d.nred; ++q) red_total *= d.red_res[q];
  const int64_t scan = red_total * d.in_row_words;
  for (int64_t ow = bid; ow < total; ow += nblk) {
    if (threadIdx.x < 2) s_bits[threadIdx.x] = 0;
    __syncthreads();
    const int64_t orow = ow / d.out_row_words, w = ow % d.out_row_words;
    int64_t brow = 0, rest = orow;
    for (int a = outer - 1; a >= 0; --a) {
      brow += rest % d.out_res[a] * d.row_stride[a];
      rest /= d.out_res[a];
    }
    for (int bit = warp; bit < 64; bit += nwarps) {
      const int64_t ocol = w * 64 + bit;
      if (ocol >= d.out_rowlen) break;
      int64_t row = brow, rest2 = ocol;
      for (int a = d.out_ndim - 1; a >= outer; --a) {
        row += rest2 % d.out_res[a] * d.row_stride[a];
        rest2 /= d.out_res[a];
      }
      bool any = false;
      for (int64_t s0 = 0; s0 < scan && !any; s0 += 32) {
        const int64_t s = s0 + lane;
        uint64_t v = 0;
        if (s < scan) {
          int64_t r = row, srest = s / d.in_row_words;
          const int64_t k = s - srest * d.in_row_words;
          for (int q = d.nred - 1; q >= 0; --q) {
            r += srest % d.red_res[q] * d.red_row_stride[q];
            srest /= d.red_res[q];
          }
          v = __ldg(d.in + r * d.in_row_words + k);
        }
        any = __any_sync(0xffffffffu, v != 0ull);
      }
      if (any && lane == 0) atomicOr(&s_bits[bit >> 5], 1u << (bit & 31));
    }
    __syncthreads();
    if (threadIdx.x == 0) d.out[ow] = (uint64_t)s_bits[0] | ((uint64_t)s_bits[1] << 32);
    __syncthreads();
  }
}

// Words scanned per output bit of a row_any reshape.
__host__ __device__ __forceinline__ int64_t any_scan(const ReshapeDesc& d) {
  int64_t n = d.in_row_words;
  for (int q = 0; q < d.nred; ++q) n *= d.red_res[q];
  return n;
}

__global__ void reshape_kernel(const ReshapeDesc* __restrict__ descs, const int64_t* __restrict__ cta0,
                               int n) {
  __shared__ ReshapeDesc sd;
  const RsCtx rc = rs_pick(descs, cta0, n, &sd);
  const ReshapeDesc& d = sd;
  if (d.row_any && any_scan(d) >= kAnyScan) {
    any_rows(d, rc.bid, rc.nblk);
    return;
  }
  const int lane = threadIdx.x & 31;
  const int64_t total = d.out_nrows * d.out_row_words;
  const int outer = d.out_ndim - d.out_inner;
  int64_t red_total = 1;
  for (int q = 0; q < d.nred; ++q) red_total *= d.red_res[q];
  const int64_t nwarps = rc.nblk * (blockDim.x >> 5);
  for (int64_t ow = rc.bid * (blockDim.x >> 5) + (threadIdx.x >> 5); ow < total; ow += nwarps) {
    const int64_t orow = ow / d.out_row_words, w = ow % d.out_row_words;
    int64_t brow = 0, bcol = 0, rest = orow;
    for (int a = outer - 1; a >= 0; --a) {
      const int64_t v = rest % d.out_res[a];
      rest /= d.out_res[a];
      brow += v * d.row_stride[a];
      bcol += v * d.col_stride[a];
    }
    uint32_t half[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t ocol = w * 64 + h * 32 + lane;
      bool bit = false;
      if (ocol < d.out_rowlen) {
        int64_t rr = brow, cc = bcol, rest2 = ocol;
        for (int a = d.out_ndim - 1; a >= outer; --a) {
          const int64_t v = rest2 % d.out_res[a];
          rest2 /= d.out_res[a];
          rr += v * d.row_stride[a];
          cc += v * d.col_stride[a];
        }
        int64_t cnt[2 * kMaxDim] = {};
        for (int64_t s = 0; s < red_total && !bit; ++s) {
          if (d.row_any) {
            const uint64_t* row = d.in + rr * d.in_row_words;
            uint64_t acc = 0;
            for (int64_t k = 0; k < d.in_row_words && !acc; ++k) acc = row[k];
            bit = acc != 0;
          } else {
            bit = (d.in[rr * d.in_row_words + (cc >> 6)] >> (cc & 63)) & 1ull;
          }
          for (int q = d.nred - 1; q >= 0; --q) {
            rr += d.red_row_stride[q];
            cc += d.red_col_stride[q];
            if (++cnt[q] < d.red_res[q]) break;
            rr -= d.red_row_stride[q] * d.red_res[q];
            cc -= d.red_col_stride[q] * d.red_res[q];
            cnt[q] = 0;
          }
        }
      }
      half[h] = __ballot_sync(0xffffffffu, bit);
    }
    if (lane == 0) d.out[ow] = (uint64_t)half[0] | ((uint64_t)half[1] << 32);
  }
}

// Words mode: output word index -> input word index through the mixed-radix
// decomposition (u_res, u_in), then an OR over the reduced axes.  A thread takes
// V = 4, 2 or 1 consecutive words (the last axis runs along the words of both
// sides), which spreads the divisions of the decomposition over them; a
// reduction over many values with few output words is dealt over the lanes of a
// warp.  Index type I is 32-bit when every word index fits.  Bound by HBM and the
// index arithmetic: 38 networks' word reshapes 0.96 -> 0.28 ms, a reduction of
// 75^2 values into 2 words each 47 -> 6 us (ncu, cold; a thread per word before).
template <int V>
struct WordRun {
  uint64_t v[V];
};
template <int V>
__device__ __forceinline__ WordRun<V> load_run(const uint64_t* __restrict__ p) {
  WordRun<V> r;
  if constexpr (V == 1) {
    r.v[0] = *p;
  } else {
#pragma unroll
    for (int k = 0; k < V; k += 2) {
      const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p + k);
      r.v[k] = t.x;
      r.v[k + 1] = t.y;
    }
  }
  return r;
}
template <int V>
__device__ __forceinline__ void store_run(uint64_t* p, const WordRun<V>& r) {
  if constexpr (V == 1) {
    *p = r.v[0];
  } else {
#pragma unroll
    for (int k = 0; k < V; k += 2)
      *reinterpret_cast<ulonglong2*>(p + k) = make_ulonglong2(r.v[k], r.v[k + 1]);
  }
}

template <class I, int V>
__device__ __forceinline__ void reshape_words(const ReshapeDesc& d, I bid, I nblk) {
  const I units = (I)(d.out_nrows * d.out_row_words) / V;
  const int last = d.nu - 1;
  auto src_of = [&](I u) -> I {
    I r = (I)d.u_res[last] / V;
    I q = u / r;
    I src = (u - q * r) * V;  // (u_in[last] is 1)
    I rest = q;
    for (int a = last - 1; a >= 0; --a) {
      r = (I)d.u_res[a];
      q = rest / r;
      src += (rest - q * r) * (I)d.u_in[a];
      rest = q;
    }
    return src;
  };
  I red_total = 1;
  for (int q = 0; q < d.nred; ++q) red_total *= (I)d.red_res[q];
  const I gid = bid * blockDim.x + threadIdx.x, gthreads = nblk * blockDim.x;
  if (red_total == 1) {
    // a pure permutation: 4 words in flight per thread
    constexpr int U = 4 / V;
    I u = gid;
    for (; u + (U - 1) * gthreads < units; u += U * gthreads) {
      WordRun<V> v[U];
#pragma unroll
      for (int k = 0; k < U; ++k) v[k] = load_run<V>(d.in + src_of(u + (I)k * gthreads));
#pragma unroll
      for (int k = 0; k < U; ++k) store_run<V>(d.out + (u + (I)k * gthreads) * V, v[k]);
    }
    for (; u < units; u += gthreads) store_run<V>(d.out + u * V, load_run<V>(d.in + src_of(u)));
    return;
  }
  // lanes per unit: a power of two, as long as there are values and idle threads
  int g = 1;
  while (g < 32 && (I)(2 * g) <= red_total && units * (I)(2 * g) <= (I)(152 * 2048)) g *= 2;
  const int sub = threadIdx.x & (g - 1);
  // (whole warps run the loop: the lanes of a unit combine with shuffles)
  const I uend = (units + 32 / g - 1) / (32 / g) * (32 / g);
  for (I u = gid / g; u < uend; u += gthreads / g) {
    WordRun<V> acc;
#pragma unroll
    for (int k = 0; k < V; ++k) acc.v[k] = 0;
    if (u < units) {
      const I src = src_of(u);
#pragma unroll 4
      for (I s = sub; s < red_total; s += g) {
        I at = src, rest = s;
        for (int q = d.nred - 1; q > 0; --q) {
          const I r = (I)d.red_res[q], t = rest / r;
          at += (rest - t * r) * (I)d.red_in_w[q];
          rest = t;
        }
        at += rest * (I)d.red_in_w[0];
        const WordRun<V> v = load_run<V>(d.in + at);
#pragma unroll
        for (int k = 0; k < V; ++k) acc.v[k] |= v.v[k];
      }
    }
    for (int o = 1; o < g; o <<= 1)
#pragma unroll
      for (int k = 0; k < V; ++k) acc.v[k] |= __shfl_xor_sync(0xffffffffu, acc.v[k], o);
    if (u < units && sub == 0) store_run<V>(d.out + u * V, acc);
  }
}

template <class I>
__global__ void __launch_bounds__(256)
reshape_words_kernel(const ReshapeDesc* __restrict__ descs, const int64_t* __restrict__ cta0, int n) {
  __shared__ ReshapeDesc sd;
  const RsCtx rc = rs_pick(descs, cta0, n, &sd);
  const ReshapeDesc& d = sd;
  const bool aligned = ((reinterpret_cast<uintptr_t>(d.in) | reinterpret_cast<uintptr_t>(d.out)) & 15) == 0;
  if (d.vec == 4 && aligned) reshape_words<I, 4>(d, (I)rc.bid, (I)rc.nblk);
  else if (d.vec >= 2 && aligned) reshape_words<I, 2>(d, (I)rc.bid, (I)rc.nblk);
  else reshape_words<I, 1>(d, (I)rc.bid, (I)rc.nblk);
}

// Transpose of a 32 x 32 bit block in a thread's registers: x[i] is row i,
// afterwards column i.  Recursive block swap: for block size s the rows k and
// k + s (k & s == 0) exchange the columns c + s of row k with the columns c of
// row k + s (c & s == 0); whole bytes by permutes, the rest by a shift and a
// select each: 256 instructions for 32 blocks of a warp.
__device__ __forceinline__ void transpose32(uint32_t (&x)[32]) {
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const uint32_t a = x[k], b = x[k + 16];
    x[k] = __byte_perm(a, b, 0x5410);
    x[k + 16] = __byte_perm(a, b, 0x7632);
  }
#pragma unroll
  for (int k = 0; k < 32; ++k)
    if (!(k & 8)) {
      const uint32_t a = x[k], b = x[k + 8];
      x[k] = __byte_perm(a, b, 0x6240);
      x[k + 8] = __byte_perm(a, b, 0x7351);
    }
#pragma unroll
  for (int s = 4; s >= 1; s >>= 1) {
    const uint32_t m = s == 4 ? 0x0F0F0F0Fu : s == 2 ? 0x33333333u : 0x55555555u;
#pragma unroll
    for (int k = 0; k < 32; ++k)
      if (!(k & s)) {
        const uint32_t a = x[k], b = x[k + s];
        x[k] = (a & m) | ((b << s) & ~m);
        x[k + s] = ((a >> s) & m) | (b & ~m);
      }
  }
}

// Transpose mode.  A CTA tile is 64 TW values of L (TW output words) x 64 TW
// values of J (TW input words) at one value of the other axes.  A thread takes a
// 32 x 32 block: its 32 rows come straight from the input (a tile row is read by
// 2 TW neighbouring lanes), are transposed in its registers and go to a shared
// tile, from which the output rows are stored whole.  TW = 4 (256 x 256), or 8
// where both axes have more than 256 values: rows of 512 bits are then read and
// written whole instead of in 32-byte halves.  The shared tile is skewed by 16 / TW
// words per 32 rows, which makes the block stores (32 rows apart) and the row
// loads free of conflicts.  Index type I is 32-bit when every word and tile index
// fits.  Bound by short accesses at the arrays' pitches.  With 32 x 32 blocks
// transposed across a warp's lanes (five shuffles each) between two shared tiles,
// L1 and shared memory were 77-82 % busy (ncu); 38 networks' whole replay 5.60 ->
// 5.21 ms.
template <class I, int TW>
__global__ void __launch_bounds__(4 * TW * TW)
reshape_transpose_kernel(const ReshapeDesc* __restrict__ descs, const int64_t* __restrict__ cta0, int n) {
  constexpr int kThreads = 4 * TW * TW, kSkew = 16 / TW;
  __shared__ __align__(16) uint32_t tile32[64 * TW * 2 * TW + 2 * TW * kSkew];
  __shared__ ReshapeDesc sd;
  const RsCtx rc = rs_pick(descs, cta0, n, &sd);
  const ReshapeDesc& d = sd;
  const int tid = threadIdx.x;
  const int c = tid % (2 * TW), br = tid / (2 * TW);  // 32 columns of J, 32 rows of L
  const I tQ = (I)d.tQ, tR = (I)d.tR, t_in_L = (I)d.t_in_L, t_out_J = (I)d.t_out_J;
  const I nJT = (tQ + 64 * TW - 1) / (64 * TW), nLT = (tR + 64 * TW - 1) / (64 * TW);
  const I tiles = (I)d.n_other * nJT * nLT;
  const I nblk = (I)rc.nblk;
  for (I tile = (I)rc.bid; tile < tiles; tile += nblk) {
    // (L tile, J tile, first input and output word of the other axes)
    const I r = tile / nLT;
    const I lt = tile - r * nLT;
    I rest = r / nJT;
    const I jt = r - rest * nJT;
    I base_in = 0, base_out = 0;
    for (int a = d.nu - 1; a >= 0; --a) {
      const I res = (I)d.u_res[a], q = rest / res, v = rest - q * res;
      rest = q;
      base_in += v * (I)d.u_in[a];
      base_out += v * (I)d.u_out[a];
    }
    const I jb = jt * TW + c / 2, L0 = lt * (64 * TW) + br * 32;
    const bool in = jb * 64 < tQ;
    uint32_t x[32];
#pragma unroll
    for (int i = 0; i < 32; ++i)
      x[i] = in && L0 + i < tR
                 ? __ldg(reinterpret_cast<const uint32_t*>(d.in + (base_in + (L0 + i) * t_in_L + jb)) + (c & 1))
                 : 0u;
    transpose32(x);
    uint32_t* st = tile32 + c * (32 * 2 * TW + kSkew) + br;
#pragma unroll
    for (int i = 0; i < 32; ++i) st[i * (2 * TW)] = x[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int idx = tid + kThreads * i, t = idx / TW, w = idx % TW;
      const I J = jt * (64 * TW) + t, lw = lt * TW + w;
      if (J < tQ && lw * 64 < tR)
        d.out[base_out + J * t_out_J + lw] =
            *reinterpret_cast<const uint64_t*>(tile32 + t * (2 * TW) + (t / 32) * kSkew + 2 * w);
    }
    __syncthreads();
  }
}

// In-register transpose of 32 x 32 bit blocks held by one warp: lane l holds row
// l; afterwards column l.  Recursive block swap: for block size s the rows r and
// r + s (r & s == 0) exchange the columns c + s of row r with the columns c of
// row r + s (c & s == 0).  Each step is one shuffle, one rotation and one select:
// a lane keeps the columns of `keep` and takes the others from its partner's
// row, rotated by s (rows without s) or back (rows with s); no kept column wraps.
struct Transpose32 {
  uint32_t keep[5];
  uint32_t rot[5];
  __device__ __forceinline__ explicit Transpose32(int lane) {
    const uint32_t masks[5] = {0x0000FFFFu, 0x00FF00FFu, 0x0F0F0F0Fu, 0x33333333u, 0x55555555u};
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const int s = 16 >> i;
      keep[i] = (lane & s) ? ~masks[i] : masks[i];
      rot[i] = (lane & s) ? 32 - s : s;
    }
  }
  __device__ __forceinline__ uint32_t operator()(uint32_t x) const {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const uint32_t y = __shfl_xor_sync(0xffffffffu, x, 16 >> i);
      x = (x & keep[i]) | (__funnelshift_l(y, y, rot[i]) & ~keep[i]);
    }
    return x;
  }
};

// Transposes of few 256 x 256 tiles: a tile's 32 x 32 blocks go to warps, a lane
// per row, so that 256 threads share a tile's loads and stores and no thread has
// a chain of 32 rows of its own.
__global__ void __launch_bounds__(256)
reshape_transpose_few_kernel(const ReshapeDesc* __restrict__ descs, const int64_t* __restrict__ cta0, int n) {
  using I = uint32_t;
  constexpr int TW = 4, kThreads = 64 * TW, kPad = TW + 1;  // a thread per value of an axis
  __shared__ uint64_t s_in[64 * TW * kPad], s_out[64 * TW * kPad];
  __shared__ ReshapeDesc sd;
  const RsCtx rc = rs_pick(descs, cta0, n, &sd);
  const ReshapeDesc& d = sd;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const Transpose32 tr(lane);
  const I tQ = (I)d.tQ, tR = (I)d.tR, t_in_L = (I)d.t_in_L, t_out_J = (I)d.t_out_J;
  const I nJT = (tQ + 64 * TW - 1) / (64 * TW), nLT = (tR + 64 * TW - 1) / (64 * TW);
  const I tiles = (I)d.n_other * nJT * nLT;
  const I nblk = (I)rc.nblk;
  // tile -> (L tile, J tile, first input and output word of its other axes)
  auto locate = [&](I tile, I& lt, I& jt, I& base_in, I& base_out) {
    const I r = tile / nLT;
    lt = tile - r * nLT;
    I rest = r / nJT;
    jt = r - rest * nJT;
    base_in = 0;
    base_out = 0;
    for (int a = d.nu - 1; a >= 0; --a) {
      const I res = (I)d.u_res[a], q = rest / res, v = rest - q * res;
      rest = q;
      base_in += v * (I)d.u_in[a];
      base_out += v * (I)d.u_out[a];
    }
  };
  // the TW input words this thread loads for a tile
  auto load = [&](I lt, I jt, I base_in, uint64_t* v) {
#pragma unroll
    for (int i = 0; i < TW; ++i) {
      const int idx = tid + kThreads * i, b = idx / TW, c = idx % TW;
      const I L = lt * (64 * TW) + b, jb = jt * TW + c;
      v[i] = (L < tR && jb * 64 < tQ) ? d.in[base_in + L * t_in_L + jb] : 0ull;
    }
  };
  // the next tile's loads are issued before the current tile is transposed
  // and stored, so that their latency overlaps that work
  I lt = 0, jt = 0, base_in = 0, base_out = 0;
  uint64_t nv[TW];
  if ((I)rc.bid < tiles) {
    locate((I)rc.bid, lt, jt, base_in, base_out);
    load(lt, jt, base_in, nv);
  }
  for (I tile = (I)rc.bid; tile < tiles; tile += nblk) {
#pragma unroll
    for (int i = 0; i < TW; ++i) {
      const int idx = tid + kThreads * i;
      s_in[idx / TW * kPad + idx % TW] = nv[i];
    }
    const I clt = lt, cjt = jt, cbase_out = base_out;
    if (tile + nblk < tiles) {
      locate(tile + nblk, lt, jt, base_in, base_out);
      load(lt, jt, base_in, nv);
    }
    __syncthreads();
    // warp w: the 32 columns w of J, all 32-row blocks of L
    if ((cjt * (2 * TW) + warp) * 32 < tQ) {
      const uint32_t* in32 = reinterpret_cast<const uint32_t*>(s_in) + lane * (2 * kPad) + warp;
      uint32_t* out32 = reinterpret_cast<uint32_t*>(s_out) + (warp * 32 + lane) * (2 * kPad);
#pragma unroll
      for (int i = 0; i < 2 * TW; ++i) out32[i] = tr(in32[i * 32 * (2 * kPad)]);
    }
    __syncthreads();
#pragma unroll
    for (int i = 0; i < TW; ++i) {
      const int idx = tid + kThreads * i, t = idx / TW, w = idx % TW;
      const I J = cjt * (64 * TW) + t, lw = clt * TW + w;
      if (J < tQ && lw * 64 < tR) d.out[cbase_out + J * t_out_J + lw] = s_out[t * kPad + w];
    }
    __syncthreads();
  }
}

// Up to two tiles per SM the launch lasts as long as one tile does; more tiles are
// bound by L1 and shared memory, where a block per thread is the cheaper way.  Whole
// solves with the line at 0 / 304 / 608 / 2432 tiles, us: 3-D arrays at 88 px 63.3 /
// 62.5 / 62.6 / 62.5, at 100 px 81.1 / 80.5 / 80.4 / 80.2; random networks, 2 of them
// 308 / 300 / 299 / 299, 3: 836 / 826 / 826 / 826, 5: 700 / 698 / 698 / 712, 16: 2466 /
// 2465 / 2463 / 2508, 38: 5220 / 5215 / 5216 / 5256.
constexpr int64_t kFewTiles = 304;

constexpr int64_t kMaxReshapeBlocks = 152 * 16;

// A transpose's tiles of 64 tw x 64 tw values.
int64_t transpose_tiles(const ReshapeDesc& d, int tw) {
  const int64_t side = 64 * tw;
  return d.n_other * ((d.tQ + side - 1) / side) * ((d.tR + side - 1) / side);
}

int reshape_kind(const ReshapeDesc& d) {
  if (d.mode == kReshapeBits) return kRsBits;
  const int64_t total = d.out_nrows * d.out_row_words, blocks = kMaxReshapeBlocks;
  int64_t in_max = 0;  // largest input word index + 1 (bounded by the sums below)
  for (int a = 0; a < d.nu; ++a) in_max += (d.u_res[a] - 1) * d.u_in[a];
  if (d.mode == kReshapeTranspose) {
    in_max += (d.tR + 511) * d.t_in_L + d.tQ / 64 + 8;
    const bool fits = in_max < (1ll << 31) && total < (1ll << 31) &&
                      transpose_tiles(d, 4) + blocks < (1ll << 31);
    return !fits ? kRsTranspose64 : d.tQ > 256 && d.tR > 256 ? kRsTranspose32Wide : kRsTranspose32;
  }
  for (int q = 0; q < d.nred; ++q) in_max += (d.red_res[q] - 1) * d.red_in_w[q];
  return (total + 1024 * blocks < (1ll << 31) && in_max < (1ll << 31)) ? kRsWords32 : kRsWords64;
}

int64_t reshape_units(const ReshapeDesc& d) {
  const int64_t total = d.out_nrows * d.out_row_words;
  if (total <= 0) return 0;
  if (d.mode == kReshapeTranspose) return transpose_tiles(d, reshape_kind(d) == kRsTranspose32Wide ? 8 : 4);
  if (d.mode == kReshapeWords) {
    // a thread per run of words, or more for a reduction (see the kernel)
    int64_t red = 1;
    for (int q = 0; q < d.nred; ++q) red *= d.red_res[q];
    const int64_t threads = total / d.vec * std::min<int64_t>(32, red);
    return (threads + 255) / 256;
  }
  if (d.row_any && any_scan(d) >= kAnyScan) return total;
  return (total + 7) / 8;  // one warp per word
}

int64_t reshape_blocks(const ReshapeDesc& d, int64_t per) {
  const int64_t n = reshape_units(d);
  return n <= 0 ? 0 : std::min<int64_t>((n + per - 1) / per, kMaxReshapeBlocks);
}

void launch_reshape(const ReshapeDesc* d_descs, const int64_t* d_cta0, int n, int kind,
                    int64_t grid, cudaStream_t s) {
  if (n <= 0 || grid <= 0) return;
  switch (kind) {
    case kRsTranspose32:
      if (grid <= kFewTiles) {
        reshape_transpose_few_kernel<<<(unsigned)grid, 256, 0, s>>>(d_descs, d_cta0, n);
        break;
      }
      reshape_transpose_kernel<uint32_t, 4>
          <<<(unsigned)grid, 64, 0, s>>>(d_descs, d_cta0, n);
      break;
    case kRsTranspose32Wide:
      reshape_transpose_kernel<uint32_t, 8>
          <<<(unsigned)grid, 256, 0, s>>>(d_descs, d_cta0, n);
      break;
    case kRsTranspose64:
      reshape_transpose_kernel<uint64_t, 4>
          <<<(unsigned)grid, 64, 0, s>>>(d_descs, d_cta0, n);
      break;
    case kRsWords32:
      reshape_words_kernel<uint32_t><<<(unsigned)grid, 256, 0, s>>>(d_descs, d_cta0, n);
      break;
    case kRsWords64:
      reshape_words_kernel<uint64_t><<<(unsigned)grid, 256, 0, s>>>(d_descs, d_cta0, n);
      break;
    default:
      reshape_kernel<<<(unsigned)grid, 256, 0, s>>>(d_descs, d_cta0, n);
      break;
  }
}

// Long dot rows (more than 16 words) are split into runs of this many words.
constexpr int64_t kDotRun = 256;

// ------------------------------------------- outer / dot / and, batched
// Every such cluster of one tree level in one launch: job p owns blocks
// [cta0[p], cta0[p+1]) and runs the loop of its kind over them.
// Index type I is 32-bit when every word and row index of the launch's jobs
// fits (a 64-bit division is 100 instructions, and an outer product's element
// takes two: 38 networks 0.73 -> 0.54 ms).
template <class I>
__global__ void __launch_bounds__(256)
ewise_kernel(const EwJob* __restrict__ jobs, const int64_t* __restrict__ cta0, int n) {
  const int lo = find_entry([&](int k) { return cta0[k]; }, n, (int64_t)blockIdx.x);
  const EwJob& j = jobs[lo];
  const I bid = (I)((int64_t)blockIdx.x - cta0[lo]), nblk = (I)(cta0[lo + 1] - cta0[lo]);
  const int lane = threadIdx.x & 31;
  const I gwarp = bid * (blockDim.x >> 5) + (threadIdx.x >> 5), nwarps = nblk * (blockDim.x >> 5);
  const I rows = (I)j.rows, m = (I)j.m, nw = (I)j.nw;
  const uint64_t* __restrict__ A = j.a;
  const uint64_t* __restrict__ B = j.b;
  uint64_t* __restrict__ C = j.c;
  const int kind = j.kind;
  if (kind == kEwAnd) {
    // two words at a time, four loads in flight, where the arrays allow it
    const bool vec = ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B) |
                       reinterpret_cast<uintptr_t>(C)) & 15) == 0;
    const I pairs = vec ? rows / 2 : 0;
    const ulonglong2* A2 = reinterpret_cast<const ulonglong2*>(A);
    const ulonglong2* B2 = reinterpret_cast<const ulonglong2*>(B);
    ulonglong2* C2 = reinterpret_cast<ulonglong2*>(C);
    const I step = nblk * blockDim.x;
    for (I i = bid * blockDim.x + threadIdx.x; i < pairs; i += step) {
      const ulonglong2 a = A2[i], b = B2[i];
      C2[i] = make_ulonglong2(a.x & b.x, a.y & b.y);
    }
    for (I i = 2 * pairs + bid * blockDim.x + threadIdx.x; i < rows; i += step) C[i] = A[i] & B[i];
  } else if (kind == kEwOuter) {
    // C[r][w] = bit r of A ? B[r / M][w] : 0
    const I total = rows * nw;
    for (I i = bid * blockDim.x + threadIdx.x; i < total; i += nblk * blockDim.x) {
      const I r = i / nw, w = i - r * nw;
      const uint64_t bit = (A[r >> 6] >> (r & 63)) & 1ull;
      C[i] = bit ? B[(r / m) * nw + w] : 0ull;
    }
  } else if (kind == kEwDot) {
    // one warp per word of C: lanes take bits r and r + 32
    const I words = (rows + 63) / 64;
    for (I cw = gwarp; cw < words; cw += nwarps) {
      uint32_t half[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const I r = cw * 64 + h * 32 + lane;
        uint64_t acc = 0;
        if (r < rows) {
          const uint64_t* a = A + r * nw;
          const uint64_t* b = B + (r / m) * nw;
          // (four words at a time: the loads of a run are in flight together)
          for (I w = 0; w < nw && !acc; w += 4) {
#pragma unroll
            for (int k = 0; k < 4; ++k)
              if (w + k < nw) acc |= a[w + k] & b[w + k];
          }
        }
        half[h] = __ballot_sync(0xffffffffu, acc != 0);
      }
      if (lane == 0) C[cw] = (uint64_t)half[0] | ((uint64_t)half[1] << 32);
    }
  } else {
    // long rows: one warp per (row, run of 256 words) into the cleared C
    const I nruns = (nw + (I)kDotRun - 1) / (I)kDotRun;
    const I items = rows * nruns;
    for (I it = gwarp; it < items; it += nwarps) {
      const I r = it / nruns, w0 = (it - r * nruns) * (I)kDotRun;
      const I w1 = min(nw, w0 + (I)kDotRun);
      const uint64_t* a = A + r * nw;
      const uint64_t* b = B + (r / m) * nw;
      uint64_t acc = 0;
      for (I w = w0 + lane; w < w1; w += 32) acc |= a[w] & b[w];
      if (__any_sync(0xffffffffu, acc != 0) && lane == 0)
        atomicOr(reinterpret_cast<unsigned long long*>(&C[r >> 6]), 1ull << (r & 63));
    }
  }
}

int64_t ewise_blocks(const EwJob& j) {
  int64_t items;
  switch (j.kind) {
    case kEwAnd: items = (j.rows / 2 + 255) / 256 + 1; break;
    case kEwOuter: items = (j.rows * j.nw + 255) / 256; break;
    case kEwDot: items = ((j.rows + 63) / 64 + 7) / 8; break;
    default: items = (j.rows * ((j.nw + kDotRun - 1) / kDotRun) + 7) / 8; break;
  }
  return std::min<int64_t>(items, 152 * 16);
}

bool ewise_fits32(const EwJob& j) {
  // (word indexes of every array, and a grid-stride past the end)
  return j.rows * std::max<int64_t>(1, j.nw) < (1ll << 31) - (1ll << 24) && j.m < (1ll << 31);
}

void launch_ewise(const EwJob* d_jobs, const int64_t* d_cta0, int n, int64_t grid, bool wide,
                  cudaStream_t s) {
  if (n <= 0 || grid <= 0) return;
  if (wide) ewise_kernel<uint64_t><<<(unsigned)grid, 256, 0, s>>>(d_jobs, d_cta0, n);
  else ewise_kernel<uint32_t><<<(unsigned)grid, 256, 0, s>>>(d_jobs, d_cta0, n);
}

// ---------------------------------------------------------------- row-OR
// One CTA owns the tile B[b][k0 .. k0+Kc)[n0 .. n0+G) in shared memory, staged
// by bulk copies when the tile is one run of memory, by 2-D boxes of 64 rows x
// G words (tensor map) when the row pitch allows it, else by 8-byte
// asynchronous copies.  Next to it the CTA
// builds the ORs of aligned blocks of 4, 16 and 64 tile rows (tables T2, T4,
// T6; T0 is the tile itself), plus an all-zero sentinel row.  A run of set bits
// in a row of A selects a run of B rows, whose OR is the OR of the maximal
// aligned blocks covering it: the plotted relations are thick curves, so most
// set bits lie in long runs and a row needs a few block lookups instead of one
// per bit.  Each warp takes a batch of R consecutive output rows at a time, a
// group of L lanes per row for its K range's L A words (L <= 32, R = 32 / L):
//   1. the lanes load one A word each and split it into maximal all-ones
//      aligned blocks of 64, 16, 4 and 1 bits (a few bit operations);
//   2. a prefix sum over the lanes gives every block its slot in the warp's
//      list in shared memory, the rows' entries one after another;
//   3. the warp splits into groups of G/2 lanes (two words each: one 16-byte
//      load per lookup); a group ORs a row's table rows, three loads in flight
//      per lane.  With more groups than rows a row's list is dealt over several
//      groups and their words are OR-ed together with shuffles.
// A batch whose blocks exceed the list goes row by row through it in windows.
// What bounds it: instruction issue (2 to 2.6 per clock and SM in the rows).  A
// row by itself costs about 200 warp instructions whatever its length, most of
// it on lanes without an A word; in batches a row of 8 or 9 words costs 50 to
// 70.  Against one row per warp, one launch per tile width and 1024-thread CTAs
// throughout (ncu, cold): 4096 chains 2.92 -> 0.78 ms, 38 networks 3.89 -> 1.02
// ms, two 4001^3 joins 41 -> 24 us, four 2048^3 joins 20 -> 16 us.
namespace {

constexpr int kRowOrThreads = 1024;  // at most; see rowor_plan
constexpr int kRowOrMaxKc = 2048;    // K range of a CTA: one A word per lane
// Entries of a warp's list per window, plus sentinel padding.
constexpr int kListWin = 256;
constexpr int kListCap = kListWin + 4 * 32;  // (a window is padded to 4 entries per group)

// Tile rows of the tables for a K range staged in `staged` rows: T0 (rounded
// up to whole 64-row groups), the sentinel, T2, T4 and T6.
__host__ __device__ __forceinline__ int64_t rowor_r64(int64_t staged) { return (staged + 63) / 64 * 64; }
__host__ __device__ __forceinline__ int64_t rowor_table_rows(int64_t staged) {
  const int64_t r64 = rowor_r64(staged);
  return r64 + 1 + r64 / 4 + r64 / 16 + r64 / 64;
}

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Wait for phase `parity` of an mbarrier, giving up after about `limit_ns`.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity, long long limit_ns) {
  const long long t0 = clock64();
  const long long limit_cycles = limit_ns * 2;  // >= 1 cycle per ns at <= 2.1 GHz
  for (long long it = 0; it < (1ll << 26); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_u32(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > limit_cycles) return false;
  }
  return false;
}

// The words a lane holds of an output row: two adjacent ones (one 16-byte
// shared-memory load per lookup) except on one-word rows.
template <int W>
struct Words {
  uint64_t v[W];
};
__device__ __forceinline__ void or_row(Words<1>& w, const uint64_t* p) { w.v[0] |= *p; }
__device__ __forceinline__ void or_row(Words<2>& w, const uint64_t* p) {
  const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(p);
  w.v[0] |= t.x;
  w.v[1] |= t.y;
}

// The output rows of one CTA: its tile's tables are in bs (G words per row).
template <int G>
__device__ __forceinline__ void rowor_rows(const RowOrDesc& d, const uint64_t* __restrict__ bs,
                                           uint16_t* list, int64_t b, int64_t k0, int kc_len,
                                           int64_t n0, int rs, int r64) {
  constexpr int W = G >= 2 ? 2 : 1, GL = G / W;  // words per lane, lanes per row
  constexpr int P = 32 / GL;                     // lookup groups per warp
  const int nwarps = blockDim.x >> 5, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sent = r64, t2 = r64 + 1, t4 = t2 + r64 / 4, t6 = t4 + r64 / 16;
  const int grp = lane / GL, lig = lane % GL;
  const uint64_t* mine = bs + W * lig;
  // lanes per row and rows per batch
  const int kw0 = (int)(k0 / 64);
  const int kw1 = (int)min(d.a_row_words, (k0 + kc_len + 63) / 64);
  const int kw = kw1 - kw0;
  // (no more rows per batch than leave every warp a batch: with few rows the
  // batches would run on a few of the warps, one after another)
  const int L = kw;  // at most 32: a K range is at most kRowOrMaxKc
  const int all_warps = (int)d.row_splits * nwarps;
  const RowWalk walk(d.M, all_warps, L);
  const int R = (int)walk.batch;
  // groups per row (gpr, a power of two) of a lookup round, rows per round and
  // rounds
  int gpr = 1;
  while (2 * gpr * R <= P) gpr *= 2;
  const int rpr = P / gpr, rounds = (R + rpr - 1) / rpr;
  const int sub = grp % gpr, rin = grp / gpr;
  // batches of rows are dealt out cyclically over every warp of the CTAs
  // sharing this tile, so that runs of dense rows (curves are locally thick)
  // are spread out.  The A words of the next three batches are always in
  // flight while one is processed.
  const int gw = rs * nwarps + warp;
  const uint32_t rstep = walk.step, M = walk.M;
  const int64_t arw = d.a_row_words;
  const int my_row = lane / L, my_word = lane - my_row * L;
  const bool busy = my_row < R;  // lanes past the last whole row are idle
  const int64_t Nw = d.Nw;
  uint64_t* const cbase = d.C + b * d.M * Nw + n0 + W * lig;
  const int cols = (int)min((int64_t)W, max((int64_t)0, Nw - n0 - W * lig));  // of this lane's words
  const bool vec = W == 2 && Nw % 2 == 0 && reinterpret_cast<uintptr_t>(d.C) % 16 == 0;
  const bool atomic = d.atomic != 0;
  auto store = [&](uint32_t row, const Words<W>& w) {
    uint64_t* c = cbase + (int64_t)row * Nw;
    if (atomic) {
#pragma unroll
      for (int k = 0; k < W; ++k)
        if (k < cols && w.v[k]) atomicOr((unsigned long long*)(c + k), (unsigned long long)w.v[k]);
    } else if (W == 2 && vec) {
      if (cols > 0) *reinterpret_cast<ulonglong2*>(c) = make_ulonglong2(w.v[0], w.v[W - 1]);
    } else {
#pragma unroll
      for (int k = 0; k < W; ++k)
        if (k < cols) c[k] = w.v[k];
    }
  };
  // OR over the groups that share a row (lane distances GL .. to)
  auto combine = [&](Words<W>& w, int to) {
    for (int o = GL; o < to; o <<= 1)
#pragma unroll
      for (int k = 0; k < W; ++k) w.v[k] |= __shfl_xor_sync(0xffffffffu, w.v[k], o);
  };
  const uint64_t* __restrict__ abase = d.A + (b * d.M) * arw + kw0 + my_word;
  uint32_t lrow = (uint32_t)(gw * R + my_row);  // row of the next batch to fetch
  auto fetch = [&]() -> uint64_t {
    const uint64_t v = (busy && lrow < M) ? __ldg(abase + (int64_t)lrow * arw) : 0ull;
    lrow += rstep;
    return v;
  };
  uint64_t pre0 = fetch(), pre1 = fetch(), pre2 = fetch();
  Words<W> zero;
#pragma unroll
  for (int k = 0; k < W; ++k) zero.v[k] = 0;
  // tile row of this lane's word's bit 0 (a multiple of 64), and the word's
  // bits inside the K range
  const int base = (kw0 + my_word) * 64 - (int)k0;
  const uint64_t in_range = base + 64 <= kc_len ? ~0ull : base >= kc_len ? 0ull : (1ull << (kc_len - base)) - 1ull;
  for (uint32_t row0 = (uint32_t)(gw * R); row0 < M; row0 += rstep) {
    const int live = (int)min((uint32_t)R, M - row0);  // rows of this batch
    uint64_t a = pre0;
    pre0 = pre1;
    pre1 = pre2;
    pre2 = fetch();
    a &= in_range;
    if (__any_sync(0xffffffffu, a != 0ull)) {
      // maximal all-ones aligned blocks of the word: bit 4i of f4 when bits
      // 4i..4i+3 are set, bit 16i of f16 when bits 16i..16i+15 are set, f1 the
      // set bits in neither; a full word is one 64-block
      const bool full = (a == ~0ull);
      uint64_t f16 = 0, f4 = 0, f1 = 0;
      if (!full) {
        uint64_t t = a & (a >> 1);
        t &= t >> 2;
        f4 = t & 0x1111111111111111ull;
        uint64_t u4 = f4 & (f4 >> 4);
        u4 &= u4 >> 8;
        f16 = u4 & 0x0001000100010001ull;
        const uint64_t m16 = f16 * 0xFFFFull;
        f4 &= ~m16;
        f1 = a & ~(m16 | f4 * 0xFull);
      }
      const int c = full ? 1 : __popcll(f16 | f4 | f1);  // (three disjoint sets of positions)
      int incl = c;
#pragma unroll
      for (int sh = 1; sh < 32; sh <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, incl, sh);
        if (lane >= sh) incl += v;
      }
      const int excl = incl - c;
      const int T = __shfl_sync(0xffffffffu, incl, 31);
      if (d.stat && lane == 0) atomicAdd(d.stat, (unsigned long long)T * G);
      // the table rows of this lane's blocks, in a fixed order
      auto entries = [&](auto&& put) {
        if (full) put(t6 + (base >> 6));
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          for (uint32_t m = (uint32_t)(f16 >> (32 * h)); m;) {
            const int p = 31 - __clz(m);
            m ^= 1u << p;
            put(t4 + ((base + 32 * h + p) >> 4));
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          for (uint32_t m = (uint32_t)(f4 >> (32 * h)); m;) {
            const int p = 31 - __clz(m);
            m ^= 1u << p;
            put(t2 + ((base + 32 * h + p) >> 2));
          }
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          for (uint32_t m = (uint32_t)(f1 >> (32 * h)); m;) {
            const int p = 31 - __clz(m);
            m ^= 1u << p;
            put(base + 32 * h + p);
          }
        }
      };
      if (T <= kListWin) {
        uint16_t* to = list + excl;
        entries([&](int row) { *to++ = (uint16_t)row; });
        __syncwarp();
        for (int rd = 0; rd < rounds; ++rd) {
          const int r = rd * rpr + rin;  // r >= R (the last round's spare groups): no row
          const int o0 = __shfl_sync(0xffffffffu, excl, (r * L) & 31);
          int o1 = __shfl_sync(0xffffffffu, incl, (r * L + L - 1) & 31);
          if (r >= R) o1 = 0;
          Words<W> w = zero;
          for (int e = o0 + sub; e < o1; e += 3 * gpr) {
            const int i0 = list[e];
            const int i1 = e + gpr < o1 ? list[e + gpr] : sent;
            const int i2 = e + 2 * gpr < o1 ? list[e + 2 * gpr] : sent;
            or_row(w, mine + i0 * G);
            or_row(w, mine + i1 * G);
            or_row(w, mine + i2 * G);
          }
          __syncwarp();
          combine(w, GL * gpr);
          if (sub == 0 && r < live) store(row0 + r, w);
        }
      } else {
        // more blocks than the list holds: row by row, in windows of the list;
        // this lane's entries are [excl, incl) of the batch's T
        for (int r = 0; r < R; ++r) {
          const int ro0 = __shfl_sync(0xffffffffu, excl, r * L);
          const int ro1 = __shfl_sync(0xffffffffu, incl, r * L + L - 1);
          Words<W> w = zero;
          for (int w0 = ro0; w0 < ro1; w0 += kListWin) {
            const int w1 = min(ro1, w0 + kListWin);
            if (my_row == r && excl < w1 && incl > w0) {
              int e = excl;
              entries([&](int row) {
                if (e >= w0 && e < w1) list[e - w0] = (uint16_t)row;
                ++e;
              });
            }
            const int n = w1 - w0;
            // pad to a whole number of rounds with the sentinel row (4P entries,
            // which is more than one per lane when the groups are narrow)
            for (int t = lane; t < 4 * P; t += 32) list[n + t] = (uint16_t)sent;
            __syncwarp();
            for (int e = grp; e < n; e += 4 * P) {
              or_row(w, mine + list[e] * G);
              or_row(w, mine + list[e + P] * G);
              or_row(w, mine + list[e + 2 * P] * G);
              or_row(w, mine + list[e + 3 * P] * G);
            }
            __syncwarp();
          }
          combine(w, 32);
          if (grp == 0 && r < live) store(row0 + r, w);
        }
      }
    } else if (!atomic) {
      for (int r = grp; r < live; r += P) store(row0 + r, zero);  // nothing selected: zero rows
    }
  }
}

// Launch description: problem p owns CTAs [cta0[p], cta0[p+1]); its
// descriptor and tensor map (used by kStageTile) live in global memory.  One
// launch serves every tile width (a branch on the problem's width).
__global__ void __launch_bounds__(kRowOrThreads)
rowor_kernel(const RowOrDesc* __restrict__ descs, const CUtensorMap* __restrict__ maps,
             const int64_t* __restrict__ cta0s, int nprob) {
  extern __shared__ __align__(1024) uint64_t bs[];
  __shared__ RowOrDesc sd;
  __shared__ int s_p;
  // the next launch may be scheduled onto SMs this grid frees; it waits for
  // this grid's completion before it touches any data
  asm volatile("griddepcontrol.launch_dependents;");
  const int tid = threadIdx.x;
  {
    const int lo = find_entry([&](int i) { return cta0s[i]; }, nprob, (int64_t)blockIdx.x);
    const uint32_t* src = reinterpret_cast<const uint32_t*>(descs + lo);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&sd);
    if (tid < (int)(sizeof(RowOrDesc) / 4)) dst[tid] = src[tid];
    if (tid == 0) s_p = lo;
  }
  __syncthreads();
  const int p = s_p;
  const RowOrDesc& d = sd;
  const CUtensorMap* tmap = maps + p;
  const int G = d.Nt;
  const int r64 = (int)rowor_r64(d.Kc);
  uint16_t* lists = reinterpret_cast<uint16_t*>(bs + rowor_table_rows(d.Kc) * G);
  uint64_t* bar = reinterpret_cast<uint64_t*>(lists + (size_t)(blockDim.x >> 5) * kListCap);

  int64_t cta = (int64_t)blockIdx.x - cta0s[p];
  const int rs = (int)(cta % d.row_splits);
  cta /= d.row_splits;
  const int64_t kc = cta % d.k_chunks;
  cta /= d.k_chunks;
  const int64_t nt = cta % d.n_tiles;
  const int64_t b = cta / d.n_tiles;
  const int64_t k0 = kc * d.Kc;
  const int kc_len = (int)min((int64_t)d.Kc, d.K - k0);
  const int64_t n0 = nt * G;

  // ---- stage the B tile
  if (d.stage != kStageWords) {
    if (tid == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(1) : "memory");
      asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      // the tensor map was written to global memory by a copy before the launch
      if (d.stage == kStageTile)
        asm volatile("fence.proxy.tensormap::generic.acquire.gpu [%0], 128;" ::"l"(tmap) : "memory");
    }
    // everything the earlier kernels of the stream wrote (A, B) is complete
    // and visible past this point, and C may be overwritten
    asm volatile("griddepcontrol.wait;" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      if (d.stage == kStageTile) {
        const int nbox = (kc_len + 63) / 64;
        const uint32_t bytes = (uint32_t)nbox * 64u * (uint32_t)G * 8u;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                     "r"(bytes)
                     : "memory");
        for (int j = 0; j < nbox; ++j) {
          const int x = (int)n0;
          const int y = (int)(b * d.K + k0 + 64 * j);
          asm volatile(
              "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
              " [%0], [%1, {%2, %3}], [%4];" ::"r"(smem_u32(bs + (size_t)j * 64 * G)),
              "l"(reinterpret_cast<uint64_t>(tmap)), "r"(x), "r"(y), "r"(smem_u32(bar))
              : "memory");
        }
      } else {
        // the tile is one run of memory (G words per row in both)
        const uint32_t bytes = (uint32_t)kc_len * (uint32_t)G * 8u;
        const uint64_t* src = d.B + (b * d.K + k0) * G;
        asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
                     "r"(bytes)
                     : "memory");
        for (uint32_t at = 0; at < bytes; at += 16384u) {
          const uint32_t n = min(bytes - at, 16384u);
          asm volatile(
              "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes"
              " [%0], [%1], %2, [%3];" ::"r"(smem_u32(bs) + at),
              "l"(reinterpret_cast<const char*>(src) + at), "r"(n), "r"(smem_u32(bar))
              : "memory");
        }
      }
    }
    const bool ok = mbar_wait(bar, 0, 1000000000ll);
    if (__syncthreads_or(!ok)) {
      if (tid == 0) atomicExch(d.err, 1);
      return;
    }
  } else {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    // 8-byte asynchronous copies, all in flight at once; words past the row
    // and rows past the K range are filled with zeros
    const int lg = 31 - __clz(G);
    for (int idx = tid; idx < r64 << lg; idx += blockDim.x) {
      const int r = idx >> lg, c = idx & (G - 1);
      const int64_t n = n0 + c;
      const bool in = r < kc_len && n < d.Nw;
      const uint64_t* src = in ? d.B + (b * d.K + k0 + r) * d.Nw + n : d.B;
      asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(smem_u32(bs + idx)),
                   "l"(src), "r"(in ? 8 : 0)
                   : "memory");
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
    asm volatile("cp.async.wait_group 0;" ::: "memory");
  }
  if (tid < G) bs[(size_t)r64 * G + tid] = 0ull;  // sentinel row
  __syncthreads();
  // block tables: a thread per (16-row block, column) ORs its four 4-row
  // blocks and the block itself, then the 64-row blocks follow
  {
    const int lg = 31 - __clz(G);
    uint64_t* T2 = bs + (size_t)(r64 + 1) * G;
    uint64_t* T4 = T2 + (size_t)(r64 / 4) * G;
    uint64_t* T6 = T4 + (size_t)(r64 / 16) * G;
    for (int idx = tid; idx < (r64 / 16) << lg; idx += blockDim.x) {
      const int q = idx >> lg, c = idx & (G - 1);
      const uint64_t* s0 = bs + (size_t)(16 * q) * G + c;
      uint64_t all = 0;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const uint64_t v = s0[(4 * j) * G] | s0[(4 * j + 1) * G] | s0[(4 * j + 2) * G] | s0[(4 * j + 3) * G];
        T2[(size_t)(4 * q + j) * G + c] = v;
        all |= v;
      }
      T4[idx] = all;
    }
    __syncthreads();
    for (int idx = tid; idx < (r64 / 64) << lg; idx += blockDim.x) {
      const int q = idx >> lg, c = idx & (G - 1);
      const uint64_t* s0 = T4 + (size_t)(4 * q) * G + c;
      T6[idx] = s0[0] | s0[G] | s0[2 * G] | s0[3 * G];
    }
    __syncthreads();
  }
  uint16_t* list = lists + (size_t)(tid >> 5) * kListCap;
  switch (G) {
    case 1: rowor_rows<1>(d, bs, list, b, k0, kc_len, n0, rs, r64); break;
    case 2: rowor_rows<2>(d, bs, list, b, k0, kc_len, n0, rs, r64); break;
    case 4: rowor_rows<4>(d, bs, list, b, k0, kc_len, n0, rs, r64); break;
    case 8: rowor_rows<8>(d, bs, list, b, k0, kc_len, n0, rs, r64); break;
    case 16: rowor_rows<16>(d, bs, list, b, k0, kc_len, n0, rs, r64); break;
    default: rowor_rows<32>(d, bs, list, b, k0, kc_len, n0, rs, r64); break;
  }
}

}  // namespace

namespace {

// cuTensorMapEncodeTiled from the driver (null when unavailable)
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn encode_fn() {
  static const EncodeTiledFn fn = [] {  // looked up once, whatever thread comes first
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(p);
    cudaGetLastError();
    return EncodeTiledFn(nullptr);
  }();
  return fn;
}

// Shared memory of one CTA: the tables plus the warps' lists and the mbarrier,
// within the 227 KB a CTA may opt into.
constexpr size_t kSmemLimit = 227 * 1024 - 2048;  // the kernel's static shared memory stays out
constexpr size_t kSmemHalf = 113 * 1024 - 1024;     // two CTAs to an SM
constexpr size_t kSmemQuarter = 56 * 1024 - 1024;   // four
constexpr size_t list_bytes(int threads) { return (size_t)(threads / 32) * kListCap * 2 + 16; }

size_t table_bytes(int64_t staged, int Nt) { return (size_t)rowor_table_rows(staged) * Nt * 8; }

}  // namespace

cudaError_t smem_limit(const void* fn, size_t bytes) {
  static std::mutex mu;
  static std::map<std::pair<const void*, int>, size_t> set;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  std::lock_guard<std::mutex> lock(mu);
  size_t& have = set[{fn, dev}];
  if (bytes <= have) return cudaSuccess;
  e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)bytes);
  if (e == cudaSuccess) have = bytes;
  return e;
}

int64_t rowor_max_kc(int Nt, int threads) {
  const size_t limit = (threads < kRowOrThreads ? kSmemHalf : kSmemLimit) - list_bytes(threads);
  // table_bytes(kc) = ((1 + 1/4 + 1/16 + 1/64) kc + 1) rows of Nt words
  const int64_t kc = (int64_t)(((double)limit / (8.0 * Nt) - 1.0) / 1.328125) / 64 * 64;
  return std::min<int64_t>(kRowOrMaxKc, std::max<int64_t>(64, kc));
}

void rowor_plan(RowOrDesc& d, double share, bool free_clear) {
  // the widest power-of-two tile (<= 32 words, <= the row): a row of A is
  // split into blocks and listed once per tile, so wide tiles cut that work
  // (32-word tiles took the chain's 2048^3 joins from 19.3 to 16.0 us per
  // launch against 8-word tiles over the whole K range).  When the whole K
  // range does not fit next to it, K is split into chunks whose results are
  // OR-ed into C (cleared beforehand).
  int Nt = 1;
  while (Nt < 32 && Nt < d.Nw) Nt <<= 1;
  d.Nt = Nt;
  // A problem with SMs to itself takes a CTA of 1024 threads per SM (64
  // registers a thread: an SM holds 1024), which shorten the set-up
  // (descriptor, copies, tables).  One with more CTAs than its share of SMs
  // takes smaller ones, whose set-up overlaps the rows of the others on the
  // SM: four of 256 threads for the many small tiles of a shared batch axis
  // (38 networks: 1.49 against 1.79 ms with two of 512), two of 512 otherwise
  // (4096 chains: 0.99 against 1.31 ms with four of 256, whose last ones run
  // long).
  const int64_t tiles = d.nbatch * ((d.Nw + Nt - 1) / Nt);
  const int64_t whole_max = rowor_max_kc(Nt, kRowOrThreads);
  d.threads = (double)(tiles * ((d.K + whole_max - 1) / whole_max)) <= share              ? kRowOrThreads
              : d.nbatch >= 8 && table_bytes(d.K, Nt) + list_bytes(256) <= kSmemQuarter ? 256
                                                                                      : 512;
  // K in chunks of equal length; many chunks take a power of two of rows, so
  // that whole batches of rows fill the lanes.  A problem with SMs left over
  // takes more chunks (down to 512 rows of K), each staging its own part of B
  // only, before its rows are split over CTAs that all stage the same one; but a
  // second chunk has C cleared first, which as a launch of its own costs more than
  // it gains (6611 x 653 x 911, a call among others 39.0 -> 43.1 us).
  int64_t kmax = rowor_max_kc(Nt, d.threads);
  if (d.K >= 4 * kmax)
    while (kmax & (kmax - 1)) kmax &= kmax - 1;
  int64_t chunks = (d.K + kmax - 1) / kmax;
  if (d.threads == kRowOrThreads && (free_clear || chunks > 1))
    chunks = std::max(chunks, std::min<int64_t>((int64_t)(share / (double)tiles), (d.K + 511) / 512));
  d.Kc = chunks <= 1 ? (int32_t)d.K : (int32_t)(((d.K + chunks - 1) / chunks + 63) / 64 * 64);
  // How the tile is staged.  A tile as wide as the rows is one run of memory
  // (bulk copies; narrow 2-D boxes move one 8- or 16-byte row per request);
  // other tiles are 2-D boxes, or 8-byte copies where the row pitch is not a
  // multiple of 16 bytes.
  const bool aligned = reinterpret_cast<uintptr_t>(d.B) % 16 == 0;
  if (d.Nw == Nt && aligned && (d.Nw % 2 == 0 || d.K % 2 == 0))
    d.stage = kStageRun;  // (every chunk starts and ends on 16 bytes: Kc is even or all of K)
  else if (Nt % 2 == 0 && d.Nw % 2 == 0 && aligned && d.nbatch * d.K < (1ll << 31) &&
           encode_fn() != nullptr)
    d.stage = kStageTile;
  else
    d.stage = kStageWords;
  d.n_tiles = (d.Nw + Nt - 1) / Nt;
  d.k_chunks = (d.K + d.Kc - 1) / d.Kc;
  d.atomic = d.k_chunks > 1 ? 1 : 0;
  const int64_t base = d.nbatch * d.n_tiles * d.k_chunks;
  // small CTAs: about twice as many as the problem's share of the slots, so
  // that the last ones to finish are short; at least 64 rows each
  const bool whole = d.threads == kRowOrThreads;
  const int64_t target = whole ? (int64_t)share : (int64_t)(2.0 * share * (kRowOrThreads / d.threads) + 0.5);
  // round down: a launch of more CTAs than fit at once would run a short
  // second wave and nearly double its time
  int64_t splits = target / base;
  const int64_t min_rows = whole ? 16 : 64;
  splits = std::max<int64_t>(1, std::min<int64_t>(splits, (d.M + min_rows - 1) / min_rows));
  d.rows_per_split = (d.M + splits - 1) / splits;
  d.row_splits = (d.M + d.rows_per_split - 1) / d.rows_per_split;
}

size_t rowor_smem_bytes(const RowOrDesc& d) { return table_bytes(d.Kc, d.Nt) + list_bytes(d.threads); }

int64_t rowor_ctas(const RowOrDesc& d) { return d.nbatch * d.n_tiles * d.k_chunks * d.row_splits; }

cudaError_t rowor_encode_map(const RowOrDesc& d, CUtensorMap* map) {
  memset(map, 0, sizeof *map);
  if (d.stage != kStageTile) return cudaSuccess;
  const cuuint64_t dims[2] = {(cuuint64_t)d.Nw, (cuuint64_t)(d.nbatch * d.K)};
  const cuuint64_t strides[1] = {(cuuint64_t)d.Nw * 8};
  const cuuint32_t box[2] = {(cuuint32_t)d.Nt, 64u};
  const cuuint32_t estr[2] = {1u, 1u};
  CUresult r = encode_fn()(map, CU_TENSOR_MAP_DATA_TYPE_UINT64, 2, const_cast<uint64_t*>(d.B), dims,
                           strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                           CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? cudaSuccess : cudaErrorInvalidValue;
}

// Failure-path check of the bounded waits: one thread waits on an mbarrier
// that nothing arrives at, gives up after limit_ns as every wait of the
// contraction kernels does, and sets the error word.
__global__ void wait_selftest_kernel(int* err, long long limit_ns) {
  __shared__ uint64_t bar;
  if (threadIdx.x != 0) return;
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(&bar)), "r"(1) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (!mbar_wait(&bar, 0, limit_ns)) atomicExch(err, 1);
}

cudaError_t launch_wait_selftest(int* err, long long limit_ns, cudaStream_t s) {
  wait_selftest_kernel<<<1, 32, 0, s>>>(err, limit_ns);
  return cudaGetLastError();
}

cudaError_t launch_rowor(const RowOrDesc* d_descs, const CUtensorMap* d_maps,
                         const int64_t* d_cta0, int nprob, int64_t grid, size_t smem, int threads,
                         cudaStream_t s) {
  if (nprob <= 0 || grid <= 0) return cudaSuccess;
  if (grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  // programmatic dependent launch: CTAs may start on SMs the previous kernel
  // has left and set up while it finishes (the kernel waits before any data)
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  smem_limit(reinterpret_cast<const void*>(rowor_kernel), smem);
  cudaLaunchKernelEx(&cfg, rowor_kernel, d_descs, d_maps, d_cta0, nprob);
  return cudaGetLastError();
}

// -------------------------------------------------------------- popcount
__global__ void popcount_kernel(const uint64_t* __restrict__ w, int64_t n,
                                unsigned long long* __restrict__ out) {
  unsigned long long c = 0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    c += (unsigned long long)__popcll(w[i]);
  for (int o = 16; o > 0; o >>= 1) c += __shfl_xor_sync(0xffffffffu, c, o);
  if ((threadIdx.x & 31) == 0 && c) atomicAdd(out, c);
}

void launch_popcount(const uint64_t* w, int64_t nwords, unsigned long long* out, cudaStream_t s) {
  if (nwords <= 0) return;
  int64_t blocks = (nwords + 255) / 256;
  if (blocks > 152 * 4) blocks = 152 * 4;
  popcount_kernel<<<(unsigned)blocks, 256, 0, s>>>(w, nwords, out);
}


}  // namespace pa
