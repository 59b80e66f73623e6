// A small fully connected network (FP32) that predicts the time of a join
// from its shape and operand densities: the learned cost model behind the
// PA_ORDER_LEARNED join order.  Forward, backward and Adam kernels are plain
// CUDA; all reductions are deterministic (no atomics), so a gradient computed
// twice is the same bit for bit.
//
// Layout of the parameters (one flat FP32 vector): for every layer l, the
// weights W_l[out][in] row-major, then the biases b_l[out].  Hidden layers use
// ReLU, the output layer is linear with one output.
//
// Every sum has one order, whatever the batch and the launch: a unit's sum starts
// with its bias and adds its inputs in their order, a delta adds the units above
// in theirs, a weight's gradient the samples in theirs (fused multiply-adds).  A
// sum that ends within its rounding of zero decides a unit's ReLU mask, and with
// it whole contributions to the gradients, so the order is part of the result.
//
// A pass is bound by latency (a 256-sample minibatch is 70 MFLOP), so it takes
// few launches and every launch keeps its chain short: one block carries a few
// samples through every layer and back with the activations in shared memory,
// each layer's weights fetched while the one before is summed (mlp_pass), and one
// launch forms every layer's weight gradients (mlp_grads).  3 x 128 units,
// prediction, loss and gradients with both read-backs: 256 samples 1520 -> 91 us,
// 4210 samples 3.75 ms -> 216 us, against a launch per layer whose threads each
// walked a weight row (the same sums, bit for bit).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "mlp.h"
#include "pa_internal.h"

namespace pa {

namespace {

constexpr int kPassThreads = 256;
constexpr int kMaxLayers = 10;     // at most 8 hidden layers, the output layer
constexpr int kWTile = 128;        // outputs and inputs of a weight tile
constexpr int kWPitch = kWTile + 4;  // (16-byte reads down a column of rows: no bank conflicts)

// Sizes and offsets of the network, and the buffers of a training pass (sample
// major): act[l] the output of layer l - 1 (l >= 1), delta[l] the loss's
// derivative with respect to layer l's sums.
struct Net {
  int L;                           // layers
  int size[kMaxLayers + 1];
  int64_t woff[kMaxLayers], boff[kMaxLayers];
  float* act[kMaxLayers + 1];
  float* delta[kMaxLayers];
};

// A 128 x 128 tile of one layer's weights, by asynchronous copies.
__device__ __forceinline__ void stage_weights(const Net& net, const float* __restrict__ p, int l, int o0,
                                              int i0, float* buf) {
  const int ni = net.size[l], rows = min(kWTile, net.size[l + 1] - o0), cols = min(kWTile, ni - i0);
  const float* __restrict__ W = p + net.woff[l] + (size_t)o0 * ni + i0;
  const int lane = threadIdx.x & 31;
  const bool vec = ni % 4 == 0 && net.woff[l] % 4 == 0;
  for (int r = threadIdx.x >> 5; r < rows; r += kPassThreads / 32) {
    const float* src = W + (size_t)r * ni;
    const uint32_t dst = (uint32_t)__cvta_generic_to_shared(buf + r * kWPitch);
    if (vec) {
      if (4 * lane < cols)
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst + 16u * lane), "l"(src + 4 * lane)
                     : "memory");
    } else {
      for (int c = lane; c < cols; c += 32)
        asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(dst + 4u * c), "l"(src + c) : "memory");
    }
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
}

// S samples per block through every layer; with t, back again, writing the
// activations and deltas that the weight gradients need and the samples' squared
// errors.  The pass walks 128 x 128 weight tiles: forward layer by layer, 128
// outputs at a time along their inputs; backward 128 inputs at a time along the
// outputs above.  A thread owns one output (input) of the tile for S / GROUPS
// samples and adds its terms in order; the next tile's copies run meanwhile.
template <int S>
__global__ void __launch_bounds__(kPassThreads)
mlp_pass(const Net net, const float* __restrict__ p, const float* __restrict__ x,
         const float* __restrict__ t, int n, int width, float* __restrict__ y,
         float* __restrict__ sq_err) {
  constexpr int GROUPS = S >= 4 ? kPassThreads / kWTile : 1, SPT = S / GROUPS;
  extern __shared__ __align__(16) float sm[];
  // two weight tiles, two activation buffers [S][width] (width a multiple of 4)
  float* in = sm + 2 * kWTile * kWPitch;
  float* out = in + S * width;
  const int tid = threadIdx.x;
  const int n0 = blockIdx.x * S, rows = min(S, n - n0);
  const int u = tid % kWTile, g = tid / kWTile;  // the thread's unit of a tile, its samples' group
  const bool works = g < GROUPS;
  const int r0 = g * SPT;
  // the tile after (l, o0, i0); l = -1: none
  int l = 0, o0 = 0, i0 = 0;
  bool back = false;
  auto advance = [&](int& al, int& ao, int& ai, bool& ab) {
    const int ni = net.size[al], no = net.size[al + 1];
    if (!ab) {
      if ((ai += kWTile) < ni) return;
      ai = 0;
      if ((ao += kWTile) < no) return;
      ao = 0;
      if (++al < net.L) return;
      ab = true;
      al = t && net.L > 1 ? net.L - 1 : -1;
    } else {
      if ((ao += kWTile) < no) return;
      ao = 0;
      if ((ai += kWTile) < ni) return;
      ai = 0;
      if (--al < 1) al = -1;
    }
  };
  stage_weights(net, p, l, o0, i0, sm);
  for (int k = tid; k < S * net.size[0]; k += kPassThreads) {
    const int r = k / net.size[0], i = k - r * net.size[0];
    in[r * width + i] = r < rows ? x[(size_t)(n0 + r) * net.size[0] + i] : 0.0f;
  }
  float acc[SPT];
  for (int turn = 0; l >= 0; ++turn) {
    const float* w = sm + (turn & 1) * (kWTile * kWPitch);
    int nl = l, no0 = o0, ni0 = i0;
    bool nback = back;
    advance(nl, no0, ni0, nback);
    if (nl >= 0) {
      stage_weights(net, p, nl, no0, ni0, sm + ((turn + 1) & 1) * (kWTile * kWPitch));
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const int ni = net.size[l], no = net.size[l + 1];
    if (!back) {
      const int o = o0 + u, cols = min(kWTile, ni - i0);
      if (works && o < no) {
        if (i0 == 0) {
          const float b = __ldg(p + net.boff[l] + o);
#pragma unroll
          for (int s = 0; s < SPT; ++s) acc[s] = b;
        }
        const float* wr = w + u * kWPitch;
        const float* xr = in + r0 * width + i0;
        int i = 0;
#pragma unroll 4
        for (; i + 4 <= cols; i += 4) {
          const float4 wv = *reinterpret_cast<const float4*>(wr + i);
#pragma unroll
          for (int s = 0; s < SPT; ++s) {
            const float4 xv = *reinterpret_cast<const float4*>(xr + s * width + i);
            acc[s] = fmaf(wv.x, xv.x, acc[s]);
            acc[s] = fmaf(wv.y, xv.y, acc[s]);
            acc[s] = fmaf(wv.z, xv.z, acc[s]);
            acc[s] = fmaf(wv.w, xv.w, acc[s]);
          }
        }
        for (; i < cols; ++i)
#pragma unroll
          for (int s = 0; s < SPT; ++s) acc[s] = fmaf(wr[i], xr[s * width + i], acc[s]);
        if (i0 + cols == ni) {
          const bool relu = l + 1 < net.L;
#pragma unroll
          for (int s = 0; s < SPT; ++s) {
            const int r = r0 + s;
            const float a = (relu && acc[s] < 0.0f) ? 0.0f : acc[s];
            out[r * width + o] = a;
            if (r < rows) {
              if (t && relu) net.act[l + 1][(size_t)(n0 + r) * no + o] = a;
              if (!relu && y) y[n0 + r] = a;
            }
          }
        }
      }
    } else {
      // deltas of the layer below: d_l-1[i] = (sum_o d_l[o] W_l[o][i]) [act_l[i] > 0]
      const int i = i0 + u, cnt = min(kWTile, no - o0);
      if (works && i < ni) {
        if (o0 == 0)
#pragma unroll
          for (int s = 0; s < SPT; ++s) acc[s] = 0.0f;
        const float* dr = in + r0 * width + o0;
        int o = 0;
#pragma unroll 4
        for (; o + 4 <= cnt; o += 4) {
          float wv[4];
#pragma unroll
          for (int q = 0; q < 4; ++q) wv[q] = w[(o + q) * kWPitch + u];
#pragma unroll
          for (int s = 0; s < SPT; ++s) {
            const float4 dv = *reinterpret_cast<const float4*>(dr + s * width + o);
            acc[s] = fmaf(dv.x, wv[0], acc[s]);
            acc[s] = fmaf(dv.y, wv[1], acc[s]);
            acc[s] = fmaf(dv.z, wv[2], acc[s]);
            acc[s] = fmaf(dv.w, wv[3], acc[s]);
          }
        }
        for (; o < cnt; ++o)
#pragma unroll
          for (int s = 0; s < SPT; ++s) acc[s] = fmaf(dr[s * width + o], w[o * kWPitch + u], acc[s]);
        if (o0 + cnt == no) {
#pragma unroll
          for (int s = 0; s < SPT; ++s) {
            const int r = r0 + s;
            float v = 0.0f;
            if (r < rows) {
              const size_t k = (size_t)(n0 + r) * ni + i;
              v = net.act[l][k] > 0.0f ? acc[s] : 0.0f;
              net.delta[l - 1][k] = v;
            }
            out[r * width + i] = v;
          }
        }
      }
    }
    __syncthreads();
    if (nl != l || nback != back) {
      // the layer is complete: its outputs are the next one's inputs
      float* swap = in;
      in = out;
      out = swap;
      if (nback && !back && t) {
        // squared errors and the derivative of the loss 0.5 mean (y - t)^2
        if (tid < S) {
          const float e = tid < rows ? in[tid * width] - t[n0 + tid] : 0.0f;
          if (tid < rows) {
            sq_err[n0 + tid] = e * e;
            net.delta[net.L - 1][n0 + tid] = e / (float)n;
          }
          in[tid * width] = e / (float)n;
        }
        __syncthreads();
      }
    }
    l = nl;
    o0 = no0;
    i0 = ni0;
    back = nback;
  }
}

// Weight gradients of every layer: dW[o][i] = sum_r delta[r][o] in[r][i], and
// dW[o][ni] the bias gradients (a column of ones).  A block forms a 16 x 16 tile
// of one layer over all samples in their order; 128 threads, two sums each, 32
// samples of both operands in shared memory at a time, sample-minor so that one
// read brings a row's next four.  (Small tiles and few sums per thread, because
// the order of a sum leaves only the weights to spread over the GPU: 3 x 128 units
// are 169 blocks, and a sum is a chain of n multiply-adds.)  Block 0 also sums the
// loss.
constexpr int kGradTile = 16;
constexpr int kGradRows = 32;
constexpr int kGradThreads = 128;
__global__ void __launch_bounds__(kGradThreads)
mlp_grads(const Net net, const float* __restrict__ x, int n, float* __restrict__ g,
          const float* __restrict__ sq_err, float* __restrict__ loss) {
  __shared__ __align__(16) float ds[kGradTile][kGradRows + 4], xs[kGradTile][kGradRows + 4];
  __shared__ float part[256];
  const int tid = threadIdx.x;
  int tile = blockIdx.x, l = 0, it = 0;
  for (; l < net.L; ++l) {
    it = (net.size[l] + 1 + kGradTile - 1) / kGradTile;
    const int tiles = it * ((net.size[l + 1] + kGradTile - 1) / kGradTile);
    if (tile < tiles) break;
    tile -= tiles;
  }
  const int ni = net.size[l], no = net.size[l + 1];
  const int i0 = (tile % it) * kGradTile, o0 = (tile / it) * kGradTile;
  const float* __restrict__ in = l == 0 ? x : net.act[l];
  const float* __restrict__ d = net.delta[l];
  const int c = tid % kGradTile, w = tid / kGradTile;  // loads: column c of rows w, w + 8, ..
  // sums: rows to and to + 1, column ti; a warp's are 8 x 8
  const int warp = tid / 32, lane = tid % 32;
  const int to = (warp / 2) * 8 + (lane / 8) * 2, ti = (warp % 2) * 8 + lane % 8;
  float a0 = 0.0f, a1 = 0.0f;
  constexpr int kStep = kGradThreads / kGradTile, kLoads = kGradRows / kStep;
  float dv[kLoads], xv[kLoads];
  auto load = [&](int r) {
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      const int row = r + w + kStep * k;
      dv[k] = (row < n && o0 + c < no) ? __ldg(d + (size_t)row * no + o0 + c) : 0.0f;
      xv[k] = row >= n ? 0.0f : i0 + c < ni ? __ldg(in + (size_t)row * ni + i0 + c) : i0 + c == ni ? 1.0f : 0.0f;
    }
  };
  load(0);
  for (int r = 0; r < n; r += kGradRows) {
#pragma unroll
    for (int k = 0; k < kLoads; ++k) {
      ds[c][w + kStep * k] = dv[k];
      xs[c][w + kStep * k] = xv[k];
    }
    __syncthreads();
    load(r + kGradRows);
    if (r + kGradRows <= n) {
#pragma unroll
      for (int k = 0; k < kGradRows; k += 4) {
        const float4 d0 = *reinterpret_cast<const float4*>(&ds[to][k]);
        const float4 d1 = *reinterpret_cast<const float4*>(&ds[to + 1][k]);
        const float4 xx = *reinterpret_cast<const float4*>(&xs[ti][k]);
        a0 = fmaf(d0.x, xx.x, a0);
        a1 = fmaf(d1.x, xx.x, a1);
        a0 = fmaf(d0.y, xx.y, a0);
        a1 = fmaf(d1.y, xx.y, a1);
        a0 = fmaf(d0.z, xx.z, a0);
        a1 = fmaf(d1.z, xx.z, a1);
        a0 = fmaf(d0.w, xx.w, a0);
        a1 = fmaf(d1.w, xx.w, a1);
      }
    } else {
      for (int k = 0; k < n - r; ++k) {
        a0 = fmaf(ds[to][k], xs[ti][k], a0);
        a1 = fmaf(ds[to + 1][k], xs[ti][k], a1);
      }
    }
    __syncthreads();
  }
#pragma unroll
  for (int a = 0; a < 2; ++a) {
    const int o = o0 + to + a, i = i0 + ti;
    if (o < no && i <= ni) g[i < ni ? net.woff[l] + (int64_t)o * ni + i : net.boff[l] + o] = a ? a1 : a0;
  }
  if (blockIdx.x == 0) {
    // 256 sums of every 256th sample, then a tree over them
    for (int q = tid; q < 256; q += kGradThreads) {
      float s = 0.0f;
      for (int k = q; k < n; k += 256) s += sq_err[k];
      part[q] = s;
    }
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
      for (int q = tid; q < k; q += kGradThreads) part[q] += part[q + k];
      __syncthreads();
    }
    if (tid == 0) *loss = 0.5f * part[0] / (float)n;
  }
}

}  // namespace

// Adam (Kingma and Ba): m = b1 m + (1-b1) g; v = b2 v + (1-b2) g^2;
// p -= lr * mhat / (sqrt(vhat) + eps), with bias corrections c1, c2.
__global__ void mlp_adam(float* __restrict__ p, const float* __restrict__ g, float* __restrict__ m,
                         float* __restrict__ v, int np, float lr, float b1, float b2, float eps,
                         float c1, float c2) {
  const int k = blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= np) return;
  const float gk = g[k];
  const float mk = b1 * m[k] + (1.0f - b1) * gk;
  const float vk = b2 * v[k] + (1.0f - b2) * gk * gk;
  m[k] = mk;
  v[k] = vk;
  p[k] -= lr * (mk / c1) / (sqrtf(vk / c2) + eps);
}

// ------------------------------------------------------------------ host
Mlp::Mlp(int nin_, int hidden_, int nlayers_) : nin(nin_), hidden(hidden_), nlayers(nlayers_) {
  sizes.push_back(nin);
  for (int l = 0; l < nlayers; ++l) sizes.push_back(hidden);
  sizes.push_back(1);
  np = 0;
  for (size_t l = 0; l + 1 < sizes.size(); ++l) {
    woff.push_back(np);
    np += (int64_t)sizes[l + 1] * sizes[l];
    boff.push_back(np);
    np += sizes[l + 1];
  }
}

cudaError_t Mlp::alloc_params() {
  cudaError_t e;
  if ((e = cudaMalloc(&p, np * 4)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&g, np * 4)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&m, np * 4)) != cudaSuccess) return e;
  if ((e = cudaMalloc(&v, np * 4)) != cudaSuccess) return e;
  if ((e = cudaMemset(m, 0, np * 4)) != cudaSuccess) return e;
  if ((e = cudaMemset(v, 0, np * 4)) != cudaSuccess) return e;
  if ((e = cudaMemset(g, 0, np * 4)) != cudaSuccess) return e;
  return cudaMalloc(&loss, 4);
}

cudaError_t Mlp::reserve(int n) {
  if (n <= cap) return cudaSuccess;
  free_acts();
  const int L = (int)sizes.size() - 1;
  acts.assign(L + 1, nullptr);
  deltas.assign(L, nullptr);
  cudaError_t e;
  for (int l = 0; l < L; ++l) {
    // act[l + 1] of the hidden layers, delta[l] of every layer
    if (l + 1 < L && (e = cudaMalloc(&acts[l + 1], (size_t)n * sizes[l + 1] * 4)) != cudaSuccess) return e;
    if ((e = cudaMalloc(&deltas[l], (size_t)n * sizes[l + 1] * 4)) != cudaSuccess) return e;
  }
  if ((e = cudaMalloc(&sq_err, (size_t)n * 4)) != cudaSuccess) return e;
  cap = n;
  return cudaSuccess;
}

void Mlp::free_acts() {
  for (float* a : acts) if (a) cudaFree(a);
  for (float* a : deltas) if (a) cudaFree(a);
  acts.clear();
  deltas.clear();
  if (sq_err) cudaFree(sq_err);
  sq_err = nullptr;
  cap = 0;
}

Mlp::~Mlp() {
  free_acts();
  if (p) cudaFree(p);
  if (g) cudaFree(g);
  if (m) cudaFree(m);
  if (v) cudaFree(v);
  if (loss) cudaFree(loss);
}

// One launch of mlp_pass.  Samples per block: as few as leave every block an SM
// (the weight tiles and activations leave room for one block), sixteen beyond
// that, since every block reads all the weights; eight where sixteen samples of
// the widest layer do not fit (1024 units: 200 KB with eight).
static cudaError_t launch_pass(const Net& net, const float* p, const float* x, const float* t, int n,
                               float* y, float* sq_err, cudaStream_t s) {
  int width = 0;
  for (int l = 0; l <= net.L; ++l) width = std::max(width, (net.size[l] + 3) / 4 * 4);
  auto smem_of = [&](int S) { return ((size_t)2 * kWTile * kWPitch + (size_t)2 * S * width) * 4; };
  auto run = [&](auto kernel, int S) {
    cudaError_t e = smem_limit(reinterpret_cast<const void*>(kernel), smem_of(S));
    if (e != cudaSuccess) return e;
    kernel<<<(unsigned)((n + S - 1) / S), kPassThreads, smem_of(S), s>>>(net, p, x, t, n, width, y, sq_err);
    return cudaGetLastError();
  };
  if (n <= 2 * 152) return run(mlp_pass<2>, 2);
  if (n <= 4 * 152) return run(mlp_pass<4>, 4);
  if (n <= 8 * 152 || smem_of(16) > 227 * 1024) return run(mlp_pass<8>, 8);
  return run(mlp_pass<16>, 16);
}

static Net net_of(const Mlp& m) {
  Net net;
  memset(&net, 0, sizeof net);
  net.L = (int)m.sizes.size() - 1;
  for (int l = 0; l <= net.L; ++l) net.size[l] = m.sizes[l];
  for (int l = 0; l < net.L; ++l) {
    net.woff[l] = m.woff[l];
    net.boff[l] = m.boff[l];
  }
  for (size_t l = 0; l < m.acts.size(); ++l) net.act[l] = m.acts[l];
  for (size_t l = 0; l < m.deltas.size(); ++l) net.delta[l] = m.deltas[l];
  return net;
}

cudaError_t Mlp::forward(const float* x, int n, float* y, cudaStream_t s) {
  return launch_pass(net_of(*this), p, x, nullptr, n, y, nullptr, s);
}

cudaError_t Mlp::backward(const float* x, const float* t, int n, cudaStream_t s) {
  cudaError_t e = reserve(n);
  if (e != cudaSuccess) return e;
  const Net net = net_of(*this);
  e = launch_pass(net, p, x, t, n, nullptr, sq_err, s);
  if (e != cudaSuccess) return e;
  int tiles = 0;
  for (int l = 0; l < net.L; ++l)
    tiles += ((net.size[l] + 1 + kGradTile - 1) / kGradTile) *
             ((net.size[l + 1] + kGradTile - 1) / kGradTile);
  mlp_grads<<<(unsigned)tiles, kGradThreads, 0, s>>>(net, x, n, g, sq_err, loss);
  return cudaGetLastError();
}

cudaError_t Mlp::adam(float lr, float b1, float b2, float eps, cudaStream_t s) {
  ++step;
  const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  mlp_adam<<<(unsigned)((np + 255) / 256), 256, 0, s>>>(p, g, m, v, (int)np, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

}  // namespace pa
