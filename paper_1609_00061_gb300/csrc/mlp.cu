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
// A pass is bound by latency (a 256-sample minibatch is 70 MFLOP), so it takes
// few launches and every launch keeps its chain short: one block carries a few
// samples through every layer and back with the activations in shared memory
// (mlp_pass), and one launch forms every layer's weight gradients (mlp_grads),
// with a second that adds up parts when the samples are split.  256 samples,
// prediction and gradients of 3 x 128 units: 1520 us with a launch per layer
// whose threads each walked a weight row, 93 us now (both read-backs included).
#include <math.h>
#include <string.h>

#include <algorithm>
#include <vector>

#include "mlp.h"
#include "pa_internal.h"

namespace pa {

namespace {

constexpr int kPassThreads = 512;
constexpr int kMaxLayers = 10;     // at most 8 hidden layers, the output layer

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

// S samples per block through every layer; with t, back again, writing the
// activations and deltas that the weight gradients need and the block's part of
// the squared error.
template <int S>
__global__ void __launch_bounds__(kPassThreads)
mlp_pass(const Net net, const float* __restrict__ p, const float* __restrict__ x,
         const float* __restrict__ t, int n, int width, float* __restrict__ y,
         float* __restrict__ loss_part) {
  extern __shared__ __align__(16) float sm[];
  // two activation buffers [S][width] (width a multiple of 4), then the partial
  // sums of the backward layers
  float* in = sm;
  float* out = sm + S * width;
  float* red = sm + 2 * S * width;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int n0 = blockIdx.x * S, rows = min(S, n - n0);
  for (int k = tid; k < S * net.size[0]; k += kPassThreads) {
    const int r = k / net.size[0], i = k - r * net.size[0];
    in[r * width + i] = r < rows ? x[(size_t)(n0 + r) * net.size[0] + i] : 0.0f;
  }
  __syncthreads();
  for (int l = 0; l < net.L; ++l) {
    const int ni = net.size[l], no = net.size[l + 1];
    const float* __restrict__ W = p + net.woff[l];
    const bool relu = l + 1 < net.L;
    // eight lanes per output: 64 outputs per pass of the block, each lane four
    // consecutive weights at a time
    const bool vec = ni % 4 == 0 && net.woff[l] % 4 == 0;
    const int sub = lane & 7;
    for (int o0 = 0; o0 < no; o0 += kPassThreads / 8) {
      const int o = o0 + warp * 4 + (lane >> 3);
      float acc[S];
#pragma unroll
      for (int r = 0; r < S; ++r) acc[r] = 0.0f;
      if (o < no) {
        const float* w = W + (size_t)o * ni;
        if (vec) {
#pragma unroll 4
          for (int i = sub * 4; i < ni; i += 32) {
            const float4 wv = __ldg(reinterpret_cast<const float4*>(w + i));
#pragma unroll
            for (int r = 0; r < S; ++r) {
              const float4 xv = *reinterpret_cast<const float4*>(in + r * width + i);
              acc[r] = fmaf(wv.x, xv.x, acc[r]);
              acc[r] = fmaf(wv.y, xv.y, acc[r]);
              acc[r] = fmaf(wv.z, xv.z, acc[r]);
              acc[r] = fmaf(wv.w, xv.w, acc[r]);
            }
          }
        } else {
          for (int i = sub; i < ni; i += 8) {
            const float wv = __ldg(w + i);
#pragma unroll
            for (int r = 0; r < S; ++r) acc[r] = fmaf(wv, in[r * width + i], acc[r]);
          }
        }
      }
#pragma unroll
      for (int r = 0; r < S; ++r)
#pragma unroll
        for (int m = 4; m > 0; m >>= 1) acc[r] += __shfl_xor_sync(0xffffffffu, acc[r], m);
      if (o < no) {
        const float b = __ldg(p + net.boff[l] + o);
#pragma unroll
        for (int r = 0; r < S; ++r) {
          if (sub != r % 8) continue;
          const float v = acc[r] + b;
          const float a = (relu && v < 0.0f) ? 0.0f : v;
          out[r * width + o] = a;
          if (r < rows) {
            if (t && relu) net.act[l + 1][(size_t)(n0 + r) * no + o] = a;
            if (!relu && y) y[n0 + r] = a;
          }
        }
      }
    }
    __syncthreads();
    float* swap = in;
    in = out;
    out = swap;
  }
  if (!t) return;
  // loss 0.5 mean (y - t)^2 and its derivative
  if (tid < S) {
    const float e = tid < rows ? in[tid * width] - t[n0 + tid] : 0.0f;
    red[tid] = e * e;
    out[tid * width] = e / (float)n;
    if (tid < rows) net.delta[net.L - 1][n0 + tid] = e / (float)n;
  }
  __syncthreads();
  if (tid == 0) {
    float s = 0.0f;
    for (int r = 0; r < S; ++r) s += red[r];
    loss_part[blockIdx.x] = s;
  }
  __syncthreads();
  // deltas of the layers below: d_l-1[i] = (sum_o d_l[o] W_l[o][i]) [act_l[i] > 0].
  // Threads along i; the sum over o is dealt over the groups of threads that are
  // left and added up in shared memory.
  float* d = out;
  float* dn = in;
  for (int l = net.L - 1; l > 0; --l) {
    const int ni = net.size[l], no = net.size[l + 1];
    const float* __restrict__ W = p + net.woff[l];
    const int lanes = min((ni + 31) / 32 * 32, kPassThreads), groups = kPassThreads / lanes;
    const int g = tid / lanes;
    for (int i0 = 0; i0 < ni; i0 += lanes) {
      const int i = i0 + tid % lanes;
      float acc[S];
#pragma unroll
      for (int r = 0; r < S; ++r) acc[r] = 0.0f;
      if (g < groups && i < ni) {
#pragma unroll 8
        for (int o = g; o < no; o += groups) {
          const float wv = __ldg(W + (size_t)o * ni + i);
#pragma unroll
          for (int r = 0; r < S; ++r) acc[r] = fmaf(d[r * width + o], wv, acc[r]);
        }
      }
#pragma unroll
      for (int r = 0; r < S; ++r) red[r * kPassThreads + tid] = acc[r];
      __syncthreads();
      for (int k = tid; k < S * lanes; k += kPassThreads) {
        const int r = k / lanes, j = k - r * lanes;
        if (i0 + j < ni && r < rows) {
          float s = 0.0f;
          for (int q = 0; q < groups; ++q) s += red[r * kPassThreads + q * lanes + j];
          if (!(net.act[l][(size_t)(n0 + r) * ni + i0 + j] > 0.0f)) s = 0.0f;
          dn[r * width + i0 + j] = s;
          net.delta[l - 1][(size_t)(n0 + r) * ni + i0 + j] = s;
        } else if (i0 + j < ni) {
          dn[r * width + i0 + j] = 0.0f;
        }
      }
      __syncthreads();
    }
    float* swap = d;
    d = dn;
    dn = swap;
  }
}

// Weight gradients of every layer: dW[o][i] = sum_r delta[r][o] in[r][i], and
// dW[o][ni] the bias gradients (a column of ones).  A block forms a 32 x 32 tile
// of one layer over one part of the samples; 256 threads, 2 x 2 sums each, 32
// samples of both operands in shared memory at a time.  parts > 1: part q's
// sums go to g + q * np of a scratch vector (mlp_add_parts adds them up in
// order).  Block 0 also sums the loss.
constexpr int kGradTile = 32;
__global__ void __launch_bounds__(256)
mlp_grads(const Net net, const float* __restrict__ x, int n, int parts, int64_t np,
          float* __restrict__ g, const float* __restrict__ loss_part, int nloss,
          float* __restrict__ loss) {
  __shared__ float ds[32][kGradTile + 1], xs[32][kGradTile + 1];
  __shared__ float part[256];
  const int tid = threadIdx.x;
  const int q = blockIdx.x % parts;
  int tile = blockIdx.x / parts, l = 0, it = 0;
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
  const int per = ((n + parts - 1) / parts + 31) / 32 * 32;
  const int r0 = q * per, r1 = min(n, r0 + per);
  const int c = tid & 31, w = tid >> 5;  // loads: column c of rows w, w + 8, ..
  const int to = (tid >> 4) * 2, ti = (tid & 15) * 2;
  float acc[2][2] = {{0.0f, 0.0f}, {0.0f, 0.0f}};
  float dv[4], xv[4];
  auto load = [&](int r) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const int row = r + w + 8 * k;
      dv[k] = (row < r1 && o0 + c < no) ? __ldg(d + (size_t)row * no + o0 + c) : 0.0f;
      xv[k] = row >= r1 ? 0.0f : i0 + c < ni ? __ldg(in + (size_t)row * ni + i0 + c) : i0 + c == ni ? 1.0f : 0.0f;
    }
  };
  load(r0);
  for (int r = r0; r < r1; r += 32) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      ds[w + 8 * k][c] = dv[k];
      xs[w + 8 * k][c] = xv[k];
    }
    __syncthreads();
    load(r + 32);
#pragma unroll
    for (int k = 0; k < 32; ++k)
#pragma unroll
      for (int a = 0; a < 2; ++a)
#pragma unroll
        for (int b = 0; b < 2; ++b) acc[a][b] = fmaf(ds[k][to + a], xs[k][ti + b], acc[a][b]);
    __syncthreads();
  }
  float* dst = g + (parts > 1 ? (int64_t)q * np : 0);
#pragma unroll
  for (int a = 0; a < 2; ++a)
#pragma unroll
    for (int b = 0; b < 2; ++b) {
      const int o = o0 + to + a, i = i0 + ti + b;
      if (o >= no || i > ni) continue;
      dst[i < ni ? net.woff[l] + (int64_t)o * ni + i : net.boff[l] + o] = acc[a][b];
    }
  if (blockIdx.x == 0) {
    float s = 0.0f;
    for (int k = tid; k < nloss; k += 256) s += loss_part[k];
    part[tid] = s;
    __syncthreads();
    for (int k = 128; k > 0; k >>= 1) {
      if (tid < k) part[tid] += part[tid + k];
      __syncthreads();
    }
    if (tid == 0) *loss = 0.5f * part[0] / (float)n;
  }
}

__global__ void mlp_add_parts(const float* __restrict__ parts, int nparts, int64_t np,
                              float* __restrict__ g) {
  const int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (k >= np) return;
  float s = 0.0f;
  for (int q = 0; q < nparts; ++q) s += parts[(int64_t)q * np + k];
  g[k] = s;
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

int Mlp::max_parts() const { return (int)std::max<int64_t>(1, std::min<int64_t>(16, (4 << 20) / np)); }

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
  // the blocks' squared errors, then the parts of the weight gradients
  if ((e = cudaMalloc(&scratch, ((size_t)n + (size_t)max_parts() * np) * 4)) != cudaSuccess) return e;
  cap = n;
  return cudaSuccess;
}

void Mlp::free_acts() {
  for (float* a : acts) if (a) cudaFree(a);
  for (float* a : deltas) if (a) cudaFree(a);
  acts.clear();
  deltas.clear();
  if (scratch) cudaFree(scratch);
  scratch = nullptr;
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

// One launch of mlp_pass.  Samples per block: few while the blocks do not fill
// the GPU (a block's chain of layers is what a small pass waits for), more where
// every block would read all the weights again for them; all that fit in shared
// memory for wide layers.
static cudaError_t launch_pass(const Net& net, const float* p, const float* x, const float* t, int n,
                               float* y, float* loss_part, int* nblocks, cudaStream_t s) {
  int width = 0;
  for (int l = 0; l <= net.L; ++l) width = std::max(width, (net.size[l] + 3) / 4 * 4);
  auto run = [&](auto kernel, int S) {
    const size_t smem = ((size_t)2 * S * width + (size_t)S * kPassThreads) * 4;
    cudaError_t e = smem_limit(reinterpret_cast<const void*>(kernel), smem);
    if (e != cudaSuccess) return e;
    *nblocks = (n + S - 1) / S;
    kernel<<<(unsigned)*nblocks, kPassThreads, smem, s>>>(net, p, x, t, n, width, y, loss_part);
    return cudaGetLastError();
  };
  if (n <= 2 * 304) return run(mlp_pass<2>, 2);
  if (n <= 4 * 608) return run(mlp_pass<4>, 4);
  return run(mlp_pass<8>, 8);
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
  int nblocks = 0;
  return launch_pass(net_of(*this), p, x, nullptr, n, y, nullptr, &nblocks, s);
}

cudaError_t Mlp::backward(const float* x, const float* t, int n, cudaStream_t s) {
  cudaError_t e = reserve(n);
  if (e != cudaSuccess) return e;
  const Net net = net_of(*this);
  int nblocks = 0;
  e = launch_pass(net, p, x, t, n, nullptr, scratch, &nblocks, s);
  if (e != cudaSuccess) return e;
  int tiles = 0;
  for (int l = 0; l < net.L; ++l)
    tiles += ((net.size[l] + 1 + kGradTile - 1) / kGradTile) *
             ((net.size[l + 1] + kGradTile - 1) / kGradTile);
  // parts of at least 64 samples while the tiles leave SMs idle
  const int parts = std::max(1, std::min({(n + 63) / 64, (4 * 152 + tiles - 1) / tiles, max_parts()}));
  float* part = scratch + cap;
  mlp_grads<<<(unsigned)(tiles * parts), 256, 0, s>>>(net, x, n, parts, np, parts > 1 ? part : g, scratch,
                                                      nblocks, loss);
  if (parts > 1)
    mlp_add_parts<<<(unsigned)((np + 255) / 256), 256, 0, s>>>(part, parts, np, g);
  return cudaGetLastError();
}

cudaError_t Mlp::adam(float lr, float b1, float b2, float eps, cudaStream_t s) {
  ++step;
  const float c1 = 1.0f - powf(b1, (float)step), c2 = 1.0f - powf(b2, (float)step);
  mlp_adam<<<(unsigned)((np + 255) / 256), 256, 0, s>>>(p, g, m, v, (int)np, lr, b1, b2, eps, c1, c2);
  return cudaGetLastError();
}

}  // namespace pa
