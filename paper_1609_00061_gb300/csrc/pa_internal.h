// Internal declarations shared by the CUDA translation units of the pixel array
// engine.  Nothing here is part of the public C interface (include/pa.h).
#pragma once

#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/pa.h"

namespace pa {

// Raise kernel `fn`'s dynamic shared-memory limit on the current device only
// when a launch needs more than any earlier one did (the attribute call costs
// host time on every launch otherwise).  Thread-safe.
cudaError_t smem_limit(const void* fn, size_t bytes);

constexpr int kMaxDim = PA_MAX_DIM;
constexpr int kMaxDeg = PA_MAX_DEGREE;

#ifdef __CUDACC__
// The last entry of an ascending table (entry i at first(i), i < n, first(0) <=
// block) that is at most `block`, found by every thread of the block together:
// each compares one of an evenly spaced sample, then the gap is searched the
// same way.  (Two rounds of independent loads up to 65536 entries; a binary
// search is a chain of as many L2 latencies as log2(n).)
template <class F>
__device__ __forceinline__ int find_entry(F&& first, int n, int64_t block) {
  int p = 0;
  while (n > 1) {
    const int step = (n + (int)blockDim.x - 1) / (int)blockDim.x;
    const int64_t at = (int64_t)threadIdx.x * step;
    const int below = at < n && first(p + (int)at) <= block;
    const int skip = (__syncthreads_count(below) - 1) * step;
    p += skip;
    n = min(step, n - skip);
  }
  return p;
}
#endif

// ------------------------------------------------------------------ plotting
// One relation to plot.  Coefficients are in "nest order": the order in which
// the nested evaluation visits the monomials (last port outermost, every
// exponent ascending), so the device reads them front to back.
//
// Pixel centres are computed on the device as lo + ((double)i + 0.5) * delta
// with delta = (hi - lo) / res divided on the host (IEEE division is correctly
// rounded on both, so the value is the one pa.h defines).
struct PlotJob {
  const double* coeffs;             // device, nest order
  // filtered jobs: ports in units of 2^k_p and f in units of 2^q (plot.cu)
  const float* c32;                 // the coefficients in those units, rounded to FP32
  uint64_t* out;                    // device, pa_array layout
  double lo[kMaxDim];               // per port: range start of its variable
  double delta[kMaxDim];            // per port: pixel width of its variable
  float lo_hi[kMaxDim], lo_lo[kMaxDim];  // lo and delta in units of the port, as sums of two floats
  float d_hi[kMaxDim], d_lo[kMaxDim];
  int64_t nrows;                    // rows = product of all but the last array axis
  int64_t row_words;                // ceil(res_last / 64)
  int64_t tile0;                    // first block of this job in the plot launch
  int32_t rows_per_tile;
  int32_t arity, degree, kind, strict;
  int32_t filter;                   // 1: FP32 filter (plot.cu); 0: FP64 at every pixel
  int32_t ndim;                     // array axes (distinct variables)
  int32_t res[kMaxDim];             // array axis resolutions
  int32_t port_axis[kMaxDim];       // port -> array axis
  double eps;
  float eps32;                      // eps in units of f, rounded to FP32
  float bound;                      // B: FP32 against FP64, eps rounding included (plot.cu)
  float dabs;                       // 1.01 x the last port's pixel width in its unit
};

// One expression relation to plot (expr.cu): the postfix program and its
// constants on the device, the pixel grid as for PlotJob; word0 is the first
// word of this job in the launch's flat word space.
struct ExprJob {
  const int32_t* prog;
  const double* consts;
  const float2* c32;                // per constant an FP32 interval that holds it
  uint64_t* out;
  double lo[kMaxDim];
  double delta[kMaxDim];
  double eps;
  int64_t nrows, row_words, word0;
  int32_t nops, arity, kind, strict, ndim;
  int32_t res[kMaxDim];
  int32_t port_axis[kMaxDim];
};
// Every expression plot of a call in one launch.
void launch_plot_expr(const ExprJob* d_jobs, int njobs, int64_t total_words, cudaStream_t s);

// One relation plotted by the corner rule (pa.h, pa_rule): a polynomial
// (prog == nullptr; coefficients in nest order) or an expression program.
// lo and delta are per port; port_axis maps a port to its axis of `out`.
struct CornerJob {
  const int32_t* prog;
  const double* consts;
  const double* coeffs;
  uint64_t* out;
  double lo[kMaxDim];
  double delta[kMaxDim];
  double eps;
  int64_t nrows, row_words, word0;
  int32_t nops, degree, arity, kind, strict, ndim;
  int32_t res[kMaxDim];
  int32_t port_axis[kMaxDim];
};
// Every corner-rule plot of a call in one launch, one thread per output byte.
void launch_plot_corner(const CornerJob* d_jobs, int njobs, int64_t total_words, cudaStream_t s);

// A range of words to clear: words [w0, w0 + words) of the launch's flat
// index space are p[0 .. words).
struct ZeroRange {
  uint64_t* p;
  int64_t words;
  int64_t w0;
};
// One launch plots every job: blocks of rows_per_tile rows, each computing its
// rows' polynomials in shared memory first.  common_degree: the degree shared
// by every job (selects a specialised kernel), or -1 when they differ.
// The same launch also clears the `nzero` ranges (zero_words words in all)
// that later contractions OR their results into, so that no separate memset
// sits between the launches.
// Plot blocks the GPU holds at once (all SMs), for the kernel of this degree.
int plot_resident_blocks(int common_degree);
void launch_plot(const PlotJob* d_jobs, int njobs, int64_t total_tiles, int max_rows_per_tile,
                 int max_degree, int common_degree, const ZeroRange* d_zero, int nzero,
                 int64_t zero_words, cudaStream_t s);

// ------------------------------------------------------------- bit arrays
// A bit-packed array with `inner` trailing axes flattened into packed rows:
// rowlen = prod(res[ndim-inner..]), row_words = ceil(rowlen / 64),
// nrows = prod(res[..ndim-inner]).  The public pa_array layout is inner = 1
// (inner = 0 for ndim = 0).
struct BitArr {
  uint64_t* w = nullptr;
  int ndim = 0;
  int inner = 0;
  int vars[2 * kMaxDim] = {};
  int64_t res[2 * kMaxDim] = {};
  int64_t rowlen() const {
    int64_t r = 1;
    for (int a = ndim - inner; a < ndim; ++a) r *= res[a];
    return r;
  }
  int64_t row_words() const { return (rowlen() + 63) / 64; }
  int64_t nrows() const {
    int64_t r = 1;
    for (int a = 0; a < ndim - inner; ++a) r *= res[a];
    return r;
  }
  int64_t words() const { return nrows() * row_words(); }
  int64_t bits() const { return nrows() * rowlen(); }
};

// Reshape modes (contract.cu):
//  kReshapeBits       any mapping; every output bit gathered on its own
//  kReshapeWords      the last output axis runs along input words: every output
//                     word is one input word (OR-ed over reduced axes), found
//                     through word strides u_in over the output-word axes u_res
//  kReshapeTranspose  the last output axis L steps by input rows or whole
//                     input words and the input's last axis J is kept: 64 x 64
//                     bit blocks are transposed; u_res / u_in / u_out cover
//                     the other axes
enum { kReshapeBits = 0, kReshapeWords = 1, kReshapeTranspose = 2 };

// General gather: out bit (axes of `out`) = OR over the reduced input axes of
// the input bit with the same values of the shared axes.  An output axis that
// is missing from the input has zero strides (broadcast).
struct ReshapeDesc {
  const uint64_t* in;
  uint64_t* out;
  int64_t out_nrows, out_row_words, out_rowlen;
  int32_t out_ndim, out_inner;
  int64_t out_res[2 * kMaxDim];
  int64_t row_stride[2 * kMaxDim];  // per output axis: input row-index stride
  int64_t col_stride[2 * kMaxDim];  // per output axis: input column (bit) stride
  int32_t nred;
  int64_t red_res[2 * kMaxDim];
  int64_t red_row_stride[2 * kMaxDim];
  int64_t red_col_stride[2 * kMaxDim];
  int64_t in_row_words;
  int32_t mode;                      // kReshape*
  int32_t row_any;                   // bit mode: all packed input axes reduced (see contract.cu)
  int32_t nu;                        // axes of the word / tile decomposition
  int64_t u_res[2 * kMaxDim];
  int64_t u_in[2 * kMaxDim];         // input words per step of the axis
  int64_t u_out[2 * kMaxDim];        // output words per step (transpose mode)
  int64_t red_in_w[2 * kMaxDim];     // words mode: input words per reduced step
  int64_t vec;                       // words mode: consecutive words that stay together (1, 2, 4)
  int64_t tQ, tR;                    // transpose: resolutions of J and L
  int64_t t_in_L, t_out_J;           // input words per L step, output words per J step
  int64_t n_other;                   // transpose: product of u_res
};
// Kernel variant of a reshape (kRs*) and its block count; a launch runs a
// table of n descriptors of one kind, problem p on blocks [cta0[p], cta0[p+1])
// (device arrays), grid = cta0[n].
enum { kRsBits = 0, kRsWords32, kRsWords64, kRsTranspose32, kRsTranspose32Wide, kRsTranspose64,
       kRsKinds };
int reshape_kind(const ReshapeDesc& d);
int64_t reshape_units(const ReshapeDesc& d);   // block-sized pieces of its work
int64_t reshape_blocks(const ReshapeDesc& d, int64_t per);  // blocks of `per` pieces each
void launch_reshape(const ReshapeDesc* d_descs, const int64_t* d_cta0, int n, int kind,
                    int64_t grid, cudaStream_t s);

// cudaSuccess when the library holds kernel code the current device can run
cudaError_t probe_kernel_image();

// Clusters that are not matrix products, batched like the contractions:
// kEwOuter  C row r (r = b * M + m) is B row b (nw words) when bit r of A is set;
// kEwDot    bit r of C = any(A row r AND B row r / M), rows of nw <= 16 words;
// kEwDotWide the same for longer rows, OR-ed into a cleared C;
// kEwAnd    C = A AND B over `rows` words.
enum { kEwOuter = 0, kEwDot = 1, kEwDotWide = 2, kEwAnd = 3 };
struct EwJob {
  const uint64_t* a;
  const uint64_t* b;
  uint64_t* c;
  int64_t rows, m, nw;
  int32_t kind;
};
int64_t ewise_blocks(const EwJob& j);
bool ewise_fits32(const EwJob& j);  // 32-bit indexes suffice (else launch with wide)
void launch_ewise(const EwJob* d_jobs, const int64_t* d_cta0, int n, int64_t grid, bool wide,
                  cudaStream_t s);

// C[b*M + m, :] |= B[b*K + k, :] for every set bit k of A[b*M + m, :].
// One CTA owns a tile of B (Kc rows x Nt words of batch b) in shared memory and
// a run of output rows; see contract.cu.
struct RowOrDesc {
  const uint64_t* A;
  const uint64_t* B;
  uint64_t* C;
  int64_t nbatch, M, K, Nw;   // Nw = words per B / C row
  int64_t a_row_words;        // = ceil(K / 64)
  int32_t Nt;                 // words per tile (power of two <= 32)
  int32_t Kc;                 // B rows per tile (a multiple of 64 unless it is all of K)
  int32_t threads;            // per CTA: 256, 512 or 1024
  int64_t n_tiles, k_chunks, row_splits, rows_per_split;
  int32_t atomic;             // 1: C pre-zeroed, results OR-ed in atomically
  int32_t stage;              // kStage*: how the tile reaches shared memory
  int* err;                   // device error word: set when a bounded wait runs out
  unsigned long long* stat;   // when not null: += shared-memory words OR-ed (timing mode)
};
enum { kStageWords = 0, kStageTile = 1, kStageRun = 2 };
// Longest K range whose tables fit next to the lists of a CTA of `threads`.
int64_t rowor_max_kc(int Nt, int threads);
// Choose the tile shape and grid for a contraction of this shape, which has
// `share` SMs (a fraction when many contractions share one launch).  free_clear: a
// result that has to start at zero costs no launch of its own.
void rowor_plan(RowOrDesc& d, double share, bool free_clear);
size_t rowor_smem_bytes(const RowOrDesc& d);
int64_t rowor_ctas(const RowOrDesc& d);
// TMA descriptor of d.B (all zero unless d.stage is kStageTile)
cudaError_t rowor_encode_map(const RowOrDesc& d, CUtensorMap* map);
// Independent contractions with the same CTA size in one launch: descriptors,
// tensor maps and CTA offsets (nprob + 1 entries) on the device.
cudaError_t launch_rowor(const RowOrDesc* d_descs, const CUtensorMap* d_maps,
                         const int64_t* d_cta0, int nprob, int64_t grid, size_t smem, int threads,
                         cudaStream_t s);

// Tensor-core contraction (mma.cu): the same problem as RowOrDesc, from the
// same bit-packed layouts, as a 0/1 matrix product on E4M3 operands thresholded
// at > 0.
struct MmaDesc {
  const uint64_t* A;          // [nbatch][M][a_row_words], K bits per row
  const uint64_t* B;          // [nbatch][K][Nw], N bits per row
  uint64_t* C;                // [nbatch][M][Nw]
  int64_t M, N, K, Nw, a_row_words, nbatch;
  int64_t m_tiles, n_tiles;
  // Occupancy bitmaps, kb_words 32-bit words for every row tile of A and then
  // every column tile of B, per batch value: bit kb when K values 128 kb ..
  // hold a set bit.  The product skips the K blocks either one lacks.  Null: the
  // product looks at the words themselves.
  uint8_t* occ;
  int64_t kb_words;
  int32_t BN;                 // columns per tile: 128 or 256
  // K split: ksplit CTAs per output tile, each summing kchunk consecutive
  // 128-value K blocks and OR-ing its bits into C, which starts at zero
  // (Boolean products only; 1 when every tile is summed by one CTA)
  int32_t ksplit, kchunk;
  int* err;                   // device error word: set when a bounded wait runs out
  uint32_t* counts;           // when not null: the sums themselves, [nbatch][M][N]
                              // (counting semiring), and C is not written
};
void mma_plan(MmaDesc& d);    // BN, Nw and the tile counts from M, N, K, nbatch
int64_t mma_ctas(const MmaDesc& d);
bool mma_wants_occ(const MmaDesc& d);      // occupancy bitmaps for this problem?
int64_t mma_occ_blocks(const MmaDesc& d);  // their bytes, and the blocks that write them
// Independent problems in one launch, or two when some want occupancy bitmaps
// (occ_grid > 0): descriptors, CTA offsets and bitmap block offsets (nprob + 1
// entries each; no blocks for problems without) on the device.
cudaError_t launch_mma(const MmaDesc* d_descs, const int64_t* d_cta0, const int64_t* d_occ0, int nprob,
                       int64_t grid, int64_t occ_grid, cudaStream_t s);
// out[i] = in[src(i)] for a row-major array whose axes are a permutation of
// the input's: out axis a has extent d_ext[a] and steps d_stride[a] elements
// of the input (one thread per output element; d_ext and d_stride are DEVICE
// arrays of ndim entries).
void launch_permute_u32(const uint32_t* in, uint32_t* out, int ndim, const int64_t* d_ext,
                        const int64_t* d_stride, int64_t total, cudaStream_t s);
// Throughput probe `which` (0: 32-bit LOP3, 1: shared-memory load bytes,
// 2: FP32 FMA flops, 3: FP64 mul + add flops) over every SM: operations per
// second, per SM per cycle, and the SM clock it ran at.
cudaError_t run_probe(int which, int sms, cudaStream_t s, double* per_s, double* per_clk_sm,
                      double* clock_hz);
// Random bit rows of the given density (autotuning inputs); padding stays zero.
void launch_random_bits(uint64_t* w, int64_t nwords, int64_t row_words, int64_t valid,
                        double density, uint64_t seed, cudaStream_t s);

// *out += number of set bits in w[0..nwords) (padding bits are zero)
void launch_popcount(const uint64_t* w, int64_t nwords, unsigned long long* out, cudaStream_t s);
// One bounded mbarrier wait that nothing completes (sets *err after limit_ns).
cudaError_t launch_wait_selftest(int* err, long long limit_ns, cudaStream_t s);

// ----------------------------------------------------------- host helpers
int64_t coeff_count(int n, int degree);
// graded lex rank of every monomial in nest order (host)
std::vector<int64_t> nest_order(int n, int degree);
// A valid tolerance: (1 + 2^-30) sum_p S_p delta_p width, width = 1/2 for the
// centre rule (a pixel's points lie within delta_p / 2 of its centre) and 1
// for the corner rule.
double valid_tolerance(int n, int degree, const double* coeffs, const double* lo,
                       const double* hi, const int32_t* res, double width);

}  // namespace pa
