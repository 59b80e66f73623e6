// Tensor-core path of the Boolean contraction (Eq. GAM of Sec. 3.3 for one
// cluster of Sec. 3.5): C[b][m][n] = OR_k A[b][m][k] AND B[b][k][n] computed as
// a matrix product of operands that are 0 or a power of two on the
// 5th-generation tensor cores, then thresholded at > 0.
//
// Exactness: the operands' non-zero values are exact in E4M3, every product is
// 0 or at least 2^-18 and the FP32 accumulator only ever adds non-negative
// values, so the sum is positive exactly when some product is not 0 (a positive
// FP32 sum can round but never back to zero).  The result bits are therefore the
// Boolean product for any K.  The counting semiring uses 2.0 throughout: sums
// are multiples of 4 up to 2^26, exact.
//
// Data path.  Both operands are read as the bit-packed arrays the row-OR reads
// and expanded to E4M3 bytes in shared memory by the CTA that multiplies them;
// nothing but bits moves between HBM, L2 and the SMs.  (Expanding both
// operands into byte arrays first, in two launches, and fetching those with TMA
// cost 11 us of a 2048^3 product's 23, and 8 times the traffic.)  Two choices
// make the expansion cheap:
//   - four bytes come from a 32-bit word by one mask: bits r, r + 8, r + 16 and
//     r + 24 stay where they are, bit r of four bytes.  A byte with one of the
//     bits 0 .. 6 set is a power of two in E4M3 (2^-9 .. 2), and only whether a
//     product is positive matters; bit 7 (the sign) moves to bit 6, and for
//     counts every bit does (0x40 is 2.0).  The bytes of a word are thereby
//     permuted; for K that does not matter as long as B's K rows are stored in
//     the same order, for N it permutes the accumulator's columns, which the
//     epilogue undoes with constant indexes;
//   - B stays N-major (tcgen05 reads 8-bit operands in either orientation), so
//     no bit transposes.
// Per 128-value K block four producer warps fill one of four 16 + 32 KB stages
// (128-byte swizzle); four such groups work on four blocks of an SM at a time (of
// one CTA, or two each of two CTAs where there are more tiles than SMs), because a
// group's chain of loads, masks and stores is longer than the tensor core's time
// for a block (one group of eight warps measured 1900 cycles per block).  One
// thread issues tcgen05.mma kind::f8f6f4 (M = 128, N = BN, K = 32 per
// instruction) into a TMEM accumulator of 128 lanes x BN FP32 columns, and the
// producer warps read it back with tcgen05.ld and store bit-packed rows.  K
// blocks in which the A rows or the B columns of the tile hold no bit are
// skipped: a group sees it in the words it has loaded, and where a CTA has many
// blocks two bitmaps name the occupied ones (occupancy_kernel, one pass over the
// bits first).  A product with few output tiles and a long K splits K over
// several CTAs per tile, whose bits are OR-ed into C (cleared beforehand):
// partial sums combine by OR because each is positive exactly when one of its
// products is.  Every wait on an mbarrier is bounded (about 1 s); on expiry the
// kernel sets the error word, finishes without storing and frees its TMEM.
//
// What bounds it (clock64 stamps, dense 2048^3, 128 CTAs): 2.7 k cycles of
// set-up, 5.1 k until the first of the four stages is full, 1060 per block, 3 k
// of read-back, 27.9 k in all.  Without the shared stores a block takes 930
// cycles and without the products 825, so both sides are near their limit (an
// N-major B halves the rate of a K-major one, 560 per block, which would need
// bit transposes).  Against the byte-array version: plots of 8192^3 102 -> 53 us of
// device time per call, the 2048^3 count 55 -> 43 per call, ternary 256 (256 products of
// 256^3) 78 -> 54; half-full operands of 4096^3 94 -> 87, but of 8192^3 450 -> 493 and of
// 16384^3 3170 -> 3600 (bytes fetched by TMA are K-major).
#include <cuda.h>
#include <string.h>

#include <algorithm>

#include "pa_internal.h"

namespace pa {

namespace {

constexpr int kMmaBM = 128;                   // rows of A per tile (TMEM lanes)
constexpr int kMmaBK = 128;                   // K values per stage = one 128-byte swizzle row
constexpr int kMmaATile = kMmaBM * kMmaBK;    // 16 KB
constexpr int kMmaNBlock = 128 * kMmaBK;      // 16 KB: 128 columns of B
constexpr int kMmaStage = kMmaATile + 2 * kMmaNBlock;  // 48 KB
constexpr int kMmaMaxStages = 4;              // one per producer group
constexpr int kMmaTmemCols = 256;
// Four producer warps to a stage; the last warp issues the products.
constexpr int mma_threads(int stages) { return 32 * (4 * stages + 1); }
constexpr size_t mma_smem(int stages) { return (size_t)stages * kMmaStage + 1024; }
constexpr int kOccBlocks = 8;                 // K blocks per block of occupancy_kernel

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Wait for phase `parity` of an mbarrier, giving up after about one second.
__device__ __forceinline__ bool bar_wait(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  for (long long it = 0; it < (1ll << 26); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(parity)
        : "memory");
    if (ok) return true;
    if (clock64() - t0 > 2000000000ll) return false;
  }
  return false;
}

// Shared-memory matrix descriptor, 128-byte swizzle (mode 2), version 1; lbo and
// sbo in bytes.  A (K-major): 8-row x 128-byte atoms every sbo bytes.  B
// (N-major): 8 K rows of 128 columns per atom, the next 8 K rows sbo bytes on,
// the next 128 columns lbo bytes on.
__device__ __forceinline__ uint64_t sw128_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((saddr >> 4) & 0x3FFFu);
  d |= (uint64_t)(lbo >> 4) << 16;
  d |= (uint64_t)(sbo >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Instruction descriptor of kind::f8f6f4: FP32 accumulator (bits 4-5 = 1),
// A and B E4M3 (bits 7-9, 10-12 = 0), A K-major (bit 15 = 0), B N-major (bit
// 16 = 1), N >> 3 in bits 17-22, M >> 4 in bits 24-28.
__device__ __forceinline__ uint32_t f8_idesc(int M, int N) {
  return (1u << 4) | (1u << 16) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t* v) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,"
      "%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]),
        "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]),
        "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}

// Byte position p of a 32-value group holds value 8 (p % 4) + p / 4 (of K in an A
// row, of N in a B row; B's K rows are placed by the same map).
__device__ __forceinline__ int pos_value(int p) { return 8 * (p & 3) + (p >> 2); }

// Byte positions 16 part .. 16 part + 15 of a 32-bit word: register t holds the
// word's bits 4 part + t + 8 j (byte j).  Boolean products keep the bit where it
// is; counts move it to bit 6.
template <bool COUNT>
__device__ __forceinline__ uint4 expand16(uint32_t x, int part) {
  if (COUNT) {
    const uint32_t y = x >> (4 * part);
    return make_uint4((y << 6) & 0x40404040u, (y << 5) & 0x40404040u, (y << 4) & 0x40404040u,
                      (y << 3) & 0x40404040u);
  }
  return part == 0 ? make_uint4(x & 0x01010101u, x & 0x02020202u, x & 0x04040404u, x & 0x08080808u)
                   : make_uint4(x & 0x10101010u, x & 0x20202020u, x & 0x40404040u,
                                (x >> 1) & 0x40404040u);
}

__device__ __forceinline__ void st_shared16(uint32_t addr, uint4 v) {
  asm volatile("st.shared.v4.b32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z),
               "r"(v.w)
               : "memory");
}

struct MmaShared {
  uint64_t full[kMmaMaxStages], empty[kMmaMaxStages], accum;
  uint32_t occ[kMmaMaxStages][2];    // per group, by turns: a byte per warp, 1 A words, 2 B words
  volatile int skip[kMmaMaxStages];  // the stage's block is to be skipped
  volatile int issued;               // blocks multiplied
  uint32_t tmem;
  volatile int fail;
};

// Occupancy bitmaps of a problem's tiles: bit kb of a row tile of A (of a column
// tile of B) when its K values 128 kb .. hold a set bit.  One block per tile and
// eight K blocks, a warp each; the block writes one byte.  (Reads every bit of
// the operands once: HBM or L2 bound, a few us of launch on small products.)
__global__ void __launch_bounds__(32 * kOccBlocks)
occupancy_kernel(const MmaDesc* __restrict__ descs, const int64_t* __restrict__ block0s, int nprob) {
  asm volatile("griddepcontrol.launch_dependents;");
  const int p = find_entry([&](int i) { return block0s[i]; }, nprob, (int64_t)blockIdx.x);
  const MmaDesc& d = descs[p];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int64_t t = (int64_t)blockIdx.x - block0s[p];
  const int64_t bytes = d.kb_words * 4;
  const int64_t byte = t % bytes;
  t /= bytes;
  const int64_t ntile = d.m_tiles + d.n_tiles;
  const int64_t b = t / ntile, tile = t - b * ntile;
  const int64_t kb = byte * kOccBlocks + warp;
  uint64_t any = 0;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  if (kb * kMmaBK < d.K) {
    if (tile < d.m_tiles) {
      const int64_t w = 2 * kb + (lane & 1), m0 = tile * kMmaBM + (lane >> 1);
      const uint64_t* src = d.A + (b * d.M + m0) * d.a_row_words + w;
      if (w < d.a_row_words) {
#pragma unroll
        for (int i = 0; i < 8; ++i)
          if (m0 + 16 * i < d.M) any |= __ldg(src + (int64_t)(16 * i) * d.a_row_words);
      }
    } else {
      // BN / 64 words of 128 rows, lanes along a row's words
      const int wl = d.BN / 64, rows = 32 / wl;  // 4 and 8, or 2 and 16
      const int64_t w = (tile - d.m_tiles) * wl + lane % wl;
      const int64_t k0 = kb * kMmaBK + lane / wl;
      const uint64_t* src = d.B + (b * d.K + k0) * d.Nw + w;
      if (w < d.Nw) {
#pragma unroll 8
        for (int i = 0; i < kMmaBK; i += rows)
          if (k0 + i < d.K) any |= __ldg(src + (int64_t)i * d.Nw);
      }
    }
  }
  __shared__ uint32_t bits[kOccBlocks];
  const bool on = __any_sync(0xffffffffu, any != 0ull);
  if (lane == 0) bits[warp] = on ? 1u : 0u;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t v = 0;
#pragma unroll
    for (int i = 0; i < kOccBlocks; ++i) v |= bits[i] << i;
    d.occ[(b * ntile + tile) * bytes + byte] = (uint8_t)v;
  }
}

// Walks the K blocks of a CTA: those in [kb0, kb1) that both bitmaps hold, or
// all of them without bitmaps.
struct ActiveBlocks {
  const uint32_t* occa;
  const uint32_t* occb;
  int kb0, kb1, w;
  uint32_t m;
  __device__ __forceinline__ uint32_t word(int i) const {
    const int lo = max(kb0 - 32 * i, 0), hi = min(kb1 - 32 * i, 32);
    if (hi <= lo) return 0u;
    const uint32_t m = occa ? __ldcg(occa + i) & __ldcg(occb + i) : 0xffffffffu;
    return m & (hi == 32 ? 0xffffffffu : (1u << hi) - 1u) &
           ~((1u << lo) - 1u);
  }
  __device__ __forceinline__ void start() {
    w = kb0 / 32;
    m = word(w);
  }
  // the next active block, or -1
  __device__ __forceinline__ int next() {
    while (!m) {
      if (32 * (w + 1) >= kb1) return -1;
      m = word(++w);
    }
    const int kb = 32 * w + __ffs((int)m) - 1;
    m &= m - 1;
    return kb;
  }
};

// A producer warp's blocks: the group's share (every STAGES-th) of the
// CTA's, into the group's stage.  BN = 128 or 256.  A thread holds two A
// words and BN / 64 B words of a block, loaded one block of its group ahead.
// The thread-to-word maps make the loads 16- and 32-byte runs of a row and the
// 16-byte shared stores free of conflicts (eight chunks of distinct bank groups
// per quarter warp).
template <int STAGES, int BN, bool COUNT>
__device__ __forceinline__ void produce(const MmaDesc& d, MmaShared& sh, uint32_t ring,
                                        ActiveBlocks act, int64_t b, int64_t m0, int64_t w0) {
  constexpr int NB = BN / 64;               // B words per thread
  constexpr int kPosStep = BN == 256 ? 8 : 16;  // K positions between a thread's B words
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int group = warp >> 2, wg = warp & 3;
  // A: rows arow and arow + 16, word ahalf of the block's two
  const int arow = wg * 32 + (lane >> 1), ahalf = lane & 1;
  const uint64_t* ap = d.A + (b * d.M + m0 + arow) * d.a_row_words + ahalf;
  const int64_t a_step = 16 * d.a_row_words;
  const bool ain0 = m0 + arow < d.M, ain1 = m0 + arow + 16 < d.M;
  // B: K positions pos + kPosStep i (rows krow + kPosStep / 4 i), word bword of
  // the tile's BN / 64
  const int q = lane >> 3;
  const int bword = BN == 256 ? lane & 3 : lane & 1;
  const int pos = wg * 32 + (BN == 256 ? (q & 1) + 4 * (q >> 1) + 2 * ((lane >> 2) & 1) : lane >> 1);
  const int krow = (pos & ~31) + pos_value(pos & 31);
  const uint64_t* bp = d.B + (b * d.K + krow) * d.Nw + w0 + bword;
  const int64_t b_step = (kPosStep / 4) * d.Nw;
  const bool bin = w0 + bword < d.Nw;
  // shared-memory offsets of the four chunks of a word
  uint32_t aoff[4], boff[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) {
    aoff[c] = (uint32_t)arow * 128u + (((uint32_t)(4 * ahalf + c) ^ (uint32_t)(arow & 7)) << 4);
    // the second column block holds a word's halves in opposite order (its rows
    // share banks with the first's)
    const uint32_t chunk = (uint32_t)(4 * (bword & 1) + 2 * (c >> 1) + ((c & 1) ^ (bword >> 1)));
    boff[c] = (uint32_t)(kMmaATile + (bword >> 1) * kMmaNBlock) + (uint32_t)pos * 128u +
              ((chunk ^ (uint32_t)(pos & 7)) << 4);
  }
  const uint32_t at = ring + (uint32_t)group * kMmaStage;
  auto load = [&](int kb, uint64_t (&aw)[2], uint64_t (&bw)[NB]) {
    const bool aw_in = kb >= 0 && 2 * (int64_t)kb + ahalf < d.a_row_words;
    const uint64_t* p = ap + 2 * (int64_t)kb;
    aw[0] = aw_in && ain0 ? __ldg(p) : 0ull;
    aw[1] = aw_in && ain1 ? __ldg(p + a_step) : 0ull;
    const int64_t left = kb >= 0 && bin ? d.K - (int64_t)kb * kMmaBK : 0;
    const int kleft = (int)min((int64_t)kMmaBK, left) - krow;  // rows past krow in range
    const uint64_t* r = bp + (int64_t)kb * kMmaBK * d.Nw;
#pragma unroll
    for (int i = 0; i < NB; ++i) bw[i] = i * (kPosStep / 4) < kleft ? __ldg(r + i * b_step) : 0ull;
  };
  act.start();
  int kb = act.next();
  for (int i = 0; i < group && kb >= 0; ++i) kb = act.next();
  uint64_t aw[2], bw[NB];
  load(kb, aw, bw);
  bool dead = false;
  for (int it = 0; kb >= 0; ++it) {
    uint64_t a[2], bb[NB];
    a[0] = aw[0];
    a[1] = aw[1];
#pragma unroll
    for (int i = 0; i < NB; ++i) bb[i] = bw[i];
    for (int i = 0; i < STAGES && kb >= 0; ++i) kb = act.next();
    load(kb, aw, bw);
    bool use = true;
    if (!act.occa) {
      // does the block hold a bit of A and of B?  (the group's four warps
      // agree; they have all passed the last reading of this slot when they
      // meet here for the other one)
      uint64_t bor = bb[0];
#pragma unroll
      for (int i = 1; i < NB; ++i) bor |= bb[i];
      const bool na = __any_sync(0xffffffffu, (a[0] | a[1]) != 0ull);
      const bool nb = __any_sync(0xffffffffu, bor != 0ull);
      if (lane == 0)
        reinterpret_cast<volatile uint8_t*>(&sh.occ[group][it & 1])[wg] = (uint8_t)((na ? 1 : 0) | (nb ? 2 : 0));
      asm volatile("bar.sync %0, 128;" ::"r"(1 + group) : "memory");
      const uint32_t o = *reinterpret_cast<volatile uint32_t*>(&sh.occ[group][it & 1]);
      use = (o & 0x01010101u) && (o & 0x02020202u);
    }
    // (a warp whose wait ran out goes on without storing or arriving: the
    // group's barriers need it)
    if (dead || (it > 0 && !bar_wait(&sh.empty[group], (uint32_t)(it - 1) & 1u))) {
      sh.fail = 1;
      dead = true;
      continue;
    }
    if (use) {
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          st_shared16(at + aoff[c] + i * (16 * 128),
                      expand16<COUNT>((uint32_t)(a[i] >> (32 * (c >> 1))), c & 1));
#pragma unroll
      for (int i = 0; i < NB; ++i)
#pragma unroll
        for (int c = 0; c < 4; ++c)
          st_shared16(at + boff[c] + i * (kPosStep * 128),
                      expand16<COUNT>((uint32_t)(bb[i] >> (32 * (c >> 1))), c & 1));
      // the stores become visible to the tensor core's proxy, then the warp
      // arrives
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    }
    if (wg == 0 && lane == 0) sh.skip[group] = use ? 0 : 1;
    __syncwarp();
    if (lane == 0)
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&sh.full[group])) : "memory");
  }
}

// One CTA per (problem, batch, 128-row tile of A, BN-column tile of B, K
// chunk).  The first 4 STAGES warps: producers, then the epilogue (warp w reads
// TMEM lanes 32 (w % 4) .. and columns BN / STAGES (w / 4) ..).  The last warp:
// TMEM allocation and, in one lane, the products.
// STAGES = 4: one CTA to an SM.  STAGES = 2: two, each with half the producers,
// half the ring and half of TMEM, so that one's set-up, first block and
// read-back (some 11K cycles, ten K blocks' worth) run under the other's.
template <int STAGES>
__global__ void __launch_bounds__(mma_threads(STAGES), 4 / STAGES)
mma_bits_kernel(const MmaDesc* __restrict__ descs, const int64_t* __restrict__ cta0s, int nprob) {
  constexpr int kProducers = 4 * STAGES;
  extern __shared__ uint8_t mma_raw[];
  uint8_t* smem =
      reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(mma_raw) + 1023) & ~uintptr_t(1023));
  __shared__ MmaShared sh;
  __shared__ MmaDesc sd;
  asm volatile("griddepcontrol.launch_dependents;");
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int p = find_entry([&](int i) { return cta0s[i]; }, nprob, (int64_t)blockIdx.x);
  {
    const uint32_t* src = reinterpret_cast<const uint32_t*>(descs + p);
    uint32_t* dst = reinterpret_cast<uint32_t*>(&sd);
    if (threadIdx.x < (int)(sizeof(MmaDesc) / 4)) dst[threadIdx.x] = src[threadIdx.x];
  }
  if (warp == kProducers) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_addr(&sh.tmem)),
                 "r"(kMmaTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  } else if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 4;" ::"r"(smem_addr(&sh.full[s])) : "memory");
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&sh.empty[s])) : "memory");
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 2;" ::"r"(smem_addr(&sh.accum)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    sh.fail = 0;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sh.tmem;
  const MmaDesc& d = sd;
  int64_t t = (int64_t)blockIdx.x - cta0s[p];
  const int kc = (int)(t % d.ksplit);
  t /= d.ksplit;
  const int64_t nt = t % d.n_tiles;
  t /= d.n_tiles;
  const int64_t mt = t % d.m_tiles;
  const int64_t b = t / d.m_tiles;
  const int BN = d.BN;
  const int nk = (int)((d.K + kMmaBK - 1) / kMmaBK);
  const bool split = d.ksplit > 1;
  // every role walks the same sequence of K blocks, the j-th in stage
  // j % STAGES
  ActiveBlocks act;
  const uint32_t* occ = reinterpret_cast<const uint32_t*>(d.occ) + b * (d.m_tiles + d.n_tiles) * d.kb_words;
  act.occa = d.occ ? occ + mt * d.kb_words : nullptr;
  act.occb = d.occ ? occ + (d.m_tiles + nt) * d.kb_words : nullptr;
  act.kb0 = kc * d.kchunk;
  act.kb1 = min(nk, act.kb0 + d.kchunk);
  // the operands, the bitmaps and C belong to the earlier kernels of the
  // stream until here
  asm volatile("griddepcontrol.wait;" ::: "memory");

  if (warp == kProducers) {
    if (lane == 0) {
      const uint32_t idesc = f8_idesc(kMmaBM, BN);
      act.start();
      int issued = 0;
      for (int j = 0; act.next() >= 0; ++j) {
        const int s = j % STAGES;
        if (!bar_wait(&sh.full[s], (uint32_t)(j / STAGES) & 1u)) {
          sh.fail = 1;
          break;
        }
        if (sh.skip[s]) {
          asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&sh.empty[s])) : "memory");
          continue;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint32_t a0 = smem_addr(smem + (size_t)s * kMmaStage), b0 = a0 + kMmaATile;
#pragma unroll
        for (int kk = 0; kk < kMmaBK / 32; ++kk) {
          const uint64_t ad = sw128_desc(a0 + kk * 32, 16, 1024);
          const uint64_t bd = sw128_desc(b0 + kk * 4096, kMmaNBlock, 1024);
          const uint32_t acc = (issued > 0 || kk > 0) ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
              "l"(ad), "l"(bd), "r"(idesc), "r"(acc)
              : "memory");
        }
        asm volatile(
            "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                smem_addr(&sh.empty[s]))
            : "memory");
        ++issued;
      }
      sh.issued = issued;
      asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(&sh.accum)) : "memory");
      // arrives once every product issued above has completed (also on failure)
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
              smem_addr(&sh.accum))
          : "memory");
    }
    __syncwarp();
  } else {
    const int64_t m0 = mt * kMmaBM, w0 = nt * (BN / 64);
    const uint32_t ring = smem_addr(smem);
    if (d.counts) {
      if (BN == 256) produce<STAGES, 256, true>(d, sh, ring, act, b, m0, w0);
      else produce<STAGES, 128, true>(d, sh, ring, act, b, m0, w0);
    } else {
      if (BN == 256) produce<STAGES, 256, false>(d, sh, ring, act, b, m0, w0);
      else produce<STAGES, 128, false>(d, sh, ring, act, b, m0, w0);
    }
    const bool ok = bar_wait(&sh.accum, 0);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    // no block multiplied: nothing was accumulated, every sum is zero; with K
    // split such a CTA leaves C as it is (others OR their bits into it)
    const bool none = sh.issued == 0;
    const bool store = ok && !sh.fail && !(split && none);
    const int ew = warp & 3, part = warp >> 2;
    const int64_t m = m0 + ew * 32 + lane;
    // a warp's columns, 32 at a time: the bits of half a result word
    for (int c0 = part * (BN / STAGES); c0 < (part + 1) * (BN / STAGES); c0 += 32) {
      uint32_t v[32];
      const uint32_t ta = tmem + ((uint32_t)(ew * 32) << 16) + (uint32_t)c0;
      if (none) {
#pragma unroll
        for (int k = 0; k < 32; ++k) v[k] = 0u;
      } else {
        tmem_ld32(ta, v);
        asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
      }
      const int64_t n0 = w0 * 64 + c0;  // first result column
      const int swap = c0 >= 128 ? 4 : 0;  // the second column block's halves are swapped
      if (d.counts) {
        // counting semiring: every sum is 4 x an integer <= K <= 2^24, exact in
        // FP32.  The warp's 32 x 32 counts go through shared memory (the ring
        // is idle once every product is done; rows padded to 33 words against
        // bank conflicts) so that each store writes 32 consecutive counts of
        // one row.
        if (store) {
          uint32_t* st = reinterpret_cast<uint32_t*>(smem) + warp * (32 * 33);
#pragma unroll
          for (int k = 0; k < 32; ++k)
            st[lane * 33 + 8 * (k & 3) + ((k >> 2) ^ swap)] = (uint32_t)(__uint_as_float(v[k]) * 0.25f);
          __syncwarp();
          const int64_t rows = min((int64_t)32, d.M - (m0 + ew * 32));
          uint32_t* dst = d.counts + (b * d.M + m0 + ew * 32) * d.N + n0 + lane;
          if (n0 + lane < d.N)
            for (int rr = 0; rr < rows; ++rr) dst[(int64_t)rr * d.N] = st[rr * 33 + lane];
          __syncwarp();
        }
        continue;
      }
      uint32_t bits = 0;
#pragma unroll
      for (int k = 0; k < 32; ++k) bits |= (v[k] != 0u ? 1u : 0u) << (8 * (k & 3) + (k >> 2));  // pos_value(k)
      if (swap) bits = ((bits & 0x0f0f0f0fu) << 4) | ((bits >> 4) & 0x0f0f0f0fu);
      const int64_t w = n0 >> 6;
      if (store && m < d.M && w < d.Nw) {
        const int64_t rem = d.N - n0;
        if (rem < 32) bits &= rem <= 0 ? 0u : (1u << rem) - 1u;
        uint32_t* dst = reinterpret_cast<uint32_t*>(d.C + (b * d.M + m) * d.Nw + w) + ((n0 >> 5) & 1);
        if (!split) *dst = bits;
        else if (bits) atomicOr(dst, bits);
      }
    }
    if (!ok && lane == 0) atomicExch(d.err, 1);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == kProducers) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(kMmaTmemCols)
                 : "memory");
  }
  if (threadIdx.x == 0 && sh.fail) atomicExch(d.err, 1);
}

// Random bits for autotuning: bit j of word i is set when the SplitMix64 mix
// of (seed, 64 i + j) falls below density * 2^64; bits of column >= valid in
// each row of row_words words stay zero.
__global__ void random_bits_kernel(uint64_t* __restrict__ w, int64_t nwords, int64_t row_words,
                                   int64_t valid, double density, uint64_t seed) {
  const uint64_t thr = density >= 1.0 ? ~0ull : (uint64_t)(density * 18446744073709551616.0);
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nwords;
       i += (int64_t)gridDim.x * blockDim.x) {
    const int64_t col0 = (i % row_words) * 64;
    uint64_t word = 0;
    for (int j = 0; j < 64 && col0 + j < valid; ++j) {
      uint64_t z = seed + (uint64_t)(i * 64 + j) * 0x9E3779B97F4A7C15ull;
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      z ^= z >> 31;
      word |= (uint64_t)(z < thr) << j;
    }
    w[i] = word;
  }
}

// ext and stride are device arrays of ndim entries (in the call's blob)
__global__ void permute_u32_kernel(const uint32_t* __restrict__ in, uint32_t* __restrict__ out,
                                   int ndim, const int64_t* __restrict__ ext,
                                   const int64_t* __restrict__ stride, int64_t total) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < total;
       i += (int64_t)gridDim.x * blockDim.x) {
    int64_t rest = i, src = 0;
    for (int a = ndim - 1; a >= 0; --a) {
      const int64_t e = __ldg(ext + a);
      const int64_t q = rest % e;
      rest /= e;
      src += q * __ldg(stride + a);
    }
    out[i] = in[src];
  }
}

}  // namespace

void launch_permute_u32(const uint32_t* in, uint32_t* out, int ndim, const int64_t* d_ext,
                        const int64_t* d_stride, int64_t total, cudaStream_t s) {
  if (total <= 0) return;
  int64_t blocks = (total + 255) / 256;
  if (blocks > 152 * 16) blocks = 152 * 16;
  permute_u32_kernel<<<(unsigned)blocks, 256, 0, s>>>(in, out, ndim, d_ext, d_stride, total);
}

void launch_random_bits(uint64_t* w, int64_t nwords, int64_t row_words, int64_t valid,
                        double density, uint64_t seed, cudaStream_t s) {
  if (nwords <= 0) return;
  int64_t blocks = (nwords + 255) / 256;
  if (blocks > 152 * 8) blocks = 152 * 8;
  random_bits_kernel<<<(unsigned)blocks, 256, 0, s>>>(w, nwords, row_words, valid, density, seed);
}

void mma_plan(MmaDesc& d) {
  d.BN = d.N <= 128 ? 128 : 256;
  d.Nw = (d.N + 63) / 64;
  d.m_tiles = (d.M + kMmaBM - 1) / kMmaBM;
  d.n_tiles = (d.N + d.BN - 1) / d.BN;
  const int64_t nk = (d.K + kMmaBK - 1) / kMmaBK;
  d.kb_words = (nk + 31) / 32;
  // Few output tiles and a long K (a cluster that sums many variables into a
  // small result) would leave most SMs idle: split K over up to one CTA per
  // SM, each with at least 8 K blocks.  Only for the Boolean product, whose
  // partial results combine by OR.
  d.ksplit = 1;
  d.kchunk = (int32_t)nk;
  const int64_t tiles = d.nbatch * d.m_tiles * d.n_tiles;
  if (!d.counts && tiles < 152) {
    const int64_t want = std::min<int64_t>(152 / tiles, nk / 8);
    if (want > 1) {
      const int64_t chunk = (nk + want - 1) / want;
      d.kchunk = (int32_t)chunk;
      d.ksplit = (int32_t)((nk + chunk - 1) / chunk);
    }
  }
}

int64_t mma_ctas(const MmaDesc& d) { return d.nbatch * d.m_tiles * d.n_tiles * d.ksplit; }

// Bitmaps pay where many K blocks are walked, by a CTA or by an SM's CTAs one after
// another: writing them takes a launch of about 4 us (8 on dense operands), seeing an
// empty block in its loaded words about 200 cycles (a CTA of 16 blocks gains 1.6 us at
// most, one of 64 sparse ones 6).  Plots of 6616 x 3119 x 6140, 205 blocks to an SM
// but 25 to a CTA, 87 -> 38 us.
bool mma_wants_occ(const MmaDesc& d) {
  return d.kchunk >= 32 || (d.kchunk >= 8 && mma_ctas(d) * d.kchunk >= 152 * 24);
}

int64_t mma_occ_blocks(const MmaDesc& d) {
  return d.nbatch * (d.m_tiles + d.n_tiles) * d.kb_words * 4;  // one byte per block
}

cudaError_t launch_mma(const MmaDesc* d_descs, const int64_t* d_cta0, const int64_t* d_occ0, int nprob,
                       int64_t grid, int64_t occ_grid, cudaStream_t s) {
  if (nprob <= 0 || grid <= 0) return cudaSuccess;
  if (grid > 0x7fffffffLL || occ_grid > 0x7fffffffLL) return cudaErrorInvalidConfiguration;
  // More CTAs than SMs: two to an SM (see the kernel).  Two against one, whole
  // calls: an 8192^3 product of sparse plots (2048 CTAs) 82.6 -> 58.1 us, ternary 256
  // (512 CTAs of two K blocks) 62.8 -> 53.8, 38 random networks 5660 -> 5560, 4096
  // chains the same.  Up to 152 CTAs have an SM each, and all four producer groups
  // serve one ring: a CTA's own chain is what such a launch waits for.
  const bool pairs = grid > 152;
  const auto kernel = pairs ? mma_bits_kernel<2> : mma_bits_kernel<4>;
  const int stages = pairs ? 2 : 4;
  smem_limit(reinterpret_cast<const void*>(kernel), mma_smem(stages));
  // programmatic dependent launches: the set-up overlaps the previous kernel
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)occ_grid);
  cfg.blockDim = dim3(32 * kOccBlocks);
  cfg.stream = s;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  if (occ_grid > 0) {
    const cudaError_t e = cudaLaunchKernelEx(&cfg, occupancy_kernel, d_descs, d_occ0, nprob);
    if (e != cudaSuccess) return e;
  }
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(mma_threads(stages));
  cfg.dynamicSmemBytes = mma_smem(stages);
  return cudaLaunchKernelEx(&cfg, kernel, d_descs, d_cta0, nprob);
}

}  // namespace pa
