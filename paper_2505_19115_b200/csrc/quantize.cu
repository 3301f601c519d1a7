// NVFP4 quantizer kernels (Section 3 and Eq. 4-6 of the paper): block amax -> E4M3 scale ->
// E2M1 codes with round-to-nearest or Philox stochastic rounding, along the contiguous axis
// (row kernel) or along the row axis with a transposed output (transposed kernel), plus the
// per-tensor amax scale.  All kernels are HBM-bound streaming kernels.
#include <cuda_bf16.h>

#include <algorithm>
#include <type_traits>

#include "quantize_core.cuh"

namespace nvfp4 {

namespace {

// -------------------------------------------------------------------------------------------------
// Row quantizer: CTA tile = 128 rows x 32 blocks (512 columns); warp w takes rows w, w+8, ...;
// lane = block within the row segment, so a warp reads 1 KB (bf16) of one row per step (one
// 256-bit load per lane when rows are 32-byte aligned) and writes 256 contiguous code bytes.
// Several rows are in flight per thread, kept packed.  Swizzled scales are staged in shared
// memory and leave as eight contiguous 512-byte tiles.
// -------------------------------------------------------------------------------------------------
constexpr int kRowTileRows = 128;
constexpr int kSfChunkPitch = 528;  // 512 + 16: spreads the eight k-tiles over different banks

// MX = true is the MXFP4 variant (Section 3, Table 1): blocks of 32 with an E8M0 scale rounded up to a
// power of two.  A lane still encodes 16 values; the two lanes of a block share their amax by a shuffle
// and the even lane stores the scale.
template <typename T, bool SR, bool SWZ, bool MX = false>
__global__ void __launch_bounds__(kThreads, 3) quantize_row_kernel(const QuantParams p) {
  __shared__ __align__(16) uint8_t sf_s[SWZ ? 8 * kSfChunkPitch : 16];
  __shared__ float inv_table[MX ? 256 : 128];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t kb = (int64_t)blockIdx.x * 32 + lane;
  // Row tiles from the last to the first: an amax pass that ran just before left the end of the tensor in the level-two cache.
  const int64_t row_tile = gridDim.y - 1 - blockIdx.y, row0 = row_tile * kRowTileRows;
  const bool kb_ok = kb < p.nkb;
  grid_dependency_wait();
  grid_dependency_trigger();
  const float g = load_scale(p.gptr);
  const float c = __fdiv_rn(__fdiv_rn(1.0f, 6.0f), g);
  const T* x = static_cast<const T*>(p.x);
  const bool aligned32 = ((reinterpret_cast<uintptr_t>(x) | (uintptr_t)(p.ld * (int64_t)sizeof(T))) & 31u) == 0;
  // scale position of this lane inside the CTA's 128-row x 32-group tile
  const int sf_chunk = MX ? (lane >> 3) : (lane >> 2);        // k-tile within the CTA tile
  const int sf_byte = MX ? ((lane >> 1) & 3) : (lane & 3);
  const bool sf_owner = MX ? ((lane & 1) == 0) : true;
  constexpr int kTilesPerCta = MX ? 4 : 8;

  if constexpr (MX) build_inv_table_mx(inv_table, g); else build_inv_table(inv_table, g);
  if constexpr (SWZ) {
    for (int i = threadIdx.x; i < 8 * kSfChunkPitch / 16; i += kThreads)
      reinterpret_cast<uint4*>(sf_s)[i] = make_uint4(0, 0, 0, 0);
  }
  __syncthreads();

  constexpr int U = (sizeof(T) == 2) ? 4 : 2;  // rows in flight per thread (32 packed registers)
  // A CTA whose 128 x 512 tile lies wholly inside the tensor (all of them but the last row and column of the grid)
  // runs the loop without any per-row or per-block predicate.
  const bool full_tile = row0 + kRowTileRows <= p.rows && ((int64_t)blockIdx.x + 1) * 32 <= p.nkb;
  auto sweep = [&](auto full_c) {
  constexpr bool FULL = decltype(full_c)::value;
#pragma unroll 1
  for (int it = 0; it < kRowTileRows / 8; it += U) {
    Block16<T> raw[U];
    bool ok[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t r = row0 + warp + 8 * (it + u);
      ok[u] = FULL || (kb_ok && r < p.rows);
      if (ok[u]) raw[u].load(x + r * p.ld + kb * 16, aligned32);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int rl = warp + 8 * (it + u);
      const int64_t r = row0 + rl;
      float v[16];
      float amax = 0.0f;
      if (ok[u]) amax = raw[u].unpack(v);
      if constexpr (MX) amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, 1));   // Kq % 32 == 0: both lanes valid or neither
      if (!ok[u]) continue;
      uint32_t lo, hi, sf;
      if constexpr (MX) {
        sf = e8m0_encode_up(__fmul_rn(amax, c));
        encode_codes<SR>(v, inv_table[sf], p.rng, (uint64_t)(r * p.nkb + kb), lo, hi);
      } else {
        encode_block<SR>(v, amax, c, inv_table, p.rng, (uint64_t)(r * p.nkb + kb), lo, hi, sf);
      }
      *reinterpret_cast<uint2*>(p.codes + (r * p.nkb + kb) * 8) = make_uint2(lo, hi);
      if (sf_owner) {
        if constexpr (SWZ) {
          sf_s[sf_chunk * kSfChunkPitch + (rl & 31) * 16 + (rl >> 5) * 4 + sf_byte] = (uint8_t)sf;
        } else {
          p.scales[r * p.nsb + (MX ? (kb >> 1) : kb)] = (uint8_t)sf;
        }
      }
    }
  }
  };
  if (full_tile) sweep(std::true_type{}); else sweep(std::false_type{});

  if constexpr (SWZ) {
    __syncthreads();
    const int q = threadIdx.x >> 5, i = threadIdx.x & 31;
    const int64_t kt = (int64_t)blockIdx.x * kTilesPerCta + q;
    if (q < kTilesPerCta && kt < p.k_tiles) {
      const uint4 val = *reinterpret_cast<const uint4*>(sf_s + q * kSfChunkPitch + i * 16);
      *reinterpret_cast<uint4*>(p.scales + (row_tile * p.k_tiles + kt) * 512 + i * 16) = val;
    }
  }
}

// -------------------------------------------------------------------------------------------------
// Transposed quantizer: blocks run along the row axis of x[rows, cols]; the output is stored as
// [cols, rows/2] codes and [cols, rows/16] scales.  A CTA stages a (TILE_R rows x 64 cols) tile
// in shared memory with 16-byte async copies (zero-filled outside the tensor), every thread
// quantizes column pairs from it, and codes/scales leave through a second staging buffer so
// that global stores run along the output's contiguous axis.
// -------------------------------------------------------------------------------------------------
constexpr int kTCols = 64;

__device__ __forceinline__ void cp_async16_zfill(void* smem_dst, const void* gsrc, int src_bytes) {
  const uint32_t dst = (uint32_t)__cvta_generic_to_shared(smem_dst);
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(gsrc), "r"(src_bytes) : "memory");
}

template <typename T>
struct TTile {
  static constexpr int kRows = (sizeof(T) == 2) ? 256 : 128;          // 32 KB of input per tile
  static constexpr int kRowBlocks = kRows / 16;                        // 16 or 8
  static constexpr int kCodePitch = kRows / 2 + 8;                     // bytes per staged output row
  static constexpr int kChunksPerRow = kTCols * (int)sizeof(T) / 16;   // 8 or 16
};

template <typename T, bool SR, bool SWZ>
__global__ void __launch_bounds__(kThreads, 3) quantize_transposed_kernel(const QuantParams p) {
  using TT = TTile<T>;
  extern __shared__ __align__(16) uint8_t smem[];
  T* tile = reinterpret_cast<T*>(smem);                                        // [kRows][64]
  uint8_t* code_s = smem + TT::kRows * kTCols * sizeof(T);                     // [64][kCodePitch]
  uint8_t* sf_s = code_s + kTCols * TT::kCodePitch;                            // [64][kRowBlocks]

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t c0 = (int64_t)blockIdx.x * kTCols;
  const int64_t r0 = (int64_t)blockIdx.y * TT::kRows;
  const T* x = static_cast<const T*>(p.x);
  grid_dependency_wait();
  grid_dependency_trigger();
  const float g = load_scale(p.gptr);
  const float c = __fdiv_rn(__fdiv_rn(1.0f, 6.0f), g);
  __shared__ float inv_table[128];
  build_inv_table(inv_table, g);                              // published by the barrier after the tile lands

  // ---- stage the input tile ----
  constexpr int kElemsPerChunk = 16 / (int)sizeof(T);
  constexpr int kChunks = TT::kRows * TT::kChunksPerRow;
#pragma unroll
  for (int i = 0; i < kChunks / kThreads; ++i) {
    const int id = threadIdx.x + i * kThreads;
    const int row = id / TT::kChunksPerRow, ch = id % TT::kChunksPerRow;
    const int64_t gr = r0 + row, gc = c0 + (int64_t)ch * kElemsPerChunk;
    int64_t valid = (gr < p.rows) ? (p.cols - gc) : 0;
    valid = valid < 0 ? 0 : (valid > kElemsPerChunk ? kElemsPerChunk : valid);
    const T* src = (valid > 0) ? (x + gr * p.ld + gc) : x;
    cp_async16_zfill(tile + row * kTCols + ch * kElemsPerChunk, src, (int)valid * (int)sizeof(T));
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();

  // ---- quantize: lane -> columns (2*lane, 2*lane+1), warp -> row blocks ----
  // Staging rows are ordered even columns first (column cl -> row (cl & 1) * 32 + cl / 2), so that a
  // warp's 8-byte code stores and its scale bytes fall into distinct banks.
#pragma unroll 1
  for (int rb = warp; rb < TT::kRowBlocks; rb += kThreads / 32) {
    float va[16], vb[16], amax_a, amax_b;
    if constexpr (sizeof(T) == 2) {
      uint32_t w[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) w[j] = *reinterpret_cast<const uint32_t*>(tile + (rb * 16 + j) * kTCols + 2 * lane);
      uint32_t m[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) m[j] = absmax_bf16x2(w[2 * j], w[2 * j + 1]);
#pragma unroll
      for (int j = 0; j < 4; ++j) m[j] = absmax_bf16x2(m[2 * j], m[2 * j + 1]);
      const uint32_t mm = absmax_bf16x2(absmax_bf16x2(m[0], m[1]), absmax_bf16x2(m[2], m[3])) & 0x7FFF7FFFu;
      amax_a = __uint_as_float(mm << 16);                     // low halves = column 2*lane
      amax_b = __uint_as_float(mm & 0xFFFF0000u);             // high halves = column 2*lane + 1
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        va[j] = __uint_as_float(w[j] << 16);
        vb[j] = __uint_as_float(w[j] & 0xFFFF0000u);
      }
    } else {
      amax_a = amax_b = 0.0f;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float2 f = *reinterpret_cast<const float2*>(tile + (rb * 16 + j) * kTCols + 2 * lane);
        va[j] = f.x;
        vb[j] = f.y;
        amax_a = fmaxf(amax_a, fabsf(f.x));
        amax_b = fmaxf(amax_b, fabsf(f.y));
      }
    }
    const int64_t kb = r0 / 16 + rb;
    const int64_t ca = c0 + 2 * lane;
    uint32_t lo, hi, sf;
    encode_block<SR>(va, amax_a, c, inv_table, p.rng, (uint64_t)(ca * p.nkb + kb), lo, hi, sf);
    *reinterpret_cast<uint2*>(code_s + lane * TT::kCodePitch + rb * 8) = make_uint2(lo, hi);
    sf_s[rb * kTCols + lane] = (uint8_t)sf;
    encode_block<SR>(vb, amax_b, c, inv_table, p.rng, (uint64_t)((ca + 1) * p.nkb + kb), lo, hi, sf);
    *reinterpret_cast<uint2*>(code_s + (32 + lane) * TT::kCodePitch + rb * 8) = make_uint2(lo, hi);
    sf_s[rb * kTCols + 32 + lane] = (uint8_t)sf;
  }
  __syncthreads();

  // ---- codes out: 8-byte units, contiguous along the quantized row ----
  const int64_t kb0 = r0 / 16;
#pragma unroll
  for (int i = 0; i < kTCols * TT::kRowBlocks / kThreads; ++i) {
    const int id = threadIdx.x + i * kThreads;
    const int cl = id / TT::kRowBlocks, u = id % TT::kRowBlocks;
    if (c0 + cl < p.cols && kb0 + u < p.nkb) {
      const int srow = (cl & 1) * 32 + (cl >> 1);
      const uint2 val = *reinterpret_cast<const uint2*>(code_s + srow * TT::kCodePitch + u * 8);
      *reinterpret_cast<uint2*>(p.codes + ((c0 + cl) * p.nkb + kb0 + u) * 8) = val;
    }
  }
  // ---- scales out ----
  if constexpr (SWZ) {
    constexpr int kKt = TT::kRowBlocks / 4;  // k-tiles per CTA tile
    const bool fill_upper = ((c0 & 127) == 0) && (c0 + kTCols >= p.cols);  // nobody else owns rows 64..127
    for (int id = threadIdx.x; id < kTCols * kKt; id += kThreads) {
      const int cl = id / kKt, t = id % kKt;
      const int64_t kt = kb0 / 4 + t;
      if (kt >= p.k_tiles) continue;
      const int srow = (cl & 1) * 32 + (cl >> 1);
      const uint8_t* s4 = sf_s + (t * 4) * kTCols + srow;
      const uint32_t val = (uint32_t)s4[0] | ((uint32_t)s4[kTCols] << 8) | ((uint32_t)s4[2 * kTCols] << 16) |
                           ((uint32_t)s4[3 * kTCols] << 24);
      *reinterpret_cast<uint32_t*>(p.scales + sf_swizzled_offset(c0 + cl, kt * 4, p.k_tiles)) =
          scales_inside(val, c0 + cl < p.cols ? p.nkb - kt * 4 : 0);
      if (fill_upper)
        *reinterpret_cast<uint32_t*>(p.scales + sf_swizzled_offset(c0 + cl + 64, kt * 4, p.k_tiles)) = 0u;
    }
  } else {
    for (int id = threadIdx.x; id < kTCols * TT::kRowBlocks; id += kThreads) {
      const int cl = id / TT::kRowBlocks, u = id % TT::kRowBlocks;
      const int srow = (cl & 1) * 32 + (cl >> 1);
      if (c0 + cl < p.cols && kb0 + u < p.nkb) p.scales[(c0 + cl) * p.nkb + kb0 + u] = sf_s[u * kTCols + srow];
    }
  }
}

// -------------------------------------------------------------------------------------------------
// Per-tensor amax -> g = amax / (6*448)
//
// The running maximum is kept as the bit pattern of |x|: non-negative IEEE patterns order as unsigned
// integers, +Inf sits above every finite value and every NaN pattern above +Inf.  A tensor that
// holds a NaN therefore gets g = NaN, one that holds an infinity (and no NaN) g = +Inf, and every
// product computed with such a scale comes out as NaN (NaN * acc, or Inf * 0): a diverged step is
// visible in Y, dX and dW instead of being quantized into finite codes.
// -------------------------------------------------------------------------------------------------
// max |.| of two packed bf16 pairs, per half, NaN if either is (the sign bits of the result are meaningless)
__device__ __forceinline__ uint32_t absmax_nan_bf16x2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("max.NaN.xorsign.abs.bf16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}

// 32 bytes at position j, zeros past the end.
__device__ __forceinline__ void load_vec32(const uint32_t* x, int64_t j, int64_t n_vec32, uint32_t (&w)[8]) {
  if (j < n_vec32) {
    asm volatile("ld.global.L1::no_allocate.v8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
                 : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]), "=r"(w[6]), "=r"(w[7])
                 : "l"(x + j * 8));
  } else {
#pragma unroll
    for (int k = 0; k < 8; ++k) w[k] = 0u;
  }
}

// Running maximum of one thread over words of source data (bf16 pairs or fp32 values).
template <typename T>
struct AmaxBits {
  uint32_t m = 0u;
  __device__ __forceinline__ void add8(const uint32_t (&w)[8]) {
    if constexpr (sizeof(T) == 2) {
      m = absmax_nan_bf16x2(absmax_nan_bf16x2(absmax_nan_bf16x2(absmax_nan_bf16x2(w[0], w[1]), absmax_nan_bf16x2(w[2], w[3])),
                                              absmax_nan_bf16x2(absmax_nan_bf16x2(w[4], w[5]), absmax_nan_bf16x2(w[6], w[7]))),
                            m);
    } else {
#pragma unroll
      for (int k = 0; k < 8; ++k) m = max(m, w[k] & 0x7FFFFFFFu);
    }
  }
  __device__ __forceinline__ void add4(uint32_t a, uint32_t b, uint32_t c, uint32_t d) {
    if constexpr (sizeof(T) == 2) {
      m = absmax_nan_bf16x2(absmax_nan_bf16x2(absmax_nan_bf16x2(a, b), absmax_nan_bf16x2(c, d)), m);
    } else {
      m = max(max(m, a & 0x7FFFFFFFu), max(max(b & 0x7FFFFFFFu, c & 0x7FFFFFFFu), d & 0x7FFFFFFFu));
    }
  }
  // fp32 bit pattern of the maximum over the warp
  __device__ __forceinline__ uint32_t warp_bits() const {
    uint32_t bits = m;
    if constexpr (sizeof(T) == 2) {
      const uint32_t h = m & 0x7FFF7FFFu;                      // bf16 patterns widen to fp32 by a shift
      bits = max(h >> 16, h & 0xFFFFu) << 16;
    }
    return __reduce_max_sync(0xFFFFFFFFu, bits);
  }
};

// Small dense tensors: one cluster of eight blocks does it all in one launch.  The block maxima meet in the first block's
// shared memory, so no accumulator has to be zeroed before and no launch has to finish it after: three launches become one.
// A 256-token layer step 47.1 -> 42.9 us, 16 tokens through kept weights 34.1 -> 29.8.  The line lies where the eight blocks'
// own bandwidth shows: 256 x 512 2.5 -> 2.1 us, 2080 x 1056 (4.4 MB) 3.0 either way at best.
// late: wait for the kernel before this one after the loads (x is older than it), not before them.
constexpr int kSmallAmaxCluster = 8, kSmallAmaxThreads = 1024;
constexpr int64_t kSmallAmaxBytes = 2 << 20;

// The maximum of what a cluster's blocks (`block` of `blocks` on the tensor) read, in the first block's first thread.
template <typename T, int THREADS, int CLUSTER>
__device__ __forceinline__ uint32_t cluster_amax_bits(const uint32_t* x, int64_t n_vec32, int block, int blocks, int late, uint32_t rank) {
  __shared__ uint32_t warp_max[THREADS / 32];
  __shared__ uint32_t block_max[CLUSTER];                      // the first block's copy is used
  // The first block's shared memory may be written only once that block runs: every block arrives here and waits behind its
  // loads, which hide the rendezvous (256 x 512 in bf16, back to back: 1.85 -> 1.89 us).
  asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory");
  if (!late) { grid_dependency_wait(); grid_dependency_trigger(); }
  const int64_t stride = (int64_t)blocks * THREADS;
  AmaxBits<T> acc;
  for (int64_t i = (int64_t)block * THREADS + threadIdx.x; i < n_vec32; i += 4 * stride) {
    uint32_t w[4][8];
#pragma unroll
    for (int u = 0; u < 4; ++u) load_vec32(x, i + u * stride, n_vec32, w[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u) acc.add8(w[u]);
  }
  uint32_t bits = acc.warp_bits();
  if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = bits;
  __syncthreads();
  asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (threadIdx.x < 32) {
    bits = __reduce_max_sync(0xFFFFFFFFu, threadIdx.x < THREADS / 32 ? warp_max[threadIdx.x] : 0u);
    if (threadIdx.x == 0) {
      const uint32_t mine = (uint32_t)__cvta_generic_to_shared(&block_max[rank]);
      asm volatile("{\n\t.reg .b32 a;\n\tmapa.shared::cluster.u32 a, %0, 0;\n\tst.shared::cluster.u32 [a], %1;\n\t}" ::"r"(mine), "r"(bits) : "memory");
    }
  }
  if (late) { grid_dependency_wait(); grid_dependency_trigger(); }
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  uint32_t m = 0u;
  if (rank == 0 && threadIdx.x == 0) {
#pragma unroll
    for (int i = 0; i < CLUSTER; ++i) m = max(m, block_max[i]);
  }
  return m;
}
template <typename T>
__device__ __forceinline__ void amax_cluster(const uint32_t* x, int64_t n_vec32, float* g_out, int late, uint32_t rank) {
  const uint32_t m = cluster_amax_bits<T, kSmallAmaxThreads, kSmallAmaxCluster>(x, n_vec32, (int)rank, kSmallAmaxCluster, late, rank);
  if (rank == 0 && threadIdx.x == 0) *g_out = amax_to_scale(m);
}
template <typename T>
__global__ void __cluster_dims__(kSmallAmaxCluster, 1, 1) __launch_bounds__(kSmallAmaxThreads)
amax_cluster_kernel(const uint32_t* x, int64_t n_vec32, float* g_out, int late) {
  amax_cluster<T>(x, n_vec32, g_out, late, blockIdx.x);
}

// Up to three tensors in one launch: each has a cluster, or a run of blocks in proportion to its size, of its own.
struct AmaxBatch {
  struct Op {
    const uint32_t* x;
    int64_t n_vec32;
    float* g;
    unsigned int* scratch;         // two zeroed words (sweep only)
    int first_block, blocks;       // of the grid (sweep only)
  } op[3];
  int n;
};
template <typename T>
__global__ void __cluster_dims__(kSmallAmaxCluster, 1, 1) __launch_bounds__(kSmallAmaxThreads)
amax_cluster_batch_kernel(const __grid_constant__ AmaxBatch batch) {
  const AmaxBatch::Op& op = batch.op[blockIdx.x / kSmallAmaxCluster];
  amax_cluster<T>(op.x, op.n_vec32, op.g, 0, blockIdx.x % kSmallAmaxCluster);
}

// Tensors above that whose quantizer can reduce them (ScaleSource): every cluster leaves the maximum of its share in a word of
// its own, so that nothing has to be zeroed before and no ticket taken after: 2080 x 2848 with its quantizer 15.4 -> 14.0 us.
// Two blocks a cluster, one on each multiprocessor: clusters of eight do not all fit on the chip at once, and the last of them
// then run alone (16384 x 11008: 75 -> 130 us).  63 of them, 126 multiprocessors, is what a scale's slot has words for.
constexpr int kSweepCluster = 2, kSweepThreads = 1024, kSweepWords = kScaleSlotBytes / 4 - 1;
struct AmaxSweep {
  struct Op {
    const uint32_t* x;
    int64_t n_vec32;
    uint32_t* maxima;
    int first, clusters;           // of the grid
  } op[kMaxLayerOperands];
  int n;
};
template <typename T>
__global__ void __cluster_dims__(kSweepCluster, 1, 1) __launch_bounds__(kSweepThreads)
amax_sweep_kernel(const __grid_constant__ AmaxSweep p) {
  const int cluster = blockIdx.x / kSweepCluster, rank = blockIdx.x % kSweepCluster;
  const int which = (p.n > 1 && cluster >= p.op[1].first) + (p.n > 2 && cluster >= p.op[2].first);
  const AmaxSweep::Op& op = p.op[which];
  const uint32_t m = cluster_amax_bits<T, kSweepThreads, kSweepCluster>(op.x, op.n_vec32, (cluster - op.first) * kSweepCluster + rank,
                                                                        op.clusters * kSweepCluster, 0, rank);
  if (rank == 0 && threadIdx.x == 0) op.maxima[cluster - op.first] = m;
}

// Strided tensors: 16-byte loads, grid-stride.
template <typename T>
__global__ void __launch_bounds__(kThreads) amax_kernel(const T* x, int64_t rows, int64_t cols, int64_t ld,
                                                        unsigned int* out_bits) {
  constexpr int kVec = 16 / (int)sizeof(T);
  const int64_t vec_per_row = cols / kVec;
  const int64_t total = rows * vec_per_row;
  AmaxBits<T> acc;
  for (int64_t i = (int64_t)blockIdx.x * kThreads + threadIdx.x; i < total; i += (int64_t)gridDim.x * kThreads) {
    const int64_t r = i / vec_per_row, vcol = i % vec_per_row;
    const uint4 q = __ldg(reinterpret_cast<const uint4*>(x + r * ld + vcol * kVec));
    acc.add4(q.x, q.y, q.z, q.w);
  }
  const uint32_t bits = acc.warp_bits();
  grid_dependency_wait();                                      // the accumulator is zero; x is older than the kernel that zeroed it
  grid_dependency_trigger();
  if ((threadIdx.x & 31) == 0 && bits != 0u) atomicMax(out_bits, bits);
}

// Dense tensors (ld == cols, 32-byte aligned): a flat sweep with four 256-bit loads in flight per thread.
// TICKET = false: the maximum is left in out[0] for amax_finalize_kernel.
// TICKET = true: one launch does it all.  out = {running max bits, ticket}, both zero on entry; the block that
// takes the last ticket turns the maximum into g = amax / 2688 (1 for an all-zero tensor), stores it in *g_out
// and leaves the two words zero again.
// Two blocks of 512 threads per multiprocessor keep 19 MB of loads in flight, and few blocks end in few atomics on one
// word: against eight blocks of 256, 16384 x 1024 bf16 10.4 -> 8.4 us, x 4096 27.5 -> 23.7, x 11008 57.4 -> 54.6 (6.6 TB/s).
constexpr int kAmaxThreads = 512, kAmaxBlocksPerSm = 2;

template <typename T, bool TICKET>
__device__ __forceinline__ void amax_sweep(const uint32_t* x, int64_t n_vec32, unsigned int* out, float* g_out, int block, int blocks) {
  __shared__ uint32_t warp_max[kAmaxThreads / 32];
  const int64_t stride = (int64_t)blocks * kAmaxThreads;
  AmaxBits<T> acc;
  for (int64_t i = (int64_t)block * kAmaxThreads + threadIdx.x; i < n_vec32; i += 4 * stride) {
    uint32_t w[4][8];
#pragma unroll
    for (int u = 0; u < 4; ++u) load_vec32(x, i + u * stride, n_vec32, w[u]);
#pragma unroll
    for (int u = 0; u < 4; ++u) acc.add8(w[u]);
  }
  const uint32_t bits = acc.warp_bits();
  grid_dependency_wait();                                      // `out` is zero; x is older than the kernel before this one
  grid_dependency_trigger();
  if constexpr (!TICKET) {
    if ((threadIdx.x & 31) == 0 && bits != 0u) atomicMax(out, bits);
  } else {
    if ((threadIdx.x & 31) == 0) warp_max[threadIdx.x >> 5] = bits;
    __syncthreads();
    if (threadIdx.x == 0) {
      uint32_t block_bits = bits;
#pragma unroll
      for (int w = 1; w < kAmaxThreads / 32; ++w) block_bits = max(block_bits, warp_max[w]);
      if (block_bits != 0u) atomicMax(&out[0], block_bits);
      __threadfence();
      if (atomicAdd(&out[1], 1u) == (uint32_t)blocks - 1) {                // every other block's maximum is in
        __threadfence();
        *g_out = amax_to_scale(atomicExch(&out[0], 0u));
        out[1] = 0u;
      }
    }
  }
}
template <typename T, bool TICKET>
__global__ void __launch_bounds__(kAmaxThreads, kAmaxBlocksPerSm) amax_flat_kernel(const uint32_t* x, int64_t n_vec32, unsigned int* out, float* g_out) {
  amax_sweep<T, TICKET>(x, n_vec32, out, g_out, blockIdx.x, gridDim.x);
}
template <typename T>
__global__ void __launch_bounds__(kAmaxThreads, kAmaxBlocksPerSm) amax_flat_batch_kernel(const __grid_constant__ AmaxBatch batch) {
  int which = 0;
  while (which + 1 < batch.n && (int)blockIdx.x >= batch.op[which + 1].first_block) ++which;
  const AmaxBatch::Op& op = batch.op[which];
  amax_sweep<T, true>(op.x, op.n_vec32, op.scratch, op.g, (int)blockIdx.x - op.first_block, op.blocks);
}

__global__ void amax_finalize_kernel(float* out) {
  grid_dependency_wait();
  grid_dependency_trigger();
  *out = amax_to_scale(__float_as_uint(*out));
}

struct ScalePairs {
  const float* from[kMaxLayerOperands];
  float* to[kMaxLayerOperands];
};
__global__ void copy_scales_kernel(const __grid_constant__ ScalePairs p, int n) {
  grid_dependency_wait();
  grid_dependency_trigger();
  if ((int)threadIdx.x < n && p.to[threadIdx.x]) *p.to[threadIdx.x] = load_scale(p.from[threadIdx.x]);
}

__global__ void zero_words_kernel(unsigned int* words, int n) {
  grid_dependency_wait();
  grid_dependency_trigger();
  if ((int)threadIdx.x < n) words[threadIdx.x] = 0u;
}

// Dense and 32-byte aligned: what the 256-bit sweeps take.
bool amax_flat_ok(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld) {
  return ld == cols && (reinterpret_cast<uintptr_t>(x) & 31u) == 0 && (rows * cols * (dtype == NVFP4_BF16 ? 2 : 4)) % 32 == 0;
}
cudaError_t launch_amax_cluster(const void* x, int dtype, int64_t n32, float* g_out, bool late, cudaStream_t s) {
  const uint32_t* xw = static_cast<const uint32_t*>(x);
  return dtype == NVFP4_BF16
      ? launch_overlapped(amax_cluster_kernel<__nv_bfloat16>, kSmallAmaxCluster, kSmallAmaxThreads, 0, s, xw, n32, g_out, (int)late)
      : launch_overlapped(amax_cluster_kernel<float>, kSmallAmaxCluster, kSmallAmaxThreads, 0, s, xw, n32, g_out, (int)late);
}

template <typename T, bool SR, bool SWZ, bool MX = false>
cudaError_t launch_row(const QuantParams& p, cudaStream_t s) {
  dim3 grid((unsigned)ceil_div(p.nkb, 32), (unsigned)ceil_div(p.rows, kRowTileRows));
  return launch_overlapped(quantize_row_kernel<T, SR, SWZ, MX>, grid, kThreads, 0, s, p);
}

template <typename T, bool SR, bool SWZ>
cudaError_t launch_transposed(const QuantParams& p, cudaStream_t s) {
  using TT = TTile<T>;
  const size_t smem = TT::kRows * kTCols * sizeof(T) + kTCols * TT::kCodePitch + kTCols * TT::kRowBlocks;
  static DeviceFlags smem_set;   // per instantiation, per device
  if (cudaError_t e = set_max_dynamic_smem(smem_set, quantize_transposed_kernel<T, SR, SWZ>, (int)smem)) return e;
  dim3 grid((unsigned)ceil_div(p.cols, kTCols), (unsigned)ceil_div(p.rows, TT::kRows));
  return launch_overlapped(quantize_transposed_kernel<T, SR, SWZ>, grid, kThreads, smem, s, p);
}

template <typename T>
cudaError_t dispatch(const QuantParams& p, bool transposed, bool sr, bool swz, cudaStream_t s) {
  if (!transposed) {
    if (sr) return swz ? launch_row<T, true, true>(p, s) : launch_row<T, true, false>(p, s);
    return swz ? launch_row<T, false, true>(p, s) : launch_row<T, false, false>(p, s);
  }
  if (sr) return swz ? launch_transposed<T, true, true>(p, s) : launch_transposed<T, true, false>(p, s);
  return swz ? launch_transposed<T, false, true>(p, s) : launch_transposed<T, false, false>(p, s);
}

}  // namespace

}  // namespace nvfp4

using namespace nvfp4;

extern "C" size_t nvfp4_sf_bytes(int64_t Rq, int64_t Kq, int sf_layout) {
  if (Rq <= 0 || Kq <= 0 || (Kq % 16) != 0) return 0;
  if (sf_layout == NVFP4_SF_LINEAR) return (size_t)(Rq * (Kq / 16));
  if (sf_layout == NVFP4_SF_SWIZZLED_128x4) return (size_t)(ceil_div(Rq, 128) * ceil_div(Kq, 64) * 512);
  return 0;
}

extern "C" int nvfp4_quantize(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld,
                              int transposed, const float* global_scale, const nvfp4_rounding* rounding,
                              uint8_t* codes, uint8_t* scales, int sf_layout, void* cuda_stream) {
  if (!x || !rounding || !codes || !scales) return NVFP4_ERR_NULL;
  if (dtype != NVFP4_BF16 && dtype != NVFP4_FP32) return NVFP4_ERR_ENUM;
  if (transposed != 0 && transposed != 1) return NVFP4_ERR_ENUM;
  if (rounding->mode != NVFP4_RTN && rounding->mode != NVFP4_SR) return NVFP4_ERR_ENUM;
  if (rounding->reserved != 0) return NVFP4_ERR_ENUM;
  if (sf_layout != NVFP4_SF_LINEAR && sf_layout != NVFP4_SF_SWIZZLED_128x4) return NVFP4_ERR_ENUM;
  if (rows <= 0 || cols <= 0 || ld < cols) return NVFP4_ERR_SHAPE;
  const int64_t Kq = transposed ? rows : cols;
  if (Kq % 16 != 0 || cols % 8 != 0) return NVFP4_ERR_SHAPE;
  if (rows >= (int64_t)1 << 31 || cols >= (int64_t)1 << 31) return NVFP4_ERR_SHAPE;
  if (!aligned16(x) || !aligned16(codes) || !aligned16(scales) || (ld % 8) != 0) return NVFP4_ERR_ALIGN;
  if (int st = check_arch()) return st;

  QuantParams p;
  p.x = x; p.rows = rows; p.cols = cols; p.ld = ld; p.gptr = global_scale;
  philox_stream_init(&p.rng, rounding->seed, rounding->offset);
  p.codes = codes; p.scales = scales;
  p.nkb = Kq / 16; p.nsb = p.nkb; p.k_tiles = ceil_div(p.nsb, 4);
  if (ceil_div(rows, 128) > 65535) return NVFP4_ERR_SHAPE;  // grid.y limit
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  if (transposed && tile_quantizer_eligible(dtype, rows, cols, false))
    return tile_quantize(x, dtype, rows, cols, ld, global_scale, false, rounding, codes, scales, nullptr, nullptr, nullptr,
                         sf_layout, s);
  const bool sr = rounding->mode == NVFP4_SR, swz = sf_layout == NVFP4_SF_SWIZZLED_128x4;
  if (!transposed && tile_row_quantizer_eligible(dtype, rows, cols, sr))
    return tile_quantize_row(x, dtype, rows, cols, ld, global_scale, rounding, codes, scales, sf_layout, s);
  cudaError_t e = (dtype == NVFP4_BF16) ? dispatch<__nv_bfloat16>(p, transposed != 0, sr, swz, s)
                                        : dispatch<float>(p, transposed != 0, sr, swz, s);
  return e == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

extern "C" size_t nvfp4_sf_bytes_mx(int64_t Rq, int64_t Kq, int sf_layout) {
  if (Rq <= 0 || Kq <= 0 || (Kq % 32) != 0) return 0;
  if (sf_layout == NVFP4_SF_LINEAR) return (size_t)(Rq * (Kq / 32));
  if (sf_layout == NVFP4_SF_SWIZZLED_128x4) return (size_t)(ceil_div(Rq, 128) * ceil_div(Kq, 128) * 512);
  return 0;
}

extern "C" int nvfp4_quantize_mx(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, int transposed,
                                 const float* global_scale, const nvfp4_rounding* rounding,
                                 uint8_t* codes, uint8_t* scales, int sf_layout,
                                 void* workspace, size_t workspace_bytes, void* cuda_stream) {
  if (!x || !rounding || !codes || !scales) return NVFP4_ERR_NULL;
  if (dtype != NVFP4_BF16 && dtype != NVFP4_FP32) return NVFP4_ERR_ENUM;
  if (transposed != 0 && transposed != 1) return NVFP4_ERR_ENUM;
  if (transposed && dtype != NVFP4_BF16) return NVFP4_ERR_ENUM;        // the tile kernel's transposed MXFP4 form
  if ((rounding->mode != NVFP4_RTN && rounding->mode != NVFP4_SR) || rounding->reserved != 0) return NVFP4_ERR_ENUM;
  if (sf_layout != NVFP4_SF_LINEAR && sf_layout != NVFP4_SF_SWIZZLED_128x4) return NVFP4_ERR_ENUM;
  if (rows <= 0 || cols <= 0 || ld < cols || cols % 8 != 0) return NVFP4_ERR_SHAPE;
  const int64_t Rq = transposed ? cols : rows, Kq = transposed ? rows : cols;
  if (Kq % 32 != 0 || rows >= (int64_t)1 << 31 || cols >= (int64_t)1 << 31) return NVFP4_ERR_SHAPE;
  if (!aligned16(x) || !aligned16(codes) || !aligned16(scales) || (ld % 8) != 0) return NVFP4_ERR_ALIGN;
  if (ceil_div(Rq, 128) > 65535) return NVFP4_ERR_SHAPE;
  // Kq = rows is a multiple of 32: the tile kernel takes every transposed tensor but the longest, and those are refused
  const bool tile_path = transposed && tile_quantizer_eligible(dtype, rows, cols, false, /*mx=*/true);
  if (transposed && !tile_path &&
      (!workspace || workspace_bytes < (size_t)rows * cols * 2 || (reinterpret_cast<uintptr_t>(workspace) & 15u)))
    return NVFP4_ERR_WORKSPACE;
  if (int st = check_arch()) return st;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  if (tile_path)
    return tile_quantize(x, dtype, rows, cols, ld, global_scale, false, rounding, codes, scales, nullptr, nullptr, nullptr, sf_layout, s,
                         /*mx_t=*/true);
  if (!transposed && tile_row_quantizer_eligible(dtype, rows, cols, rounding->mode == NVFP4_SR, /*mx=*/true))
    return tile_quantize_row(x, dtype, rows, cols, ld, global_scale, rounding, codes, scales, sf_layout, s, /*mx=*/true);
  // what is left: large bf16 tensors rounded to nearest, and tensors of 2^31 tiles, beyond any memory
  if (transposed || dtype != NVFP4_BF16 || rounding->mode != NVFP4_RTN) return NVFP4_ERR_SHAPE;
  QuantParams p;
  p.x = x; p.rows = rows; p.cols = cols; p.ld = ld; p.gptr = global_scale;
  philox_stream_init(&p.rng, rounding->seed, rounding->offset);
  p.codes = codes; p.scales = scales;
  p.nkb = cols / 16; p.nsb = cols / 32; p.k_tiles = ceil_div(p.nsb, 4);
  using T = __nv_bfloat16;
  const cudaError_t e = sf_layout == NVFP4_SF_SWIZZLED_128x4 ? launch_row<T, false, true, true>(p, s) : launch_row<T, false, false, true>(p, s);
  return e == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

extern "C" int nvfp4_quantize_dual(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld,
                                   const float* global_scale,
                                   const nvfp4_rounding* rounding_row, uint8_t* codes_row, uint8_t* scales_row,
                                   const nvfp4_rounding* rounding_t, uint8_t* codes_t, uint8_t* scales_t,
                                   int sf_layout, void* cuda_stream) {
  if (!x || !rounding_row || !rounding_t || !codes_row || !scales_row || !codes_t || !scales_t) return NVFP4_ERR_NULL;
  if (dtype != NVFP4_BF16 && dtype != NVFP4_FP32) return NVFP4_ERR_ENUM;
  for (const nvfp4_rounding* r : {rounding_row, rounding_t})
    if ((r->mode != NVFP4_RTN && r->mode != NVFP4_SR) || r->reserved != 0) return NVFP4_ERR_ENUM;
  if (sf_layout != NVFP4_SF_LINEAR && sf_layout != NVFP4_SF_SWIZZLED_128x4) return NVFP4_ERR_ENUM;
  if (rows <= 0 || cols <= 0 || ld < cols || rows % 16 != 0 || cols % 16 != 0) return NVFP4_ERR_SHAPE;
  if (rows >= (int64_t)1 << 31 || cols >= (int64_t)1 << 31) return NVFP4_ERR_SHAPE;
  if (!aligned16(x) || !aligned16(codes_row) || !aligned16(scales_row) || !aligned16(codes_t) || !aligned16(scales_t) ||
      (ld % 8) != 0)
    return NVFP4_ERR_ALIGN;
  if (int st = check_arch()) return st;
  if (tile_quantizer_eligible(dtype, rows, cols, true))
    return tile_quantize(x, dtype, rows, cols, ld, global_scale, true, rounding_t, codes_t, scales_t, rounding_row, codes_row,
                         scales_row, sf_layout, static_cast<cudaStream_t>(cuda_stream));
  // shapes or types the tile kernel does not take: the two single-output kernels, two reads
  if (int st = nvfp4_quantize(x, dtype, rows, cols, ld, 0, global_scale, rounding_row, codes_row, scales_row, sf_layout,
                              cuda_stream))
    return st;
  return nvfp4_quantize(x, dtype, rows, cols, ld, 1, global_scale, rounding_t, codes_t, scales_t, sf_layout, cuda_stream);
}

namespace nvfp4 {
namespace {
// Per-tensor scale in one launch where the tensor allows it (dense, 32-byte aligned); `scratch_zeroed` is two
// zeroed 32-bit words in device memory that the kernel leaves zeroed.  Otherwise the three-step public path.
int tensor_amax_scale_ws(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, float* g_out,
                         unsigned int* scratch_zeroed, bool late, void* cuda_stream) {
  const int64_t total_bytes = rows * cols * (dtype == NVFP4_BF16 ? 2 : 4);
  if (!x || !g_out || !scratch_zeroed || rows <= 0 || cols <= 0 || !amax_flat_ok(x, dtype, rows, cols, ld))
    return nvfp4_tensor_amax_scale(x, dtype, rows, cols, ld, g_out, cuda_stream);
  if (dtype != NVFP4_BF16 && dtype != NVFP4_FP32) return NVFP4_ERR_ENUM;
  if (int st = check_arch()) return st;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const int64_t n32 = total_bytes / 32;
  if (total_bytes <= kSmallAmaxBytes) return launch_amax_cluster(x, dtype, n32, g_out, late, s) == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
  const int64_t fb = std::min(ceil_div(n32, (int64_t)kAmaxThreads * 4), (int64_t)sm_count() * kAmaxBlocksPerSm);
  const uint32_t* xw = static_cast<const uint32_t*>(x);
  const cudaError_t e = (dtype == NVFP4_BF16)
      ? launch_overlapped(amax_flat_kernel<__nv_bfloat16, true>, (unsigned)fb, kAmaxThreads, 0, s, xw, n32, scratch_zeroed, g_out)
      : launch_overlapped(amax_flat_kernel<float, true>, (unsigned)fb, kAmaxThreads, 0, s, xw, n32, scratch_zeroed, g_out);
  return e == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

int64_t operand_bytes(const LayerOperand& op, int dtype) { return op.rows * op.cols * (dtype == NVFP4_BF16 ? 2 : 4); }
bool needs_scratch(const LayerOperand& op, int dtype) { return operand_bytes(op, dtype) > kSmallAmaxBytes; }
cudaError_t zero_words(unsigned int* words, int n, cudaStream_t s) { return launch_overlapped(zero_words_kernel, 1, 32, 0, s, words, n); }
// Two words an operand for the passes that take a ticket, behind the first operand's scale.
unsigned int* amax_scratch(const LayerOperand* ops, int i) { return reinterpret_cast<unsigned int*>(ops[0].slot) + 16 + 2 * i; }

// One launch for the amax passes of all operands (dense, 32-byte aligned), which leaves their scales in their slots.
int amax_together(const LayerOperand* ops, int n, int dtype, cudaStream_t s) {
  AmaxBatch b = {};
  b.n = n;
  int64_t total = 0;
  bool sweep = false;
  for (int i = 0; i < n; ++i) {
    b.op[i] = {static_cast<const uint32_t*>(ops[i].x), operand_bytes(ops[i], dtype) / 32, ops[i].slot, amax_scratch(ops, i), 0, 0};
    total += b.op[i].n_vec32;
    sweep = sweep || needs_scratch(ops[i], dtype);
  }
  if (sweep && zero_words(amax_scratch(ops, 0), 2 * n, s) != cudaSuccess) return NVFP4_ERR_CUDA;
  int first = 0;
  for (int i = 0; i < n; ++i) {                              // blocks in proportion to the sizes, one wave in all
    const int64_t share = (int64_t)sm_count() * kAmaxBlocksPerSm * b.op[i].n_vec32 / total;
    b.op[i].first_block = first;
    b.op[i].blocks = (int)std::min(ceil_div(b.op[i].n_vec32, (int64_t)kAmaxThreads * 4), std::max<int64_t>(share, 1));
    first += b.op[i].blocks;
  }
  const bool bf16 = dtype == NVFP4_BF16;
  cudaError_t e;
  if (sweep) e = bf16 ? launch_overlapped(amax_flat_batch_kernel<__nv_bfloat16>, first, kAmaxThreads, 0, s, b)
                      : launch_overlapped(amax_flat_batch_kernel<float>, first, kAmaxThreads, 0, s, b);
  else e = bf16 ? launch_overlapped(amax_cluster_batch_kernel<__nv_bfloat16>, n * kSmallAmaxCluster, kSmallAmaxThreads, 0, s, b)
                : launch_overlapped(amax_cluster_batch_kernel<float>, n * kSmallAmaxCluster, kSmallAmaxThreads, 0, s, b);
  return e == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

// The same for a quantizer that reduces maxima.
int amax_sweep(const LayerOperand* ops, int n, int dtype, ScaleSource* src, cudaStream_t s) {
  AmaxSweep b = {};
  b.n = n;
  int64_t total = 0;
  for (int i = 0; i < n; ++i) total += operand_bytes(ops[i], dtype) / 32;
  int first = 0;
  for (int i = 0; i < n; ++i) {                              // clusters in proportion to the sizes, one wave in all
    const int64_t n32 = operand_bytes(ops[i], dtype) / 32, share = (int64_t)sm_count() / kSweepCluster * n32 / total;
    const int clusters = (int)std::min<int64_t>({ceil_div(n32, (int64_t)kSweepThreads * 4 * kSweepCluster), std::max<int64_t>(share, 1), kSweepWords});
    b.op[i] = {static_cast<const uint32_t*>(ops[i].x), n32, reinterpret_cast<uint32_t*>(ops[i].slot) + 1, first, clusters};
    first += clusters;
    src[i] = {nullptr, b.op[i].maxima, clusters, ops[i].slot};
  }
  const cudaError_t e = dtype == NVFP4_BF16 ? launch_overlapped(amax_sweep_kernel<__nv_bfloat16>, first * kSweepCluster, kSweepThreads, 0, s, b)
                                            : launch_overlapped(amax_sweep_kernel<float>, first * kSweepCluster, kSweepThreads, 0, s, b);
  return e == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

int quantize_operand(const LayerOperand& op, int dtype, const float* g, void* stream) {
  constexpr int kLayout = NVFP4_SF_SWIZZLED_128x4;
  if (op.rr && op.rt)
    return nvfp4_quantize_dual(op.x, dtype, op.rows, op.cols, op.cols, g, op.rr, op.codes_r, op.scales_r, op.rt, op.codes_t, op.scales_t, kLayout, stream);
  if (op.rr) return nvfp4_quantize(op.x, dtype, op.rows, op.cols, op.cols, 0, g, op.rr, op.codes_r, op.scales_r, kLayout, stream);
  return nvfp4_quantize(op.x, dtype, op.rows, op.cols, op.cols, 1, g, op.rt, op.codes_t, op.scales_t, kLayout, stream);
}
}  // namespace

// Amax by sweeps that leave maxima, and one quantizer launch for all operands, while they have at most this many bytes together.
// Beyond it the sweep with a ticket wins, whose small blocks start one by one in the tail of the kernel before, and so do the
// quantizers made for one tensor.  us, ticket / maxima: 2080 x 2848 (12 MB) with its quantizer 15.5 / 13.8, both operands of
// 4864 x 1120 x 800 (13 MB) and their step 52.9 / 51.1, 16384 x 1024 (34 MB) 21.4 / 22.2, 16384 x 3072 49.0 / 53.5, fp32 step 16384 x 2816 x 1024
// (67 MB of dY) 206.7 / 210.4.
constexpr int64_t kSweepBytes = (int64_t)24 << 20;

// Where there are no amax passes, bf16 operands of which only the transposed outputs are asked for are quantized apart from this many
// bytes on: the kernel for all has room for both outputs, the one for a single output has more blocks on a multiprocessor for
// the random stream's chains.  Weight gradient, us, apart / in one launch: 4096 x 1024 x 1024 (17 MB) 17.7 / 16.7, 8192 x 512 x 1024 (25 MB)
// 21.8 / 21.6, 2336 x 1024 x 4096 (24 MB) 20.3 / 21.3, 4096 x 4096 x 1024 25.0 / 26.7, 12288 x 4096 x 64 43.0 / 46.9; fp32 operands
// 4096 x 2048 x 2048 26.7 / 24.7, 8192 x 4096 x 1024 53.0 / 51.2.
constexpr int64_t kApartBytes = (int64_t)20 << 20;

int quantize_operands(const LayerOperand* ops, int n, int dtype, int gscale_mode, const float** g, void* cuda_stream) {
  if (int st = check_arch()) return st;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const bool amax = gscale_mode == NVFP4_G_AMAX, given = gscale_mode == NVFP4_G_GIVEN;
  ScaleSource src[kMaxLayerOperands];
  int64_t bytes = 0;
  bool flat = true, sweep = false, rows = false;
  for (int i = 0; i < n; ++i) {
    for (const nvfp4_rounding* r : {ops[i].rr, ops[i].rt})
      if (r && ((r->mode != NVFP4_RTN && r->mode != NVFP4_SR) || r->reserved != 0)) return NVFP4_ERR_ENUM;
    if (!aligned16(ops[i].x)) return NVFP4_ERR_ALIGN;
    g[i] = amax ? ops[i].slot : given ? ops[i].given : nullptr;
    src[i] = {g[i], nullptr, 0, given ? ops[i].slot : nullptr};
    bytes += operand_bytes(ops[i], dtype);
    flat = flat && amax_flat_ok(ops[i].x, dtype, ops[i].rows, ops[i].cols, ops[i].cols);
    sweep = sweep || needs_scratch(ops[i], dtype);
    rows = rows || ops[i].rr;
  }
  const bool batch = tile_batch_eligible(ops, n);
  if (!amax) {
    const bool apart = !rows && dtype == NVFP4_BF16 && bytes >= kApartBytes;
    if (batch && n > 1 && !apart) return tile_quantize_batch(ops, src, n, dtype, s);
    if (given) {
      ScalePairs p = {};
      bool any = false;
      for (int i = 0; i < n; ++i) { p.from[i] = ops[i].given; p.to[i] = ops[i].slot; any = any || ops[i].slot; }
      if (any && launch_overlapped(copy_scales_kernel, 1, 32, 0, s, p, n) != cudaSuccess) return NVFP4_ERR_CUDA;
    }
  } else if (batch && flat && bytes <= kSweepBytes && (sweep || n > 1)) {
    if (int st = sweep ? amax_sweep(ops, n, dtype, src, s) : amax_together(ops, n, dtype, s)) return st;
    return tile_quantize_batch(ops, src, n, dtype, s);
  } else if (n > 1 && flat && bytes <= (int64_t)64 << 20) {
    // Together below 64 MB the operands still lie in the level-two cache when their quantizers read them, so nothing is lost by
    // sweeping them all first, and a launch and its latency are saved for each but one.
    if (int st = amax_together(ops, n, dtype, s)) return st;
  } else {
    // One by one: the pass leaves the end of its tensor in the cache for the quantizer behind it.  Three fp32 operands begin with the
    // output gradient, the last of the list: linear_bwd, us, in the list's order / so: 12384 x 160 x 3392 108.9 / 99.5, 12864 x 864 x 2240
    // 117.9 / 114.3, 8192 x 512 x 4096 101.1 / 94.9, 16384 x 2816 x 512 148.3 / 144.2, 512 x 8192 x 8192 179.0 / 178.8; bf16 13280 x 4864 x 288
    // 147 / 155, 2048 x 8192 x 8192 206 / 211, 12384 x 160 x 3392 84.3 / 82.9.
    const int lead = n == 3 && dtype == NVFP4_FP32 ? 2 : 0;
    if (sweep && zero_words(amax_scratch(ops, 0), 2 * n, s) != cudaSuccess) return NVFP4_ERR_CUDA;
    for (int j = 0; j < n; ++j) {
      const int i = (lead + j) % n;
      if (int st = tensor_amax_scale_ws(ops[i].x, dtype, ops[i].rows, ops[i].cols, ops[i].cols, ops[i].slot, amax_scratch(ops, i), sweep || j > 0, cuda_stream))
        return st;
      if (int st = quantize_operand(ops[i], dtype, g[i], cuda_stream)) return st;
    }
    return NVFP4_OK;
  }
  for (int i = 0; i < n; ++i)
    if (int st = quantize_operand(ops[i], dtype, g[i], cuda_stream)) return st;
  return NVFP4_OK;
}
}  // namespace nvfp4

extern "C" int nvfp4_tensor_amax_scale(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld,
                                       float* global_scale_out, void* cuda_stream) {
  if (!x || !global_scale_out) return NVFP4_ERR_NULL;
  if (dtype != NVFP4_BF16 && dtype != NVFP4_FP32) return NVFP4_ERR_ENUM;
  if (rows <= 0 || cols <= 0 || ld < cols || cols % 8 != 0) return NVFP4_ERR_SHAPE;
  if (!aligned16(x) || (ld % 8) != 0 || (reinterpret_cast<uintptr_t>(global_scale_out) & 3u)) return NVFP4_ERR_ALIGN;
  if (int st = check_arch()) return st;
  cudaStream_t s = static_cast<cudaStream_t>(cuda_stream);
  const int64_t total_bytes = rows * cols * (dtype == NVFP4_BF16 ? 2 : 4);
  const bool flat = amax_flat_ok(x, dtype, rows, cols, ld);
  if (flat && total_bytes <= kSmallAmaxBytes)
    return launch_amax_cluster(x, dtype, total_bytes / 32, global_scale_out, false, s) == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
  unsigned int* bits = reinterpret_cast<unsigned int*>(global_scale_out);
  cudaError_t e = launch_overlapped(zero_words_kernel, 1, 32, 0, s, bits, 1);
  if (e != cudaSuccess) return NVFP4_ERR_CUDA;
  if (flat) {
    const int64_t n32 = total_bytes / 32;
    const int64_t fb = std::min(ceil_div(n32, (int64_t)kAmaxThreads * 4), (int64_t)sm_count() * kAmaxBlocksPerSm);
    const uint32_t* xw = static_cast<const uint32_t*>(x);
    e = (dtype == NVFP4_BF16)
        ? launch_overlapped(amax_flat_kernel<__nv_bfloat16, false>, (unsigned)fb, kAmaxThreads, 0, s, xw, n32, bits, (float*)nullptr)
        : launch_overlapped(amax_flat_kernel<float, false>, (unsigned)fb, kAmaxThreads, 0, s, xw, n32, bits, (float*)nullptr);
  } else {
    const int64_t vecs = rows * (cols / (dtype == NVFP4_BF16 ? 8 : 4));
    int64_t blocks = ceil_div(vecs, (int64_t)kThreads * 4);
    if (blocks > sm_count() * 16) blocks = sm_count() * 16;
    e = (dtype == NVFP4_BF16)
        ? launch_overlapped(amax_kernel<__nv_bfloat16>, (unsigned)blocks, kThreads, 0, s, static_cast<const __nv_bfloat16*>(x), rows, cols, ld, bits)
        : launch_overlapped(amax_kernel<float>, (unsigned)blocks, kThreads, 0, s, static_cast<const float*>(x), rows, cols, ld, bits);
  }
  if (e == cudaSuccess) e = launch_overlapped(amax_finalize_kernel, 1, 1, 0, s, global_scale_out);
  return e == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}
