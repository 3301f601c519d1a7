// Tile quantizer: one read of x[rows, cols] produces the transposed NVFP4 quantization (blocks of 16 along the row
// axis, output stored [cols, rows/2]), the row quantization (blocks along the column axis), or both.  Both is the producer fusion for the operands that Eq. 4-6 need in both orientations: dY as Q(dY) for Eq. 5 and
// Q(dY^T) for Eq. 6, X as Q(X) for Eq. 4 and Q(X^T) for Eq. 6, W as Q(W) for Eq. 4 and Q(W^T) for Eq. 5.
//
// Persistent blocks walk over tiles of 128 rows x 64 columns, or a block of its own takes each tile of 256 rows (launch_tile
// says which).  One thread fetches tiles with tiled bulk copies (128-byte swizzle, zero fill outside the tensor); all threads quantize from shared memory; the packed codes are staged
// in shared memory and leave as tiled bulk stores (which clip at the tensor edge), the scales as plain stores.
//
// Bound by instruction issue where it rounds stochastically, by memory otherwise.  Against one 256-row tile per block and,
// for fp32, two single-output passes (us): fp32 16384 x 4096, both outputs, RtN 101 -> 53 and SR 115 -> 56; bf16 256 x 512
// 3.1 -> 2.3 and 3.5 -> 2.7; 16384 x 1024 11.4 -> 9.9 and 16.0 -> 15.5; 65536 x 4096 transposed SR 118 -> 115.
#include <cuda.h>
#include <cuda_bf16.h>

#include <type_traits>

#include "quantize_core.cuh"
#include "tensor_map.cuh"

namespace nvfp4 {
namespace {

constexpr int kTileCols = 64;
constexpr int64_t kBatchElements = (int64_t)1 << 26;          // beyond it the 256-row tiles are better (launch_tile)
constexpr unsigned long long kTileWaitLimitNs = 2000000000ull;
constexpr int kLoader = kThreads - 32;                                // the thread that issues the bulk copies

// Shared memory of a block, in order: tile slots, code staging, scale staging, SLOTS of each.
// Two slots, used in turn: the tile after next lands while the present one is quantized.  One slot: the block has one tile,
// and the other blocks of the SM cover its load and its stores.
template <typename T, int ROWS, bool TR, bool ROW, int SLOTS>
struct TileSmem {
  static constexpr int kBoxBytes = ROWS * 128;                        // a copy's box is 128 bytes wide: 64 bf16 or 32 fp32 columns
  static constexpr int kBoxes = kTileCols * (int)sizeof(T) / 128;
  static constexpr int kTileBytes = kBoxes * kBoxBytes;
  static constexpr int kCodesTBytes = TR ? kTileCols * (ROWS / 2) : 0;   // 64 output rows, swizzled over their 64 or 128 bytes
  static constexpr int kCodesRBytes = ROW ? ROWS * (kTileCols / 2) : 0;   // ROWS output rows x 32 bytes
  static constexpr int kCodesBytes = kCodesTBytes + kCodesRBytes;
  static constexpr int kSfTBytes = TR ? kTileCols * (ROWS / 16) : 0;  // [four row blocks][64 columns][4]: words as scale tiles hold them
  static constexpr int kSfRBytes = ROW ? (ROWS / 128) * 512 : 0;     // whole scale tiles (128 rows x 4 blocks)
  static constexpr int kSfBytes = kSfTBytes + kSfRBytes;
  static constexpr int kCodesAt = SLOTS * kTileBytes, kSfAt = kCodesAt + SLOTS * kCodesBytes;
  static constexpr int kBytes = kSfAt + SLOTS * kSfBytes + 1024 /*align*/;
  static constexpr int kBlocksPerSm = sizeof(T) == 2 ? 4 : 2;
  static_assert(kBlocksPerSm * (kBytes + 1024 /*static*/ + 1024 /*reserved*/) <= 228 * 1024, "shared memory of an SM");
};

struct TileParams {
  const float* gptr;
  int64_t rows, cols;
  int tiles_x, tiles;         // tiles across the columns, in all
  int step_x, step_y;         // two slots: distance between two tiles of a block, gridDim.x = step_y * tiles_x + step_x
  // transposed output: quantized shape (cols, rows)
  PhiloxStream t_rng;
  uint8_t* t_scales;
  int64_t t_nkb, t_k_tiles;   // groups of 16 per quantized row (the unit of the random draws); scale tiles per quantized row
  int64_t t_nsb;              // scale blocks per quantized row: rows / 16 (NVFP4) or rows / 32 (MXFP4)
  // row output: quantized shape (rows, cols)
  PhiloxStream r_rng;
  uint8_t* r_scales;
  int64_t r_nkb, r_k_tiles, r_nsb;   // as t_*
};

__device__ unsigned int g_tile_error_word = 0;

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Shared-memory accesses with the address split into a register part and a compile-time byte offset, so that
// the unrolled loops below spend no instructions on addresses.  The loads are plain (not volatile) statements, so
// that the compiler may schedule them ahead of the arithmetic of the previous block; the tile they read is written
// by the bulk copy before the wait, and their base address is taken only after that wait (after_wait).
template <int IMM>
__device__ __forceinline__ uint32_t lds32(uint32_t addr) {
  uint32_t v;
  asm("ld.shared.b32 %0, [%1 + %2];" : "=r"(v) : "r"(addr), "n"(IMM));
  return v;
}
template <int IMM>
__device__ __forceinline__ float2 lds64(uint32_t addr) {
  float2 v;
  asm("ld.shared.v2.f32 {%0, %1}, [%2 + %3];" : "=f"(v.x), "=f"(v.y) : "r"(addr), "n"(IMM));
  return v;
}
template <int IMM>
__device__ __forceinline__ uint4 lds128(uint32_t addr) {
  uint4 v;
  asm("ld.shared.v4.b32 {%0, %1, %2, %3}, [%4 + %5];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(addr), "n"(IMM));
  return v;
}
// An address the compiler must consider produced here: every load whose address derives from it stays behind the call.
__device__ __forceinline__ uint32_t after_wait(uint32_t a) {
  asm volatile("" : "+r"(a) :: "memory");
  return a;
}
template <int IMM>
__device__ __forceinline__ void sts64(uint32_t addr, uint32_t lo, uint32_t hi) {
  asm volatile("st.shared.v2.b32 [%0 + %3], {%1, %2};" ::"r"(addr), "r"(lo), "r"(hi), "n"(IMM) : "memory");
}
template <int I>
using Const = std::integral_constant<int, I>;
// f(Const<0>) ... f(Const<N - 1>)
template <int N, int I = 0, typename F>
__device__ __forceinline__ void unrolled(F&& f) {
  if constexpr (I < N) {
    f(Const<I>{});
    unrolled<N, I + 1>(f);
  }
}

// Bounded wait for a tile; false (and an error word) when the time ran out.
__device__ __forceinline__ bool wait_tile(uint32_t bar, uint32_t parity) {
  unsigned long long t0 = 0;
  for (uint32_t spin = 0;; ++spin) {
    uint32_t done;
    asm volatile("{\n\t.reg .pred q;\n\tmbarrier.try_wait.parity.shared::cta.b64 q, [%1], %2;\n\tselp.u32 %0, 1, 0, q;\n\t}"
                 : "=r"(done) : "r"(bar), "r"(parity) : "memory");
    if (done) return true;
    if ((spin & 255u) == 255u) {
      unsigned long long now;
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
      if (t0 == 0) t0 = now;
      if (now - t0 > kTileWaitLimitNs) {
        atomicOr(&g_tile_error_word, 0x200u);
        return false;
      }
    }
  }
}

// The part of one thread in a tile's transposed output: columns (2 * cp, 2 * cp + 1) of the 16 rows of groups g16 and, in a tile
// of 256 rows, g16 + 8.  in_t, out_t, sf_t: where these lie in the tile's slot, its staged codes and its staged scales; blk0_t:
// the index of the first column's group.
template <typename T, int ROWS, bool SR_T, bool SR_R, bool MX, typename Blk>
__device__ __forceinline__ void quantize_columns(const TileParams& p, uint32_t in_t, uint32_t out_t, uint8_t* sf_t, int g16, int cp, float c,
                                                 const float* inv_table, Blk blk0_t) {
  [[maybe_unused]] const int lane = threadIdx.x & 31;
  unrolled<ROWS / 128>([&](auto I) {
    constexpr int i = decltype(I)::value;
    [[maybe_unused]] const Blk blk_a = blk0_t + 8 * i, blk_b = blk_a + (Blk)p.t_nkb;
    [[maybe_unused]] uint32_t w[16];                    // bf16: both columns packed
    float va[16], vb[16], amax_a, amax_b;
    if constexpr (sizeof(T) == 2) {
      unrolled<16>([&](auto J) {
        constexpr int j = decltype(J)::value;
        w[j] = lds32<i * 16384 + j * 128>(in_t ^ ((j & 7) << 4));
      });
      uint32_t m[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) m[j] = absmax_bf16x2(w[2 * j], w[2 * j + 1]);
#pragma unroll
      for (int j = 0; j < 4; ++j) m[j] = absmax_bf16x2(m[2 * j], m[2 * j + 1]);
      uint32_t mm = absmax_bf16x2(absmax_bf16x2(m[0], m[1]), absmax_bf16x2(m[2], m[3]));
      if constexpr (MX) mm = absmax_bf16x2(mm, __shfl_xor_sync(0xFFFFFFFFu, mm, 16));   // the block's other 16 rows
      mm &= 0x7FFF7FFFu;
      amax_a = __uint_as_float(mm << 16);
      amax_b = __uint_as_float(mm & 0xFFFF0000u);
    } else {
      amax_a = amax_b = 0.0f;
      unrolled<16>([&](auto J) {
        constexpr int j = decltype(J)::value;
        const float2 f = lds64<i * 16384 + j * 128>(in_t ^ ((j & 7) << 4));
        va[j] = f.x;
        vb[j] = f.y;
        amax_a = fmaxf(amax_a, fabsf(f.x));
        amax_b = fmaxf(amax_b, fabsf(f.y));
      });
    }
    uint32_t sfa, sfb;
    if constexpr (MX) { sfa = e8m0_encode_up(__fmul_rn(amax_a, c)); sfb = e8m0_encode_up(__fmul_rn(amax_b, c)); }
    else { sfa = e4m3_encode(__fmul_rn(amax_a, c)); sfb = e4m3_encode(__fmul_rn(amax_b, c)); }
    const float inv_a = inv_table[sfa], inv_b = inv_table[sfb];
    // Two Philox chains in flight; one after the other where the compiler has registers to overlap row blocks instead.
    constexpr bool kPairDraws = ROWS == 128 || SR_R;
    uint4 ra = make_uint4(0, 0, 0, 0), rb = ra;
    if constexpr (SR_T && kPairDraws) philox4x32_10_x2(p.t_rng, blk_a, blk_b, ra, rb);
    if constexpr (SR_T && !kPairDraws) ra = philox4x32_10(p.t_rng, blk_a);
    uint32_t lo, hi;
    if constexpr (sizeof(T) == 2) {
#pragma unroll
      for (int j = 0; j < 16; ++j) va[j] = __uint_as_float(w[j] << 16);
    }
    encode_with<SR_T>(va, inv_a, ra, lo, hi);
    const uint32_t out = out_t ^ (i * 64);
    sts64<0>(out, lo, hi);
    if constexpr (SR_T && !kPairDraws) rb = philox4x32_10(p.t_rng, blk_b);
    if constexpr (sizeof(T) == 2) {
#pragma unroll
      for (int j = 0; j < 16; ++j) vb[j] = __uint_as_float(w[j] & 0xFFFF0000u);
    }
    encode_with<SR_T>(vb, inv_b, rb, lo, hi);
    if constexpr (ROWS == 128) sts64<64>(out, lo, hi); else sts64<128>(out ^ 16u, lo, hi);
    if constexpr (MX) {
      if (lane < 16) {
        uint8_t* const dst = sf_t + i * (4 * kTileCols) + 8 * cp + (g16 >> 1);
        dst[0] = (uint8_t)sfa;
        dst[4] = (uint8_t)sfb;
      }
    } else {
      uint8_t* const dst = sf_t + ((g16 >> 2) + 2 * i) * (4 * kTileCols) + 8 * cp + (g16 & 3);
      dst[0] = (uint8_t)sfa;
      dst[4] = (uint8_t)sfb;
    }
  });
}

// The part of one thread in its row output: block kbl of the tile's four, rows t, t + 64, ...
template <typename T, int ROWS, bool SR_R, bool SWZ, bool MX, typename Blk>
__device__ __forceinline__ void quantize_rows(const TileParams& p, uint32_t in, uint32_t out, uint8_t* sf_thread, int kbl, int t, int r0, int c0, float c,
                                              const float* inv_table, Blk blk0) {
  unrolled<ROWS / 64>([&](auto I) {
    constexpr int i = decltype(I)::value;
    Block16<T> blk;
    if constexpr (sizeof(T) == 2) {
      const uint4 a = lds128<i * 8192>(in), d = lds128<i * 8192>(in ^ 16u);
      blk.w[0] = a.x; blk.w[1] = a.y; blk.w[2] = a.z; blk.w[3] = a.w;
      blk.w[4] = d.x; blk.w[5] = d.y; blk.w[6] = d.z; blk.w[7] = d.w;
    } else {
      unrolled<4>([&](auto Q) {
        constexpr int q = decltype(Q)::value;
        const uint4 a = lds128<i * 8192>(in ^ (q << 4));
        blk.f[q] = make_float4(__uint_as_float(a.x), __uint_as_float(a.y), __uint_as_float(a.z), __uint_as_float(a.w));
      });
    }
    float v[16];
    float amax = blk.unpack(v);
    uint32_t lo, hi, sf;
    if constexpr (MX) {
      amax = fmaxf(amax, __shfl_xor_sync(0xFFFFFFFFu, amax, 1));   // the block's other half is the neighbouring lane's
      sf = e8m0_encode_up(__fmul_rn(amax, c));
      encode_codes<SR_R>(v, inv_table[sf], p.r_rng, blk0 + (Blk)(i * 64) * (Blk)p.r_nkb, lo, hi);
    } else {
      encode_block<SR_R>(v, amax, c, inv_table, p.r_rng, blk0 + (Blk)(i * 64) * (Blk)p.r_nkb, lo, hi, sf);
    }
    sts64<i * 2048>(out, lo, hi);
    const int sb = MX ? kbl >> 1 : kbl;              // scale block within the tile; MXFP4: the even lane's
    if (!MX || (kbl & 1) == 0) {
      if constexpr (SWZ) {
        sf_thread[(i >> 1) * 512 + (i & 1) * 8 + sb] = (uint8_t)sf;
      } else {
        constexpr int kSb = MX ? 32 : 16;
        const int64_t r = (int64_t)r0 + t + i * 64;
        if (r < p.rows && c0 / kSb + sb < p.r_nsb) p.r_scales[r * p.r_nsb + c0 / kSb + sb] = (uint8_t)sf;
      }
    }
  });
}

// Padding of scale tiles is zero: every thread goes once more over the words it stored for its block's tiles (the loop of
// quantize_tile_kernel says which).  Out of line and after the loop, since it is hardly ever called: masking the words on their
// way out, on edge tiles alone, cost 0.3 us of a 2080-token step's 61.7 and 0.4 of 22.8 for both outputs RtN of 11008 x 4096.
template <int ROWS, bool TR, bool ROW>
__device__ __noinline__ void zero_tile_padding(const TileParams& p, int64_t r0, int64_t c0) {
  constexpr int kKtPerTile = ROWS / 64;                   // scale tiles per column
  if (TR && threadIdx.x < kTileCols * kKtPerTile) {
    const int64_t col = c0 + threadIdx.x / kKtPerTile, kt = r0 / 64 + threadIdx.x % kKtPerTile;
    if (kt < p.t_k_tiles) {
      uint32_t* const w = reinterpret_cast<uint32_t*>(p.t_scales + sf_swizzled_offset(col, kt * 4, p.t_k_tiles));
      *w = scales_inside(*w, col < p.cols ? p.t_nsb - kt * 4 : 0);
    }
  }
  if (ROW && threadIdx.x >= 128 && threadIdx.x < 128 + ROWS / 4) {
    // thread 128 + 32 * h + i: the 16 bytes of rows i, i + 32, i + 64, i + 96 of the tile's half h
    const int64_t half = r0 + ((threadIdx.x - 128) >> 5) * 128, row = half + (threadIdx.x & 31);
    if (half < p.rows) {
      uint32_t* const w = reinterpret_cast<uint32_t*>(p.r_scales + sf_swizzled_offset(row, c0 / 16, p.r_k_tiles));
      for (int j = 0; j < 4; ++j) w[j] = scales_inside(w[j], row + 32 * j < p.rows ? p.r_nsb - c0 / 16 : 0);
    }
  }
}

// Staged scales to their tiles.  Transposed output: one 32-bit word = four scale blocks of one column.
template <int ROWS, bool MX>
__device__ __forceinline__ void store_transposed_scales(const TileParams& p, const uint8_t* sf_t, int r0, int c0) {
  constexpr int kSbRows = MX ? 32 : 16;                   // rows per scale block
  constexpr int kKtPerTile = ROWS / kSbRows / 4;          // scale tiles per column
  static_assert(kTileCols * kKtPerTile <= kThreads, "one word per thread");
  if (threadIdx.x < kTileCols * kKtPerTile) {
    // sf_swizzled_offset(c0 + cl, 4 * (kt0 + q), t_k_tiles) taken apart: the tile's part and this thread's
    const int cl = threadIdx.x / kKtPerTile, q = threadIdx.x % kKtPerTile, kt0 = r0 / kSbRows / 4;
    if (kt0 + q < p.t_k_tiles) {
      uint8_t* dst = p.t_scales + ((int64_t)(c0 >> 7) * p.t_k_tiles + kt0) * 512 + ((c0 & 64) >> 3) +
                     (q * 512 + (cl & 31) * 16 + (cl >> 5) * 4);
      *reinterpret_cast<uint32_t*>(dst) = *reinterpret_cast<const uint32_t*>(sf_t + q * (4 * kTileCols) + cl * 4);
      if (((c0 & 127) == 0) && ((int64_t)c0 + kTileCols >= p.cols))        // nobody else owns rows 64..127 of the scale tile
        *reinterpret_cast<uint32_t*>(dst + 8) = 0u;
    }
  }
}
// Row output: the tile owns whole 512-byte scale tiles (128 rows x this k-tile); from the fifth warp on.
template <int ROWS>
__device__ __forceinline__ void store_row_scales(const TileParams& p, const uint8_t* sf_r, int r0, int c0) {
  const int h = (threadIdx.x >> 5) - 4, i = threadIdx.x & 31;
  if (h >= 0 && h < ROWS / 128 && (int64_t)r0 + h * 128 < p.rows)
    *reinterpret_cast<uint4*>(p.r_scales + ((int64_t)(r0 / 128 + h) * p.r_k_tiles + c0 / 64) * 512 + i * 16) =
        *reinterpret_cast<const uint4*>(sf_r + h * 512 + i * 16);
}

// MX: the output (one of the two) is MXFP4 (Section 3, Table 1): blocks of 32 with an E8M0 scale rounded up to a power
// of two; the two groups of 16 inside a block keep their own random draws (group index as for NVFP4).
// TR, ROW: which outputs are written.
template <typename T, int ROWS, int SLOTS, bool TR, bool SR_T, bool ROW, bool SR_R, bool SWZ, bool MX>
__global__ void __launch_bounds__(kThreads, TileSmem<T, ROWS, TR, ROW, SLOTS>::kBlocksPerSm)
quantize_tile_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_ct,
                     const __grid_constant__ CUtensorMap map_cr, const __grid_constant__ TileParams p) {
  using S = TileSmem<T, ROWS, TR, ROW, SLOTS>;
  static_assert(ROWS == 128 || ROWS == 256, "a staged output row is one swizzle span");
  static_assert((TR || ROW) && !(MX && TR && (ROW || sizeof(T) != 2)), "MXFP4: one output, the transposed one of bf16 tensors only");
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem = (smem_addr(smem_raw) + 1023u) & ~1023u;
  uint8_t* const smem_gen = smem_raw + (smem - smem_addr(smem_raw));
  __shared__ __align__(8) uint64_t bars[SLOTS];
  __shared__ float inv_table[MX ? 256 : 128];

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  // Tiles are walked from the last to the first: a pass over the tensor that ran just before (its amax) left the end of
  // it in the level-two cache, not the beginning.
  const int mine = SLOTS == 1 ? 1 : (p.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  int ty = (p.tiles - 1 - (int)blockIdx.x) / p.tiles_x, tx = (p.tiles - 1 - (int)blockIdx.x) - ty * p.tiles_x;
  int load_x = tx, load_y = ty;                           // the loader's position, up to two tiles ahead
  auto step_back = [&](int& x, int& y) {
    x -= p.step_x;
    y -= p.step_y;
    if (x < 0) { x += p.tiles_x; --y; }
  };
  auto load_tile = [&](int b) {
    const uint32_t bar = smem_addr(&bars[b]);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(S::kTileBytes) : "memory");
#pragma unroll
    for (int i = 0; i < S::kBoxes; ++i)
      asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                   ::"r"(smem + b * S::kTileBytes + i * S::kBoxBytes), "l"(&map_x), "r"(bar),
                     "r"(load_x * kTileCols + i * (128 / (int)sizeof(T))), "r"(load_y * ROWS) : "memory");
    step_back(load_x, load_y);
  };

  if (threadIdx.x == kLoader) {
    for (int i = 0; i < SLOTS; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&bars[i])));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  grid_dependency_wait();
  grid_dependency_trigger();
  if (threadIdx.x == kLoader) {
    load_tile(0);
    if (SLOTS > 1 && mine > 1) load_tile(1);
  }
  const float g = load_scale(p.gptr);
  const float c = __fdiv_rn(__fdiv_rn(1.0f, 6.0f), g);
  if constexpr (MX) build_inv_table_mx(inv_table, g); else build_inv_table(inv_table, g);
  __syncthreads();                                        // barriers initialised, table published

  // ---- this thread's part of a tile ----
  // Block indices (the random draws' counters) in 32 bits: the launch has fewer than 2^32 of them.  MXFP4 takes any size.
  using Blk = std::conditional_t<MX, uint64_t, uint32_t>;
  // Transposed: columns (2*cp, 2*cp + 1) of the 16 rows of groups g16 and, in a tile of 256 rows, g16 + 8.
  const int g16 = MX ? (warp >> 1) * 2 + (lane >> 4) : warp;
  const int cp = MX ? (warp & 1) * 16 + (lane & 15) : lane;
  // Row r of a tile starts at r * 128, its 16-byte piece i sits at i ^ (r & 7): for row j of the group the position is
  // (base | piece) ^ (j & 7) << 4, plus j * 128 as a compile-time offset.
  const uint32_t t_in = smem + g16 * 2048 + (sizeof(T) == 2 ? (uint32_t)cp * 4u : (uint32_t)(cp >> 4) * S::kBoxBytes + (cp & 15) * 8u);
  // Codes of a column: half g16 & 1 of piece g16 / 2 of its staged row, swizzled by the row's index (bits 1-2 of it over
  // 64 bytes, bits 0-2 over 128).  Group g16 + 8 sits four pieces further, which the swizzle turns into an XOR with 64.
  const uint32_t codes0 = smem + S::kCodesAt;
  const uint32_t t_out = codes0 + cp * ROWS + ((((uint32_t)g16 >> 1) ^ (ROWS == 128 ? cp & 3 : (2 * cp) & 7)) << 4) + (g16 & 1) * 8;
  // Row output: block kbl of the tile's 64 columns, rows t, t + 64, ...
  const int kbl = threadIdx.x & 3, t = threadIdx.x >> 2;
  const uint32_t r_piece = sizeof(T) == 2 ? 2u * kbl : 4u * (kbl & 1);
  const uint32_t r_in = smem + (sizeof(T) == 2 ? 0u : (uint32_t)(kbl >> 1) * S::kBoxBytes) + t * 128 + ((r_piece ^ (t & 7)) << 4);
  const uint32_t r_out = codes0 + S::kCodesTBytes + t * 32 + kbl * 8;

  for (int k = 0; k < mine; ++k) {
    const int b = SLOTS == 2 ? k & 1 : 0;
    const int c0 = tx * kTileCols, r0 = ty * ROWS;          // below 2^31, as rows and columns are
    if (!wait_tile(smem_addr(&bars[b]), (SLOTS == 2 ? k >> 1 : k) & 1)) break;
    uint8_t* const sf_t = smem_gen + S::kSfAt + b * S::kSfBytes;
    uint8_t* const sf_r = sf_t + S::kSfTBytes;

    if constexpr (TR)
      quantize_columns<T, ROWS, SR_T, SR_R, MX>(p, after_wait(t_in + b * S::kTileBytes), t_out + b * S::kCodesBytes, sf_t, g16, cp, c, inv_table,
                                                (Blk)((Blk)(c0 + 2 * cp) * (Blk)p.t_nkb + (Blk)(r0 / 16 + g16)));
    if constexpr (ROW)
      quantize_rows<T, ROWS, SR_R, SWZ, MX>(p, after_wait(r_in + b * S::kTileBytes), r_out + b * S::kCodesBytes, sf_r + (t & 31) * 16 + (t >> 5) * 4, kbl, t,
                                            r0, c0, c, inv_table, (Blk)((Blk)(r0 + t) * (Blk)p.r_nkb + (Blk)(c0 / 16 + kbl)));

    // ---- codes out: tiled bulk stores from this tile's staging buffer; its slot then takes the tile after next ----
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (SLOTS == 2 && threadIdx.x == kLoader)             // the previous tile's codes have left the other staging buffer
      asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
    __syncthreads();
    if (threadIdx.x == kLoader) {
      const uint32_t out = codes0 + b * S::kCodesBytes;
      if constexpr (TR)
        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];"
                     ::"l"(&map_ct), "r"(out), "r"(r0 / 2), "r"(c0) : "memory");
      if constexpr (ROW)
        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];"
                     ::"l"(&map_cr), "r"(out + S::kCodesTBytes), "r"(c0 / 2), "r"(r0) : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      if (SLOTS == 2 && k + SLOTS < mine) load_tile(b);
    }

    // ---- scales out ----
    if constexpr (SWZ) {
      if constexpr (TR) store_transposed_scales<ROWS, MX>(p, sf_t, r0, c0);
      if constexpr (ROW && MX) {
        // a scale tile holds 128 columns' scales: this tile owns bytes 0-1 or 2-3 of each of its words
        if (threadIdx.x >= 128) {
          const int w = threadIdx.x - 128;               // word: row (w & 3) * 32 + w / 4
          const uint32_t val = *reinterpret_cast<const uint16_t*>(sf_r + w * 4);
          uint8_t* const dst = p.r_scales + ((int64_t)(r0 / 128) * p.r_k_tiles + c0 / 128) * 512 + w * 4;
          if (((c0 & 127) == 0) && ((int64_t)c0 + kTileCols >= p.cols))        // nobody else owns the upper half
            *reinterpret_cast<uint32_t*>(dst) = val;
          else
            *reinterpret_cast<uint16_t*>(dst + ((c0 & 64) >> 5)) = (uint16_t)val;
        }
      } else if constexpr (ROW) {
        store_row_scales<ROWS>(p, sf_r, r0, c0);
      }
    } else if constexpr (TR) {
      constexpr int kSbRows = MX ? 32 : 16, kSbPerTile = ROWS / kSbRows;   // rows per scale block, scale blocks per column
      const int kb0 = r0 / kSbRows;
      for (int id = threadIdx.x; id < kTileCols * kSbPerTile; id += kThreads) {
        const int cl = id / kSbPerTile, u = id % kSbPerTile;
        if (c0 + cl < p.cols && kb0 + u < p.t_nsb) p.t_scales[(int64_t)(c0 + cl) * p.t_nsb + kb0 + u] = sf_t[(u >> 2) * (4 * kTileCols) + cl * 4 + (u & 3)];
      }
    }
    if constexpr (SLOTS == 2) step_back(tx, ty);
  }
  // The zeros beyond the tensor encode to zero scales by themselves unless the per-tensor scale is NaN, zero or subnormal (c is
  // then NaN, or may be infinite).  Asked of g: asked of c, 2080 x 1056 took 2.57 us instead of 2.40 in every form.
  if constexpr (SWZ && !MX)
    if (!(g >= 0x1p-126f))
      for (int tile = p.tiles - 1 - (int)blockIdx.x, k = 0; k < mine; ++k, tile -= (int)gridDim.x)
        zero_tile_padding<ROWS, TR, ROW>(p, (int64_t)(tile / p.tiles_x) * ROWS, (int64_t)(tile % p.tiles_x) * kTileCols);
  if (threadIdx.x == kLoader) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // staging must outlive the stores' reads
}

// Several operands of one layer call in one launch: their tiles (128 rows, swizzled NVFP4 scales) in one list, each with the
// outputs and the roundings of its operand.  Small operands leave most of the chip idle, and each launch costs its latency:
// one step of 256 x 512 x 512 24.9 -> 22.3 us, 2080 x 1056 x 2848 55.6 -> 54.7, 3680 x 896 x 640 with given scales 40.0 -> 34.3.
struct TileBatch {
  struct Op {
    CUtensorMap x, ct, cr;
    TileParams p;
    ScaleSource scale;
    int first;                  // its first tile in the list
    uint32_t magic;             // tile / tiles_x = the upper half of tile * magic (0: tiles_x is 1)
    bool tr, sr_t, row, sr_r;
  } op[kMaxLayerOperands];
  int n, tiles;
};
template <typename T>
__global__ void __launch_bounds__(kThreads, TileSmem<T, 128, true, true, 2>::kBlocksPerSm)
quantize_tile_batch_kernel(const __grid_constant__ TileBatch p) {
  using S = TileSmem<T, 128, true, true, 2>;
  constexpr int ROWS = 128;
  extern __shared__ uint8_t smem_raw[];
  const uint32_t smem = (smem_addr(smem_raw) + 1023u) & ~1023u;
  uint8_t* const smem_gen = smem_raw + (smem - smem_addr(smem_raw));
  __shared__ __align__(8) uint64_t bars[2];
  __shared__ float inv_tables[kMaxLayerOperands][128], scales[kMaxLayerOperands], cs[kMaxLayerOperands];

  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int mine = (p.tiles - (int)blockIdx.x + (int)gridDim.x - 1) / (int)gridDim.x;
  auto locate = [&](int tile, int& r0, int& c0) {
    const int which = (p.n > 1 && tile >= p.op[1].first) + (p.n > 2 && tile >= p.op[2].first);
    const TileBatch::Op& op = p.op[which];
    tile -= op.first;
    const int ty = op.magic ? (int)__umulhi((uint32_t)tile, op.magic) : tile;
    r0 = ty * ROWS;
    c0 = (tile - ty * op.p.tiles_x) * kTileCols;
    return which;
  };
  auto load_tile = [&](int b, int tile) {
    int r0, c0;
    const CUtensorMap* map = &p.op[locate(tile, r0, c0)].x;
    const uint32_t bar = smem_addr(&bars[b]);
    asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(S::kTileBytes) : "memory");
#pragma unroll
    for (int i = 0; i < S::kBoxes; ++i)
      asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];"
                   ::"r"(smem + b * S::kTileBytes + i * S::kBoxBytes), "l"(map), "r"(bar), "r"(c0 + i * (128 / (int)sizeof(T))), "r"(r0) : "memory");
  };
  int tile = p.tiles - 1 - (int)blockIdx.x;
  if (threadIdx.x == kLoader) {
    for (int i = 0; i < 2; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&bars[i])));
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  grid_dependency_wait();
  grid_dependency_trigger();
  if (threadIdx.x == kLoader) {
    load_tile(0, tile);
    if (mine > 1) load_tile(1, tile - (int)gridDim.x);
  }
  __syncwarp();
  if (warp < p.n) {                                       // a warp per operand: their latencies overlap
    const ScaleSource& src = p.op[warp].scale;
    const float g = read_scale(src);
    if (lane == 0) {
      scales[warp] = g;
      cs[warp] = __fdiv_rn(__fdiv_rn(1.0f, 6.0f), g);
      if (src.keep && blockIdx.x == 0) *src.keep = g;
    }
  }
  __syncthreads();                                        // barriers initialised, scales published
  for (int i = threadIdx.x; i < p.n * 128; i += kThreads) inv_tables[i >> 7][i & 127] = inv_scale((uint32_t)(i & 127), scales[i >> 7]);
  __syncthreads();

  // ---- this thread's part of a tile: as in quantize_tile_kernel ----
  const uint32_t t_in = smem + warp * 2048 + (sizeof(T) == 2 ? (uint32_t)lane * 4u : (uint32_t)(lane >> 4) * S::kBoxBytes + (lane & 15) * 8u);
  const uint32_t codes0 = smem + S::kCodesAt;
  const uint32_t t_out = codes0 + lane * ROWS + ((((uint32_t)warp >> 1) ^ (lane & 3)) << 4) + (warp & 1) * 8;
  const int kbl = threadIdx.x & 3, t = threadIdx.x >> 2;
  const uint32_t r_piece = sizeof(T) == 2 ? 2u * kbl : 4u * (kbl & 1);
  const uint32_t r_in = smem + (sizeof(T) == 2 ? 0u : (uint32_t)(kbl >> 1) * S::kBoxBytes) + t * 128 + ((r_piece ^ (t & 7)) << 4);
  const uint32_t r_out = codes0 + S::kCodesTBytes + t * 32 + kbl * 8;

  for (int k = 0; k < mine; ++k, tile -= (int)gridDim.x) {
    const int b = k & 1;
    int r0, c0;
    const int which = locate(tile, r0, c0);
    const TileBatch::Op& op = p.op[which];
    const float c = cs[which];
    const float* inv_table = inv_tables[which];
    if (!wait_tile(smem_addr(&bars[b]), (k >> 1) & 1)) break;
    uint8_t* const sf_t = smem_gen + S::kSfAt + b * S::kSfBytes;
    uint8_t* const sf_r = sf_t + S::kSfTBytes;
    if (op.tr) {
      const uint32_t in = after_wait(t_in + b * S::kTileBytes), out = t_out + b * S::kCodesBytes;
      const uint32_t blk0 = (uint32_t)(c0 + 2 * lane) * (uint32_t)op.p.t_nkb + (uint32_t)(r0 / 16 + warp);
      if (op.sr_t) quantize_columns<T, ROWS, true, true, false>(op.p, in, out, sf_t, warp, lane, c, inv_table, blk0);
      else quantize_columns<T, ROWS, false, true, false>(op.p, in, out, sf_t, warp, lane, c, inv_table, blk0);
    }
    if (op.row) {
      const uint32_t in = after_wait(r_in + b * S::kTileBytes), out = r_out + b * S::kCodesBytes;
      const uint32_t blk0 = (uint32_t)(r0 + t) * (uint32_t)op.p.r_nkb + (uint32_t)(c0 / 16 + kbl);
      uint8_t* const sf_thread = sf_r + (t & 31) * 16 + (t >> 5) * 4;
      if (op.sr_r) quantize_rows<T, ROWS, true, true, false>(op.p, in, out, sf_thread, kbl, t, r0, c0, c, inv_table, blk0);
      else quantize_rows<T, ROWS, false, true, false>(op.p, in, out, sf_thread, kbl, t, r0, c0, c, inv_table, blk0);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (threadIdx.x == kLoader) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // the other staging buffer is free
    __syncthreads();
    if (threadIdx.x == kLoader) {
      const uint32_t out = codes0 + b * S::kCodesBytes;
      if (op.tr)
        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];"
                     ::"l"(&op.ct), "r"(out), "r"(r0 / 2), "r"(c0) : "memory");
      if (op.row)
        asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.tile.bulk_group [%0, {%2, %3}], [%1];"
                     ::"l"(&op.cr), "r"(out + S::kCodesTBytes), "r"(c0 / 2), "r"(r0) : "memory");
      asm volatile("cp.async.bulk.commit_group;" ::: "memory");
      if (k + 2 < mine) load_tile(b, tile - 2 * (int)gridDim.x);
    }
    if (op.tr) store_transposed_scales<ROWS, false>(op.p, sf_t, r0, c0);
    if (op.row) store_row_scales<ROWS>(op.p, sf_r, r0, c0);
  }
  for (int i = 0; i < p.n; ++i)
    if (!(scales[i] >= 0x1p-126f))                        // as in quantize_tile_kernel
      for (int k = 0, u = p.tiles - 1 - (int)blockIdx.x; k < mine; ++k, u -= (int)gridDim.x) {
        int r0, c0;
        if (locate(u, r0, c0) != i) continue;
        if (p.op[i].tr) zero_tile_padding<ROWS, true, false>(p.op[i].p, r0, c0);
        if (p.op[i].row) zero_tile_padding<ROWS, false, true>(p.op[i].p, r0, c0);
      }
  if (threadIdx.x == kLoader) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");   // staging must outlive the stores' reads
}

bool make_map_2d(CUtensorMap* map, CUtensorMapDataType dt, const void* base, uint64_t inner, uint64_t outer,
                 uint64_t pitch_bytes, uint32_t box_inner, uint32_t box_outer, CUtensorMapSwizzle swz) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {inner, outer};
  const cuuint64_t strides[1] = {pitch_bytes};
  const cuuint32_t box[2] = {box_inner, box_outer};
  const cuuint32_t estr[2] = {1, 1};
  return fn(map, dt, 2, const_cast<void*>(base), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, swz,
            CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// What a launch reads and writes; its tensor maps depend on the tile's height.
struct TileTensors {
  const void* x;
  int64_t ld;
  uint8_t *codes_t, *codes_r;
};

// Maps of the tensor and of its outputs; the map of an output that is not written is not read either.
template <typename T, int ROWS>
bool make_tile_maps(const TileTensors& a, uint64_t rows, uint64_t cols, bool tr, bool row, CUtensorMap* mx, CUtensorMap* mct, CUtensorMap* mcr) {
  if (!make_map_2d(mx, sizeof(T) == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, a.x, cols, rows,
                   (uint64_t)a.ld * sizeof(T), 128 / (int)sizeof(T), ROWS, CU_TENSOR_MAP_SWIZZLE_128B))
    return false;
  *mct = *mcr = *mx;
  if (tr && !make_map_2d(mct, CU_TENSOR_MAP_DATA_TYPE_UINT8, a.codes_t, rows / 2, cols, rows / 2, ROWS / 2, kTileCols,
                         ROWS == 128 ? CU_TENSOR_MAP_SWIZZLE_64B : CU_TENSOR_MAP_SWIZZLE_128B))
    return false;
  return !row || make_map_2d(mcr, CU_TENSOR_MAP_DATA_TYPE_UINT8, a.codes_r, cols / 2, rows, cols / 2, kTileCols / 2, ROWS, CU_TENSOR_MAP_SWIZZLE_NONE);
}

template <typename T, int ROWS, int SLOTS, bool TR, bool SR_T, bool ROW, bool SR_R, bool SWZ, bool MX>
cudaError_t launch_rows(const TileTensors& a, TileParams& p, cudaStream_t s) {
  using S = TileSmem<T, ROWS, TR, ROW, SLOTS>;
  CUtensorMap mx, mct, mcr;
  if (!make_tile_maps<T, ROWS>(a, (uint64_t)p.rows, (uint64_t)p.cols, TR, ROW, &mx, &mct, &mcr)) return cudaErrorInvalidValue;
  static DeviceFlags smem_set;   // per instantiation, per device
  if (cudaError_t e = set_max_dynamic_smem(smem_set, quantize_tile_kernel<T, ROWS, SLOTS, TR, SR_T, ROW, SR_R, SWZ, MX>, S::kBytes)) return e;
  p.tiles_x = (int)ceil_div(p.cols, kTileCols);
  p.tiles = (int)(p.tiles_x * ceil_div(p.rows, ROWS));
  const int slots = sm_count() * S::kBlocksPerSm;
  const int grid = (SLOTS == 1 || p.tiles < slots) ? p.tiles : slots;   // one slot: a block per tile
  p.step_x = grid % p.tiles_x;
  p.step_y = grid / p.tiles_x;
  return launch_overlapped(quantize_tile_kernel<T, ROWS, SLOTS, TR, SR_T, ROW, SR_R, SWZ, MX>, grid, kThreads, S::kBytes, s, mx, mct, mcr, p);
}

template <typename T, bool SR_T, bool DUAL, bool SR_R, bool SWZ, bool MX = false>
cudaError_t launch_tile(const TileTensors& a, TileParams& p, cudaStream_t s) {
  // 128-row tiles under persistent blocks win while blocks are few or the arithmetic is heavy; on large tensors a block per
  // 256-row tile does, started in order by the hardware where walking blocks drift apart (us, 128-row / 256-row):
  //   both outputs RtN  16384 x 2816 22.9 / 25.6   x 4096 37.5 / 35.6   x 11008 115 / 90     SR  35.4 / 35.2, 50.2 / 48.7, 135 / 128
  //   transposed RtN    16384 x 1024 7.5 / 8.2     x 2816 19.7 / 19.7   x 11008 73 / 70      SR  9.9 / 11.0, 22.0 / 24.2, 79 / 84
  // fp32 tensors are bound by memory with the 128-row tile (16384 x 4096, both outputs: 6.2-6.4 TB/s).
  constexpr bool can_be_tall = sizeof(T) == 2 && (DUAL || !SR_T);
  if constexpr (can_be_tall)
    if (p.rows * p.cols >= (int64_t)1 << (DUAL ? 26 : 25))
      return launch_rows<T, 256, 1, true, SR_T, DUAL, SR_R, SWZ, MX>(a, p, s);
  return launch_rows<T, 128, 2, true, SR_T, DUAL, SR_R, SWZ, MX>(a, p, s);
}

template <typename T, bool DUAL, bool SWZ>
cudaError_t dispatch_tile(bool sr_t, bool sr_r, const TileTensors& a,
                          TileParams& p, cudaStream_t s) {
  if constexpr (DUAL) {
    if (sr_t) return sr_r ? launch_tile<T, true, true, true, SWZ>(a, p, s) : launch_tile<T, true, true, false, SWZ>(a, p, s);
    return sr_r ? launch_tile<T, false, true, true, SWZ>(a, p, s) : launch_tile<T, false, true, false, SWZ>(a, p, s);
  } else {
    return sr_t ? launch_tile<T, true, false, false, SWZ>(a, p, s) : launch_tile<T, false, false, false, SWZ>(a, p, s);
  }
}

template <typename T>
cudaError_t dispatch_tile(bool dual, bool swz, bool sr_t, bool sr_r, const TileTensors& a,
                          TileParams& p, cudaStream_t s) {
  if (dual) return swz ? dispatch_tile<T, true, true>(sr_t, sr_r, a, p, s) : dispatch_tile<T, true, false>(sr_t, sr_r, a, p, s);
  return swz ? dispatch_tile<T, false, true>(sr_t, sr_r, a, p, s) : dispatch_tile<T, false, false>(sr_t, sr_r, a, p, s);
}

}  // namespace

// True when the tile kernel can take the tensor: rows a multiple of 32 (16-byte pitch of the transposed codes) and, for
// the row output, columns a multiple of 32 as well.
bool tile_quantizer_eligible(int dtype, int64_t rows, int64_t cols, bool dual, bool mx) {
  if (rows % 32 != 0) return false;
  if (!mx && rows * cols >= (int64_t)1 << 36) return false;                          // block indices in 32 bits
  if (dual && cols % 32 != 0) return false;
  if (rows > (int64_t)65535 * (dtype == NVFP4_BF16 ? 256 : 128)) return false;       // longer tensors are refused further on
  return ceil_div(rows, 128) * ceil_div(cols, kTileCols) < (int64_t)1 << 31;   // tiles are counted in 32 bits
}

// Launches the tile kernel.  r_* arguments are ignored unless `dual`.  Arguments are validated by the callers.
int tile_quantize(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, const float* g, bool dual,
                  const nvfp4_rounding* rt, uint8_t* codes_t, uint8_t* scales_t,
                  const nvfp4_rounding* rr, uint8_t* codes_r, uint8_t* scales_r, int sf_layout, cudaStream_t s, bool mx_t) {
  const bool bf16 = dtype == NVFP4_BF16;
  const TileTensors a = {x, ld, codes_t, codes_r};
  TileParams p;
  p.gptr = g; p.rows = rows; p.cols = cols;
  philox_stream_init(&p.t_rng, rt->seed, rt->offset);
  p.t_scales = scales_t; p.t_nkb = rows / 16;
  p.t_nsb = mx_t ? rows / 32 : rows / 16;
  p.t_k_tiles = ceil_div(p.t_nsb, 4);
  const nvfp4_rounding* r2 = dual ? rr : rt;
  philox_stream_init(&p.r_rng, r2->seed, r2->offset);
  p.r_scales = scales_r; p.r_nkb = p.r_nsb = cols / 16; p.r_k_tiles = ceil_div(p.r_nsb, 4);
  const bool swz = sf_layout == NVFP4_SF_SWIZZLED_128x4;
  const bool sr_t = rt->mode == NVFP4_SR, sr_r = dual && rr->mode == NVFP4_SR;
  cudaError_t e;
  if (mx_t) {                                                 // MXFP4, transposed output of a bf16 tensor only
    if (dual || !bf16) return NVFP4_ERR_ENUM;
    using B = __nv_bfloat16;
    if (sr_t) e = swz ? launch_tile<B, true, false, false, true, true>(a, p, s) : launch_tile<B, true, false, false, false, true>(a, p, s);
    else e = swz ? launch_tile<B, false, false, false, true, true>(a, p, s) : launch_tile<B, false, false, false, false, true>(a, p, s);
  } else {
    e = bf16 ? dispatch_tile<__nv_bfloat16>(dual, swz, sr_t, sr_r, a, p, s)
             : dispatch_tile<float>(dual, swz, sr_t, sr_r, a, p, s);
  }
  return e == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

// Row output alone.  True when the kernel takes the tensor (columns a multiple of 32: 16-byte pitch of the codes) and is the
// better one: everywhere but for large bf16 tensors rounded to nearest, where the plain row kernel streams longer pieces
// (us, row kernel / this: bf16 RtN 256 x 512 4.1 / 2.0, 2080 x 1056 5.7 / 2.4, 11008 x 4096 20.0 / 20.2, 16384 x 11008
// 71 / 77; SR 7.2 / 2.9 at 2080 x 1056, 24.0 / 21.3, 80 / 75; fp32 RtN 7.0 / 3.4, 36 / 33, 126 / 122).  MXFP4 follows the same line:
// the 16384 x 1024 x 2816 forward in it 57.8 us / 55.9, 2048 x 4096 x 11008 97.7 / 93.3.
bool tile_row_quantizer_eligible(int dtype, int64_t rows, int64_t cols, bool sr, bool mx) {
  if (!mx && rows * cols >= (int64_t)1 << 36) return false;                          // block indices in 32 bits
  if (cols % 32 != 0 || ceil_div(rows, 128) * ceil_div(cols, kTileCols) >= (int64_t)1 << 31) return false;
  return dtype == NVFP4_FP32 || sr || rows * cols < (int64_t)48 << 20;
}

namespace {
template <typename T, bool MX>
cudaError_t dispatch_tile_row(bool sr, bool swz, const TileTensors& a, TileParams& p, cudaStream_t s) {
  if (sr) return swz ? launch_rows<T, 128, 2, false, false, true, true, true, MX>(a, p, s) : launch_rows<T, 128, 2, false, false, true, true, false, MX>(a, p, s);
  return swz ? launch_rows<T, 128, 2, false, false, true, false, true, MX>(a, p, s) : launch_rows<T, 128, 2, false, false, true, false, false, MX>(a, p, s);
}
}  // namespace

int tile_quantize_row(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, const float* g, const nvfp4_rounding* r,
                      uint8_t* codes, uint8_t* scales, int sf_layout, cudaStream_t s, bool mx) {
  TileParams p = {};
  p.gptr = g; p.rows = rows; p.cols = cols;
  philox_stream_init(&p.r_rng, r->seed, r->offset);
  p.r_scales = scales; p.r_nkb = cols / 16; p.r_nsb = mx ? cols / 32 : cols / 16; p.r_k_tiles = ceil_div(p.r_nsb, 4);
  const TileTensors a = {x, ld, nullptr, codes};
  const bool sr = r->mode == NVFP4_SR, swz = sf_layout == NVFP4_SF_SWIZZLED_128x4;
  const cudaError_t e = dtype == NVFP4_BF16 ? (mx ? dispatch_tile_row<__nv_bfloat16, true>(sr, swz, a, p, s) : dispatch_tile_row<__nv_bfloat16, false>(sr, swz, a, p, s))
                                            : (mx ? dispatch_tile_row<float, true>(sr, swz, a, p, s) : dispatch_tile_row<float, false>(sr, swz, a, p, s));
  return e == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

// Several operands in one launch: tensors that the 128-row tiles take, together small enough (see launch_tile) and with tile
// counts that tile * magic divides exactly.
bool tile_batch_eligible(const LayerOperand* ops, int n) {
  int64_t elements = 0;
  for (int i = 0; i < n; ++i) {
    const LayerOperand& op = ops[i];
    if ((op.rt && op.rows % 32 != 0) || (op.rr && op.cols % 32 != 0) || op.cols % 8 != 0 || op.rows > (int64_t)65535 * 128) return false;
    if (op.cols > (int64_t)1 << 20 || op.rows * op.cols > kBatchElements) return false;
    elements += op.rows * op.cols;
  }
  return n <= kMaxLayerOperands && elements <= kBatchElements;
}

namespace {
template <typename T>
cudaError_t launch_batch(const LayerOperand* ops, const ScaleSource* scale, int n, cudaStream_t s) {
  using S = TileSmem<T, 128, true, true, 2>;
  TileBatch b;
  b.n = n; b.tiles = 0;
  for (int i = 0; i < n; ++i) {
    TileBatch::Op& o = b.op[i];
    const LayerOperand& op = ops[i];
    const TileTensors a = {op.x, op.cols, op.codes_t, op.codes_r};
    o.tr = op.rt != nullptr; o.row = op.rr != nullptr;
    o.sr_t = o.tr && op.rt->mode == NVFP4_SR; o.sr_r = o.row && op.rr->mode == NVFP4_SR;
    if (!make_tile_maps<T, 128>(a, (uint64_t)op.rows, (uint64_t)op.cols, o.tr, o.row, &o.x, &o.ct, &o.cr)) return cudaErrorInvalidValue;
    TileParams& p = o.p;
    p = TileParams{};
    o.scale = scale[i]; p.rows = op.rows; p.cols = op.cols;
    p.tiles_x = (int)ceil_div(op.cols, kTileCols);
    p.tiles = (int)(p.tiles_x * ceil_div(op.rows, 128));
    if (o.sr_t) philox_stream_init(&p.t_rng, op.rt->seed, op.rt->offset);
    if (o.sr_r) philox_stream_init(&p.r_rng, op.rr->seed, op.rr->offset);
    p.t_scales = op.scales_t; p.t_nkb = p.t_nsb = op.rows / 16; p.t_k_tiles = ceil_div(p.t_nsb, 4);
    p.r_scales = op.scales_r; p.r_nkb = p.r_nsb = op.cols / 16; p.r_k_tiles = ceil_div(p.r_nsb, 4);
    o.first = b.tiles;
    o.magic = p.tiles_x > 1 ? (uint32_t)ceil_div((int64_t)1 << 32, p.tiles_x) : 0u;
    b.tiles += p.tiles;
  }
  static DeviceFlags smem_set;   // per instantiation, per device
  if (cudaError_t e = set_max_dynamic_smem(smem_set, quantize_tile_batch_kernel<T>, S::kBytes)) return e;
  const int slots = sm_count() * S::kBlocksPerSm;
  return launch_overlapped(quantize_tile_batch_kernel<T>, b.tiles < slots ? b.tiles : slots, kThreads, S::kBytes, s, b);
}
}  // namespace

int tile_quantize_batch(const LayerOperand* ops, const ScaleSource* scale, int n, int dtype, cudaStream_t s) {
  const cudaError_t e = dtype == NVFP4_BF16 ? launch_batch<__nv_bfloat16>(ops, scale, n, s) : launch_batch<float>(ops, scale, n, s);
  return e == cudaSuccess ? NVFP4_OK : NVFP4_ERR_CUDA;
}

// Reads and clears this file's device error word (set when a tile wait ran out).
int tile_error_word(unsigned int* out) {
  unsigned int w = 0, zero = 0;
  if (cudaMemcpyFromSymbol(&w, g_tile_error_word, sizeof(w)) != cudaSuccess) return NVFP4_ERR_CUDA;
  if (w != 0 && cudaMemcpyToSymbol(g_tile_error_word, &zero, sizeof(zero)) != cudaSuccess) return NVFP4_ERR_CUDA;
  *out = w;
  return NVFP4_OK;
}

}  // namespace nvfp4
