// Shared device/host helpers of the NVFP4 library (sm_100a only).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include "nvfp4.h"
#include "per_device.h"

namespace nvfp4 {

// ---------------------------------------------------------------------------------------------
// Host-side argument helpers
// ---------------------------------------------------------------------------------------------
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }
inline int64_t ceil_div(int64_t a, int64_t b) { return (a + b - 1) / b; }

// Checks that the current device is a compute-capability 10.x part (cached per device).
int check_arch();

// Ordinal of the current device (-1 if the runtime cannot tell) and its multiprocessor count (cached per device).
int current_device();
int sm_count();

// Raises the dynamic shared-memory limit of `kernel` to `bytes` on the current device, once per device:
// the attribute belongs to (function, device), so `flags` is a static of the calling instantiation.
template <class Kernel>
inline cudaError_t set_max_dynamic_smem(DeviceFlags& flags, Kernel kernel, int bytes) {
  cudaError_t err = cudaSuccess;
  once_per_device(flags, current_device(), [&] {
    err = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
    return err == cudaSuccess;
  });
  return err;
}

// Launch whose blocks may become resident while the kernel before it on the stream still runs (programmatic dependent
// launch): barrier set-up, tensor-memory allocation and descriptor fetches of a kernel then overlap the tail of the one
// before.  The rules every kernel launched this way keeps:
//   * it calls grid_dependency_wait() in every block, before its first access to memory that an earlier kernel may
//     still read or write; when that returns, the kernel before it has finished and its writes are visible;
//   * it calls grid_dependency_trigger() only after that wait.  A kernel that follows it directly therefore starts when
//     everything TWO launches back is finished, and may read that without waiting ("late" kernels), as long as it still waits
//     before it ends, so that "finished" keeps meaning "and all before it".
//   * the late one of two products (gemm_two) does not trigger: what follows starts when it and all before it are finished.  Blocks of
//     the next kernel would take its room (16384 x 11008 x 512 181 -> 182 us, 512 x 11008 x 11008 126.1 -> 128.3).
// After anything else on the stream (a kernel that does not take part, a copy) the attribute changes nothing.
// Launched the ordinary way -> this way, us: one step of a 256 x 512 x 512 layer (six kernels) 34.8 -> 22.4, of a 2080 x 1056 x 2848
// one 67.1 -> 54.6, 16 tokens through kept 11008 x 4096 weights (three kernels) 20.5 -> 14.0.
// Long products neither gain nor lose (11008 x 4096 x 65536 alone 1326 us launched the ordinary way / 1290 this way, behind its
// two quantizers 1813 / 1809; 11008 x 4096 x 16384 333 / 327 and 459 / 461).
template <class... Params, class... Args>
inline cudaError_t launch_overlapped(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t s, Args&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = s;
  cfg.attrs = &attr; cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<Params>(args)...);
}
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

// A per-tensor scale that the kernel before this one may have written (1 where there is none): an ordinary load that stays
// behind the wait.  __ldg is for data that nobody writes while the kernel is resident, and a kernel launched this way is
// resident before its wait returns; source tensors read behind the wait are loaded the same way.
__device__ __forceinline__ float load_scale(const float* g) {
  if (!g) return 1.0f;
  float v;
  asm volatile("ld.global.f32 %0, [%1];" : "=f"(v) : "l"(g) : "memory");
  return v;
}

// A product: the arguments of nvfp4_gemm.
struct GemmCall {
  const uint8_t* a_codes;
  const uint8_t* a_sf;
  const float* a_g;
  const uint8_t* b_codes;
  const uint8_t* b_sf;
  const float* b_g;
  int64_t M, N, K;
  void* d;
  int d_dtype;
  int64_t ldd;
};
// Two products that do not depend on one another, in one launch; and the two of nvfp4_linear_bwd_bf16 (gemm.cu).
int gemm_two(const GemmCall& x, const GemmCall& y, void* cuda_stream);
int gemm_bf16_gradients(const void* dY, const void* W, const void* X, int64_t M, int64_t N, int64_t K, void* dX, int dx_dtype,
                        void* dW, int dw_dtype, void* cuda_stream);

// Tile quantizer (quantize_tile.cu): transposed output, optionally the row output from the same read.
bool tile_quantizer_eligible(int dtype, int64_t rows, int64_t cols, bool dual, bool mx = false);
int tile_quantize(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, const float* g, bool dual,
                  const nvfp4_rounding* rt, uint8_t* codes_t, uint8_t* scales_t,
                  const nvfp4_rounding* rr, uint8_t* codes_r, uint8_t* scales_r, int sf_layout, cudaStream_t s,
                  bool mx_t = false);   // mx_t: MXFP4 (blocks of 32, E8M0 scales) for the transposed output, no row output
// The same kernel with the row output alone.
bool tile_row_quantizer_eligible(int dtype, int64_t rows, int64_t cols, bool sr, bool mx = false);
int tile_quantize_row(const void* x, int dtype, int64_t rows, int64_t cols, int64_t ld, const float* g, const nvfp4_rounding* r,
                      uint8_t* codes, uint8_t* scales, int sf_layout, cudaStream_t s, bool mx = false);
int tile_error_word(unsigned int* out);

// A dense operand [rows, cols] of a layer call, as its products take it: rows, columns (transposed) or both, with swizzled scales.
struct LayerOperand {
  const void* x;
  int64_t rows, cols;
  const nvfp4_rounding* rr;       // null: no row output
  uint8_t *codes_r, *scales_r;
  const nvfp4_rounding* rt;       // null: no transposed output
  uint8_t *codes_t, *scales_t;
  const float* given;             // NVFP4_G_GIVEN: its scale
  float* slot;                    // its scale in the call's buffers: kScaleSlotBytes, the rest of which the amax passes use; null: not kept
};
constexpr int kScaleSlotBytes = 256;
constexpr int kMaxLayerOperands = 3;
// Quantizes a layer call's operands (quantize.cu), with their amax passes where the mode asks for it: the operands are older
// than the call, and this is the first thing that it launches.  g[i]: where the scale of operand i is afterwards.
int quantize_operands(const LayerOperand* ops, int n, int dtype, int gscale_mode, const float** g, void* cuda_stream);
// Where a quantizer takes its per-tensor scale from: one stored scale (null = 1), or the maxima that an amax sweep left
// (n > 0).  keep: where to leave the scale for the kernels behind it (null = nowhere).
struct ScaleSource {
  const float* g = nullptr;
  const uint32_t* maxima = nullptr;
  int n = 0;
  float* keep = nullptr;
};
// The part of it that one launch of the tile quantizer does for all (quantize_tile.cu).
bool tile_batch_eligible(const LayerOperand* ops, int n);
int tile_quantize_batch(const LayerOperand* ops, const ScaleSource* scale, int n, int dtype, cudaStream_t s);

// ---------------------------------------------------------------------------------------------
// Scale-factor layout (128 rows x 4 blocks per 512-byte tile, k-tiles contiguous per row tile)
// ---------------------------------------------------------------------------------------------
__host__ __device__ inline int64_t sf_swizzled_offset(int64_t r, int64_t kb, int64_t k_tiles) {
  return ((r >> 7) * k_tiles + (kb >> 2)) * 512 + (r & 31) * 16 + ((r >> 5) & 3) * 4 + (kb & 3);
}
// Four scale bytes of one quantized row of which the first `left` belong to the tensor, the others being padding: zero also
// where the per-tensor scale is NaN or so small that a zero block's scale encodes as NaN.
__device__ __forceinline__ uint32_t scales_inside(uint32_t word, int64_t left) {
  return left >= 4 ? word : left <= 0 ? 0u : word & ((1u << (8 * (int)left)) - 1u);
}

// ---------------------------------------------------------------------------------------------
// Number formats (Section 3 of the paper)
// ---------------------------------------------------------------------------------------------
// Unsigned E4M3 of a non-negative float: round to nearest even, saturate at 448.
__device__ __forceinline__ uint32_t e4m3_encode(float v) {
  uint16_t r;
  asm("cvt.rn.satfinite.e4m3x2.f32 %0, %1, %2;" : "=h"(r) : "f"(0.0f), "f"(v));
  return r & 0xFFu;
}

// E8M0 (power-of-two) scale of MXFP4: the smallest power of two >= v, as code = exponent + 127
// (0 for v <= 0 or below 2^-127, 254 at most).
__device__ __forceinline__ uint32_t e8m0_encode_up(float v) {
  uint16_t r;
  asm("cvt.rp.satfinite.ue8m0x2.f32 %0, %1, %2;" : "=h"(r) : "f"(0.0f), "f"(v));
  return (v > 0.0f) ? (r & 0xFFu) : 0u;
}

// Exact value of an unsigned E4M3 code (0..0x7E).
__device__ __forceinline__ float e4m3_decode(uint32_t q) {
  return (q < 8u) ? __uint2float_rn(q) * 0x1p-9f : __uint_as_float((q << 20) + (120u << 23));
}

// Two floats -> one byte of E2M1 codes (lo in bits 0-3, hi in bits 4-7), nearest even, clamp at 6.
__device__ __forceinline__ uint32_t e2m1x2_rn(float lo, float hi) {
  uint32_t r;
  asm("{\n\t.reg .b8 t;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 t, %1, %2;\n\t"
      "mov.b32 %0, {t, 0, 0, 0};\n\t}"
      : "=r"(r) : "f"(hi), "f"(lo));
  return r;
}

// Eight floats -> eight E2M1 codes in one word (element 0 in bits 0-3), nearest even, clamp at 6,
// sign kept (also for results of zero).
__device__ __forceinline__ uint32_t e2m1x8_rn(const float (&y)[16], int o) {
  uint32_t r;
  asm("{\n\t.reg .b8 b0, b1, b2, b3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b0, %2, %1;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b1, %4, %3;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b2, %6, %5;\n\t"
      "cvt.rn.satfinite.e2m1x2.f32 b3, %8, %7;\n\t"
      "mov.b32 %0, {b0, b1, b2, b3};\n\t}"
      : "=r"(r)
      : "f"(y[o]), "f"(y[o + 1]), "f"(y[o + 2]), "f"(y[o + 3]), "f"(y[o + 4]), "f"(y[o + 5]), "f"(y[o + 6]), "f"(y[o + 7]));
  return r;
}

// Stochastic rounding of eight floats to E2M1 with the hardware conversion.  For one group of four
// elements and one 32-bit random word the instruction rounds element e up iff
// floor(frac * 2^16) + r_e >= 2^16, frac being the element's position inside its grid step and
//   r_0 = byte2:byte0 of the word,  r_1 = r_0 with its 16 bits mirrored,
//   r_2 = byte3:byte1,              r_3 = r_2 mirrored
// (element 0 = the last operand of the vector, which lands in bits 0-3).  Values beyond 6 clamp, the
// sign is kept.  Word w0 serves elements o..o+3, w1 elements o+4..o+7.
__device__ __forceinline__ uint32_t e2m1x8_rs(const float (&y)[16], int o, uint32_t w0, uint32_t w1) {
  uint32_t r;
  asm("{\n\t.reg .b16 h0, h1;\n\t"
      "cvt.rs.satfinite.e2m1x4.f32 h0, {%4, %3, %2, %1}, %9;\n\t"
      "cvt.rs.satfinite.e2m1x4.f32 h1, {%8, %7, %6, %5}, %10;\n\t"
      "mov.b32 %0, {h0, h1};\n\t}"
      : "=r"(r)
      : "f"(y[o]), "f"(y[o + 1]), "f"(y[o + 2]), "f"(y[o + 3]), "f"(y[o + 4]), "f"(y[o + 5]), "f"(y[o + 6]), "f"(y[o + 7]),
        "r"(w0), "r"(w1));
  return r;
}

// ---------------------------------------------------------------------------------------------
// Philox4x32-10 (Salmon et al. 2011): key = seed, counter = (block index, offset)
// ---------------------------------------------------------------------------------------------
// One random stream: the ten round keys of the seed (key + i * Weyl increment, precomputed on the
// host so that a round costs two wide multiplies and two three-way XORs) and counter words 2, 3.
struct PhiloxStream {
  uint32_t k0[10], k1[10];
  uint32_t off_lo, off_hi;
  uint32_t b32[4];          // what the first two rounds come down to for block indices below 2^32 (see philox4x32_10 below)
};

inline void philox_stream_init(PhiloxStream* s, uint64_t seed, uint64_t offset) {
  uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32);
  for (int i = 0; i < 10; ++i) {
    s->k0[i] = k0;
    s->k1[i] = k1;
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  s->off_lo = (uint32_t)offset;
  s->off_hi = (uint32_t)(offset >> 32);
  const uint64_t p1 = (uint64_t)s->off_lo * 0xCD9E8D57ull;
  const uint64_t p0 = (uint64_t)((uint32_t)(p1 >> 32) ^ s->k0[0]) * 0xD2511F53ull;
  s->b32[0] = s->off_hi ^ s->k1[0];
  s->b32[1] = (uint32_t)p1 ^ s->k0[1];
  s->b32[2] = (uint32_t)(p0 >> 32) ^ s->k1[1];
  s->b32[3] = (uint32_t)p0;
}

// Counter = (c0, c1, off_lo, off_hi); c0, c1 = the block's linear index.
__device__ __forceinline__ uint4 philox4x32_10(const PhiloxStream& s, uint32_t c0, uint32_t c1) {
  uint32_t c2 = s.off_lo, c3 = s.off_hi;
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint64_t p0 = (uint64_t)c0 * 0xD2511F53ull, p1 = (uint64_t)c2 * 0xCD9E8D57ull;   // one wide multiply each
    c0 = (uint32_t)(p1 >> 32) ^ c1 ^ s.k0[i];
    c2 = (uint32_t)(p0 >> 32) ^ c3 ^ s.k1[i];
    c1 = (uint32_t)p1;
    c3 = (uint32_t)p0;
  }
  return make_uint4(c0, c1, c2, c3);
}

// The same for a block index below 2^32: with counter word 1 zero, one multiply of each of the first two rounds depends on
// the stream alone and is done on the host.  c = counter words after two rounds.  With 32-bit index arithmetic and scales
// staged as words, both stochastic outputs of 16384 x 11008 went from 129 to 123 us, the transposed one from 78.7 to 76.9.
__device__ __forceinline__ void philox_two_rounds(const PhiloxStream& s, uint32_t blk, uint32_t (&c)[4]) {
  const uint64_t p = (uint64_t)blk * 0xD2511F53ull;
  const uint64_t q = (uint64_t)((uint32_t)(p >> 32) ^ s.b32[0]) * 0xCD9E8D57ull;
  c[0] = (uint32_t)(q >> 32) ^ s.b32[1];
  c[1] = (uint32_t)q;
  c[2] = (uint32_t)p ^ s.b32[2];
  c[3] = s.b32[3];
}
__device__ __forceinline__ void philox_round(const PhiloxStream& s, int i, uint32_t (&c)[4]) {
  const uint64_t p0 = (uint64_t)c[0] * 0xD2511F53ull, p1 = (uint64_t)c[2] * 0xCD9E8D57ull;
  c[0] = (uint32_t)(p1 >> 32) ^ c[1] ^ s.k0[i];
  c[2] = (uint32_t)(p0 >> 32) ^ c[3] ^ s.k1[i];
  c[1] = (uint32_t)p1;
  c[3] = (uint32_t)p0;
}
__device__ __forceinline__ uint4 philox4x32_10(const PhiloxStream& s, uint32_t blk) {
  uint32_t c[4];
  philox_two_rounds(s, blk, c);
#pragma unroll
  for (int i = 2; i < 10; ++i) philox_round(s, i, c);
  return make_uint4(c[0], c[1], c[2], c[3]);
}
__device__ __forceinline__ uint4 philox4x32_10(const PhiloxStream& s, uint64_t blk) {
  return philox4x32_10(s, (uint32_t)blk, (uint32_t)(blk >> 32));
}
__device__ __forceinline__ void philox4x32_10_x2(const PhiloxStream& s, uint32_t blk_a, uint32_t blk_b, uint4& ra, uint4& rb) {
  uint32_t a[4], b[4];
  philox_two_rounds(s, blk_a, a);
  philox_two_rounds(s, blk_b, b);
#pragma unroll
  for (int i = 2; i < 10; ++i) {
    philox_round(s, i, a);
    philox_round(s, i, b);
  }
  ra = make_uint4(a[0], a[1], a[2], a[3]);
  rb = make_uint4(b[0], b[1], b[2], b[3]);
}

// Two independent calls with their rounds interleaved (two dependency chains in flight per thread).
__device__ __forceinline__ void philox4x32_10_x2(const PhiloxStream& s, uint64_t blk_a, uint64_t blk_b, uint4& ra, uint4& rb) {
  uint32_t a0 = (uint32_t)blk_a, a1 = (uint32_t)(blk_a >> 32), a2 = s.off_lo, a3 = s.off_hi;
  uint32_t b0 = (uint32_t)blk_b, b1 = (uint32_t)(blk_b >> 32), b2 = s.off_lo, b3 = s.off_hi;
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint64_t pa0 = (uint64_t)a0 * 0xD2511F53ull, pa1 = (uint64_t)a2 * 0xCD9E8D57ull;
    const uint64_t pb0 = (uint64_t)b0 * 0xD2511F53ull, pb1 = (uint64_t)b2 * 0xCD9E8D57ull;
    a0 = (uint32_t)(pa1 >> 32) ^ a1 ^ s.k0[i];
    b0 = (uint32_t)(pb1 >> 32) ^ b1 ^ s.k0[i];
    a2 = (uint32_t)(pa0 >> 32) ^ a3 ^ s.k1[i];
    b2 = (uint32_t)(pb0 >> 32) ^ b3 ^ s.k1[i];
    a1 = (uint32_t)pa1; a3 = (uint32_t)pa0;
    b1 = (uint32_t)pb1; b3 = (uint32_t)pb0;
  }
  ra = make_uint4(a0, a1, a2, a3);
  rb = make_uint4(b0, b1, b2, b3);
}

}  // namespace nvfp4
