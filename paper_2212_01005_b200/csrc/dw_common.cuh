// Depthwise 3x3 building blocks of the fused kernels: CUDA-core arithmetic on bf16 channel pairs held in
// shared memory as planes of [pixel][8 channels] (16 bytes per pixel), mixed-precision FMAs (bf16 operands as
// stored, fp32 accumulate), bias and ReLU6 fused into the store (Section III-A: simple operators are applied right
// after the window sum).
#pragma once
#include <cstdint>

namespace ago {
namespace dw {

// bf16x2(min(max(lo, 0), 6), min(max(hi, 0), 6)): the conversion clamps at 0, one packed min caps at 6.
__device__ __forceinline__ uint32_t relu6_pack(float lo, float hi) {
  uint32_t r;
  asm("{\n\t.reg .b32 t;\n\tcvt.rn.relu.bf16x2.f32 t, %2, %1;\n\tmin.bf16x2 %0, t, %3;\n\t}"
      : "=r"(r) : "f"(lo), "f"(hi), "r"(0x40C040C0u));   // the packed 6.0 is an operand, so one register serves every call
  return r;
}

// Shared-memory word loads / stores with an immediate byte offset.
template <int OFF>
__device__ __forceinline__ uint32_t lds32(uint32_t saddr) {
  uint32_t v;
  asm volatile("ld.shared.u32 %0, [%1+%2];" : "=r"(v) : "r"(saddr), "n"(OFF));
  return v;
}
template <int OFF = 0>
__device__ __forceinline__ void sts32(uint32_t saddr, uint32_t v) {
  asm volatile("st.shared.u32 [%0+%1], %2;" ::"r"(saddr), "n"(OFF), "r"(v) : "memory");
}

// acc += x * w for a packed pair of bf16 channels: the mixed-precision FMA takes the bf16 operands
// as they are (exact product, fp32 accumulate) -- no unpacking of the activations or the weights.
__device__ __forceinline__ void fma_pair(float2& acc, uint32_t x, uint32_t w) {
  asm("{\n\t.reg .b16 xl, xh, wl, wh;\n\t"
      "mov.b32 {xl, xh}, %2;\n\tmov.b32 {wl, wh}, %3;\n\t"
      "fma.rn.f32.bf16 %0, xl, wl, %0;\n\tfma.rn.f32.bf16 %1, xh, wh, %1;\n\t}"
      : "+f"(acc.x), "+f"(acc.y) : "r"(x), "r"(w));
}

// c + x * w without touching c: the first tap of a window starts from the bias.
__device__ __forceinline__ float2 fma_pair_from(float2 c, uint32_t x, uint32_t w) {
  float2 r;
  asm("{\n\t.reg .b16 xl, xh, wl, wh;\n\t"
      "mov.b32 {xl, xh}, %2;\n\tmov.b32 {wl, wh}, %3;\n\t"
      "fma.rn.f32.bf16 %0, xl, wl, %4;\n\tfma.rn.f32.bf16 %1, xh, wh, %5;\n\t}"
      : "=f"(r.x), "=f"(r.y) : "r"(x), "r"(w), "f"(c.x), "f"(c.y));
  return r;
}

struct Row3 { uint32_t v0, v1, v2; };   // three horizontally adjacent pixels of one channel pair
template <int PIX_STEP>
__device__ __forceinline__ Row3 load_row3(uint32_t a) {
  Row3 r;
  r.v0 = lds32<0>(a); r.v1 = lds32<PIX_STEP>(a); r.v2 = lds32<2 * PIX_STEP>(a);
  return r;
}
__device__ __forceinline__ uint32_t depthwise_point(const Row3& a, const Row3& b, const Row3& c, const uint32_t (&w)[9],
                                                    float2 bias) {
  float2 acc = bias;
  fma_pair(acc, a.v0, w[0]); fma_pair(acc, a.v1, w[1]); fma_pair(acc, a.v2, w[2]);
  fma_pair(acc, b.v0, w[3]); fma_pair(acc, b.v1, w[4]); fma_pair(acc, b.v2, w[5]);
  fma_pair(acc, c.v0, w[6]); fma_pair(acc, c.v1, w[7]); fma_pair(acc, c.v2, w[8]);
  return relu6_pack(acc.x, acc.y);
}

// E and D chunks are two planes of [pixel][8 channels] (16 bytes per pixel), which is also the
// un-swizzled K-major operand layout; all addresses below are 32-bit shared-memory addresses.
//
// Stride-2 depthwise 3x3 for one (channel pair, output column) and output rows [r0, r1), r1 > r0:
// consecutive output rows share one input row, which stays packed in registers (the loop body is
// unrolled over the two roles of that row).
__device__ __forceinline__ void depthwise_column_s2(uint32_t e_col, uint32_t d_col, int r0, int r1, int IW, int Wo,
                                                    const uint32_t (&w)[9], float2 bias) {
  const uint32_t e_pitch = (uint32_t)IW * 16u, d_pitch = (uint32_t)Wo * 16u;
  uint32_t src = e_col + (uint32_t)(r0 * 2) * e_pitch;
  uint32_t dst = d_col + (uint32_t)r0 * d_pitch;
  int n = r1 - r0;
  Row3 a = load_row3<16>(src), b, c;
  src += e_pitch;
  while (true) {
    b = load_row3<16>(src); c = load_row3<16>(src + e_pitch); src += 2 * e_pitch;
    sts32(dst, depthwise_point(a, b, c, w, bias)); dst += d_pitch;
    if (--n == 0) break;
    b = load_row3<16>(src); a = load_row3<16>(src + e_pitch); src += 2 * e_pitch;
    sts32(dst, depthwise_point(c, b, a, w, bias)); dst += d_pitch;
    if (--n == 0) break;
  }
}

// Stride-1 depthwise 3x3 for one channel pair and a block of 2 output rows x up to 7 output columns. The block is walked
// by INPUT column: the four pixels of a column are loaded, used for every tap they meet (outputs of three columns are in
// flight, their accumulators rotate by renaming) and dropped. All shared-memory offsets are immediates. `segw` is the
// block width the caller cuts rows into (the same for all threads: the walk ends there); `ncol` <= segw columns and
// `nrows` <= 2 rows are stored, by predicated stores, so that ragged blocks take the same instructions as whole ones.
// (The previous form held three columns of pixels and had a second copy of the code for ragged blocks: a warp with both
// kinds ran both, 5.9k cycles instead of 3.4k for two 14 x 56 chunks of 16 channels on one SM. This one: 3.3k for
// either; alone in its scheduler a block of width 7 takes 620 cycles instead of 710 / 1420, one of width 4 490.
// Measured and not taken: 4 output rows, the same; packed fp32 pairs, 30 % slower: their unpacking costs more slots.)
// e_row: address of the block's first input pixel in the row above the first output row; d_row: address of its first
// output pixel. The loads of a block with fewer valid rows or columns run past the valid pixels, inside shared memory.
constexpr int kSegCols = 7;       // the widest block
constexpr int kMinSegCols = 3;    // the narrowest one the early ends below know
// Width of the blocks a row of `wo` outputs is cut into: the narrowest that keeps the number of blocks, made odd -- a warp
// works on four neighbouring blocks, whose 16-byte pixels then lie in different banks.
inline int seg_width(int wo) {
  const int n = (wo + kSegCols - 1) / kSegCols, w = (wo + n - 1) / n;
  return w < kMinSegCols ? kMinSegCols : (w | 1);
}

template <int J>
__device__ __forceinline__ void depthwise_input_column(const uint32_t (&e)[4], uint32_t d0, uint32_t d1, int ncol, bool two,
                                                       const uint32_t (&w)[9], float2 bias, float2 (&done)[2], float2 (&mid)[2],
                                                       float2 (&first)[2]) {
  uint32_t x[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = lds32<J * 16>(e[i]);
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    if (J < kSegCols) {               // left tap of output column J
      first[r] = bias;
      fma_pair(first[r], x[r], w[0]); fma_pair(first[r], x[r + 1], w[3]); fma_pair(first[r], x[r + 2], w[6]);
    }
    if (J >= 1 && J <= kSegCols) {    // middle tap of output column J - 1
      fma_pair(mid[r], x[r], w[1]); fma_pair(mid[r], x[r + 1], w[4]); fma_pair(mid[r], x[r + 2], w[7]);
    }
    if (J >= 2) {                     // right tap of output column J - 2: complete
      fma_pair(done[r], x[r], w[2]); fma_pair(done[r], x[r + 1], w[5]); fma_pair(done[r], x[r + 2], w[8]);
    }
  }
  if constexpr (J >= 2) {
    if (J - 2 < ncol) {
      sts32<(J - 2) * 16>(d0, relu6_pack(done[0].x, done[0].y));
      if (two) sts32<(J - 2) * 16>(d1, relu6_pack(done[1].x, done[1].y));
    }
  }
}

__device__ __forceinline__ void depthwise_block(uint32_t e_row, uint32_t d_row, uint32_t e_pitch, uint32_t d_pitch, int segw, int ncol,
                                                int nrows, const uint32_t (&w)[9], float2 bias) {
  const uint32_t e[4] = {e_row, e_row + e_pitch, e_row + 2 * e_pitch, e_row + 3 * e_pitch};
  const uint32_t d0 = d_row, d1 = d_row + d_pitch;
  const bool two = nrows > 1;
  float2 a[2], b[2], c[2];
  depthwise_input_column<0>(e, d0, d1, ncol, two, w, bias, b, c, a);
  depthwise_input_column<1>(e, d0, d1, ncol, two, w, bias, c, a, b);
  depthwise_input_column<2>(e, d0, d1, ncol, two, w, bias, a, b, c);
  depthwise_input_column<3>(e, d0, d1, ncol, two, w, bias, b, c, a);
  depthwise_input_column<4>(e, d0, d1, ncol, two, w, bias, c, a, b);
  if (segw <= 3) return;
  depthwise_input_column<5>(e, d0, d1, ncol, two, w, bias, a, b, c);
  if (segw <= 4) return;
  depthwise_input_column<6>(e, d0, d1, ncol, two, w, bias, b, c, a);
  if (segw <= 5) return;
  depthwise_input_column<7>(e, d0, d1, ncol, two, w, bias, c, a, b);
  if (segw <= 6) return;
  depthwise_input_column<8>(e, d0, d1, ncol, two, w, bias, a, b, c);
}

}  // namespace dw
}  // namespace ago
