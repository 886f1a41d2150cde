// Fused pair of pointwise convolutions: 1x1 conv + bias [+ ReLU6] -> 1x1 conv + bias [+ ReLU6], one kernel
// (the "two pointwise convolutions" subgraph of the micro-benchmark, Section VI-B; in MobileNetV2-like networks
// the linear bottleneck of one block followed by the expansion of the next).
//
// Both operators are matrix multiplications over the pixel rows, so the link is the "downstream pointwise"
// category of Section III-B: the downstream tile keeps all its output channels and is tiled over rows, the upstream
// tile it needs is the same rows with all middle channels -- nothing is recomputed. CTAs are persistent (two per SM
// where the operands leave room) and walk over tiles of up to 128 pixel rows with three kinds of warps:
//   copy warp      TMA: the X tile as K-major blocks of 64 channels (128-byte swizzle); rows past the tensor and
//                  channels past C0 read as zero. The next X tile is requested as soon as the first product of this one
//                  is complete.
//   MMA warp       P2: mid[128 x C1] = X[128 x C0] * W1^T; P4: out[128 x C2] = mid[128 x C1] * W2^T (TMEM, fp32). The
//                  first product of the next tile runs while this tile's outputs are stored.
//   epilogue warps P3: TMEM -> registers: + b1 [ReLU6], bf16 -> shared memory as the swizzled A operand of the second
//                  product; P5: TMEM -> registers: + b2 [ReLU6], bf16 -> device memory, a 32-byte sector per store.
// Both weight matrices are fetched once per CTA into the same layout: by the copy warp's TMA loads where few CTAs ask for them,
// else by the epilogue threads' asynchronous copies through L1 (weights_by_tma). 1200 pixels x 64 -> 16 -> 64 3.15 -> 2.65 us,
// 1936 x 192 -> 40 -> 192 5.50 -> 4.93, the chain below on 1568 rows x 120 -> 240 5.79 -> 5.22, 17248 x 64 -> 128 4.53 -> 4.14.
// What bounds it: the stores and loads on large tensors, the chain weights -> product -> epilogue -> product -> epilogue
// of one tile on small ones. With block-wide barriers between the steps, the outputs staged in shared memory and the X
// tile's buffer busy until they had left it, a tile took 4.0-4.8 us with every unit idle most of that time; now 2.2-2.7.
// 100352 pixels x 144 -> 24 -> 144: 20.6 -> 14.1 us (8.8 us of memory traffic); the chain below on 32768 rows x
// 96 -> 192: 12.4 -> 7.7 us (3.9).
//
// The same kernel serves the projection chain of a patch-unfolded attention block (Section VI-B: matrix
// multiplication, reshape, add, reshape, transpose, reshape, matrix multiplication, reshape): the reshapes are
// views, the add takes a second input tensor, and the transpose of two leading axes only permutes the rows between
// the products -- so the tile's output rows are stored at their permuted positions and no layout operator costs a
// pass over memory. There the weights are GEMM operands ([K][N], used as N-major B operands as they lie in memory)
// and the tensor to add arrives by TMA in the buffer of the second product's A operand, which the first epilogue
// updates in place.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <unordered_map>

#include "fused.h"
#include "tc_common.cuh"
#include "tmap.h"

namespace ago {

namespace {

using namespace tc;

constexpr int kColWarps = 2;   // warps that share the 16-column groups of one tensor-memory lane quarter; 3 or 4: 2-5% slower
constexpr int kEpiThreads = 128 * kColWarps;      // epilogue threads; then the MMA warp and the copy warp
constexpr int kThreads = kEpiThreads + 64;
constexpr int kBM = 128, kBK = 64;
constexpr int kXBlock = kBM * kBK * 2;   // one K block of the X / mid tile: 16 KB

struct PwPwParams {
  const __nv_bfloat16* w1;   // [C1][C0]
  const __nv_bfloat16* w2;   // [C2][C1]
  const float* b1;
  const float* b2;
  __nv_bfloat16* out;        // [M][C2]
  unsigned int* status;
  int M, C0, C1, C2;
  int BR;                    // rows per tile (<= 128)
  int C0p, C1p, C2p;         // padded to the MMA granularity (16)
  int nkb0, nkb1;            // 64-channel K blocks of the first / second product
  int act1, act2;            // ReLU6 after the first / second convolution
  int perm_a, perm_b;        // output row ((g * a + i) * b + j) is stored as row ((g * b + j) * a + i); 0: no permutation
  int w1_block, w2_block;    // byte distance between the 64-wide blocks of the weight tiles
  uint32_t c0_recip, c1_recip;   // reciprocals of the 16-byte pieces per row of W1 / W2 as they lie in memory
  int x_tx, r_tx;            // bytes one X tile / its tile of the added tensor brings in (TMA transaction counts)
  int tmem_cols, acc2_col;   // tensor-memory columns; first column of the second product (0: both share their columns)
  int wide_store;            // output rows start at multiples of 32 bytes
  int off_x, off_a, off_w1, off_w2, off_b, off_bar;
  int tma_weights;           // the weights come by TMA (the kernel template's TMA)
  int w1_rows, w2_rows, w1_box, w2_box, w1_tx, w2_tx;     // rows of a block of the weight tiles and of one load, bytes of all blocks
};

// ReLU6 of two bf16 values: rounding is monotone and both bounds are bf16 numbers, so it may follow the rounding.
__device__ __forceinline__ uint32_t relu6_bf16x2(uint32_t w) {
  const __nv_bfloat162 lo = __float2bfloat162_rn(0.0f), hi = __float2bfloat162_rn(6.0f);
  const __nv_bfloat162 v = __hmin2(__hmax2(*reinterpret_cast<const __nv_bfloat162*>(&w), lo), hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

// 16 fp32 sums + 16 bias values of shared memory
__device__ __forceinline__ void add_bias16(uint32_t (&v)[16], const float* bias) {
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const float4 t4 = *reinterpret_cast<const float4*>(bias + 4 * j);
    v[4 * j] = __float_as_uint(__uint_as_float(v[4 * j]) + t4.x);
    v[4 * j + 1] = __float_as_uint(__uint_as_float(v[4 * j + 1]) + t4.y);
    v[4 * j + 2] = __float_as_uint(__uint_as_float(v[4 * j + 2]) + t4.z);
    v[4 * j + 3] = __float_as_uint(__uint_as_float(v[4 * j + 3]) + t4.w);
  }
}

template <bool TMA> struct WeightMaps { CUtensorMap w1, w2; };
template <> struct WeightMaps<false> {};

// CHAIN: the GEMM -> + tensor -> row permutation -> GEMM chain: [K][N] weights, no biases, no activations.
// Otherwise two 1x1 convolutions: [N][K] weights, biases and optional activations.
// TMA: the copy warp fetches the weights too, and nothing but the barriers' set-up is ahead of the roles; otherwise the epilogue
// threads copy them through L1 (weights_by_tma).
template <bool CHAIN, bool TMA>
__global__ void __launch_bounds__(kThreads, 2)
pwpw_fused_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_r,
                  const __grid_constant__ WeightMaps<TMA> tmap_w, const PwPwParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sX = smem + p.off_x;
  uint8_t* sA = smem + p.off_a;
  uint8_t* sW1 = smem + p.off_w1;
  uint8_t* sW2 = smem + p.off_w2;
  float* sB1 = reinterpret_cast<float*>(smem + p.off_b);
  float* sB2 = sB1 + p.C1p;
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.off_bar);
  uint64_t* bar_x = bars;        // X tile landed
  uint64_t* bar_r = bars + 1;    // tile of the added tensor landed
  uint64_t* bar_m1 = bars + 2;   // first product complete
  uint64_t* bar_m2 = bars + 3;   // second product complete
  uint64_t* bar_a = bars + 4;    // A operand of the second product written, columns of the first product drained
  uint64_t* bar_d = bars + 5;    // columns of the second product drained (used where both products share their columns)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 6);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(bars + 7);
  uint64_t* bar_w = bars + 8;    // TMA: [2] W1, W2 landed

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  constexpr int kMmaWarp = kEpiThreads / 32, kCopyWarp = kMmaWarp + 1;
  const int ntiles = (p.M + p.BR - 1) / p.BR;   // tiles of BR <= 128 rows: the MMAs still span 128 rows, the rest is ignored
  const bool shared_cols = p.acc2_col == 0;

  if (tid == kCopyWarp * 32) {
    *abort_flag = 0u;
    for (int i = 0; i < 4; ++i) mbar_init(bars + i, 1);
    mbar_init(bar_a, kEpiThreads / 32);
    mbar_init(bar_d, kEpiThreads / 32);
    if (TMA) { mbar_init(bar_w, 1); mbar_init(bar_w + 1, 1); }
    fence_mbar_init();
    fence_proxy_async_smem();
    tma_prefetch_desc(&tmap_x);
    if (CHAIN) tma_prefetch_desc(&tmap_r);
    if constexpr (TMA) { tma_prefetch_desc(&tmap_w.w1); tma_prefetch_desc(&tmap_w.w2); }
  }
  if (warp == kMmaWarp) {
    tmem_alloc(tmem_slot, (uint32_t)p.tmem_cols);
    tmem_relinquish();
  }
  auto load_x = [&](int tile) {   // one thread
    mbar_arrive_expect_tx(bar_x, (uint32_t)p.x_tx);
    for (int kb = 0; kb < p.nkb0; ++kb) tma_load_2d(sX + kb * kXBlock, &tmap_x, bar_x, kb * kBK, tile * p.BR);
  };
  auto load_r = [&](int tile) {   // one thread
    mbar_arrive_expect_tx(bar_r, (uint32_t)p.r_tx);
    for (int kb = 0; kb < p.nkb1; ++kb) tma_load_2d(sA + kb * kXBlock, &tmap_r, bar_r, kb * kBK, tile * p.BR);
  };
  // the blocks of 64 columns of a weight matrix as it lies in memory; rows and columns that the padding adds read as zeros
  auto load_w = [&](const CUtensorMap* map, uint64_t* bar, uint8_t* dst, int rows, int box, int tx) {   // one thread
    mbar_arrive_expect_tx(bar, (uint32_t)tx);
    for (int at = 0, n0 = 0; at < tx; at += rows * 128, n0 += kBK)
      for (int r0 = 0; r0 < rows; r0 += box) tma_load_2d(dst + at + r0 * 128, map, bar, n0, r0);
  };
  auto meet = [&]() {
    tcgen05_fence_before_sync();
    __syncthreads();
    tcgen05_fence_after_sync();
  };
  if (TMA) meet();
  grid_dependency_wait();
  grid_launch_dependents_if(warp == kMmaWarp);
  if (tid == kCopyWarp * 32 && (int)blockIdx.x < ntiles) {
    load_x(blockIdx.x);
    if constexpr (TMA) load_w(&tmap_w.w1, bar_w, sW1, p.w1_rows, p.w1_box, p.w1_tx);
    if (CHAIN) load_r(blockIdx.x);
    if constexpr (TMA) load_w(&tmap_w.w2, bar_w + 1, sW2, p.w2_rows, p.w2_box, p.w2_tx);
  }
  auto stage_biases = [&]() {       // by the epilogue threads
    for (int i = tid; i < p.C1p + p.C2p; i += kEpiThreads)
      sB1[i] = i < p.C1p ? (i < p.C1 && p.b1 ? __ldg(p.b1 + i) : 0.0f) : (i - p.C1p < p.C2 && p.b2 ? __ldg(p.b2 + i - p.C1p) : 0.0f);
  };
  // Weights: 16-byte asynchronous copies into the swizzled blocks, W1 as one group and W2 as a second one that is
  // only waited for before the first tile's second product; rows and reduction channels added by the padding are
  // zero-filled. All CTAs read the same few lines at the same moment, which the lines' L2 slices serve one after the
  // other: the copies go through L1, so that a line is requested once per SM (27783 pixels x 112/24 channels: 5.1 us,
  // 7.5 us past L1, from sector to sector).
  if (!TMA && tid < kEpiThreads) {
    // [N][K] weights: a piece is (row n, 16-byte chunk of k) -> K-major block k / 64, row n;
    // [K][N] weights: a piece is (row k, 16-byte chunk of n) -> N-major block n / 64, row k
    // The valid pieces lie one after the other in memory.
    auto stage = [&](const __nv_bfloat16* w, uint8_t* dst, int block, int rows, int cols, int vrows, int vcols, uint32_t recip) {
      auto place = [&](int row, int ch) { return (uint32_t)((ch >> 3) * block) + swz_offset((uint32_t)row, (uint32_t)(ch & 7), 128); };
      const int vcpr = vcols >> 3, cpr = cols >> 3;
      const uint32_t d0 = smem_u32(dst);
      for (int i = tid; i < vrows * vcpr; i += kEpiThreads) {
        const int row = (int)fast_div((uint32_t)i, (uint32_t)vcpr, recip);
        cp_async_16_l1(d0 + place(row, i - row * vcpr), w + i * 8);
      }
      cp_async_commit();
      if (vcpr < cpr)   // one chunk of reduction channels or columns
        for (int i = tid; i < rows; i += kEpiThreads) *reinterpret_cast<uint4*>(dst + place(i, vcpr)) = make_uint4(0, 0, 0, 0);
      if (vrows < rows)   // eight rows; their products meet the zero columns of the other operand, which cancel finite values only
        for (int i = tid; i < 8 * cpr; i += kEpiThreads) *reinterpret_cast<uint4*>(dst + place(vrows + (i & 7), i >> 3)) = make_uint4(0, 0, 0, 0);
    };
    if (CHAIN) {
      stage(p.w1, sW1, p.w1_block, p.C0p, p.C1p, p.C0, p.C1, p.c0_recip);
      stage(p.w2, sW2, p.w2_block, p.C1p, p.C2p, p.C1, p.C2, p.c1_recip);
    } else {
      stage(p.w1, sW1, p.w1_block, p.C1p, p.C0p, p.C1, p.C0, p.c0_recip);
      stage(p.w2, sW2, p.w2_block, p.C2p, p.C1p, p.C2, p.C1, p.c1_recip);
      stage_biases();
    }
    cp_async_wait_but_one();
    fence_proxy_async_smem();
  }
  if (!TMA) meet();
  const uint32_t tmem_base = *tmem_slot;

  if (warp == kCopyWarp) {
    if (lane == 0)
      for (int tile = blockIdx.x + gridDim.x, it = 0; tile < ntiles; tile += gridDim.x, ++it) {
        mbar_wait(bar_m1, (uint32_t)it & 1u, abort_flag, p.status, 0x903);   // the first product has read the X tile
        load_x(tile);
        if (CHAIN) {
          mbar_wait(bar_m2, (uint32_t)it & 1u, abort_flag, p.status, 0x905);   // the second product has read the buffer
          load_r(tile);
        }
      }
  } else if (warp == kMmaWarp) {   // converged; MMAs predicated on one elected lane, see tc_common.cuh
    const uint32_t elected = elect_one();
    const uint32_t idesc1 = make_idesc_bf16(128, (uint32_t)p.C1p, 0, CHAIN ? 1u : 0u);
    const uint32_t idesc2 = make_idesc_bf16(128, (uint32_t)p.C2p, 0, CHAIN ? 1u : 0u);
    // K-major B: one block per 64 reduction channels, 32 bytes per step; N-major B: 16 rows of 128 bytes per step, the
    // 64-column blocks w_block apart (LBO)
    auto product = [&](uint32_t acc, const uint8_t* a, const uint8_t* w, int w_block, int nkb, int Kp, uint32_t idesc) {
      for (int kb = 0; kb < nkb; ++kb) {
        const uint64_t ad = make_smem_desc(smem_u32(a + kb * kXBlock), 0, 1024, SW_128B);
        const uint64_t bd = CHAIN ? make_smem_desc(smem_u32(w + kb * 4 * 2048), (uint32_t)w_block, 1024, SW_128B)
                                  : make_smem_desc(smem_u32(w + kb * w_block), 0, 1024, SW_128B);
        const uint32_t bstep = CHAIN ? 2048u >> 4 : 2u;
        const int ksteps = min(4, (Kp - kb * kBK) / 16);
        for (int ks = 0; ks < ksteps; ++ks) umma_bf16_elected_acc(acc, ad + 2u * ks, bd + bstep * ks, idesc, elected, (kb | ks) != 0);
      }
    };
    for (int tile = blockIdx.x, it = 0; tile < ntiles; tile += gridDim.x, ++it) {
      const uint32_t par = (uint32_t)it & 1u;
      if (shared_cols && it) mbar_wait(bar_d, par ^ 1u, abort_flag, p.status, 0x906);
      // ---- P2: first product ----
      mbar_wait(bar_x, par, abort_flag, p.status, 0x900);
      if (TMA && it == 0) mbar_wait(bar_w, 0, abort_flag, p.status, 0x908);
      tcgen05_fence_after_sync();
      product(tmem_base, sX, sW1, p.w1_block, p.nkb0, p.C0p, idesc1);
      umma_commit_elected(bar_m1, elected);
      // ---- P4: second product ----
      mbar_wait(bar_a, par, abort_flag, p.status, 0x907);
      if (TMA && it == 0) mbar_wait(bar_w + 1, 0, abort_flag, p.status, 0x909);
      tcgen05_fence_after_sync();
      product(tmem_base + (uint32_t)p.acc2_col, sA, sW2, p.w2_block, p.nkb1, p.C1p, idesc2);
      umma_commit_elected(bar_m2, elected);
    }
  } else {
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const int quarter_rows = (warp & 3) * 32;   // first row of this warp's tensor-memory lane quarter
    const int half = warp >> 2;                 // the warps of a lane quarter take the 16-column groups of an epilogue round-robin
    const int r = quarter_rows + lane;          // this thread's row of the tile = its tensor-memory lane
    if (TMA && !CHAIN) {                        // while the first tile and the weights travel
      stage_biases();
      named_barrier_sync(1, kEpiThreads);
    }
    for (int tile = blockIdx.x, it = 0; tile < ntiles; tile += gridDim.x, ++it) {
      const uint32_t par = (uint32_t)it & 1u;
      const int row0 = tile * p.BR, rows = min(p.BR, p.M - row0);
      int m = row0 + r;   // output row
      if (CHAIN) {
        const int ab = p.perm_a * p.perm_b;
        const int g = m / ab, rem = m - g * ab, i = rem / p.perm_b, j = rem - i * p.perm_b;
        m = (g * p.perm_b + j) * p.perm_a + i;
      }
      mbar_wait(bar_m1, par, abort_flag, p.status, 0x901);
      if (CHAIN) mbar_wait(bar_r, par, abort_flag, p.status, 0x904);
      tcgen05_fence_after_sync();
      // ---- P3: [+ b1, ReLU6 | + tensor] -> swizzled A operand of the second product (no rows past the tile) ----
      if (quarter_rows < rows)
        for (int g = half; g < p.C1p / 16; g += kColWarps) {
          uint32_t v[16], w[8];
          tmem_ld_x16(tmem_base + lane_base + g * 16, v);
          uint8_t* blk = sA + (g >> 2) * kXBlock;              // 64 channels per block = 4 groups = 8 chunks of 16 bytes
          const uint32_t ch = (uint32_t)(g & 3) * 2u;
          uint4* d0 = reinterpret_cast<uint4*>(blk + swz_offset((uint32_t)r, ch, 128));
          uint4* d1 = reinterpret_cast<uint4*>(blk + swz_offset((uint32_t)r, ch + 1u, 128));
          if (CHAIN) {   // the tensor to add lies where the result goes
            const uint4 a0 = *d0, a1 = *d1;
            const uint32_t add[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
            tmem_ld_wait_on(v);
#pragma unroll
            for (int j = 0; j < 8; ++j)
              w[j] = pack_bf16x2(__uint_as_float(v[2 * j]) + bf16_lo(add[j]), __uint_as_float(v[2 * j + 1]) + bf16_hi(add[j]));
          } else {
            tmem_ld_wait_on(v);
            add_bias16(v, sB1 + g * 16);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              w[j] = pack_bf16x2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
              if (p.act1) w[j] = relu6_bf16x2(w[j]);
            }
          }
          *d0 = make_uint4(w[0], w[1], w[2], w[3]);
          *d1 = make_uint4(w[4], w[5], w[6], w[7]);
        }
      if (!TMA && it == 0) cp_async_wait_all();   // W2 (this thread's pieces; the arrivals below cover everybody's)
      fence_proxy_async_smem();
      tcgen05_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(bar_a);
      mbar_wait(bar_m2, par, abort_flag, p.status, 0x902);
      tcgen05_fence_after_sync();
      // ---- P5: [+ b2, ReLU6] -> device memory; every thread its row, 32 bytes at a time ----
      if (quarter_rows < rows) {
        __nv_bfloat16* orow = p.out + (int64_t)m * p.C2;
        for (int g = half; g < p.C2p / 16; g += kColWarps) {
          uint32_t v[16], w[8];
          tmem_ld_x16(tmem_base + (uint32_t)p.acc2_col + lane_base + g * 16, v);
          tmem_ld_wait_on(v);
          if (!CHAIN) add_bias16(v, sB2 + g * 16);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            w[j] = pack_bf16x2(__uint_as_float(v[2 * j]), __uint_as_float(v[2 * j + 1]));
            if (!CHAIN && p.act2) w[j] = relu6_bf16x2(w[j]);
          }
          if (r < rows) {
            if (p.wide_store) {
              store_global_32(orow + g * 16, w);
            } else {
              *reinterpret_cast<uint4*>(orow + g * 16) = make_uint4(w[0], w[1], w[2], w[3]);
              if (g * 16 + 8 < p.C2) *reinterpret_cast<uint4*>(orow + g * 16 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
            }
          }
        }
      }
      if (shared_cols) {
        tcgen05_fence_before_sync();
        __syncwarp();
        if (lane == 0) mbar_arrive(bar_d);
      }
    }
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  if (warp == kMmaWarp) tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
}

int round_up(int v, int m) { return (v + m - 1) / m * m; }

// Whether the weights come by TMA. That takes one thread and starts at once, where the copies take every thread 1.5k to 3.7k
// cycles; but each row of a block is a request to L2 past L1, and all CTAs make them for the same lines at the same moment.
// Against the copies, 134 pairs and 123 chains of 1 to 60000 rows, time by TMA over time by copies:
//   pairs    up to 40 CTAs 0.78 to 0.96; with 12 KB of weights up to 64 CTAs (16 KB: 72) 0.83 to 0.95, but 1.10 at 72 with 13.8 KB;
//            rows of whole 64 bytes and tiles of up to 64 rows 0.9 to 0.97 up to one CTA per SM; else 1.0 to 1.26 from 86 CTAs on
//   chains   up to 24 CTAs 0.84 to 0.97; with less than 20 KB of weights 1.01 to 1.10 from 31 CTAs on, with more 0.82 to 1.0 up to 72;
//            rows of whole 64 bytes 0.89 to 1.02 up to one CTA per SM, 1.01 to 1.02 with tiles of more than 120 rows; else up to 1.2;
//            weights in rows of 16 bytes (8 columns) 1.02 to 1.12 whatever the CTAs
// and 1.0 to 1.4 with two CTAs per SM.
bool weights_by_tma(const PwPwParams& q, bool chain, int grid, int sms) {
  const int bytes = 2 * q.C1 * (q.C0 + q.C2);
  const bool whole = q.C0 % 32 == 0 && q.C1 % 32 == 0 && q.C2 % 32 == 0 && q.BR <= (chain ? 120 : 64);
  if (chain && std::min(q.C1, q.C2) < 16) return false;
  if (grid <= (chain ? 24 : 40)) return true;
  if (bytes < (chain ? 20 : 12) * 1024) return false;
  return grid <= (whole ? sms : bytes >= 16 * 1024 ? 72 : 64);
}

struct PwPwHost {
  PwPwParams prm;
  int smem_bytes = 0;
  int grid = 0;   // persistent CTAs: two per SM
  bool chain = false;   // the GEMM -> + input -> row transpose -> GEMM chain instead of two 1x1 convolutions
  std::unordered_map<const void*, CUtensorMap> maps, maps_r, maps_w1, maps_w2;   // tensor maps of X / the added tensor / the weights by base address
};

}  // namespace

ago_status_t pwpw_plan(Plan* plan, FusedState* st, std::string* err) {
  const auto& ops = plan->ops;
  auto* host = new PwPwHost();
  PwPwParams& q = host->prm;
  q = PwPwParams{};
  auto bad = [&](const char* m) { *err = std::string("fused pointwise pair: ") + m; delete host; return AGO_ERR_UNSUPPORTED; };
  const OpInfo& a = ops[0];
  q.C0 = (int)a.in.last();
  q.M = (int)(a.in.numel() / q.C0);
  q.C1 = a.op.p[0];
  if (plan->fused_kernel == AGO_KERNEL_GEMM_PERMUTE_GEMM) {
    // gemm, reshape, add_input, reshape [G, A, B, C1], transpose (A, B), reshape, gemm, reshape
    host->chain = true;
    q.C2 = ops[6].op.p[0];
    q.perm_a = (int)ops[3].out.d[1]; q.perm_b = (int)ops[3].out.d[2];
    if (a.in.numel() >= (1ll << 31) || ops[7].out.numel() >= (1ll << 31)) return bad("tensors of 2^31 elements or more are not supported");
  } else {
    // conv, bias, [relu6], conv, bias, [relu6]
    int i2 = 2;
    if (ops[2].op.kind == AGO_OP_RELU6) { q.act1 = 1; i2 = 3; }
    q.act2 = (int)ops.size() > i2 + 2 ? 1 : 0;
    q.C2 = ops[i2].op.p[0];
  }
  if (q.C0 % 8 || q.C1 % 8 || q.C2 % 8) return bad("channel counts must be multiples of 8");
  q.C0p = round_up(q.C0, 16); q.C1p = round_up(q.C1, 16); q.C2p = round_up(q.C2, 16);
  if (q.C1p > 256 || q.C2p > 256) return bad("more than 256 middle or output channels is not supported");
  q.nkb0 = (q.C0 + kBK - 1) / kBK; q.nkb1 = (q.C1p + kBK - 1) / kBK;
  const int w1_chunks = (host->chain ? q.C1p : q.C0p) / 8, w2_chunks = (host->chain ? q.C2p : q.C1p) / 8;
  const int w1_rows = host->chain ? q.C0p : q.C1p, w2_rows = host->chain ? q.C1p : q.C2p;
  q.c0_recip = fast_div_recip((host->chain ? q.C1 : q.C0) / 8); q.c1_recip = fast_div_recip((host->chain ? q.C2 : q.C1) / 8);
  q.w1_block = w1_rows * 128; q.w2_block = w2_rows * 128;
  q.w1_rows = w1_rows; q.w2_rows = w2_rows;
  q.w1_tx = (w1_chunks + 7) / 8 * q.w1_block; q.w2_tx = (w2_chunks + 7) / 8 * q.w2_block;
  // a load brings up to 256 rows: the fewest equal pieces of whole swizzle patterns
  auto box_rows = [](int rows) { int n = (rows + 255) / 256; while (rows % (8 * n) != 0) ++n; return rows / n; };
  q.w1_box = box_rows(w1_rows); q.w2_box = box_rows(w2_rows);
  int off = 0;
  auto take = [&](int bytes) { int o = off; off = round_up(off + bytes, 1024); return o; };
  q.off_x = take(q.nkb0 * kXBlock);
  q.off_a = take(q.nkb1 * kXBlock);
  q.off_w1 = take(q.w1_tx);
  q.off_w2 = take(q.w2_tx);
  q.off_b = take((q.C1p + q.C2p) * 4);
  q.off_bar = take(128);
  host->smem_bytes = off + 1024;
  if (host->smem_bytes > 227 * 1024) return bad("the operands of one row tile do not fit shared memory");
  if ((long)w1_rows * w1_chunks > 65535 || (long)w2_rows * w2_chunks > 65535)
    return bad("operands too large for the copy index arithmetic");
  // Rows per tile. Up to one 128-row tile per SM: an even share for one CTA per SM, but no less than 32 rows, the share
  // of one warp -- a tile takes as long with fewer, and every further CTA reads the same weights at the same moment
  // (2523 rows x 176/40 channels on 79 CTAs 5.3 us, on 141 5.7 us, on 281 6.7 us). Beyond: with k = rounds of 128-row
  // tiles over the resident CTAs, the smallest height that still needs k rounds -- less work in each.
  const long sms = device_sm_count(), slots = (host->smem_bytes <= 113 * 1024 ? 2 : 1) * sms;
  const bool one_round = q.M <= sms * kBM;
  const long k = ((long)(q.M + kBM - 1) / kBM + slots - 1) / slots;
  q.BR = one_round ? std::max(32, (int)((q.M + sms - 1) / sms)) : (int)std::min<long>(kBM, (q.M + k * slots - 1) / (k * slots));
  // Each product has tensor-memory columns of its own, so that the next tile's first product need not wait for this
  // tile's outputs -- unless there is none, or two CTAs would then not find room on an SM
  auto columns = [](int n) { int c = 32; while (c < n) c *= 2; return c; };
  q.acc2_col = !one_round && columns(q.C1p + q.C2p) * (slots / sms) <= 512 ? q.C1p : 0;
  q.tmem_cols = columns(q.acc2_col ? q.C1p + q.C2p : std::max(q.C1p, q.C2p));
  q.x_tx = q.nkb0 * q.BR * 128;
  q.r_tx = q.nkb1 * q.BR * 128;
  host->grid = (int)std::min<long>((q.M + q.BR - 1) / q.BR, slots);
  q.tma_weights = weights_by_tma(q, host->chain, host->grid, (int)sms) ? 1 : 0;
  st->impl = host;
  st->impl_free = [](void* p) { delete static_cast<PwPwHost*>(p); };
  st->tile_rows = q.BR; st->grid = host->grid; st->smem_bytes = host->smem_bytes;
  plan->tile_rows = q.BR; plan->smem_bytes = host->smem_bytes; plan->fused_variant = q.tma_weights;
  return AGO_OK;
}

namespace {
template <bool CHAIN, bool TMA>
cudaError_t launch_pwpw(const PwPwHost& host, const PwPwParams& q, const CUtensorMap& mx, const CUtensorMap& mr, const WeightMaps<TMA>& mw, cudaStream_t stream) {
  static int smem_opt_in[64] = {};
  const cudaError_t e = ensure_max_dynamic_smem(reinterpret_cast<const void*>(pwpw_fused_kernel<CHAIN, TMA>), smem_opt_in);
  if (e != cudaSuccess) return e;
  FusedLaunch launch(dim3((unsigned)host.grid), kThreads, (size_t)host.smem_bytes, stream);
  return cudaLaunchKernelEx(&launch.config, pwpw_fused_kernel<CHAIN, TMA>, mx, mr, mw, q);
}
}  // namespace

ago_status_t pwpw_run(const Plan& plan, FusedState* st, const void* const* inputs, const void* const* weights,
                      void* output, unsigned int* status_word, cudaStream_t stream, std::string* err) {
  (void)plan;
  PwPwHost* host = static_cast<PwPwHost*>(st->impl);
  PwPwParams q = host->prm;
  if (host->chain) {
    q.w1 = static_cast<const __nv_bfloat16*>(weights[0]); q.w2 = static_cast<const __nv_bfloat16*>(weights[1]);
    q.b1 = nullptr; q.b2 = nullptr;
  } else {
    q.w1 = static_cast<const __nv_bfloat16*>(weights[0]); q.b1 = static_cast<const float*>(weights[1]);
    q.w2 = static_cast<const __nv_bfloat16*>(weights[2]); q.b2 = static_cast<const float*>(weights[3]);
  }
  q.out = static_cast<__nv_bfloat16*>(output);
  q.status = status_word;
  q.wide_store = q.C2 % 16 == 0 && reinterpret_cast<uintptr_t>(output) % 32 == 0;
  // [M][C] bf16 matrices as tiles of 64 columns: BR rows of X and of the added tensor, blocks of the weights
  auto get_map = [&](std::unordered_map<const void*, CUtensorMap>& cache, const void* base, int M, int C, int box_rows, CUtensorMap* out) -> bool {
    auto it = cache.find(base);
    if (it == cache.end()) {
      CUtensorMap m;
      const uint64_t dims[2] = {(uint64_t)C, (uint64_t)M};
      const uint64_t strides[1] = {(uint64_t)C * 2};
      const uint32_t box[2] = {(uint32_t)kBK, (uint32_t)box_rows};
      if (!encode_tmap_bf16(&m, base, 2, dims, strides, box, 128, err)) return false;
      if (cache.size() > 4096) cache.clear();
      it = cache.emplace(base, m).first;
    }
    *out = it->second;
    return true;
  };
  CUtensorMap mx, mr;
  WeightMaps<true> mw;
  if (!get_map(host->maps, inputs[0], q.M, q.C0, q.BR, &mx)) return AGO_ERR_CUDA;
  mr = mx;
  if (host->chain && !get_map(host->maps_r, inputs[1], q.M, q.C1, q.BR, &mr)) return AGO_ERR_CUDA;
  if (q.tma_weights) {      // 1x1 convolutions: [N][K]; the chain's operands: [K][N]
    if (!get_map(host->maps_w1, q.w1, host->chain ? q.C0 : q.C1, host->chain ? q.C1 : q.C0, q.w1_box, &mw.w1)) return AGO_ERR_CUDA;
    if (!get_map(host->maps_w2, q.w2, host->chain ? q.C1 : q.C2, host->chain ? q.C2 : q.C1, q.w2_box, &mw.w2)) return AGO_ERR_CUDA;
  }
  cudaError_t e = host->chain ? (q.tma_weights ? launch_pwpw<true, true>(*host, q, mx, mr, mw, stream) : launch_pwpw<true, false>(*host, q, mx, mr, {}, stream))
                              : (q.tma_weights ? launch_pwpw<false, true>(*host, q, mx, mr, mw, stream) : launch_pwpw<false, false>(*host, q, mx, mr, {}, stream));
  if (e != cudaSuccess) { *err = std::string("fused pointwise pair launch: ") + cudaGetErrorString(e); return AGO_ERR_CUDA; }
  return AGO_OK;
}

}  // namespace ago
