// Fused feed-forward chain on a thread-block cluster: Y = GELU(X W1 + b1) W2 + b2; the hidden activations H never leave
// the SMs. With enough row blocks to fill the device nothing is reduced through device memory and the run is one kernel;
// with few row blocks each row block's hidden tiles are split over J clusters, whose output shares meet in an fp32 buffer
// (J additions per element), and a second, small launch turns the buffer into the output. There the run is a chain of
// latencies, so a cluster of one step requests everything it needs at once, keeps only the rows that exist and takes hidden
// tiles of 64 where they put more clusters to work: 768 -> 3072 -> 768 with 1 row 14.6 -> 7.9 us, 128 rows 18.1 -> 10.8,
// 256 rows 18.7 -> 11.6, 512 rows 19.9 -> 15.7 (of which 3.8 us are the 9.4 MB of additions at the rate of the L2).
//
// Tile choice (Section III-B, "downstream pointwise / matmul"): the second GEMM reuses H only along its output
// columns, so the downstream tile keeps ALL output columns of a block of 128 rows. Those (768 fp32 columns for
// BERT-base) do not fit the tensor memory of one SM next to the first GEMM's accumulator -- but they fit the tensor
// memory of a CLUSTER: CS CTAs (CS = 2..4) work on the same 128 rows, CTA r owns output columns
// [r N2/CS, (r+1) N2/CS) and computes every CS-th tile of 128 (or 64) hidden units. A finished H tile (bias, GELU, bf16,
// 32 KB as a swizzled K-major operand) is copied to the same shared-memory slot of every peer with one bulk
// shared-to-shared copy per peer (distributed shared memory), so every H tile is computed once and multiplied
// into all N2 output columns without recomputation and without reductions outside the SM.
//
// Per CTA (rank r), T = hidden tiles / CS steps:
//   ring   two TMA warps, every second load each (ffn_cluster_shape.h, kLoadsOfOneStage): X [RP x 64] + W1 [64 x BH] for the first
//          GEMM, W2 [64 x N2/CS] for the second; a third one for W2 tiles with memory of their own. Converged, an elected lane issuing, one load per operand: a thread in a lane-0 branch that loaded
//          every 64 columns by themselves took 350 cycles per stage, 4.5k of a one-step run's 34k (512 rows 17.4 -> 15.7 us,
//          64 rows 11.2 -> 9.5, 1815 rows 40 -> 36)
//   MMA    one warp: G1(t+1): Hacc[(t+1) & 1] = X W1[:, tile (t+1) CS + r]; then for k = 0..CS-1
//          G2(k): out += H slot k * W2[tile t CS + k, own columns]; its completion is committed onto CTA k's
//          "slot consumed" barrier
//   epi    8 or 16 warps: Hacc[t & 1] -> + b1, GELU, bf16 -> own slot r (after every CTA has consumed its previous
//          content) -> announce locally, bulk-copy to the peers' slot r with completion on their "slot full" barrier
//   end    out (TMEM) -> + b2 -> bf16 -> device memory
// Every wait is bounded; a CTA leaves only after a cluster barrier, so no peer copies into an exited CTA.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <unordered_map>

#include "ffn_cluster_shape.h"
#include "fused.h"
#include "tc_common.cuh"
#include "tmap.h"

namespace ago {

namespace {

using namespace tc;
using namespace ffn_cluster;

// Epilogue warps: four per tensor-memory lane quarter, each with a quarter of a tile's columns; two where the epilogue hides
// behind the next step's products (whole row blocks in several steps).
constexpr int epi_warps_of(int bh, bool full) { return full && bh == 128 ? 8 : 16; }
constexpr int threads_of(int bh, bool full) { return epi_warps_of(bh, full) * 32 + 128; }   // + MMA warp + three TMA warps
constexpr uint32_t kOutCol = 256;            // tensor memory: [0, 256) two first-GEMM accumulators, [256, 256 + NC) the output

struct FfnClusterParams : FfnClusterShape {
  const float* b1;
  const float* b2;
  __nv_bfloat16* out;
  unsigned int* status;
  float* acc;              // J > 1: fp32 [M x N2] partial sums, zero between launches
  int wide_out;            // out starts on a 32-byte boundary (its rows then do too)
};

__device__ __forceinline__ float gelu_tanh_fast(float v) {
  const float u = v * (0.7978845608028654f + 0.7978845608028654f * 0.044715f * v * v);
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(u));
  const float w = 0.5f * v;
  return w + w * t;
}

__device__ __forceinline__ void red_add_v4(float* addr, float a, float b, float c, float d) {
  asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(addr), "f"(a), "f"(b), "f"(c), "f"(d) : "memory");
}

// BH: hidden units per tile; FULL: all 128 rows of a block are kept (RP == 128).
template <int BH, bool FULL>
__global__ void __launch_bounds__(threads_of(BH, FULL), 1)
ffn_cluster_kernel(const __grid_constant__ CUtensorMap tmap_x, const __grid_constant__ CUtensorMap tmap_w1,
                   const __grid_constant__ CUtensorMap tmap_w2, const FfnClusterParams p) {
  extern __shared__ uint8_t smem_raw[];
  // the same offset in every CTA of the cluster: peers address each other's slots and barriers by it
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int CS = p.CS, stages = p.stages;
  constexpr int kEpiWarps = epi_warps_of(BH, FULL), kEpiThreads = kEpiWarps * 32;
  constexpr int halves = BH / 64;
  constexpr bool kWhole = FULL && BH == 128;       // then a stage is 32 KB, and layout() gives W2 no stages of its own
  const int RP = FULL ? kBM : p.RP, stage_bytes = kWhole ? 32768 : p.stage_bytes, slot_bytes = RP * BH * 2;
  uint8_t* sRing = smem;                                   // stages x stage_bytes
  uint8_t* sH = smem + p.slots_off;                        // CS slots x ([RP x 64] bf16 per 64 hidden units, 128-byte-swizzled)
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.bars_off);
  const bool own_w2 = !kWhole && p.w2_off > 0;
  uint64_t* bar_full = bars;                       // [kMaxStages] ring stage landed
  uint64_t* bar_empty = bars + kMaxStages;         // [kMaxStages] ring stage consumed
  uint64_t* bar_hacc = bars + 2 * kMaxStages;      // [2] first GEMM complete in accumulator b
  uint64_t* bar_hfree = bar_hacc + 2;              // [2] accumulator b drained
  uint64_t* bar_hfull = bar_hacc + 4;              // [kMaxCS] H tile present in slot k (from CTA k)
  uint64_t* bar_hdone = bar_hfull + kMaxCS;        // own slot consumed by every CTA of the cluster (count CS)
  uint64_t* bar_out = bar_hdone + 1;               // second GEMM of a row block complete
  uint64_t* bar_outfree = bar_out + 1;             // output accumulators drained: the next row block may overwrite them
  uint64_t* bar_w2 = bar_outfree + 1;              // [kMaxCS * 2] a W2 stage of its own has landed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_w2 + 2 * kMaxCS);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(bar_w2 + 2 * kMaxCS + 1);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int r = (int)cluster_ctarank();
  const int T = p.Tp, J = p.J;
  // A unit of work is (row block, one of the J parts of its hidden tiles): T steps. A cluster walks over the units
  // blockIdx.y, + gridDim.y, ...: its steps form one sequence, so the first GEMM of the next unit overlaps the tail of
  // the current one. With J = 1 a unit is a whole row block and its output is final; with J > 1 (few row blocks: the
  // hidden dimension is what fills the SMs) the J clusters of a row block add their outputs in device memory; each of them
  // has one unit (launched_clusters).
  const int row_blocks = (p.M + kBM - 1) / kBM;
  const int units = row_blocks * J;
  const int my_units = ((int)blockIdx.y < units) ? (units - 1 - (int)blockIdx.y) / (int)gridDim.y + 1 : 0;
  const int steps = my_units * T;
  // A cluster of one step expects the tiles of the others right away; with more steps the sender announces each tile on the
  // receiver's barrier (0.4 us each for its thread: 9.2 against 8.5 us for 16 rows, where nothing hides it).
  const bool one_step = steps == 1;
  auto unit_of = [&](int step) { return (int)blockIdx.y + (step / T) * (int)gridDim.y; };
  auto row0_of = [&](int step) { return (unit_of(step) / J) * kBM; };
  auto tile0_of = [&](int step) { return ((unit_of(step) % J) * T + step % T) * CS; };   // first of the step's CS hidden tiles
  if (tid == kEpiThreads) {
    *abort_flag = 0u;
    for (int i = 0; i < kMaxStages; ++i) { mbar_init(bar_full + i, 1); mbar_init(bar_empty + i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar_hacc + i, 1); mbar_init(bar_hfree + i, 1); }
    for (int i = 0; i < kMaxCS; ++i) mbar_init(bar_hfull + i, 1);
    mbar_init(bar_hdone, (uint32_t)CS);
    mbar_init(bar_out, 1);
    mbar_init(bar_outfree, 1);
    for (int i = 0; i < 2 * kMaxCS; ++i) mbar_init(bar_w2 + i, 1);
    fence_mbar_init();
    if (one_step)
      for (int i = 0; i < CS; ++i)
        if (i != r) mbar_arrive_expect_tx(bar_hfull + i, (uint32_t)slot_bytes);
    fence_proxy_async_smem();
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, 512);
    tmem_relinquish();
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  // Every CTA's barriers exist before a peer signals them: the arrival is here (relaxed: fence_mbar_init published them), each
  // role waits before it first touches another CTA.
  cluster_arrive();
  tcgen05_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
  // The set-up above overlaps the previous grid's tail (the second launch of the previous run leaves the SM room for this CTA).
  grid_dependency_wait();      // the previous grid of the stream has completed; device memory may be touched
  grid_launch_dependents();
  const int n0 = r * p.NC;     // first output column of this CTA

  if (warp > kEpiWarps) {
    // ================================ TMA producers: two for every second ring stage each, one for W2 tiles with memory of their own ================================
    const int w = warp - kEpiWarps - 1;
    const uint32_t elected = elect_one();
    if (elected) { tma_prefetch_desc(&tmap_x); tma_prefetch_desc(&tmap_w1); tma_prefetch_desc(&tmap_w2); }
    __syncwarp();
    if (w == 2) {
      if (own_w2 && steps > 0) {             // the whole second GEMM's operand
        for (int i = 0; i < CS; ++i) {
          const int hid0 = (tile0_of(0) + (int)((r + CS - i) % CS)) * BH;
          for (int h = 0; h < halves; ++h) {
            const uint32_t bar = smem_u32(bar_w2 + i * halves + h), st = smem_u32(smem) + (uint32_t)(p.w2_off + (i * halves + h) * p.NC * 128);
            mbar_arrive_expect_tx_elected(bar, (uint32_t)(p.NC * 128), elected);
            tma_load_3d_elected(st, &tmap_w2, bar, 0, hid0 + h * 64, n0 >> 6, elected);
          }
        }
      }
    } else {
      const uint32_t ring = smem_u32(sRing), full0 = smem_u32(bar_full);
      int s = 0, round = 0;
      bool mine = w == 0;                    // loads go to the two warps in turn
      auto acquire = [&](uint32_t bytes) -> uint32_t {
        if (round > 0) mbar_wait_poll(bar_empty + s, (uint32_t)(round - 1) & 1u, abort_flag, p.status, 0x701);
        mbar_arrive_expect_tx_elected(full0 + (uint32_t)(s * 8), bytes, elected);
        return ring + (uint32_t)(s * stage_bytes);
      };
      auto advance = [&]() { mine = !mine; if (++s == stages) { s = 0; ++round; } };
      auto load_g1 = [&](int step) {         // first GEMM of this CTA's hidden tile of that step
        const int hid0 = (tile0_of(step) + r) * BH, row0 = row0_of(step);
        for (int kb = 0; kb < p.kblocks; ++kb, advance()) {
          if (!mine) continue;
          const uint32_t st = acquire((uint32_t)(RP * 128 + BH * 128)), full = full0 + (uint32_t)(s * 8);
          tma_load_2d_elected(st, &tmap_x, full, kb * kBK, row0, elected);                                              // X [RP rows x 64 k]
          tma_load_3d_elected(st + (uint32_t)(RP * 128), &tmap_w1, full, 0, kb * kBK, hid0 >> 6, elected);              // W1 [64 k x 64 n] blocks
        }
      };
      if (steps > 0) load_g1(0);
      for (int step = 0; step < steps && !own_w2; ++step) {
        if (step + 1 < steps) load_g1(step + 1);
        for (int i = 0; i < CS; ++i) {      // second GEMM over hidden tile t CS + k: two stages of 64 hidden units
          const int k = (int)((r + CS - i) % CS);   // in the order the MMA warp consumes the slots: own tile first
          const int hid0 = (tile0_of(step) + k) * BH;
          for (int h = 0; h < halves; ++h, advance()) {
            if (!mine) continue;
            const uint32_t st = acquire((uint32_t)(p.NC * 128));
            tma_load_3d_elected(st, &tmap_w2, full0 + (uint32_t)(s * 8), 0, hid0 + h * 64, n0 >> 6, elected);           // W2 [64 k x 64 n] blocks
          }
        }
      }
    }
    __syncwarp();
    cluster_wait();
  } else if (warp == kEpiWarps) {
    // ================================ MMA issuer ================================
    // the whole warp, converged; MMAs and commits predicated on one elected lane (see tc_common.cuh)
    {
      const uint32_t elected = elect_one();
      const uint32_t idesc1 = make_idesc_bf16(128, (uint32_t)BH, 0, 1);     // A K-major, B N-major (weights as they lie in memory)
      const uint32_t idesc2 = make_idesc_bf16(128, (uint32_t)p.NC, 0, 1);
      int s = 0, round = 0;
      auto advance = [&]() { if (++s == stages) { s = 0; ++round; } };
      auto g1 = [&](int step) {
        const int b = step & 1;
        if (step >= 2) {
          mbar_wait(bar_hfree + b, (uint32_t)((step - 2) >> 1) & 1u, abort_flag, p.status, 0x702);
          tcgen05_fence_after_sync();
        }
        for (int kb = 0; kb < p.kblocks; ++kb) {
          mbar_wait(bar_full + s, (uint32_t)round & 1u, abort_flag, p.status, 0x703);
          tcgen05_fence_after_sync();
          const uint32_t st = smem_u32(sRing + s * stage_bytes);
          const uint64_t ad = make_smem_desc(st, 0, 1024, SW_128B);
          const uint64_t bd = make_smem_desc(st + (uint32_t)(RP * 128), 8192, 1024, SW_128B);
#pragma unroll
          for (int ks = 0; ks < kBK / 16; ++ks)
            umma_bf16_elected_acc(tmem_base + b * BH, ad + 2u * ks, bd + (uint64_t)((ks * 2048) >> 4), idesc1, elected, (kb | ks) != 0);
          umma_commit_elected(bar_empty + s, elected);
          advance();
        }
        umma_commit_elected(bar_hacc + b, elected);
      };
      if (steps > 0) g1(0);
      cluster_wait();
      for (int step = 0; step < steps; ++step) {
        if (step + 1 < steps) g1(step + 1);
        const int t = step % T, bi = step / T;
        if (t == 0 && bi >= 1) {   // the output accumulators of the previous row block have been drained
          mbar_wait(bar_outfree, (uint32_t)(bi - 1) & 1u, abort_flag, p.status, 0x709);
          tcgen05_fence_after_sync();
        }
        // Slots in the order their tiles arrive: this CTA's own tile first (no copy), then the tiles of ranks r - 1,
        // r - 2, ... -- every producer sends to rank + 1 first, so rank r - q's tile is the q-th to land here.
        for (int i = 0; i < CS; ++i) {
          const int k = (int)((r + CS - i) % CS);
          mbar_wait(bar_hfull + k, (uint32_t)step & 1u, abort_flag, p.status, 0x704);   // H tile t CS + k is in slot k
          for (int h = 0; h < halves; ++h) {
            if (own_w2) mbar_wait(bar_w2 + i * halves + h, 0, abort_flag, p.status, 0x70a);
            else mbar_wait(bar_full + s, (uint32_t)round & 1u, abort_flag, p.status, 0x705);
            tcgen05_fence_after_sync();
            const uint64_t hd = make_smem_desc(smem_u32(sH + k * slot_bytes + h * (RP * 128)), 0, 1024, SW_128B);
            const uint64_t bd = make_smem_desc(own_w2 ? smem_u32(smem) + (uint32_t)(p.w2_off + (i * halves + h) * p.NC * 128) : smem_u32(sRing + s * stage_bytes),
                                               8192, 1024, SW_128B);
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
              umma_bf16_elected_acc(tmem_base + kOutCol, hd + 2u * ks, bd + (uint64_t)((ks * 2048) >> 4), idesc2, elected, (t | i | h | ks) != 0);
            if (!own_w2) {
              umma_commit_elected(bar_empty + s, elected);
              advance();
            }
          }
          // slot k of this CTA has been read: tell its producer (CTA k)
          umma_commit_cluster_elected(cluster_map(smem_u32(bar_hdone), (uint32_t)k), elected);
        }
        if (t == T - 1) umma_commit_elected(bar_out, elected);
      }
    }
    __syncwarp();
  } else {
    // ================ epilogue warps: thread = (row, quarter of a tile's columns) ================
    const int row = (warp & 3) * 32 + lane;
    const int part = warp >> 2;
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const bool warp_rows = (warp & 3) * 32 < RP;   // some row of this warp exists
    uint8_t* slot = sH + r * slot_bytes;           // this CTA produces into slot r everywhere
    constexpr int kParts = kEpiWarps / 4;
    constexpr int pc = BH / kParts;                        // columns per thread: 16 or 32
    cluster_wait();

    for (int step = 0; step < steps; ++step) {
      const int b = step & 1, t = step % T;
      const int col0 = part * pc;
      const float* bb = p.b1 + (size_t)(tile0_of(step) + r) * BH + col0;
      float4 bv4[pc / 4];                          // the tile's biases travel while its product is made
#pragma unroll
      for (int q = 0; q < pc / 4; ++q) bv4[q] = __ldg(reinterpret_cast<const float4*>(bb) + q);
      mbar_wait(bar_hacc + b, (uint32_t)(step >> 1) & 1u, abort_flag, p.status, 0x706);
      tcgen05_fence_after_sync();
      // every CTA has multiplied the previous content of slot r (and the copies that delivered it are complete)
      if (step >= 1) mbar_wait(bar_hdone, (uint32_t)(step - 1) & 1u, abort_flag, p.status, 0x707);
      uint8_t* tile = slot + (col0 >> 6) * (RP * 128);
      if (warp_rows) {
        constexpr int kLd = pc >= 32 ? 32 : 16;    // columns per tensor-memory load
#pragma unroll
        for (int c0 = 0; c0 < pc; c0 += kLd) {
          uint32_t v[kLd];
          if constexpr (kLd == 32) tmem_ld_x32(tmem_base + lane_base + b * BH + col0 + c0, v);
          else tmem_ld_x16(tmem_base + lane_base + b * BH + col0 + c0, v);
          tmem_ld_wait();
          if (row < RP) {
#pragma unroll
            for (int q = 0; q < kLd / 8; ++q) {
              const float4 lo = bv4[c0 / 4 + 2 * q], hi = bv4[c0 / 4 + 2 * q + 1];
              const float bv[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
              uint32_t w[4];
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                const int e = q * 8 + j * 2;
                w[j] = pack_bf16x2(gelu_tanh_fast(__uint_as_float(v[e]) + bv[2 * j]),
                                   gelu_tanh_fast(__uint_as_float(v[e + 1]) + bv[2 * j + 1]));
              }
              *reinterpret_cast<uint4*>(tile + swz_offset(row, (((col0 & 63) + c0) >> 3) + q, 128)) = make_uint4(w[0], w[1], w[2], w[3]);
            }
          }
        }
      }
      fence_proxy_async_smem();      // the MMA and the bulk copies read the tile through the async proxy
      tcgen05_fence_before_sync();
      named_barrier_sync(1, kEpiThreads);
      if (tid == 0) {
        mbar_arrive(bar_hfree + b);
        mbar_arrive(bar_hfull + r);                                   // the local consumer
        const uint32_t src = smem_u32(slot), bar = smem_u32(bar_hfull + r);
        for (int q = 1; q < CS; ++q) {                                // the peers, starting with the next rank
          const uint32_t peer = (uint32_t)((r + q) % CS);
          const uint32_t rbar = cluster_map(bar, peer);
          if (!one_step) mbar_remote_arrive_expect_tx(rbar, (uint32_t)slot_bytes);
          bulk_copy_to_cluster(cluster_map(src, peer), src, (uint32_t)slot_bytes, rbar);
        }
      }
      if (t == T - 1) {
        // ---- output of the row block: out (TMEM) -> + b2 -> bf16 -> device memory; thread = (row, quarter of the CTA's columns) ----
        const int bi = step / T, row0 = row0_of(step);
        const bool row_ok = row0 + row < p.M;
        mbar_wait(bar_out, (uint32_t)bi & 1u, abort_flag, p.status, 0x708);
        tcgen05_fence_after_sync();
        const int hc = p.NC / kParts;                                          // columns per thread: 16, 32, 48 or 64
        if (J > 1) {
          // ---- split row block: this cluster's share is added into the fp32 buffer; the second launch turns the buffer
          // into the output (+ b2, bf16) and zeroes it. ----
          if (RP < kStagedRows) {
            // few rows: every thread adds from its registers (one barrier less than below: 10.9 against 12.0 us for one row)
            float* arow = p.acc + (size_t)(row0 + row) * p.N2 + n0 + part * hc;
            if (warp_rows) {
              for (int c0 = 0; c0 < hc; c0 += 16) {
                uint32_t v[16];
                tmem_ld_x16(tmem_base + lane_base + kOutCol + part * hc + c0, v);
                tmem_ld_wait();
                if (row_ok) {
#pragma unroll
                  for (int q = 0; q < 4; ++q)
                    red_add_v4(arow + c0 + q * 4, __uint_as_float(v[4 * q]), __uint_as_float(v[4 * q + 1]),
                               __uint_as_float(v[4 * q + 2]), __uint_as_float(v[4 * q + 3]));
                }
              }
            }
          } else {
            // Blocks of 64 columns go through shared memory (two buffers over the ring, which this cluster's one unit has
            // used up; where they reach past it, the copies of this CTA's tile to its peers must have left), so that a half-warp adds 256 contiguous bytes of a row: additions of 16 bytes per row took the L2 twice
            // as long. The clusters of a row block start with different blocks, not to meet on the same addresses.
            if (p.wait_copies) mbar_wait(bar_hdone, (uint32_t)step & 1u, abort_flag, p.status, 0x70b);
            const int blocks = p.NC >> 6, first = (unit_of(step) % J) % blocks, rows_here = min(RP, p.M - row0);
            for (int k = 0; k < blocks; ++k) {
              int cb = first + k;
              if (cb >= blocks) cb -= blocks;
              uint8_t* buf = sRing + (k & 1) * (RP * 256);
              if (warp_rows) {
                for (int c0 = part * (64 / kParts); c0 < (part + 1) * (64 / kParts); c0 += 16) {
                  uint32_t v[16];
                  tmem_ld_x16(tmem_base + lane_base + kOutCol + cb * 64 + c0, v);
                  tmem_ld_wait();
                  if (row < RP) {
#pragma unroll
                    for (int q = 0; q < 4; ++q)
                      *reinterpret_cast<uint4*>(buf + row * 256 + ((((c0 / 4 + q) ^ row) & 15) << 4)) = make_uint4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
                  }
                }
              }
              named_barrier_sync(1, kEpiThreads);
              float* ablk = p.acc + (size_t)row0 * p.N2 + n0 + cb * 64;
              for (int i = tid; i < rows_here * 16; i += kEpiThreads) {
                const int rr = i >> 4, c = i & 15;
                const float4 f = *reinterpret_cast<const float4*>(buf + rr * 256 + (((c ^ rr) & 15) << 4));
                red_add_v4(ablk + (size_t)rr * p.N2 + c * 4, f.x, f.y, f.z, f.w);
              }
            }
          }
          tcgen05_fence_before_sync();
          named_barrier_sync(1, kEpiThreads);
          if (tid == 0) mbar_arrive(bar_outfree);
          continue;
        }
        __nv_bfloat16* orow = p.out + (size_t)(row0 + row) * p.N2 + n0 + part * hc;
        const float* b2 = p.b2 + n0 + part * hc;
        if (warp_rows) {
          for (int c0 = 0; c0 < hc; c0 += 16) {
            uint32_t v[16];
            tmem_ld_x16(tmem_base + lane_base + kOutCol + part * hc + c0, v);
            tmem_ld_wait();
            if (row_ok) {
              uint32_t w[8];
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const float4 b = __ldg(reinterpret_cast<const float4*>(b2 + c0 + q * 4));
                w[2 * q] = pack_bf16x2(__uint_as_float(v[q * 4]) + b.x, __uint_as_float(v[q * 4 + 1]) + b.y);
                w[2 * q + 1] = pack_bf16x2(__uint_as_float(v[q * 4 + 2]) + b.z, __uint_as_float(v[q * 4 + 3]) + b.w);
              }
              if (p.wide_out) store_global_32(orow + c0, w);      // a whole sector
              else {
                *reinterpret_cast<uint4*>(orow + c0) = make_uint4(w[0], w[1], w[2], w[3]);
                *reinterpret_cast<uint4*>(orow + c0 + 8) = make_uint4(w[4], w[5], w[6], w[7]);
              }
            }
          }
        }
        tcgen05_fence_before_sync();
        named_barrier_sync(1, kEpiThreads);
        if (tid == 0) mbar_arrive(bar_outfree);
      }
    }
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  cluster_meet();              // no CTA leaves while a peer may still copy into it or signal its barriers
  if (warp == 0) tmem_dealloc(tmem_base, 512);
}

// Second launch of a split run: out = bf16(acc + b2), acc = 0. One float4 per thread and iteration, coalesced. (A sweep that
// follows per-slice arrival counters instead of the end of the first grid was slower at every size: 16.6 against 16.3 us at 256
// rows, 56 against 53 at 2048; the counters' fences wait for the additions, which keep the L2 busy.)
__global__ void __launch_bounds__(256) ffn_cluster_finalize_kernel(float* acc, const float* b2, __nv_bfloat16* out, long long total4, int n2) {
  grid_dependency_wait();      // the additions of the first launch are complete and visible
  grid_launch_dependents();
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total4; i += stride) {
    const float4 a = __ldcg(reinterpret_cast<const float4*>(acc) + i);
    const float4 bb = __ldg(reinterpret_cast<const float4*>(b2 + (int)((i * 4) % n2)));
    reinterpret_cast<float4*>(acc)[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    reinterpret_cast<uint2*>(out)[i] = make_uint2(pack_bf16x2(a.x + bb.x, a.y + bb.y), pack_bf16x2(a.z + bb.z, a.w + bb.w));
  }
}

struct FfnClusterHost {
  FfnClusterParams prm;
  int smem_bytes = 0;
  int clusters = 0;   // clusters launched; 0: the device has not been asked yet
  size_t acc_bytes = 0, ws_bytes = 0;   // split row blocks: fp32 partial sums
  const void* clean_ws = nullptr;   // workspace known to be zeroed (kept so by the kernel itself) ...
  unsigned clean_epoch = 0;         // ... as of this attach (FusedState::workspace_epoch)
  struct Key { const void* p; int which; bool operator==(const Key& o) const { return p == o.p && which == o.which; } };
  struct KeyHash { size_t operator()(const Key& k) const { return std::hash<const void*>()(k.p) ^ (size_t)k.which * 0x9e3779b97f4a7c15ull; } };
  std::unordered_map<Key, CUtensorMap, KeyHash> maps;
};

using ClusterKernel = void (*)(CUtensorMap, CUtensorMap, CUtensorMap, FfnClusterParams);
ClusterKernel kernel_of(int bh, bool full) {
  if (bh == 64) return full ? ffn_cluster_kernel<64, true> : ffn_cluster_kernel<64, false>;
  return full ? ffn_cluster_kernel<128, true> : ffn_cluster_kernel<128, false>;
}

void fill_launch(cudaLaunchConfig_t* cfg, cudaLaunchAttribute* attr, const FfnClusterParams& q, int clusters, int smem_bytes,
                 cudaStream_t stream) {
  *cfg = cudaLaunchConfig_t{};
  cfg->gridDim = dim3((unsigned)q.CS, (unsigned)clusters, 1);
  cfg->blockDim = dim3((unsigned)threads_of(q.BH, q.RP == kBM), 1, 1);
  cfg->dynamicSmemBytes = (size_t)smem_bytes;
  cfg->stream = stream;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)q.CS; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg->attrs = attr;
  cfg->numAttrs = 2;
}

}  // namespace

namespace {
bool cluster_shape(const Plan& plan, FfnClusterParams* q) {
  q->K = (int)plan.inputs[0].last();
  q->M = (int)(plan.inputs[0].numel() / q->K);
  q->Hid = plan.ops[0].op.p[0];
  q->N2 = plan.ops[3].op.p[0];
  if (q->K % kBK != 0 || q->Hid % 128 != 0) return false;
  q->kblocks = q->K / kBK;
  q->RP = std::min(kBM, (q->M + 15) / 16 * 16);
  return choose_split(q, (q->M + kBM - 1) / kBM, kResident);
}
}  // namespace

// Set-up + steps of the longest cluster x (the first product's operands, W2's, a constant, what a W2 stage costs besides its bytes, the
// chain of hand-offs where an input of one K block does not hide it);
// split row blocks: the additions (3 T bytes/s). One step with W2 stages of its own: everything is on its way at once, which is
// a chain of latencies. 232 measured chains of 1 to 12288 rows and widths of 64 to 4096: 6 % and 3 % rms.
double ffn_cluster_estimate(const Plan& plan) {
  FfnClusterParams q{};
  if (!cluster_shape(plan, &q)) return -1.0;
  layout(&q);
  const double units = (double)((q.M + kBM - 1) / kBM) * q.J, steps = std::ceil(units / kResident[q.CS]) * q.Tp;
  const double w2_stages = q.CS * (q.BH / 64), g1 = q.kblocks * (q.RP + q.BH) / 256.0, w2 = w2_stages * q.NC / 256.0;      // in 32 KB
  const double additions = q.J > 1 ? (double)q.J * q.M * q.N2 * 4 / 3.0e6 : 0.0;
  if (q.w2_off > 0) return 5.05 + 0.096 * g1 + 0.477 * w2 + 0.089 * q.kblocks + 2.02 * q.RP / kBM + 0.72 * additions;
  return 4.53 + steps * (0.18 * g1 + 0.216 * w2 + 0.339 + 0.584 * w2_stages + (q.kblocks == 1 ? 0.38 : 0.0)) + 1.04 * additions;
}

// AGO_ERR_UNSUPPORTED (without touching *err) when the shape has no cluster split: the caller falls back to the
// kernel that tiles the second GEMM's reduction across independent CTAs.
ago_status_t ffn_cluster_plan(Plan* plan, FusedState* st, std::string* err) {
  (void)err;
  FfnClusterParams q{};
  if (!cluster_shape(*plan, &q)) return AGO_ERR_UNSUPPORTED;
  auto* host = new FfnClusterHost();
  host->smem_bytes = layout(&q);
  host->prm = q;
  st->impl = host;
  st->impl_free = [](void* p) { delete static_cast<FfnClusterHost*>(p); };
  st->variant = 1;
  st->tile_rows = kBM; st->grid = q.CS * q.J * ((q.M + kBM - 1) / kBM); st->smem_bytes = host->smem_bytes;
  plan->tile_rows = kBM; plan->smem_bytes = host->smem_bytes;
  plan->fused_variant = q.J > 1 ? 2 : 1;
  if (q.J > 1) {
    host->acc_bytes = ((size_t)q.M * q.N2 * 4 + 255) & ~size_t(255);
    host->ws_bytes = host->acc_bytes;
    // every cluster of a row block adds its share into the buffer; the second launch reads it back and zeroes it
    plan->workspace_traffic_bytes = (int64_t)(q.J + 2) * q.M * q.N2 * 4;
    plan->num_launches = 2;
  }
  return AGO_OK;
}

size_t ffn_cluster_workspace_bytes(const Plan& plan) {
  if (plan.fused_variant != 2) return 0;
  const int64_t M = plan.inputs[0].numel() / plan.inputs[0].last();
  const int64_t N2 = plan.output.last();
  return ((size_t)M * N2 * 4 + 255) & ~size_t(255);
}

ago_status_t ffn_cluster_run(const Plan& plan, FusedState* st, const void* const* inputs, const void* const* weights,
                             void* output, void* workspace, unsigned int* status_word, cudaStream_t stream, std::string* err) {
  (void)plan;
  FfnClusterHost* host = static_cast<FfnClusterHost*>(st->impl);
  FfnClusterParams q = host->prm;
  q.b1 = static_cast<const float*>(weights[1]);
  q.b2 = static_cast<const float*>(weights[3]);
  q.out = static_cast<__nv_bfloat16*>(output);
  q.status = status_word;
  q.wide_out = reinterpret_cast<uintptr_t>(output) % 32 == 0;
  if (q.J > 1) {
    if (!workspace) { *err = "fused feed-forward (cluster, split row blocks): no workspace attached"; return AGO_ERR_INVALID_ARG; }
    q.acc = static_cast<float*>(workspace);
    if (host->clean_ws != workspace || host->clean_epoch != st->workspace_epoch) {
      // a workspace is zeroed at the first run after each attach; after that every launch leaves it zeroed (the caller
      // must not touch it in between)
      cudaError_t e = cudaMemsetAsync(workspace, 0, host->ws_bytes, stream);
      if (e != cudaSuccess) { *err = std::string("cudaMemsetAsync(workspace): ") + cudaGetErrorString(e); return AGO_ERR_CUDA; }
      host->clean_ws = workspace;
      host->clean_epoch = st->workspace_epoch;
    }
  }
  auto get_map = [&](const void* base, int which, CUtensorMap* out) -> bool {
    FfnClusterHost::Key key{base, which};
    auto it = host->maps.find(key);
    if (it == host->maps.end()) {
      CUtensorMap m;
      uint64_t dims[3] = {}; uint64_t strides[2] = {}; uint32_t box[3] = {};
      if (which == 0) { dims[0] = q.K; dims[1] = q.M; strides[0] = (uint64_t)q.K * 2; box[0] = kBK; box[1] = (uint32_t)q.RP; }
      else {      // a weight matrix in blocks of 64 columns: one box brings a tile's
        const int cols = which == 1 ? q.Hid : q.N2;
        dims[0] = 64; dims[1] = which == 1 ? q.K : q.Hid; dims[2] = cols / 64; strides[0] = (uint64_t)cols * 2; strides[1] = 128;
        box[0] = 64; box[1] = 64; box[2] = (uint32_t)((which == 1 ? q.BH : q.NC) / 64);
      }
      if (!encode_tmap_bf16(&m, base, which == 0 ? 2 : 3, dims, strides, box, 128, err)) return false;
      if (host->maps.size() > 4096) host->maps.clear();
      it = host->maps.emplace(key, m).first;
    }
    *out = it->second;
    return true;
  };
  CUtensorMap mx, mw1, mw2;
  if (!get_map(inputs[0], 0, &mx) || !get_map(weights[0], 1, &mw1) || !get_map(weights[2], 2, &mw2)) return AGO_ERR_CUDA;
  {
    static int smem_opt_in[4][64] = {};
    cudaError_t e = cudaSuccess;
    for (int i = 0; i < 4 && e == cudaSuccess; ++i) e = ensure_max_dynamic_smem(reinterpret_cast<const void*>(kernel_of(i & 1 ? 128 : 64, (i & 2) != 0)), smem_opt_in[i]);
    if (e != cudaSuccess) { *err = std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(e); return AGO_ERR_CUDA; }
  }
  const auto kernel = kernel_of(q.BH, q.RP == kBM);
  cudaLaunchConfig_t cfg; cudaLaunchAttribute attr[2];
  const int row_blocks = (q.M + kBM - 1) / kBM;
  if (host->clusters == 0) {
    // persistent clusters: as many as the device keeps resident at once (one CTA per SM, CS SMs of one GPC each)
    fill_launch(&cfg, attr, q, row_blocks * q.J, host->smem_bytes, stream);
    int resident = 0;
    cudaError_t e = cudaOccupancyMaxActiveClusters(&resident, kernel, &cfg);
    if (e != cudaSuccess || resident < 1) {
      *err = std::string("fused feed-forward (cluster): no cluster of this size is schedulable: ") + cudaGetErrorString(e);
      return AGO_ERR_CUDA;
    }
    host->clusters = launched_clusters(row_blocks, q.J, resident);
  }
  fill_launch(&cfg, attr, q, host->clusters, host->smem_bytes, stream);
  cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, mx, mw1, mw2, q);
  if (e != cudaSuccess) { *err = std::string("fused feed-forward (cluster) launch: ") + cudaGetErrorString(e); return AGO_ERR_CUDA; }
  if (q.J > 1) {
    const long long total4 = (long long)q.M * q.N2 / 4;
    const int blocks = (int)std::min<long long>((total4 + 255) / 256, 4LL * device_sm_count());
    FusedLaunch fin(dim3((unsigned)blocks), 256, 0, stream);
    e = cudaLaunchKernelEx(&fin.config, ffn_cluster_finalize_kernel, q.acc, q.b2, q.out, total4, q.N2);
    if (e != cudaSuccess) { *err = std::string("fused feed-forward (cluster) finalisation launch: ") + cudaGetErrorString(e); return AGO_ERR_CUDA; }
  }
  return AGO_OK;
}

}  // namespace ago
