// Fused inverted-residual block: 1x1 conv + bias + ReLU6 -> depthwise 3x3
// (pad 1, stride 1|2) + bias + ReLU6 -> 1x1 conv + bias [+ input], one kernel.
//
// Tiling follows Section III-B. The pointwise -> depthwise link is the
// "downstream depthwise" category: the depthwise tile keeps its spatial extent
// and is tiled over channels (o1 = o2, here 16 channels per chunk). The
// depthwise -> pointwise link is the "downstream pointwise" category: the
// project tile keeps ALL output channels and is tiled over rows (a strip of R
// output rows of one image per CTA), so nothing is recomputed except the
// expand convolution on the strip's one-row halo.
//
// Wide blocks and small batches: the expanded channels of a strip are split over
// a cluster of CS CTAs (the chunks of a CTA are what its time grows with, and a
// handful of strips leaves most SMs idle). Each runs the steps below on its share;
// the partial output sums are exchanged through distributed shared memory.
// 25 images of 15 x 15, 96 -> 576 -> 96: 34 us as three launches (the weights of
// so wide a block do not fit one SM), 16.5 us on clusters of four.
//
// Per CTA (one image, R output rows, full width, its share of the channels):
//   P1  16-byte asynchronous copies bring the NHWC input strip (with its row
//       halo; rows outside the image -> 0, channels padded to the MMA K
//       granularity), W1 and W3 into swizzled K-major tiles (X and W1 by TMA for wide pixels); descriptors and work
//       mapping are computed while they travel. (A pixel is Cin * 2 bytes there,
//       e.g. 48: one TMA box row per pixel was several times slower.)
//   for each 16-channel chunk c of the expanded tensor:
//     P2  tcgen05.mma: expand[pixels x 16] = X[pixels x Cin] * W1[c]^T   (TMEM, fp32; Cin > 64: K blocks of 64)
//     P3  TMEM -> registers: + b1, ReLU6, zero outside the image (the depthwise
//         conv pads the post-activation tensor), bf16 -> shared memory; the
//         padding columns of the E chunk are written once
//     P4  CUDA cores: depthwise 3x3 + bd + ReLU6 over the resident chunk with
//         mixed-precision FMAs (bf16 activations and weights as stored, fp32
//         accumulate), result written as the K-major A operand of the project GEMM
//     P5  tcgen05.mma: out[pixels x Cout] += DW[pixels x 16] * W3[:, c]^T  (TMEM)
//   P6  TMEM -> registers: [sum over the cluster] + b3 (+ x), bf16, 16-byte stores.
// The expand MMA of chunk c+1 is issued before the CUDA-core work of chunk c.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <unordered_map>

#include "dw_common.cuh"
#include "fused.h"
#include "tc_common.cuh"
#include "tmap.h"

namespace ago {

namespace {

using namespace tc;
using namespace dw;

// Sixteen warps with 128 registers a thread; every warp computes, MMAs are issued inline by some of them. (With 32 warps the
// cap of 64 registers left the depthwise block no room to have its loads in flight: it took twice the cycles it takes alone.
// One 14 x 14 image of 32 -> 192 -> 32 channels 9.8 -> 6.5 us, 12 images of 16 x 16 10.9 -> 7.3 us; 56 x 56 strips the same.)
constexpr int kWarps = 16;
constexpr int kThreads = kWarps * 32;
// The warps form NG groups (2 or 4) that own the chunks c = g, g + NG, ...: two groups of eight warps for strips whose
// chunk is real work (their phases overlap), four groups of four warps for small strips, where a chunk is a chain of
// latencies (MMA hand-off, tensor-memory round trip, two barriers) and more chains in flight is what helps.
constexpr int kTilesPerWarp = 4;                   // expand-epilogue tiles per warp
constexpr int kExpandIssuers = 2;                  // the last two warps of a group issue its expand GEMMs
constexpr int kChunk = 16;      // expanded channels per chunk = one MMA K step of the project GEMM
constexpr int kChunkRowBytes = 32;
constexpr int kMaxPieces = 2;   // of the partial sums that the CTAs of a cluster exchange

struct Mbv2Params {
  const __nv_bfloat16* x;
  const __nv_bfloat16* w1;
  const float* b1;
  const __nv_bfloat16* wd;
  const float* bd;
  const __nv_bfloat16* w3;
  const float* b3;
  __nv_bfloat16* out;
  unsigned int* status;
  int N, H, W, Cin, Cexp, Cout, stride, Ho, Wo, residual;   // Cexp: expanded channels of one CTA
  int CS, Cfull;                // the expanded channels are split over CS CTAs; Cfull = CS * Cexp
  int PP;                       // CS > 1: output pixels of a strip that one CTA of the cluster sums up and stores (odd)
  int off_send, off_recv, recv_shared;   // CS > 1: blocks of partial sums for / from the other CTAs; recv_shared: over dead operands
  int kblocks, ksteps, cpr;     // reduction of the expand GEMM: 128-byte-row blocks, MMA steps, 16-byte chunks per row (kblocks > 1)
  int piece_cgs;                // ... sent by pieces of piece_cgs x 16 output channels
  uint32_t pp_recip, cpr_recip, c8s_recip, c8s_last_recip;
  int groups;                   // warp groups: 2 or 4 (the kernel template's NG)
  int fold_b1;                  // the expand bias rides in two spare reduction channels of the expand GEMM (Cin < Kp)
  int R, strips, IH, IW, P_x, P_in, M1, M2;   // P_x = IH * W pixels in the input tile, P_in = IH * IW in an E chunk
  int Kp, row_bytes, swizzle;   // input / W1 tiles: padded K, bytes per row, tc::SwizzleMode
  int Coutp, NC;
  // 2^32 / d + 1 for the run-time divisors of the index arithmetic: x / d == __umulhi(x, recip) for x, d < 65536
  uint32_t coutp_recip, w_recip, strips_recip, per_row_recip, cexp8_recip;   // cexp8: Cexp / 8 (>= 2)
  int per_row, nseg, segw, step_r, step_c, col_slots;   // depthwise item geometry (see the kernel), fixed per shape
  int tmem_cols, ecol0, pcol0;
  int e_plane, d_plane;         // byte distance between the two 8-channel planes of an E / D chunk
  // shared-memory byte offsets (from the 1024-aligned base)
  int off_x, off_w1, off_e, off_d, off_w3, off_wd, off_b1, off_bd, off_b3, off_bar;
  int tma, w1_box;              // X and W1 by TMA, rows of W1 per load
};

// FOLD: the expand bias rides in the expand GEMM (see the prologue). EXPAND / PROJECT select the pairs of the
// block: <true, true> the whole block, <true, false> pointwise -> depthwise
// (the depthwise result of every chunk goes to device memory), <false, true> depthwise -> pointwise (every chunk of
// the input is copied into the E buffers instead of being computed).
// TMA: the input strip and W1 come by TMA (not with FOLD, where channels of their K blocks belong to a bias). An instance of its own: with
// both ways in one kernel either ran 3 % slower.
template <bool MAPS> struct Mbv2Maps { CUtensorMap x, w1; };
template <> struct Mbv2Maps<false> {};

template <bool EXPAND, bool PROJECT, bool FOLD, int NG, bool TMA>
__global__ void __launch_bounds__(kThreads, 1)
mbv2_fused_kernel(const Mbv2Params p, const __grid_constant__ Mbv2Maps<TMA> maps) {
  constexpr int kGroupWarps = kWarps / NG;
  constexpr int kGroupThreads = kGroupWarps * 32;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sX = smem + p.off_x;
  uint8_t* sW1 = smem + p.off_w1;
  uint8_t* sE = smem + p.off_e;
  uint8_t* sD = smem + p.off_d;
  uint8_t* sW3 = smem + p.off_w3;
  const uint8_t* sWd = smem + p.off_wd;                   // [chunk][9 taps][16 channels] bf16
  float* sB1 = reinterpret_cast<float*>(smem + p.off_b1);
  float* sBd = reinterpret_cast<float*>(smem + p.off_bd);
  float* sB3 = reinterpret_cast<float*>(smem + p.off_b3);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + p.off_bar);
  uint64_t* bar_e = bars;           // [NG] expand accumulators of group g complete (MMA commit)
  uint64_t* bar_d = bars + 8;       // [NG] project MMA has consumed D[g] (MMA commit)
  uint64_t* bar_first = bars + 16;  // project GEMM of chunk 0 complete (it overwrites the output accumulators: the other groups issue after it)
  uint64_t* bar_done = bars + 17;   // every project MMA complete (the groups do not follow each other's bar_d phases)
  uint64_t* bar_chain = bars + 18;  // two groups: group 0's first expand GEMM complete. One phase only: a waiter on bar_e could
                                    // fall behind its next phase and then wait for a parity that has come and gone
  uint64_t* bar_red = bars + 12;    // [kMaxPieces] a piece of the partial sums of the other CTAs of the cluster has arrived
  uint64_t* bar_x = bars + 19;      // input strip and W1 landed (TMA)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 20);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(bars + 21);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // CS CTAs (a cluster when their partial products are to be added) work on one strip, each on its share of the channels
  const int unit = p.CS == 1 ? (int)blockIdx.x : (int)(blockIdx.x / (unsigned)p.CS), rank = (int)blockIdx.x - unit * p.CS;
  const int n = (int)fast_div((uint32_t)unit, (uint32_t)p.strips, p.strips_recip), strip = unit - n * p.strips;
  const int ch0 = rank * p.Cexp;        // first expanded channel of this CTA
  const int ho0 = strip * p.R;
  const int rows_valid = min(p.R, p.Ho - ho0);
  const int gh0 = ho0 * p.stride - 1;   // image row of tile row 0
  const int d_bytes = 2 * p.d_plane;

  if (tid == kThreads - 1) {
    *abort_flag = 0u;
    for (int i = 0; i < NG; ++i) {
      mbar_init(bar_e + i, kExpandIssuers);
      mbar_init(bar_d + i, (uint32_t)p.M2);
    }
    mbar_init(bar_first, (uint32_t)p.M2);
    mbar_init(bar_chain, kExpandIssuers);
    for (int k = 0; k < kMaxPieces; ++k) mbar_init(bar_red + k, 1);
    mbar_init(bar_done, (uint32_t)(p.M2 * min(p.NC, NG)));
    if (TMA) mbar_init(bar_x, 1);
    fence_mbar_init();
    fence_proxy_async_smem();
    if constexpr (TMA) { tma_prefetch_desc(&maps.x); tma_prefetch_desc(&maps.w1); }
  }
    // ---- P1: stage the input strip, the weights and the biases by asynchronous 16-byte copies, region by region; row and
    // column of a thread's chunks advance by fixed steps. X and W1 rows go to their swizzled K-major tiles (one tile of 16, 32
    // or 64 channels, or blocks of 64), zero beyond Cin; W3 to one [Coutp x 16 channels] slice per chunk; depthwise weights
    // and biases are copied as they are. (Pixels are Cin * 2 bytes apart in device memory: coalesced copies of the contiguous
    // strip serve that better than one TMA box row per pixel.) ----
    const int cs = p.Kp == 16 ? 1 : (p.Kp == 32 ? 2 : 3);   // log2(16-byte chunks per tile row)
    const bool wide = EXPAND && !FOLD && p.kblocks > 1;     // more than 64 input channels: K blocks of 64
    // tile pixel `pix` is image pixel gh0 * W + pix of image n (strips are full-width rows): in the image for pix in [pix_lo, pix_hi)
    const int pix_lo = max(0, -gh0 * p.W), pix_hi = min(p.P_x, (p.H - gh0) * p.W);
    const uint8_t* x0 = reinterpret_cast<const uint8_t*>(p.x) + ((int64_t)n * p.H + gh0) * p.W * p.Cin * 2;   // not dereferenced outside the image
    const int cin_chunks = p.Cin >> 3;
    const uint32_t cin_bytes = (uint32_t)p.Cin * 2u, swz_mask = ((uint32_t)p.row_bytes >> 4) - 1u;
    const uint8_t* w1p = reinterpret_cast<const uint8_t*>(p.w1) + (size_t)ch0 * cin_bytes;
    auto stage_region = [&](int rows, int cpr, uint32_t recip, auto&& put) {      // put(row, chunk of the row)
      int row = (int)fast_div((uint32_t)tid, (uint32_t)cpr, recip), ch = tid - row * cpr;
      const int dr = (int)fast_div((uint32_t)kThreads, (uint32_t)cpr, recip), dc = kThreads - dr * cpr;
      for (; row < rows; row += dr) {
        put(row, ch);
        if ((ch += dc) >= cpr) { ch -= cpr; ++row; }
      }
    };
    auto stage = [&]() {
      const uint8_t* none = reinterpret_cast<const uint8_t*>(p.wd);      // never read: the copies from it have no bytes
      const uint32_t s0 = smem_u32(smem);
      const float fold_b = FOLD && tid < p.Cexp ? __ldg(p.b1 + ch0 + tid) : 0.0f;     // on its way while the copies are issued
      if (EXPAND && !TMA) {
        const int xblk = p.M1 * 128 * 128, wblk = p.Cexp * 128;
        auto place = [&](int row, int ch, int blk) -> uint32_t {
          if (wide) return (uint32_t)((ch >> 3) * blk + row * 128 + (((ch ^ row) & 7) << 4));
          const uint32_t i = ((uint32_t)row << cs) + (uint32_t)ch;
          return (i << 4) ^ (((i >> 3) & swz_mask) << 4);
        };
        stage_region(p.P_x, p.cpr, p.cpr_recip, [&](int row, int ch) {
          const uint32_t d = p.off_x + place(row, ch, xblk);
          // two channels of ones multiply the folded bias
          if (FOLD && ch == cin_chunks) { *reinterpret_cast<uint4*>(smem + d) = make_uint4(0x3F803F80u, 0, 0, 0); return; }
          const bool in = ch < cin_chunks && row >= pix_lo && row < pix_hi;
          cp_async_16(s0 + d, in ? x0 + (uint32_t)row * cin_bytes + ch * 16 : none, in ? 16u : 0u);
        });
        stage_region(p.Cexp, p.cpr, p.cpr_recip, [&](int row, int ch) {
          const uint32_t d = p.off_w1 + place(row, ch, wblk);
          if (FOLD && ch == cin_chunks) return;     // the bias, below
          const bool in = ch < cin_chunks;
          cp_async_16(s0 + d, in ? w1p + (uint32_t)row * cin_bytes + ch * 16 : none, in ? 16u : 0u);
        });
      }
      const uint8_t* wdp = reinterpret_cast<const uint8_t*>(p.wd + ch0);
      stage_region(9, p.Cexp >> 3, p.cexp8_recip, [&](int tap, int c8) {      // [chunk][tap][16 channels]: a thread's nine taps lie 32 bytes apart
        cp_async_16(s0 + p.off_wd + (c8 >> 1) * (9 * kChunkRowBytes) + tap * kChunkRowBytes + (c8 & 1) * 16, wdp + ((uint32_t)tap * p.Cfull + c8 * 8) * 2, 16u);
      });
      if (PROJECT) {
        const uint8_t* w3p = reinterpret_cast<const uint8_t*>(p.w3 + ch0);
        stage_region(p.Coutp, 2 * p.NC, p.cexp8_recip, [&](int row, int j) {      // 2 NC == Cexp / 8
          const bool in = row < p.Cout;
          cp_async_16(s0 + p.off_w3 + (j >> 1) * p.Coutp * kChunkRowBytes + swz_offset(row, j & 1, kChunkRowBytes),
                      in ? w3p + ((uint32_t)row * p.Cfull + j * 8) * 2 : none, in ? 16u : 0u);
        });
      }
      // the biases, each by warps of its own: what a few warps run alone they also fetch the instructions for alone
      auto stage_bias = [&](int first_warp, int off, const float* b, int count) {
        const int i = (tid - first_warp * 32) & (kThreads - 1);
        for (int j = i; j < (count >> 2); j += kThreads) cp_async_16(s0 + off + j * 16, reinterpret_cast<const uint8_t*>(b) + j * 16, 16u);
      };
      stage_bias(4, p.off_bd, p.bd + ch0, p.Cexp);
      if (PROJECT) stage_bias(8, p.off_b3, p.b3, p.Cout);
      if (EXPAND && !FOLD) stage_bias(12, p.off_b1, p.b1 + ch0, p.Cexp);
      if (FOLD) {
        for (int row = tid; row < p.Cexp; row += kThreads) {
          // the bias as bf16 high and low parts (their sum carries 16 mantissa bits, and 1.0 * part is exact in the fp32 accumulator)
          const float b = row == tid ? fold_b : __ldg(p.b1 + ch0 + row);
          const __nv_bfloat16 hi = __float2bfloat16_rn(b);
          const __nv_bfloat16 lo = __float2bfloat16_rn(b - __bfloat162float(hi));
          const uint32_t i = ((uint32_t)row << cs) + (uint32_t)cin_chunks;
          *reinterpret_cast<uint4*>(smem + p.off_w1 + ((i << 4) ^ (((i >> 3) & swz_mask) << 4))) =
              make_uint4((uint32_t)__bfloat16_as_ushort(hi) | ((uint32_t)__bfloat16_as_ushort(lo) << 16), 0, 0, 0);
        }
      }
    };
    // ---- per-thread work mapping: needs no device memory, so it runs before the wait for the previous grid of the
    // stream (with back-to-back launches it overlaps that grid's tail) ----
    const int g = warp / kGroupWarps;
    const int gwarp0 = g * kGroupWarps;           // first warp of the group
    const int gt = tid - gwarp0 * 32;             // thread index in the group
    const uint32_t gbar = 1u + (uint32_t)g;       // named barrier of the group
    const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
    const int gw = warp - gwarp0;                 // warp index in the group
    const int xi = gw - (kGroupWarps - kExpandIssuers);   // >= 0: this warp issues expand tiles xi, xi + 2, ...
    // Depthwise work split: thread = (channel pair, slot). Stride 1: an item is a block of 2 output rows x segw output
    // columns. Stride 2: an item is one output column
    // of one row group.
    constexpr int kSlots = kGroupThreads / 8;
    const int cp = gt & 7, slot = gt >> 3;
    const int cp_off = (cp & 3) * 4;   // byte offset inside a 16-byte pixel entry
    const uint32_t e_pitch = (uint32_t)p.IW * 16u, d_pitch = (uint32_t)p.Wo * 16u;
    const int per_row = p.per_row;                                         // items per output row (stride 1: column segments) / per row group
    int groups = 1, rows_per_group = rows_valid;                           // stride 2: row groups
    if (p.stride != 1) {
      groups = max(1, min(rows_valid, p.col_slots));
      rows_per_group = (rows_valid + groups - 1) / groups;
    }
    const int dw_items = per_row * (p.stride == 1 ? (rows_valid + 1) / 2 : groups);   // stride 1: blocks of two rows
    const int item0_r = (int)fast_div((uint32_t)slot, (uint32_t)per_row, p.per_row_recip), item0_c = slot - item0_r * per_row;   // the thread's first item
    const int step_r = p.step_r, step_c = p.step_c;                        // item += kSlots in (row, column) form
    const int e_bytes = 2 * p.e_plane;
    // Expand-epilogue tiles of this warp: the group's warps of one tensor-memory lane quarter (warp & 3) share the M1
    // tiles round-robin, at most kTilesPerWarp each. e_pix[k]: pixel index in an E plane (the tile has no padding
    // columns, the E chunk does), -1: no such pixel; bit k of e_inimg: the row lies inside the image (the rest is the
    // zero padding of the intermediate tensor).
    const int q_first = (((warp & 3) - gwarp0) & 3);                // group-relative index of the quarter's first warp
    const int q_mates = (kGroupWarps - q_first + 3) >> 2;           // warps of this quarter in the group (3 or 4)
    const int q_rank = (warp - gwarp0 - q_first) >> 2;              // this warp's rank among them
    constexpr uint32_t kNone = 0xffffffffu;
    uint32_t e_off[kTilesPerWarp];   // shared-memory address of the thread's pixel in plane 0 of the group's E buffer
    uint32_t e_inimg = 0;
#pragma unroll
    for (int k = 0; k < kTilesPerWarp; ++k) {
      const int t = q_rank + k * q_mates;
      const int pix = t * 128 + (warp & 3) * 32 + lane;
      const int ih = (int)fast_div((uint32_t)pix, (uint32_t)p.W, p.w_recip), iw = pix - ih * p.W;
      const int gh = gh0 + ih;
      e_off[k] = kNone;
      if (t < p.M1 && pix < p.P_x) {
        e_off[k] = smem_u32(sE) + (uint32_t)(g * e_bytes + (ih * p.IW + iw + 1) * 16);
        if (gh >= 0 && gh < p.H) e_inimg |= 1u << k;
      }
    }

    // Without the expand GEMM a chunk is 16 channels of the input strip, copied asynchronously into one of the
    // group's two E buffers two chunks ahead: 16-byte pieces (pixel, 8-channel plane), rows outside the image
    // zero-filled. The piece geometry is the same for every chunk.
    constexpr int kPieces = 8;                      // P_x * 2 pieces over the group's threads
    uint32_t ld_src[kPieces], ld_dst[kPieces], ld_ok = 0u, ld_in = 0u;
    const uint8_t* xin = reinterpret_cast<const uint8_t*>(p.x) + ((int64_t)n * p.H + gh0) * p.W * p.Cfull * 2 + ch0 * 2;   // row gh0 may lie outside
    if (!EXPAND) {
#pragma unroll
      for (int k = 0; k < kPieces; ++k) {
        const int i = gt + k * kGroupThreads;
        ld_src[k] = 0u; ld_dst[k] = 0u;
        if (i < p.P_x * 2) {
          const int pix = i >> 1, plane = i & 1;
          const int ih = (int)fast_div((uint32_t)pix, (uint32_t)p.W, p.w_recip), iw = pix - ih * p.W;
          ld_ok |= 1u << k;
          ld_dst[k] = (uint32_t)(plane * p.e_plane + (ih * p.IW + iw + 1) * 16);
          if (gh0 + ih >= 0 && gh0 + ih < p.H) { ld_in |= 1u << k; ld_src[k] = (uint32_t)(pix * p.Cfull * 2 + plane * 16); }
        }
      }
    }
    auto load_chunk = [&](int c, int b) {   // chunk c -> E buffer (g, b); always one commit group
      if (c < p.NC) {
        const uint32_t e0 = smem_u32(sE) + (uint32_t)((g * 2 + b) * e_bytes);   // two buffers per group
#pragma unroll
        for (int k = 0; k < kPieces; ++k) {
          if ((ld_ok >> k) & 1u) {
            const bool in = (ld_in >> k) & 1u;
            cp_async_16(e0 + ld_dst[k], in ? xin + ld_src[k] + c * kChunkRowBytes : reinterpret_cast<const uint8_t*>(p.x), in ? 16u : 0u);
          }
        }
      }
      cp_async_commit();
    };
    if (warp == kWarps - 2) {      // before the wait: an allocation takes 400 cycles
      tmem_alloc(tmem_slot, (uint32_t)p.tmem_cols);
      tmem_relinquish();
    }
    grid_dependency_wait();      // first access to device memory below
    grid_launch_dependents_if(warp == kWarps - 2);
    if constexpr (TMA) {
      if (warp == kWarps - 1) {      // the warp that set the barrier up
        __syncwarp();
        const uint32_t one = elect_one(), bar = smem_u32(bar_x), s0 = smem_u32(smem), rb = (uint32_t)p.row_bytes;
        mbar_arrive_expect_tx_elected(bar, (uint32_t)(p.kblocks * (p.M1 * 128 + p.Cexp)) * rb, one);
        for (int kb = 0; kb < p.kblocks; ++kb) {
          for (int t = 0; t < p.M1; ++t)
            tma_load_3d_elected(s0 + (uint32_t)p.off_x + (uint32_t)(kb * p.M1 + t) * 128u * rb, &maps.x, bar, kb * 64, gh0 * p.W + t * 128, n, one);
          for (int r0 = 0; r0 < p.Cexp; r0 += p.w1_box)
            tma_load_2d_elected(s0 + (uint32_t)p.off_w1 + (uint32_t)(kb * p.Cexp + r0) * rb, &maps.w1, bar, kb * 64, ch0 + r0, one);
        }
      }
    }
    if (!EXPAND) { load_chunk(g, 0); load_chunk(g + NG, 1); }   // the first two chunks travel while the weights are staged
    stage();
    // the zero padding columns of the two E chunk buffers (written once: every chunk reuses them)
    constexpr int kEPlanes = (EXPAND ? NG : 2 * NG) * 2;   // one E buffer per group (two when the chunks are copied in), two planes each
    for (int i = tid; i < p.IH * 2 * kEPlanes; i += kThreads) {
      const int ih = i / (2 * kEPlanes), side = (i / kEPlanes) & 1, plane = i % kEPlanes;
      *reinterpret_cast<uint4*>(sE + plane * p.e_plane + (ih * p.IW + side * (p.W + 1)) * 16) = make_uint4(0, 0, 0, 0);
    }

    // Group g owns the chunks c = g, g + NG, ... (expand buffer, E buffer and D buffer g). A group alternates expand epilogue and
    // depthwise stage with a group-wide barrier after each; the groups are out of phase, so one group's barrier and
    // tensor-memory latencies hide behind the others' arithmetic.
    // MMAs are issued inline, right after the barrier that makes their operands ready: the expand GEMM of chunk c + NG
    // by the group's last two warps (the first to run out of depthwise items), the project GEMM of chunk c by M2 warps,
    // one tile each -- a parked issuer warp would share its scheduler with busy warps and issue an MMA every few
    // hundred cycles, and the project GEMM is urgent: it must be through before the depthwise stage of chunk c + NG
    // may overwrite its operand.
    // Descriptors as (low, high) words: start address and LBO live in the low word, so an operand advances with one
    // 32-bit add (shared-memory addresses >> 4 stay below the 14-bit field limit).
    uint32_t e_tm[kTilesPerWarp];   // tensor-memory address of this warp's k-th expand tile (buffer g)
#pragma unroll
    for (int k = 0; k < kTilesPerWarp; ++k) {
      const int t = q_rank + k * q_mates;
      e_tm[k] = t < p.M1 ? lane_base + p.ecol0 + (t * NG + g) * kChunk : kNone;
    }
    const uint32_t sbo_x = 8u * (uint32_t)p.row_bytes;
    const uint64_t xdesc0 = make_smem_desc(smem_u32(sX), 0, sbo_x, p.swizzle);
    const uint64_t w1desc0 = make_smem_desc(smem_u32(sW1), 0, sbo_x, p.swizzle);
    // D: un-swizzled K-major; the two 8-channel planes are the two K core-matrix columns
    const uint64_t ddesc0 = make_smem_desc(smem_u32(sD), (uint32_t)p.d_plane, 128, SW_NONE);
    const uint64_t w3desc0 = make_smem_desc(smem_u32(sW3), 0, 256, SW_32B);
    // MMAs are issued by whole, converged warps: the MMA itself is predicated on one elected lane, its descriptors are
    // ready 64-bit values (see tc_common.cuh: several times the issue rate of a lane-0 branch next to busy warps).
    const uint32_t elected = elect_one();
    // Expand issue state of the group's last two warps: tiles xi, xi + 2, ... of the group's chunks -> buffer g.
    const uint32_t idesc_e = make_idesc_bf16(128, kChunk);
    const uint64_t exp_a_step = (uint64_t)((uint32_t)(kExpandIssuers * 128 * p.row_bytes) >> 4);
    const uint64_t exp_a0 = xdesc0 + (uint64_t)((uint32_t)(max(xi, 0) * 128 * p.row_bytes) >> 4);
    uint32_t exp_d_tmem0 = p.ecol0 + (max(xi, 0) * NG + g) * kChunk;
    const uint64_t exp_b_step = (uint64_t)((uint32_t)(NG * kChunk * p.row_bytes) >> 4);   // the group's next chunk is c + NG
    uint64_t exp_b = w1desc0 + (uint64_t)((uint32_t)(g * kChunk * p.row_bytes) >> 4);
    const int ksteps = p.ksteps;
    const int exp_tiles = xi >= 0 ? (p.M1 - xi + kExpandIssuers - 1) / kExpandIssuers : 0;   // tiles this warp issues per chunk
    auto issue_expand_as = [&](uint32_t idesc_e) {   // whole warp. Straight-line per reduction length.
      uint64_t a = exp_a0;
      uint32_t d_tmem = exp_d_tmem0;
      const uint64_t b = exp_b;
      if (ksteps == 2) {
#pragma unroll 1
        for (int t = 0; t < exp_tiles; ++t, a += exp_a_step, d_tmem += kExpandIssuers * NG * kChunk) {
          umma_bf16_elected<false>(d_tmem, a, b, idesc_e, elected);
          umma_bf16_elected<true>(d_tmem, a + 2u, b + 2u, idesc_e, elected);
        }
      } else if (ksteps == 4) {
#pragma unroll 1
        for (int t = 0; t < exp_tiles; ++t, a += exp_a_step, d_tmem += kExpandIssuers * NG * kChunk) {
          umma_bf16_elected<false>(d_tmem, a, b, idesc_e, elected);
          umma_bf16_elected<true>(d_tmem, a + 2u, b + 2u, idesc_e, elected);
          umma_bf16_elected<true>(d_tmem, a + 4u, b + 4u, idesc_e, elected);
          umma_bf16_elected<true>(d_tmem, a + 6u, b + 6u, idesc_e, elected);
        }
      } else if (ksteps == 1) {
#pragma unroll 1
        for (int t = 0; t < exp_tiles; ++t, a += exp_a_step, d_tmem += kExpandIssuers * NG * kChunk)
          umma_bf16_elected<false>(d_tmem, a, b, idesc_e, elected);
      } else {                                 // K blocks of four steps (the last one may have fewer)
        const uint64_t a_blk = (uint64_t)((uint32_t)(p.M1 * 128 * 128) >> 4), b_blk = (uint64_t)((uint32_t)(p.Cexp * 128) >> 4);
#pragma unroll 1
        for (int t = 0; t < exp_tiles; ++t, a += exp_a_step, d_tmem += kExpandIssuers * NG * kChunk) {
          uint64_t ak = a, bk = b;
#pragma unroll 1
          for (int ks = 0; ks < ksteps; ks += 4, ak += a_blk, bk += b_blk) {
            umma_bf16_elected_acc(d_tmem, ak, bk, idesc_e, elected, ks > 0 ? 1u : 0u);
            if (ks + 1 < ksteps) umma_bf16_elected<true>(d_tmem, ak + 2u, bk + 2u, idesc_e, elected);
            if (ks + 2 < ksteps) umma_bf16_elected<true>(d_tmem, ak + 4u, bk + 4u, idesc_e, elected);
            if (ks + 3 < ksteps) umma_bf16_elected<true>(d_tmem, ak + 6u, bk + 6u, idesc_e, elected);
          }
        }
      }
    };
    auto issue_expand = [&]() {      // one chunk; advances to the group's next one
      issue_expand_as(idesc_e);
      umma_commit_elected(bar_e + g, elected);
      exp_b += exp_b_step;
    };
    // Project issue state of warp gw < M2 (tile gw), kept in three registers: a warp that runs a serial instruction
    // chain next to warps with dense arithmetic gets an issue slot only every few tens of cycles, so the path from
    // the barrier to the MMA is one add, the MMA and the commit.
    const uint32_t idesc_p = make_idesc_bf16(128, (uint32_t)p.Coutp);
    const uint64_t proj_a = ddesc0 + (uint64_t)((uint32_t)(g * d_bytes + gw * 128 * 16) >> 4);
    uint32_t proj_d_tmem = p.pcol0 + gw * p.Coutp;
    const uint64_t proj_b_step = (uint64_t)((uint32_t)(NG * p.Coutp * kChunkRowBytes) >> 4);     // the group's next chunk is c + NG
    uint64_t proj_b = w3desc0 + (uint64_t)((uint32_t)(g * p.Coutp * kChunkRowBytes) >> 4);
    // The thread's first depthwise item (for most shapes its only one) is the same for every chunk: offsets of its
    // first input / output pixel inside a plane and its extent (stride 1: columns, rows; stride 2: first and last row).
    const bool has_item = slot < dw_items;
    uint32_t it_e, it_d; int it_a, it_b;
    if (p.stride == 1) {
      const int wo = item0_c * p.segw;
      it_e = (uint32_t)(2 * item0_r) * e_pitch + wo * 16; it_d = (uint32_t)(2 * item0_r) * d_pitch + wo * 16;
      it_a = min(p.segw, p.Wo - wo); it_b = min(2, rows_valid - 2 * item0_r);
    } else {
      it_e = item0_c * 32; it_d = item0_c * 16;
      it_a = item0_r * rows_per_group; it_b = min(rows_valid, it_a + rows_per_group);
    }
    const uint32_t e_plane0 = smem_u32(sE) + (uint32_t)((EXPAND ? g : g * 2) * e_bytes + (cp >> 2) * p.e_plane + cp_off);
    const uint32_t d_plane = smem_u32(sD) + (uint32_t)(g * d_bytes + (cp >> 2) * p.d_plane + cp_off);
    // running shared-memory addresses of this thread's depthwise weights / bias and of the chunk's expand bias
    uint32_t wd_addr = smem_u32(sWd) + (uint32_t)(g * 9 * kChunkRowBytes + cp * 4);
    uint32_t bd_addr = smem_u32(sBd) + (uint32_t)((g * kChunk + cp * 2) * 4);
    uint32_t b1_addr = smem_u32(sB1) + (uint32_t)(g * kChunk * 4);
    // All of the above needs nothing that the copies bring: it runs (and its instructions are fetched) while they travel.
    cp_async_wait_all();
    fence_proxy_async_smem();
  tcgen05_fence_before_sync();
  __syncthreads();
  tcgen05_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;
    if (PROJECT && p.CS > 1) {
      if (tid == 0)
        for (int k = 0, cg = 0; cg < (p.Coutp >> 4); ++k, cg += p.piece_cgs)
          mbar_arrive_expect_tx(bar_red + k, (uint32_t)((p.CS - 1) * min(p.piece_cgs, (p.Coutp >> 4) - cg) * 64 * p.PP));
      __syncwarp();
      if (!p.recv_shared) cluster_arrive();       // the barrier is armed: the others may send from now on
    }
    exp_d_tmem0 += tmem_base;
    proj_d_tmem += tmem_base;
#pragma unroll
    for (int k = 0; k < kTilesPerWarp; ++k) if (e_tm[k] != kNone) e_tm[k] += tmem_base;
    if (EXPAND && xi >= 0) {
      if (TMA) mbar_wait(bar_x, 0, abort_flag, p.status, 0x109);
      if (NG == 2) {
        // group 1 issues its first expand GEMM once group 0's is through the tensor pipe: group 0 has the longer chain
        // of chunks, and its first epilogue would otherwise wait for both groups' MMAs
        if (g < p.NC) {
          if (g == 1) {
            if (lane == 0) mbar_wait(bar_chain, 0, abort_flag, p.status, 0x107);
            __syncwarp();
          }
          issue_expand();
          if (g == 0) umma_commit_elected(bar_chain, elected);
        }
      } else {
        // The first chunks of all groups lie side by side in W1 and in tensor memory: one product with N = 16 x groups
        // makes them all (an MMA costs about the same with N = 16 and N = 64: its operand fetch bounds it).
        if (g == 0) {
          const int first = min(NG, p.NC);
          issue_expand_as(make_idesc_bf16(128, (uint32_t)(kChunk * first)));
          for (int i = 0; i < first; ++i) umma_commit_elected(bar_e + i, elected);
        }
        exp_b += exp_b_step;
      }
    }
    __syncwarp();
    // Waits on MMA completion are taken by ONE warp of the group, just before it arrives at the group barrier that
    // the others are parked at: a polling warp spends issue slots, sixteen of them a large share of the SM's.
    const bool waiter = gw == kGroupWarps - 1;
    if (EXPAND && g < p.NC) {
      if (waiter) mbar_wait(bar_e + g, 0, abort_flag, p.status, 0x102);   // the group's first expand GEMM
      named_barrier_sync(gbar, kGroupThreads);
    }
    for (int c = g, it = 0; c < p.NC; c += NG, ++it) {
      // ---- P3: expand epilogue of chunk c -> E[g]: + b1, ReLU6, zero outside the image, bf16 ----
      if (!EXPAND) cp_async_wait_but_one();   // this thread's pieces of chunk c have landed
      if (EXPAND) {
      tcgen05_fence_after_sync();
#pragma unroll
      for (int k = 0; k < kTilesPerWarp; ++k) {
        if (e_tm[k] == kNone) break;   // warp-uniform
        uint32_t acc[16];
        tmem_ld_x16(e_tm[k], acc);
        tmem_ld_wait();
        if (e_off[k] != kNone) {
          uint32_t w[8];
          if (FOLD && ((e_inimg >> k) & 1u)) {   // the bias came out of the expand GEMM
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] = relu6_pack(__uint_as_float(acc[2 * j]), __uint_as_float(acc[2 * j + 1]));
          } else if ((e_inimg >> k) & 1u) {
            const float4 b0 = lds128f<0>(b1_addr), b1v = lds128f<16>(b1_addr), b2 = lds128f<32>(b1_addr), b3v = lds128f<48>(b1_addr);
            w[0] = relu6_pack(__uint_as_float(acc[0]) + b0.x, __uint_as_float(acc[1]) + b0.y);
            w[1] = relu6_pack(__uint_as_float(acc[2]) + b0.z, __uint_as_float(acc[3]) + b0.w);
            w[2] = relu6_pack(__uint_as_float(acc[4]) + b1v.x, __uint_as_float(acc[5]) + b1v.y);
            w[3] = relu6_pack(__uint_as_float(acc[6]) + b1v.z, __uint_as_float(acc[7]) + b1v.w);
            w[4] = relu6_pack(__uint_as_float(acc[8]) + b2.x, __uint_as_float(acc[9]) + b2.y);
            w[5] = relu6_pack(__uint_as_float(acc[10]) + b2.z, __uint_as_float(acc[11]) + b2.w);
            w[6] = relu6_pack(__uint_as_float(acc[12]) + b3v.x, __uint_as_float(acc[13]) + b3v.y);
            w[7] = relu6_pack(__uint_as_float(acc[14]) + b3v.z, __uint_as_float(acc[15]) + b3v.w);
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) w[j] = 0u;
          }
          sts128(e_off[k], w[0], w[1], w[2], w[3]);
          sts128(e_off[k] + (uint32_t)p.e_plane, w[4], w[5], w[6], w[7]);
        }
      }
      b1_addr += (uint32_t)NG * kChunk * 4u;
      tcgen05_fence_before_sync();
      }
      // D[g] was read by the project GEMM of chunk c - 2
      if (PROJECT && waiter && it >= 1) mbar_wait(bar_d + g, (uint32_t)(it - 1) & 1u, abort_flag, p.status, 0x103);
      named_barrier_sync(gbar, kGroupThreads);
      if (EXPAND && xi >= 0 && c + NG < p.NC) {   // expand buffer g is drained: the expand GEMM of the group's next chunk
        tcgen05_fence_after_sync();
        issue_expand();
      }

      // ---- P4: depthwise 3x3 + bias + ReLU6 on CUDA cores: E[g] -> D[g] (A operand of the project GEMM) ----
      {
        uint32_t wgt[9];   // packed bf16 pairs
        wgt[0] = lds32<0>(wd_addr); wgt[1] = lds32<32>(wd_addr); wgt[2] = lds32<64>(wd_addr);
        wgt[3] = lds32<96>(wd_addr); wgt[4] = lds32<128>(wd_addr); wgt[5] = lds32<160>(wd_addr);
        wgt[6] = lds32<192>(wd_addr); wgt[7] = lds32<224>(wd_addr); wgt[8] = lds32<256>(wd_addr);
        const float2 bias = make_float2(__uint_as_float(lds32<0>(bd_addr)), __uint_as_float(lds32<4>(bd_addr)));
        wd_addr += (uint32_t)NG * 9u * kChunkRowBytes; bd_addr += (uint32_t)NG * kChunk * 4u;   // the group's next chunk is c + NG
        const uint32_t e_plane = e_plane0 + (EXPAND ? 0u : (uint32_t)((it & 1) * e_bytes));
        if (has_item) {
          // the geometry of the thread's first item was fixed before the chunk loop; shapes with more items than slots
          // go around with that of the next ones (one copy of the unrolled block: the code of a chunk stays small)
          uint32_t e = e_plane + it_e, d = d_plane + it_d;
          int ia = it_a, ib = it_b, r = item0_r, col = item0_c;
#pragma unroll 1
          for (int item = slot;;) {
            if (p.stride == 1) depthwise_block(e, d, e_pitch, d_pitch, p.segw, ia, ib, wgt, bias);
            else if (ia < ib) depthwise_column_s2(e, d, ia, ib, p.IW, p.Wo, wgt, bias);
            if ((item += kSlots) >= dw_items) break;
            r += step_r; col += step_c;
            if (col >= per_row) { col -= per_row; ++r; }
            if (p.stride == 1) {
              const int wo = col * p.segw;
              e = e_plane + (uint32_t)(2 * r) * e_pitch + wo * 16; d = d_plane + (uint32_t)(2 * r) * d_pitch + wo * 16;
              ia = min(p.segw, p.Wo - wo); ib = min(2, rows_valid - 2 * r);
            } else {
              ia = r * rows_per_group; ib = min(rows_valid, ia + rows_per_group);
              e = e_plane + col * 32; d = d_plane + col * 16;
            }
          }
        }
      }
      fence_proxy_async_smem();
      // the expand GEMM of the group's next chunk (issued after the previous barrier) is complete
      if (EXPAND && waiter && c + NG < p.NC) mbar_wait(bar_e + g, (uint32_t)(it + 1) & 1u, abort_flag, p.status, 0x105);
      named_barrier_sync(gbar, kGroupThreads);
      if (!EXPAND) load_chunk(c + 2 * NG, it & 1);   // the E buffer of chunk c is free
      if (!PROJECT) {
        // the depthwise result of the chunk is the output: 16-byte pieces (pixel, plane) of D[g] to device memory
        const int pieces = rows_valid * p.Wo * 2;
        __nv_bfloat16* o0 = p.out + ((size_t)n * p.Ho + ho0) * p.Wo * p.Cfull + ch0 + c * kChunk;
        for (int i = gt; i < pieces; i += kGroupThreads) {
          const int pix = i >> 1, plane = i & 1;
          *reinterpret_cast<uint4*>(o0 + (size_t)pix * p.Cfull + plane * 8) =
              *reinterpret_cast<const uint4*>(sD + g * d_bytes + plane * p.d_plane + pix * 16);
        }
      }
      if (PROJECT && gw < p.M2) {   // D[g] is complete: the project GEMM of chunk c, one tile per warp
        // chunk 0 overwrites the accumulators: everything else is issued after it
        if (c >= 1 && c < NG) {
          if (lane == 0) mbar_wait(bar_first, 0, abort_flag, p.status, 0x106);
          __syncwarp();
        }
        tcgen05_fence_after_sync();
        umma_bf16_elected_acc(proj_d_tmem, proj_a, proj_b, idesc_p, elected, c > 0 ? 1u : 0u);
        umma_commit_elected(bar_d + g, elected);
        if (c == 0) umma_commit_elected(bar_first, elected);
        if (c + NG >= p.NC && !skip_signal_for_test(p.status, 0x104)) umma_commit_elected(bar_done, elected);
      }
      proj_b += proj_b_step;
    }

    // ---- P6: project epilogue: + b3 (+ residual), bf16, 16-byte stores ----
    if (PROJECT) {
      if (warp == kWarps - 1) mbar_wait(bar_done, 0, abort_flag, p.status, 0x104);
      __syncthreads();
      tcgen05_fence_after_sync();
      const int valid_pix = rows_valid * p.Wo;
      const size_t gpix0 = ((size_t)n * p.Ho + ho0) * p.Wo;
      if (p.CS > 1) {
        // ---- the channel shares of the cluster's CTAs are added: CTA r sums and stores pixels [r PP, (r + 1) PP) of the
        // strip. A CTA lays its fp32 partial sums out as one block [4 channels][pixel] per owner (over its own operands,
        // which are dead now) and sends each block by bulk copies (single 16-byte stores into the other CTAs took
        // three times as long), a piece of some output channels at a time: a piece travels while the next is laid out and the
        // previous one summed up. Where the incoming blocks have no memory of their own they go over operands too, so the
        // cluster meets once more before anything is sent. ----
        const int ncg = p.Coutp >> 4;
        const uint32_t out0 = smem_u32(smem) + (uint32_t)p.off_send, in0 = smem_u32(smem) + (uint32_t)p.off_recv;
        const uint32_t block = (uint32_t)(p.Coutp * p.PP * 4);
        for (int k = 0, cg0 = 0; cg0 < ncg; ++k, cg0 += p.piece_cgs) {
          const int cgs = min(p.piece_cgs, ncg - cg0);
          for (int u = warp >> 2; u < p.M2 * cgs; u += kWarps / 4) {
            const int t = u / cgs, cg = cg0 + u - t * cgs;
            const int po = t * 128 + (warp & 3) * 32 + lane;
            uint32_t acc[16];
            tmem_ld_x16(tmem_base + lane_base + p.pcol0 + t * p.Coutp + cg * 16, acc);
            tmem_ld_wait();
            if (po < valid_pix) {
              const uint32_t owner = fast_div((uint32_t)po, (uint32_t)p.PP, p.pp_recip);
              const uint32_t a = out0 + owner * block + (uint32_t)((cg * 4 * p.PP + po - (int)owner * p.PP) * 16);
#pragma unroll
              for (int q = 0; q < 4; ++q) sts128(a + (uint32_t)(q * p.PP * 16), acc[4 * q], acc[4 * q + 1], acc[4 * q + 2], acc[4 * q + 3]);
            }
          }
          fence_proxy_async_smem();
          __syncthreads();
          if (k == 0) {
            if (p.recv_shared) cluster_arrive();   // this CTA's operands are dead
            cluster_wait();                        // ... every CTA's, or: every CTA has started (it arrived when its barriers were set up)
          }
          if (tid < p.CS - 1) {
            const uint32_t peer = (uint32_t)((rank + 1 + tid) % p.CS), at = (uint32_t)(cg0 * 64 * p.PP);
            bulk_copy_to_cluster(cluster_map(in0 + (uint32_t)rank * block + at, peer), out0 + peer * block + at, (uint32_t)(cgs * 64 * p.PP),
                                 cluster_map(smem_u32(bar_red + k), peer));
          }
        }
        const int own0 = rank * p.PP, own = min(p.PP, valid_pix - own0), c8n = p.Cout >> 3;
        for (int k = 0, cg0 = 0; cg0 < ncg; ++k, cg0 += p.piece_cgs) {
          const int c80 = cg0 * 2, c8s = min(2 * p.piece_cgs, c8n - c80);      // 16-byte pieces of a pixel
          const uint32_t recip = c8s == 2 * p.piece_cgs ? p.c8s_recip : p.c8s_last_recip;
          int i = tid, lp = (int)fast_div((uint32_t)i, (uint32_t)c8s, recip), c8 = c80 + i - lp * c8s;
          auto residual_of = [&]() -> uint4 {       // stride 1, Cin == Cout: the input at the same place
            if (!(EXPAND && p.residual) || i >= own * c8s) return make_uint4(0, 0, 0, 0);
            return __ldg(reinterpret_cast<const uint4*>(p.x + (gpix0 + own0 + lp) * p.Cout + c8 * 8));
          };
          uint4 xr = residual_of();                 // travels while the blocks do
          mbar_wait(bar_red + k, 0, abort_flag, p.status, 0x108);
          if (cg0 + p.piece_cgs >= ncg) { __syncwarp(); cluster_arrive(); }      // this thread has seen everything arrive
          while (i < own * c8s) {
            float v[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) v[q] = sB3[c8 * 8 + q];
            v[0] += bf16_lo(xr.x); v[1] += bf16_hi(xr.x); v[2] += bf16_lo(xr.y); v[3] += bf16_hi(xr.y);
            v[4] += bf16_lo(xr.z); v[5] += bf16_hi(xr.z); v[6] += bf16_lo(xr.w); v[7] += bf16_hi(xr.w);
            const uint32_t at = (uint32_t)((c8 * 2 * p.PP + lp) * 16);
            for (int src = 0; src < p.CS; ++src) {
              const uint32_t a = (src == rank ? out0 : in0) + (uint32_t)src * block + at;
              const float4 lo = lds128f<0>(a), hi = lds128f<0>(a + (uint32_t)(p.PP * 16));
              v[0] += lo.x; v[1] += lo.y; v[2] += lo.z; v[3] += lo.w; v[4] += hi.x; v[5] += hi.y; v[6] += hi.z; v[7] += hi.w;
            }
            *reinterpret_cast<uint4*>(p.out + (gpix0 + own0 + lp) * p.Cout + c8 * 8) =
                make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
            if ((i += kThreads) >= own * c8s) break;
            lp = (int)fast_div((uint32_t)i, (uint32_t)c8s, recip); c8 = c80 + i - lp * c8s;
            xr = residual_of();
          }
        }
        cluster_wait();                           // the copies out of this CTA have arrived: it may leave
      } else {
      if (TMA && p.residual) mbar_wait(bar_x, 0, abort_flag, p.status, 0x10a);      // complete since the first product: the strip is read below
      for (int t = warp >> 2; t < p.M2; t += kWarps / 4) {
        const int po = t * 128 + (warp & 3) * 32 + lane;
        for (int j0 = 0; j0 < p.Coutp; j0 += 16) {
          const uint8_t* sXk = wide ? sX + (j0 >> 6) * (p.M1 * 128 * 128) : sX;     // the K block of these channels
          uint32_t acc[16];
          tmem_ld_x16(tmem_base + lane_base + p.pcol0 + t * p.Coutp + j0, acc);
          tmem_ld_wait();
          if (po < valid_pix) {
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int j = j0 + h * 8;
              if (j < p.Cout) {
                float v[8];
#pragma unroll
                for (int q = 0; q < 8; ++q) v[q] = __uint_as_float(acc[h * 8 + q]) + sB3[j + q];
                const size_t off = (gpix0 + po) * p.Cout + j;
                if (EXPAND && p.residual) {
                  // stride 1, Cin == Cout: output pixel po is pixel po + W of the input tile (one halo row above)
                  const uint4 xr = *reinterpret_cast<const uint4*>(sXk + swz_offset(po + p.W, (j >> 3) & 7, p.row_bytes));
                  v[0] += bf16_lo(xr.x); v[1] += bf16_hi(xr.x); v[2] += bf16_lo(xr.y); v[3] += bf16_hi(xr.y);
                  v[4] += bf16_lo(xr.z); v[5] += bf16_hi(xr.z); v[6] += bf16_lo(xr.w); v[7] += bf16_hi(xr.w);
                }
                *reinterpret_cast<uint4*>(p.out + off) =
                    make_uint4(pack_bf16x2(v[0], v[1]), pack_bf16x2(v[2], v[3]), pack_bf16x2(v[4], v[5]), pack_bf16x2(v[6], v[7]));
              }
            }
          }
        }
      }
      }
    }
  tcgen05_fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem_base, (uint32_t)p.tmem_cols);
}

int round_up(int v, int m) { return (v + m - 1) / m * m; }

constexpr int kMaxSplit = 8;     // CTAs per strip (the portable cluster size)
// clusters of 1-CTA-per-SM kernels a B200 keeps resident at once, as cudaOccupancyMaxActiveClusters reports them
constexpr int kResident[kMaxSplit + 1] = {0, 148, 74, 45, 33, 26, 22, 15, 15};

struct Mbv2Host {
  Mbv2Params prm;
  int smem_bytes = 0;
  bool expand = true, project = true;
  std::unordered_map<const void*, CUtensorMap> maps_x, maps_w1;   // by base address
};

bool layout(Mbv2Params& q, int R, bool expand, bool project, int* smem_bytes) {
  const int NG = q.groups, group_threads = kThreads / NG;
  q.R = R;
  q.strips = (q.Ho + R - 1) / R;
  q.strips_recip = fast_div_recip(q.strips);
  q.IH = (R - 1) * q.stride + 3;
  q.IW = q.W + 2;
  if (q.nseg < 4) q.IW |= 1;     // an odd pitch: the warp's blocks in two rows use other banks
  q.P_in = q.IH * q.IW;
  q.P_x = q.IH * q.W;
  q.M1 = (q.P_x + 127) / 128;
  q.M2 = (R * q.Wo + 127) / 128;
  if (q.IH > 256 || q.IW > 256 || q.M1 > 8) return false;
  // per group: at most kTilesPerWarp expand tiles per warp of a lane quarter, one project tile per warp, and (when the
  // chunks are copied in) eight 16-byte pieces per thread
  if (q.M1 > kTilesPerWarp * (kWarps / NG / 4) || q.M2 > kWarps / NG || (!expand && q.P_x * 2 > 8 * group_threads)) return false;
  const int cols = (expand ? NG * q.M1 * kChunk : 0) + (project ? q.M2 * q.Coutp : 0);
  if (cols > 512) return false;
  q.tmem_cols = 32;
  while (q.tmem_cols < cols) q.tmem_cols *= 2;
  q.ecol0 = 0;
  q.pcol0 = expand ? NG * q.M1 * kChunk : 0;
  int off = 0;
  auto take = [&](int bytes) { int o = off; off = round_up(off + bytes, 1024); return o; };
  q.off_x = take(expand ? q.M1 * 128 * q.row_bytes * q.kblocks : 0);
  q.off_w1 = take(expand ? q.Cexp * q.row_bytes * q.kblocks : 0);
  // two 8-channel planes per chunk, offset by 64 mod 128 bytes so that a warp's
  // 2 x 64-byte accesses (4 pixels x 4 channel pairs per plane) never share a bank
  q.e_plane = round_up(q.P_in * 16, 128) + 64;
  q.d_plane = q.M2 * 128 * 16 + 64;
  q.off_e = take((expand ? NG : 2 * NG) * 2 * q.e_plane);   // one chunk buffer per group, two when the chunks are copied in
  q.off_d = take(NG * 2 * q.d_plane);
  q.off_w3 = take(project ? q.NC * q.Coutp * kChunkRowBytes : 0);
  q.off_wd = take(9 * q.Cexp * 2);
  q.off_b1 = take(expand ? q.Cexp * 4 : 0);
  q.off_bd = take(q.Cexp * 4);
  q.PP = ((R * q.Wo + q.CS - 1) / q.CS) | 1;
  q.pp_recip = fast_div_recip(q.PP);
  {
    // A second piece costs 0.1 to 0.9 us of hand-over and hides a layout and a summation: worth it from some 56 KB on (65 KB of
    // 25 images 15 x 15 x 96: one piece 16.3, two 15.5, three 15.6 us; 45 KB of 39 images 11 x 11 x 96: 15.17, 15.16, 15.7;
    // 38 KB of 32 images 14 x 14 x 64: 9.7, 9.9, 9.9; 5 KB of one image 14 x 14 x 32: 5.9, 6.8).
    const int ncg = q.Coutp / 16, pieces = (q.CS - 1) * q.PP * q.Coutp * 4 >= 56 * 1024 ? 2 : 1;
    q.piece_cgs = (ncg + pieces - 1) / pieces;
    const int last = q.Cout / 8 - (ncg - 1) / q.piece_cgs * q.piece_cgs * 2;
    q.c8s_recip = fast_div_recip(2 * q.piece_cgs); q.c8s_last_recip = fast_div_recip(std::max(1, last));
  }
  q.off_send = q.off_recv = q.recv_shared = 0;
  if (project && q.CS > 1) {
    const int blocks = round_up(q.CS * q.PP * q.Coutp * 4, 1024);
    if (std::max(off, blocks) + blocks + 4096 <= 227 * 1024) {      // incoming blocks in memory of their own
      q.off_recv = std::max(off, blocks);
      off = q.off_recv + blocks;
    } else {                                                        // outgoing and incoming blocks over the operands
      q.recv_shared = 1;
      q.off_recv = blocks;
      off = std::max(off, 2 * blocks);
    }
  }
  q.off_b3 = take(project ? q.Coutp * 4 : 0);
  q.off_bar = take(256);
  *smem_bytes = off + 1024;  // slack for the 1024-byte alignment of the base
  return *smem_bytes <= 227 * 1024;
}

// Estimated cycles of a launch with the tiling in `t` (for comparisons between tilings). Per wave of resident CTAs or clusters:
// staging (the bytes a CTA copies), the chunk loop, the output. The chunk loop is the larger of its instruction issue (NC chunks)
// and the chain of a group's chunks, each a chain of latencies. Constants fitted to 23 shapes (7 to 78 pixels wide, 16 to 160
// input channels, batches of 1 to 64) x all their tilings, 1900 launches in all: 6.5 % rms, and the tiling of the least estimate
// is on average 0.3 % slower than the best one measured.
double estimated_cycles(const Mbv2Params& t, bool expand, bool project, int sms) {
  const bool split = project && t.CS > 1;
  const long resident = split ? kResident[t.CS] * (long)sms / kDefaultSMs : sms / t.CS;
  const long units = (long)t.N * t.strips, waves = (units + std::max(1l, resident) - 1) / std::max(1l, resident);
  const int slots = kThreads / t.groups / 8;
  double dw_issue, dw_chain;       // depthwise stage of one chunk: warp instructions, cycles of a warp's own chain
  if (t.stride == 1) {
    const int items = t.nseg * ((t.R + 1) / 2);
    const double block = (t.segw + 2) / 9.0;
    dw_issue = items * 8 / 32.0 * 360.0 * block;
    dw_chain = (items + slots - 1) / slots * 800.0 * block;
  } else {
    const int rows = (t.R + std::max(1, std::min(t.R, t.col_slots)) - 1) / std::max(1, std::min(t.R, t.col_slots));
    const int items = t.Wo * std::max(1, std::min(t.R, t.col_slots));
    dw_issue = t.Wo * t.R * 8 / 32.0 * 45.0;
    dw_chain = (items + slots - 1) / slots * (rows * 130.0 + 100.0);
  }
  const double issue = t.NC * (dw_issue + t.M1 * 4 * 30.0 + t.M2 * 370.0) / 4 / 0.59;
  const double chain = (t.NC + t.groups - 1) / t.groups * (515.0 + 1.5 * dw_chain + 68.0 * t.M1);
  const double loop = std::pow(std::pow(issue, 4) + std::pow(chain, 4), 0.25);
  const double bytes = (expand ? (double)(t.P_x + t.Cexp) * t.Cin * 2 : 0.0) + (project ? t.Cexp * t.Cout * 2.0 : 0.0) + t.Cexp * 26.0;
  const double out = split ? 1100.0 + 0.066 * (t.CS - 1) / t.CS * (t.R * t.Wo * t.Coutp * 4.0) : 42.0 * t.M2 * t.Cout / 4;
  return waves * (7500.0 + 0.069 * bytes + loop + out);
}

}  // namespace

ago_status_t mbv2_plan(Plan* plan, FusedState* st, std::string* err) {
  // operator indices of the three convolutions in the chain (-1: the pair has none)
  const bool expand = plan->fused_kernel != AGO_KERNEL_DW_PW, project = plan->fused_kernel != AGO_KERNEL_PW_DW;
  const int i_dw = expand ? 3 : 0, i_pr = expand ? 6 : 3;
  const OpInfo& first = plan->ops[0];
  const OpInfo& d = plan->ops[i_dw];
  auto* host = new Mbv2Host();
  host->expand = expand; host->project = project;
  Mbv2Params& q = host->prm;
  q = Mbv2Params{};
  q.N = (int)first.in.d[0]; q.H = (int)first.in.d[1]; q.W = (int)first.in.d[2];
  q.Cfull = (int)d.in.d[3];
  q.Cin = expand ? (int)first.in.d[3] : 16;
  q.Cout = project ? plan->ops[i_pr].op.p[0] : 16;
  q.stride = d.op.p[3];
  q.Ho = (int)d.out.d[1]; q.Wo = (int)d.out.d[2];
  q.residual = plan->fused_kernel == AGO_KERNEL_MBV2_BLOCK && plan->ops.size() == 9 ? 1 : 0;
  auto bad = [&](const char* m) { *err = std::string("fused inverted-residual block: ") + m; delete host; return AGO_ERR_UNSUPPORTED; };
  if (q.Cin > 256) return bad("more than 256 input channels is not supported");
  if (q.Cfull % kChunk != 0) return bad("expanded channels must be a multiple of 16");
  if (q.Cout > 256) return bad("more than 256 output channels is not supported");
  if (q.residual && (q.stride != 1 || q.Cin != q.Cout)) return bad("residual needs stride 1 and Cin == Cout");
  q.Kp = q.Cin <= 16 ? 16 : (q.Cin <= 32 ? 32 : 64);
  q.ksteps = q.Cin <= 64 ? q.Kp / 16 : (q.Cin + 15) / 16;
  q.kblocks = (q.ksteps + 3) / 4;
  q.cpr = 2 * q.ksteps;      // Cin <= 64: Kp / 8
  q.row_bytes = q.Kp * 2;
  q.swizzle = q.Kp == 16 ? tc::SW_32B : (q.Kp == 32 ? tc::SW_64B : tc::SW_128B);
  q.Coutp = round_up(q.Cout, 16);
  q.fold_b1 = expand && q.Cin % 8 == 0 && q.Cin < q.Kp ? 1 : 0;
  auto recip = [](int d) { return tc::fast_div_recip(d); };
  q.coutp_recip = recip(q.Coutp);
  q.w_recip = recip(q.W);
  q.cpr_recip = recip(q.cpr);
  q.segw = seg_width(q.Wo);
  q.nseg = (q.Wo + q.segw - 1) / q.segw;
  q.per_row = q.stride == 1 ? q.nseg : q.Wo;
  q.per_row_recip = recip(q.per_row);
  auto set_groups = [&](Mbv2Params& t, int ng) {   // depthwise item geometry of a group of 32 / ng warps
    const int slots = kThreads / ng / 8;
    t.groups = ng;
    t.step_r = slots / t.per_row; t.step_c = slots - t.step_r * t.per_row;
    t.col_slots = slots / std::max(1, std::min(t.Wo, slots));
  };
  // Rows per CTA, warp groups and channel split: the least estimated time among all that fit.
  int best_R = 0, best_ng = 2, best_cs = 1; double best_cost = 0; int best_smem = 0;
  const int sms = device_sm_count();
  const int chunks = q.Cfull / kChunk;
  auto set_split = [&](Mbv2Params& t, int cs) {
    t.CS = cs; t.Cexp = q.Cfull / cs; t.NC = chunks / cs;
    t.cexp8_recip = recip(t.Cexp / 8);
  };
  for (int cs = 1; cs <= kMaxSplit; ++cs) {
    if (chunks % cs != 0) continue;
    for (int ng = 2; ng <= 4; ng *= 2) {
      for (int R = 1; R <= q.Ho; ++R) {
        Mbv2Params t = q; int smem = 0;
        set_groups(t, ng);
        set_split(t, cs);
        if (!layout(t, R, expand, project, &smem)) continue;
        const double cost = estimated_cycles(t, expand, project, sms);
        if (best_R == 0 || cost < best_cost) { best_R = R; best_ng = ng; best_cs = cs; best_cost = cost; best_smem = smem; }
      }
    }
  }
  if (best_R == 0) return bad("no row-strip tiling fits shared memory / tensor memory");
  set_groups(q, best_ng);
  set_split(q, best_cs);
  layout(q, best_R, expand, project, &best_smem);
  if ((long)q.N * q.strips > 65535) return bad("more than 65535 row strips in the batch");
  // Input strip and W1 by TMA where a pixel is 64 bytes or more and the strip 12.5 KB or more: the threads' 16-byte copies bring 27
  // bytes per cycle. 25 images of 15 x 15 x 96 15.5 -> 14.6 us, 40 of 20 x 20 x 64 18.6 -> 17.7, 32 of 28 x 28 x 32 at stride 2 9.7 -> 9.2, 26 of
  // 8 x 8 x 160 14.8 -> 13.2; 32 shapes on this side of the line 1.01 to 1.1x. Short strips were 1 to 1.5 % slower (one image 14 x 14 x 32:
  // 2.7 KB, 5.8 -> 5.9; two of 9 x 9 x 96 at stride 2: 5.2 KB), pixels of 32 bytes up to 7 % (8 images of 56 x 56 x 16: 7.6 -> 8.1).
  // Pixels that end inside a 32-byte sector cost their neighbours' bytes too, and boxes of 64 channels that are mostly padding bring zeros:
  // over 36 shapes each the mean of TMA over copies is 1.04 at 72 channels, 1.03 at 88, 1.01 at 104, 0.99 and 1.00 at 136 and 152 with single
  // shapes up to 1.2 (30 images of 17 x 20 x 72 10.3 -> 11.4 us, 40 of 18 x 18 x 72 expanded to 32 5.1 -> 6.1), but 0.96 to 0.98 at 120
  // and 184, in whole blocks also at 168 and 200 (pairs 1.0), and 0.93 to 0.99 for whole sectors.
  const bool whole_sectors = q.Cin % 16 == 0 || q.Cin % 64 == 56 || (project && q.Cin >= 168);
  q.tma = expand && !q.fold_b1 && whole_sectors && q.Cin >= 32 && q.P_x >= 64 && q.P_x * q.Cin * 2 >= 12800 ? 1 : 0;
  q.w1_box = std::min(q.Cexp, 256);
  while (q.Cexp % q.w1_box != 0) q.w1_box -= kChunk;
  host->smem_bytes = best_smem;
  st->impl = host;
  st->impl_free = [](void* p) { delete static_cast<Mbv2Host*>(p); };
  // cycles -> us, the constant factor of each chain over 976 measured shapes (rms 7 % blocks, 10 to 11 % pairs)
  plan->fused_us = best_cost / (project ? 1820.0 : 2170.0);
  st->tile_rows = best_R; st->grid = q.N * q.strips * q.CS; st->smem_bytes = best_smem;
  plan->tile_rows = best_R; plan->smem_bytes = best_smem; plan->fused_variant = q.tma;
  return AGO_OK;
}

namespace {

template <bool EXPAND, bool PROJECT, bool FOLD, int NG, bool TMA>
ago_status_t launch_groups(const Mbv2Params& q, const Mbv2Maps<TMA>& maps, int smem_bytes, cudaStream_t stream, std::string* err) {
  static int smem_opt_in[64] = {};
  cudaError_t e = ensure_max_dynamic_smem(reinterpret_cast<const void*>(mbv2_fused_kernel<EXPAND, PROJECT, FOLD, NG, TMA>), smem_opt_in);
  if (e != cudaSuccess) { *err = std::string("cudaFuncSetAttribute: ") + cudaGetErrorString(e); return AGO_ERR_CUDA; }
  FusedLaunch launch(dim3((unsigned)(q.N * q.strips * q.CS)), kThreads, (size_t)smem_bytes, stream);
  cudaLaunchAttribute attr[2] = {launch.attr[0], {}};
  if (PROJECT && q.CS > 1) {        // the CTAs of a strip add their partial products through distributed shared memory
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = (unsigned)q.CS; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
    launch.config.attrs = attr;
    launch.config.numAttrs = 2;
  }
  e = cudaLaunchKernelEx(&launch.config, mbv2_fused_kernel<EXPAND, PROJECT, FOLD, NG, TMA>, q, maps);
  if (e != cudaSuccess) { *err = std::string("fused inverted-residual launch: ") + cudaGetErrorString(e); return AGO_ERR_CUDA; }
  return AGO_OK;
}
template <bool EXPAND, bool PROJECT, bool FOLD, bool TMA = false>
ago_status_t launch_variant(const Mbv2Params& q, Mbv2Host* host, cudaStream_t stream, std::string* err) {
  Mbv2Maps<TMA> maps;
  if constexpr (TMA) {
    auto get = [&](std::unordered_map<const void*, CUtensorMap>& cache, const void* base, bool weights, CUtensorMap* out) -> bool {
      auto it = cache.find(base);
      if (it == cache.end()) {
        CUtensorMap m;
        const uint64_t wdims[2] = {(uint64_t)q.Cin, (uint64_t)q.Cfull}, xdims[3] = {(uint64_t)q.Cin, (uint64_t)q.H * q.W, (uint64_t)q.N};
        const uint64_t strides[2] = {(uint64_t)q.Cin * 2, (uint64_t)q.H * q.W * q.Cin * 2};
        const uint32_t wbox[2] = {(uint32_t)q.Kp, (uint32_t)q.w1_box}, xbox[3] = {(uint32_t)q.Kp, 128, 1};
        if (!encode_tmap_bf16(&m, base, weights ? 2 : 3, weights ? wdims : xdims, strides, weights ? wbox : xbox, q.row_bytes, err)) return false;
        if (cache.size() > 4096) cache.clear();
        it = cache.emplace(base, m).first;
      }
      *out = it->second;
      return true;
    };
    if (!get(host->maps_x, q.x, false, &maps.x) || !get(host->maps_w1, q.w1, true, &maps.w1)) return AGO_ERR_CUDA;
  }
  return q.groups == 4 ? launch_groups<EXPAND, PROJECT, FOLD, 4, TMA>(q, maps, host->smem_bytes, stream, err)
                       : launch_groups<EXPAND, PROJECT, FOLD, 2, TMA>(q, maps, host->smem_bytes, stream, err);
}

}  // namespace

ago_status_t mbv2_run(const Plan& plan, FusedState* st, const void* const* inputs, const void* const* weights,
                      void* output, unsigned int* status_word, cudaStream_t stream, std::string* err) {
  Mbv2Host* host = static_cast<Mbv2Host*>(st->impl);
  Mbv2Params q = host->prm;
  q.x = static_cast<const __nv_bfloat16*>(inputs[0]);
  int w = 0;   // weights in chain order: (w1, b1) (wd, bd) (w3, b3), without the pair's missing convolution
  if (host->expand) { q.w1 = static_cast<const __nv_bfloat16*>(weights[w]); q.b1 = static_cast<const float*>(weights[w + 1]); w += 2; }
  q.wd = static_cast<const __nv_bfloat16*>(weights[w]); q.bd = static_cast<const float*>(weights[w + 1]); w += 2;
  if (host->project) { q.w3 = static_cast<const __nv_bfloat16*>(weights[w]); q.b3 = static_cast<const float*>(weights[w + 1]); }
  q.out = static_cast<__nv_bfloat16*>(output);
  q.status = status_word;
  if (!host->expand) return launch_variant<false, true, false>(q, host, stream, err);
  if (!host->project)
    return q.fold_b1 ? launch_variant<true, false, true>(q, host, stream, err)
         : q.tma    ? launch_variant<true, false, false, true>(q, host, stream, err)
                    : launch_variant<true, false, false>(q, host, stream, err);
  return q.fold_b1 ? launch_variant<true, true, true>(q, host, stream, err)
       : q.tma    ? launch_variant<true, true, false, true>(q, host, stream, err)
                  : launch_variant<true, true, false>(q, host, stream, err);
}

}  // namespace ago
