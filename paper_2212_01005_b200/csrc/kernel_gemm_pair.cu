// Tensor-core GEMM of the unfused modes for large products: C[M][N] = epilogue(A[M][K] * B) on PAIRED CTAs
// (one launch per complex operator with its simple operators in the epilogue: Section III-A, "conventional
// fusion within a mini-subgraph"). The small-tile kernel (kernel_gemm_tc.cu) fetches 8 KB of operands per
// 128 x 128 x 16 product, which is all the shared memory delivers in the product's 64 cycles; this kernel is the
// one whose main loop is bound by the tensor pipe instead:
//
//   * a cluster of two CTAs computes a 256 x 256 output tile with tcgen05.mma.cta_group::2: each CTA holds 128 rows
//     of A and HALF of the B tile (128 of its 256 columns) and fetches both with its own TMA loads -- no multicast --
//     so a 256 x 256 x 16 product (128 cycles of tensor pipe) reads 8 KB per SM;
//   * persistent pairs walk over the output tiles; two accumulators in tensor memory (2 x 256 columns) let the
//     epilogue of tile i overlap the products of tile i + 1;
//   * roles per CTA: two TMA warps (every second ring stage each), one MMA warp (it issues in the leader CTA only), sixteen
//     epilogue warps (bias / activation / scale in fp32 -> the warp's own 64-byte-swizzled piece of 32 rows x 64 bytes -> TMA
//     store, clipped at the edges). All of them issue converged, on one elected lane.
//
// What bounds it: shared memory. A block of 64 k of a 256-column tile is written by TMA and read by the products once, 2 x 32 KB
// at 128 bytes per cycle = 512 cycles, as many as its products take; measured 560. With tiles of 128 columns 384 and 415.
// It took 724 and 548 with one thread in a lane-0 branch issuing three loads per stage: a wait costs such a thread 150 cycles, an
// announcement 70, a load 135 and each further one 50, so it brought 38 bytes per cycle where an SM takes 125 (and all 148
// together 113 each). GELU's epilogue went from 8.9k to 5k cycles per tile (6.1k are the products of 768 k): twice the warps,
// the bias in shared memory before the products are complete (loaded after them it cost 1.3k per 32 columns). Whole sectors
// stored straight from the registers were slower than pieces (1.4k cycles per 32 columns against 0.8k); stages of two
// blocks made no difference. 3001 x 768 -> 3072 -> 768 as two launches 36.8 -> 26.2 us, 8000 x 512 -> 2048 -> 512 42.3 -> 32.8,
// 12288 x 768 -> 3072 -> 768 102 -> 91 (1.26 PFLOP/s).
//
// Barriers (per ring stage s, per accumulator a):
//   full[s]   leader only, count 1: the leader's TMA warps announce the bytes of both CTAs, both CTAs' loads complete there
//   empty[s]  each CTA, count 1: the leader's MMA warp commits onto both after the stage's products
//   accf[a]   each CTA, count 1: accumulator a complete (committed onto both CTAs by the leader)
//   acce[a]   leader only: its epilogue warps and the peer (relayed by the peer's idle MMA warp) have read accumulator a
//   drain[a]  peer only: its epilogue warps have
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <mutex>
#include <unordered_map>

#include "fused.h"
#include "kernels.h"
#include "tc_common.cuh"
#include "tmap.h"

namespace ago {

namespace {

using namespace tc;

constexpr int kPM = 128;                 // rows per CTA (256 per pair)
constexpr int kPK = 64;                  // reduction elements per ring stage
constexpr int kPStages = 6;
constexpr int kPStageBytes = 32 * 1024;  // A [128 x 64] + this CTA's half of B [<= 128 x 64]
constexpr int kPEpiWarps = 16;           // (tensor-memory lane quarter) x (column quarter of the tile)
constexpr int kPEpiThreads = kPEpiWarps * 32;
constexpr int kPProducers = 2;           // warps that issue the loads, of every second stage each
constexpr int kPThreads = kPEpiThreads + 32 + 32 * kPProducers;
constexpr int kPPieceBytes = 32 * 64;    // staged output: 32 rows x 64 bytes per epilogue warp
constexpr int kPSmemBytes = kPStages * kPStageBytes + kPEpiWarps * kPPieceBytes + 1024 + 256 + 1024;     // ... bias, barriers, alignment

struct GemmPairParams {
  int M, N, K;
  int BN;                  // columns per tile: 128 or 256
  int b_kmajor;
  int b_blocks;            // B is mapped as blocks of 64 columns: one load brings all of a CTA's
  int c_fp32;              // output element: fp32 (else bf16)
  int kblocks, tiles_m, tiles_n, pairs;
  // the simple operators in canonical order: + bias, activation 1, * scale, + tensor, activation 2
  const float* bias;       // or null
  const void* add;         // or null: bf16 tensor [M][N] with the output's leading dimension
  int64_t ldc;
  int act1, act2;          // EPI_RELU | EPI_RELU6 | EPI_GELU | -1
  float scale;
  unsigned int* status;
};

template <int ACT>
__device__ __forceinline__ float pair_activate(float x) {
  if constexpr (ACT == EPI_RELU) return fmaxf(x, 0.0f);
  if constexpr (ACT == EPI_RELU6) return fminf(fmaxf(x, 0.0f), 6.0f);
  if constexpr (ACT == EPI_GELU) {
    const float u = x * (0.7978845608028654f + 0.7978845608028654f * 0.044715f * x * x);
    float t;
    asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(u));
    const float h = 0.5f * x;
    return h + h * t;
  }
  return x;
}
__device__ __forceinline__ void pair_activate(float (&y)[32], int act) {      // `act` is the same for the whole grid
  auto all = [&](auto f) {
#pragma unroll
    for (int j = 0; j < 32; ++j) y[j] = f(y[j]);
  };
  if (act == EPI_RELU) all(pair_activate<EPI_RELU>);
  else if (act == EPI_RELU6) all(pair_activate<EPI_RELU6>);
  else if (act == EPI_GELU) all(pair_activate<EPI_GELU>);
}

__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPThreads, 1)
gemm_pair_kernel(const __grid_constant__ CUtensorMap tmap_a, const __grid_constant__ CUtensorMap tmap_b,
                 const __grid_constant__ CUtensorMap tmap_c, const GemmPairParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sRing = smem;
  uint8_t* sPiece = smem + kPStages * kPStageBytes;
  float* sBias = reinterpret_cast<float*>(sPiece + kPEpiWarps * kPPieceBytes);      // [256 columns of the tile]
  uint64_t* bars = reinterpret_cast<uint64_t*>(sBias + 256);
  uint64_t* bar_full = bars;                   // [kPStages]
  uint64_t* bar_empty = bars + kPStages;       // [kPStages]
  uint64_t* bar_accf = bars + 2 * kPStages;    // [2]
  uint64_t* bar_acce = bar_accf + 2;           // [2]
  uint64_t* bar_drain = bar_acce + 2;          // [2] peer only: its epilogue warps have read accumulator a
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar_drain + 2);
  volatile uint32_t* abort_flag = reinterpret_cast<volatile uint32_t*>(bar_drain + 3);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = cluster_ctarank();             // 0: leader
  const int pair = (int)blockIdx.x >> 1;
  const int tiles = p.tiles_m * p.tiles_n;
  const int half_n = p.BN >> 1;                        // B columns held by each CTA

  if (tid == kPEpiThreads) {
    *abort_flag = 0u;
    for (int i = 0; i < kPStages; ++i) { mbar_init(bar_full + i, 1); mbar_init(bar_empty + i, 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(bar_accf + i, 1); mbar_init(bar_acce + i, kPEpiWarps + 1); mbar_init(bar_drain + i, kPEpiWarps); }
    fence_mbar_init();
    fence_proxy_async_smem();
  }
  if (warp == kPEpiWarps) {      // the MMA warp of either CTA allocates (a pair-wide allocation is issued by both CTAs)
    tmem_alloc_pair(tmem_slot, 512);
    tmem_relinquish_pair();
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  cluster_meet();                    // the peer's barriers exist before anything signals them
  tcgen05_fence_after_sync();
  // The set-up above overlaps the previous grid's tail. The next grid may be scheduled from here on: it can only take SMs
  // that this grid does not need (one CTA per SM).
  grid_dependency_wait();
  grid_launch_dependents();
  const uint32_t tmem_base = *tmem_slot;

  if (warp > kPEpiWarps) {
    // ================================ TMA producers (both CTAs): stages i, i + kPProducers, ... each ================================
    const uint32_t elected = elect_one();
    if (elected) { tma_prefetch_desc(&tmap_a); tma_prefetch_desc(&tmap_b); }
    __syncwarp();
    const uint32_t stage_tx = (uint32_t)(kPM * kPK * 2) + (uint32_t)half_n * kPK * 2u;
    const uint32_t announces = rank == 0 ? elected : 0u;
    const uint32_t ring = smem_u32(sRing), full0 = cluster_map(smem_u32(bar_full), 0u);   // the leader's barriers
    int s = warp - kPEpiWarps - 1, round = 0, kb = s;
    for (int t = pair; t < tiles; t += p.pairs) {
      const int tm = t % p.tiles_m, tn = t / p.tiles_m;
      const int row0 = tm * 2 * kPM + (int)rank * kPM;
      const int n0 = tn * p.BN + (int)rank * half_n;
      for (; kb < p.kblocks; kb += kPProducers) {
        if (round > 0) mbar_wait_poll(bar_empty + s, (uint32_t)(round - 1) & 1u, abort_flag, p.status, 0x601);
        const uint32_t st = ring + (uint32_t)(s * kPStageBytes), full = full0 + (uint32_t)(s * 8);
        // The leader announces both CTAs' bytes with a plain local arrival. (An arrival from the peer would have to be
        // a release at cluster scope, which costs about a thousand cycles per stage: measured 98 -> 55 us on a
        // 12288 x 768 x 3072 product.) The peer's bytes may land before the announcement -- the transaction count
        // goes negative meanwhile -- but never in an earlier phase: the peer refills a stage only after the commit
        // that follows the products of its previous content.
        mbar_arrive_expect_tx_elected(smem_u32(bar_full + s), 2u * stage_tx, announces);
        tma_load_2d_pair_elected(st, &tmap_a, full, kb * kPK, row0, elected);                       // A [128 rows x 64 k]
        if (p.b_kmajor) {
          tma_load_2d_pair_elected(st + 16384, &tmap_b, full, kb * kPK, n0, elected);               // B [half_n n x 64 k]
        } else if (p.b_blocks) {
          tma_load_3d_pair_elected(st + 16384, &tmap_b, full, 0, kb * kPK, n0 >> 6, elected);       // B [64 k x 64 n] blocks, at once
        } else {
          for (int nb = 0; nb < half_n; nb += 64)                                                   // ... or each by itself
            tma_load_2d_pair_elected(st + 16384u + (uint32_t)(nb >> 6) * 8192u, &tmap_b, full, n0 + nb, kb * kPK, elected);
        }
        if ((s += kPProducers) >= kPStages) { s -= kPStages; ++round; }
      }
      kb -= p.kblocks;
    }
    __syncwarp();
  } else if (warp == kPEpiWarps) {
    // ================================ MMA issuer (leader CTA only) ================================
    if (lane == 0 && rank != 0) {
      // The peer's MMA warp has no products to issue: it relays "accumulator drained" to the leader. (An arrival on
      // another CTA's barrier is a release at cluster scope, about a thousand cycles: kept off the epilogue warps.)
      const uint32_t acce_leader = cluster_map(smem_u32(bar_acce), 0u);
      int it = 0;
      for (int t = pair; t + 2 * p.pairs < tiles; t += p.pairs, ++it) {      // the last two accumulators are not used again
        const int a = it & 1;
        mbar_wait(bar_drain + a, (uint32_t)(it >> 1) & 1u, abort_flag, p.status, 0x605);
        mbar_remote_arrive(acce_leader + (uint32_t)(a * 8));
      }
    }
    if (rank == 0) {
      // the whole warp runs the loop converged; MMAs and commits are predicated on one elected lane (tc_common.cuh)
      const uint32_t elected = elect_one();
      const uint32_t idesc = make_idesc_bf16(256, (uint32_t)p.BN, 0, p.b_kmajor ? 0 : 1);
      int s = 0, round = 0, it = 0;
      for (int t = pair; t < tiles; t += p.pairs, ++it) {
        const int a = it & 1;
        if (it >= 2) {      // both CTAs have read accumulator a (tile it - 2) out of tensor memory
          mbar_wait_poll(bar_acce + a, (uint32_t)((it >> 1) - 1) & 1u, abort_flag, p.status, 0x602);
          tcgen05_fence_after_sync();
        }
        const uint32_t d_tmem = tmem_base + (uint32_t)(a * 256);
        for (int kb = 0; kb < p.kblocks; ++kb) {
          mbar_wait_poll(bar_full + s, (uint32_t)round & 1u, abort_flag, p.status, 0x603);
          tcgen05_fence_after_sync();
          const uint32_t st = smem_u32(sRing + s * kPStageBytes);
          const uint64_t ad = make_smem_desc(st, 0, 1024, SW_128B);
          const uint64_t bd = p.b_kmajor ? make_smem_desc(st + 16384, 0, 1024, SW_128B) : make_smem_desc(st + 16384, 8192, 1024, SW_128B);
#pragma unroll
          for (int ks = 0; ks < kPK / 16; ++ks)
            umma_bf16_pair_elected(d_tmem, ad + 2u * ks, bd + (p.b_kmajor ? (uint64_t)(2u * ks) : (uint64_t)((ks * 2048) >> 4)), idesc, elected, (kb | ks) != 0);
          const uint32_t e = smem_u32(bar_empty + s);
          umma_commit_pair_elected(cluster_map(e, 0u), elected);
          umma_commit_pair_elected(cluster_map(e, 1u), elected);
          if (++s == kPStages) { s = 0; ++round; }
        }
        if (!skip_signal_for_test(p.status, 0x604)) {
          const uint32_t f = smem_u32(bar_accf + a);
          umma_commit_pair_elected(cluster_map(f, 0u), elected);
          umma_commit_pair_elected(cluster_map(f, 1u), elected);
        }
      }
    }
    __syncwarp();
  } else {
    // ================ epilogue warps (both CTAs): thread = (row, column quarter) ================
    const int q = warp & 3, h = warp >> 2;
    const uint32_t lane_base = (uint32_t)(q * 32) << 16;
    const uint32_t piece = smem_u32(sPiece + warp * kPPieceBytes);
    const uint32_t bias_s = smem_u32(sBias);
    int it = 0;
    for (int t = pair; t < tiles; t += p.pairs, ++it) {
      const int a = it & 1;
      const int tm = t % p.tiles_m, tn = t / p.tiles_m;
      const int row0 = tm * 2 * kPM + (int)rank * kPM + q * 32;       // first row of the warp
      const int col_t = tn * p.BN;                  // first column of the tile
      if (p.bias) {      // the tile's bias on its way to shared memory while the products run; every column group has its own 64 floats
        const int c0 = h * 32 + (q & 1) * 128 + lane;
        const float b = q < 2 && col_t + c0 < p.N ? __ldg(p.bias + col_t + c0) : 0.0f;
        named_barrier_sync(1 + h, 128);             // the group is through with the previous tile's
        if (q < 2) sBias[c0] = b;
        named_barrier_sync(1 + h, 128);
      }
      mbar_wait(bar_accf + a, (uint32_t)(it >> 1) & 1u, abort_flag, p.status, 0x604);
      tcgen05_fence_after_sync();
      const uint32_t t_acc = tmem_base + lane_base + (uint32_t)(a * 256);
      // the four warps of a lane quarter take alternate blocks of 32 columns, so a narrow last tile still splits between them
#pragma unroll 1
      for (int c0 = h * 32; c0 < p.BN; c0 += 32 * (kPEpiWarps / 4)) {
        const int col = col_t + c0;
        if (col >= p.N) break;                      // uniform over the warp
        uint32_t v[32];
        tmem_ld_x32(t_acc + (uint32_t)c0, v);
        tmem_ld_wait();
        float y[32];
#pragma unroll
        for (int j = 0; j < 32; ++j) y[j] = __uint_as_float(v[j]);
        if (p.bias) {
#pragma unroll
          for (int j = 0; j < 32; j += 4) {
            const float4 b = lds128f(bias_s + (uint32_t)((c0 + j) * 4));
            y[j] += b.x; y[j + 1] += b.y; y[j + 2] += b.z; y[j + 3] += b.w;
          }
        }
        pair_activate(y, p.act1);
        if (p.scale != 1.0f) {
#pragma unroll
          for (int j = 0; j < 32; ++j) y[j] *= p.scale;
        }
        if (p.add && row0 + lane < p.M) {   // + tensor: this thread's row, 16-byte pieces (N is a multiple of 8)
          const __nv_bfloat16* arow = reinterpret_cast<const __nv_bfloat16*>(p.add) + (int64_t)(row0 + lane) * p.ldc + col;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            if (col + 8 * k < p.N) {
              const uint4 w = __ldg(reinterpret_cast<const uint4*>(arow + 8 * k));
              y[8 * k] += bf16_lo(w.x); y[8 * k + 1] += bf16_hi(w.x); y[8 * k + 2] += bf16_lo(w.y); y[8 * k + 3] += bf16_hi(w.y);
              y[8 * k + 4] += bf16_lo(w.z); y[8 * k + 5] += bf16_hi(w.z); y[8 * k + 6] += bf16_lo(w.w); y[8 * k + 7] += bf16_hi(w.w);
            }
          }
        }
        if (p.act2 >= 0) pair_activate(y, p.act2);
        // 64-byte rows of a piece of 32 rows, 64-byte swizzle, one TMA store per piece (clipped at the edges)
        auto store_piece = [&](const uint32_t (&w)[16], int col16) {
          if (lane == 0) bulk_wait_group_read_all();   // the warp's previous store has read the piece
          __syncwarp();
#pragma unroll
          for (int k = 0; k < 4; ++k) sts128(piece + swz_offset((uint32_t)lane, (uint32_t)k, 64), w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
          fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0 && row0 < p.M) { tma_store_2d(&tmap_c, sPiece + warp * kPPieceBytes, col16, row0); bulk_commit_group(); }
        };
        uint32_t w[16];
        if (p.c_fp32) {              // mapped as pairs of 16-bit elements
#pragma unroll
          for (int k = 0; k < 2; ++k) {
#pragma unroll
            for (int j = 0; j < 16; ++j) w[j] = __float_as_uint(y[16 * k + j]);
            store_piece(w, (col + 16 * k) * 2);
          }
        } else {
#pragma unroll
          for (int j = 0; j < 16; ++j) w[j] = pack_bf16x2(y[2 * j], y[2 * j + 1]);
          store_piece(w, col);
        }
      }
      // this warp's share of accumulator a is in registers: hand it back to the MMA warp
      tcgen05_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(rank == 0 ? bar_acce + a : bar_drain + a);   // the leader's MMA warp waits on bar_acce; the peer's goes through its relay
    }
    if (lane == 0) bulk_wait_group_all();           // the stores have left shared memory and are complete
  }
  tcgen05_fence_before_sync();
  __syncthreads();
  cluster_meet();              // neither CTA leaves (or frees tensor memory) while the other may still signal it or multiply into it
  if (warp == kPEpiWarps) tmem_dealloc_pair(tmem_base, 512);
}

struct PairMapKey {
  const void* p; int d0, d1, b0, b1, blocks; int64_t ld;
  bool operator==(const PairMapKey& o) const { return p == o.p && d0 == o.d0 && d1 == o.d1 && b0 == o.b0 && b1 == o.b1 && blocks == o.blocks && ld == o.ld; }
};
struct PairMapKeyHash {
  size_t operator()(const PairMapKey& k) const {
    return std::hash<const void*>()(k.p) ^ ((size_t)k.d0 * 1000003u) ^ ((size_t)k.d1 * 10007u) ^ ((size_t)k.b0 << 7) ^ (size_t)k.b1 ^ ((size_t)k.blocks << 40) ^ ((size_t)k.ld << 20);
  }
};
std::mutex g_pair_mutex;
std::unordered_map<PairMapKey, CUtensorMap, PairMapKeyHash> g_pair_maps;
int g_pair_resident[64] = {};   // pairs the device keeps resident at once (0: not asked yet)

// 16-bit elements [d1 rows][d0 columns], leading dimension ld (elements); box [b1][b0], swizzled over a row of the box (64 or 128 bytes). blocks > 0: the
// columns as blocks of b0 (d0 a multiple of it), a box holds that many of them one after the other.
bool pair_map(const void* base, int d0, int d1, int64_t ld, int b0, int b1, CUtensorMap* out, int blocks = 0) {
  std::lock_guard<std::mutex> lock(g_pair_mutex);
  const PairMapKey key{base, d0, d1, b0, b1, blocks, ld};
  auto it = g_pair_maps.find(key);
  if (it == g_pair_maps.end()) {
    CUtensorMap m;
    const uint64_t dims[3] = {(uint64_t)(blocks ? b0 : d0), (uint64_t)d1, (uint64_t)(d0 / b0)};
    const uint64_t strides[2] = {(uint64_t)ld * 2, (uint64_t)b0 * 2};
    const uint32_t box[3] = {(uint32_t)b0, (uint32_t)b1, (uint32_t)blocks};
    std::string err;
    if (!encode_tmap_bf16(&m, base, blocks ? 3 : 2, dims, strides, box, b0 * 2, &err)) return false;
    if (g_pair_maps.size() > 4096) g_pair_maps.clear();
    it = g_pair_maps.emplace(key, m).first;
  }
  *out = it->second;
  return true;
}

// (+ bias) (activation) (* scale) (+ tensor) (activation): the simple operators this kernel applies, in this order
bool pair_epilogue(const EpiProgram& e, GemmPairParams* p) {
  p->bias = nullptr; p->add = nullptr; p->act1 = -1; p->act2 = -1; p->scale = 1.0f;
  int stage = 0;
  for (int i = 0; i < e.n; ++i) {
    const int c = e.code[i];
    const bool act = c == EPI_RELU || c == EPI_RELU6 || c == EPI_GELU;
    if (c == EPI_BIAS && stage < 1) { p->bias = static_cast<const float*>(e.ptr[i]); stage = 1; }
    else if (act && stage < 2) { p->act1 = c; stage = 2; }
    else if (c == EPI_SCALE && stage < 3) { p->scale = e.f[i]; stage = 3; }
    else if (c == EPI_ADD && stage < 4) { p->add = e.ptr[i]; stage = 4; }
    else if (act && stage == 4) { p->act2 = c; stage = 5; }
    else return false;
  }
  return true;
}

}  // namespace

static long pair_tiles(const GemmArgs& a, int bn) { return (long)((a.M + 255) / 256) * ((a.N + bn - 1) / bn); }
// Columns per tile: 256 (128 flop per byte that enters the SM), or 128 where tiles of 256 would leave half of the pairs idle or
// fill a last round by less than a third (rounds x bytes per K block: 64 against 48 KB).
static int pair_columns(const GemmArgs& a) {
  if (a.N <= 128) return 128;
  const long pairs = device_sm_count() / 2;
  const long wide = (pair_tiles(a, 256) + pairs - 1) / pairs * 64, narrow = (pair_tiles(a, 128) + pairs - 1) / pairs * 48;
  return narrow < wide ? 128 : 256;
}

// Unbatched products with enough rows to fill the SM pairs (wide or narrow, long or short reductions: the narrow,
// short ones -- 1x1 convolutions of a few tens of channels -- are bound by the output stream, which the persistent
// pairs overlap with the next tile's loads and products); everything else stays on the small-tile kernel.
bool gemm_pair_supported(const GemmArgs& a) {
  GemmPairParams probe{};
  if (!pair_epilogue(a.epi, &probe)) return false;
  if (a.a_dtype != AGO_BF16 || a.batches > 1) return false;
  if (a.a_im2col && !(a.R == 1 && a.S == 1 && a.stride == 1 && a.pad == 0)) return false;
  if (a.K % 8 != 0 || a.N % 8 != 0 || a.ldb % 8 != 0 || a.ldc % 8 != 0) return false;
  if (!a.a_im2col && a.lda % 8 != 0) return false;
  if (probe.add && a.c_dtype != AGO_BF16) return false;   // the added tensor has the I/O dtype of a bf16 subgraph
  if (a.M < 512) return false;
  // worth it once the 256-row tiles (of 256 or 128 columns) fill most of the SM pairs
  return pair_tiles(a, pair_columns(a)) * 2 >= device_sm_count() / 2;
}

// The chain as two GEMM launches. Pairs of CTAs: per launch 3.2 us + rounds x the larger of the K blocks (0.33 / 0.2 us each for tiles
// of 256 / 128 columns) and a tile's epilogue (2.2 us for 256 columns with an activation, 1.3 without) + one more epilogue; single CTAs:
// 5.65 us + rounds x K blocks x 0.33 / 0.254 us (128 / 64 columns). 3.3 % rms, 11 % at most over 85 chains of 16 to 12288 rows.
double ffn_unfused_estimate(const Plan& plan) {
  GemmArgs a{};
  a.a_dtype = a.c_dtype = AGO_BF16;
  a.batches = 1;
  double us = 0.0;
  int K = (int)plan.inputs[0].last();
  a.M = (int)(plan.inputs[0].numel() / K);
  for (int i : {0, 3}) {
    a.K = K; a.N = plan.ops[i].op.p[0];
    a.lda = K; a.ldb = a.ldc = a.N;
    const int kblocks = (K + 63) / 64;
    if (gemm_pair_supported(a)) {
      const int bn = pair_columns(a);
      const long pairs = device_sm_count() / 2, rounds = (pair_tiles(a, bn) + pairs - 1) / pairs;
      const double epi = (i == 0 ? 2.2 : 1.3) * bn / 256;
      us += 3.2 + rounds * std::max(kblocks * (bn == 256 ? 0.33 : 0.2), epi) + epi;
    } else {
      const int bn = gemm_tc_columns(a);
      const long ctas = (long)((a.M + 127) / 128) * ((a.N + bn - 1) / bn), sms = device_sm_count();
      us += 5.65 + (ctas + sms - 1) / sms * kblocks * (bn == 128 ? 0.33 : 0.254);
    }
    K = a.N;
  }
  return us;
}

// Pointwise convolutions: set-up + rounds x (K blocks, or the stores of a tile where those take longer; one after the other on the
// kernel without an overlap) + the tensors' way through memory. Depthwise: set-up + tensors. 60 blocks of 16 to 160 input
// channels, 1 to 61 images of 7 to 63 pixels: 6 % rms, 13 % at most.
double conv_unfused_estimate(const Plan& plan) {
  double us = 0.0;
  for (const OpInfo& o : plan.ops) {
    if (!o.complex_op()) continue;
    const double mb = (o.in.numel() + o.out.numel()) * 2e-6;
    if (o.depthwise()) { us += 2.35 + 0.185 * mb; continue; }
    GemmArgs a{};
    a.a_dtype = a.c_dtype = AGO_BF16;
    a.batches = 1;
    a.K = (int)o.in.last(); a.N = (int)o.out.last(); a.M = (int)(o.in.numel() / a.K);
    a.lda = a.ldb = a.K; a.ldc = a.N;
    const int kblocks = (a.K + 63) / 64;
    if (gemm_pair_supported(a)) {
      const int bn = pair_columns(a);
      const long pairs = device_sm_count() / 2, rounds = (pair_tiles(a, bn) + pairs - 1) / pairs;
      us += 4.6 + rounds * std::max(kblocks * (bn == 256 ? 0.32 : 0.2), bn / 256.0 * 2.0) + 0.13 * mb;
    } else {
      const int bn = gemm_tc_columns(a);
      const long ctas = (long)((a.M + 127) / 128) * ((a.N + bn - 1) / bn), sms = device_sm_count(), rounds = (ctas + sms - 1) / sms;
      us += 4.05 + rounds * (kblocks * (bn == 128 ? 0.29 : 0.22) + bn / 128.0 * 0.81) + 0.46 * mb;
    }
  }
  return us;
}

cudaError_t launch_gemm_pair(const GemmArgs& a, cudaStream_t stream) {
  GemmPairParams p{};
  pair_epilogue(a.epi, &p);
  p.M = a.M; p.N = a.N; p.K = a.K;
  p.BN = pair_columns(a);
  p.b_kmajor = a.b_kmajor;
  p.c_fp32 = a.c_dtype == AGO_FP32 ? 1 : 0;
  p.kblocks = (a.K + kPK - 1) / kPK;
  p.tiles_m = (a.M + 2 * kPM - 1) / (2 * kPM);
  p.tiles_n = (a.N + p.BN - 1) / p.BN;
  p.status = a.status;
  p.ldc = a.ldc;
  const int64_t lda = a.a_im2col ? a.K : a.lda;
  CUtensorMap ma, mb, mc;
  if (!pair_map(a.A, a.K, a.M, lda, kPK, kPM, &ma)) return cudaErrorInvalidValue;
  p.b_blocks = !a.b_kmajor && a.N % 64 == 0 ? 1 : 0;
  if (a.b_kmajor ? !pair_map(a.B, a.K, a.N, a.ldb, kPK, p.BN / 2, &mb)
                 : !pair_map(a.B, a.N, a.K, a.ldb, 64, kPK, &mb, p.b_blocks ? p.BN / 128 : 0)) return cudaErrorInvalidValue;
  // the output as 16-bit elements: an fp32 tensor has twice the columns; pieces of 64 bytes x 32 rows
  const int cmul = p.c_fp32 ? 2 : 1;
  if (!pair_map(a.C, a.N * cmul, a.M, a.ldc * cmul, 32, 32, &mc)) return cudaErrorInvalidValue;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  {
    static int smem_opt_in[64] = {};
    e = ensure_max_dynamic_smem(reinterpret_cast<const void*>(gemm_pair_kernel), smem_opt_in);
    if (e != cudaSuccess) return e;
  }
  int resident;
  {
    std::lock_guard<std::mutex> lock(g_pair_mutex);
    if (g_pair_resident[dev] == 0) {
      cudaLaunchConfig_t cfg = cudaLaunchConfig_t{};
      cudaLaunchAttribute attr[1];
      cfg.gridDim = dim3(2 * 512, 1, 1); cfg.blockDim = dim3(kPThreads, 1, 1); cfg.dynamicSmemBytes = kPSmemBytes;
      attr[0].id = cudaLaunchAttributeClusterDimension;
      attr[0].val.clusterDim.x = 2; attr[0].val.clusterDim.y = 1; attr[0].val.clusterDim.z = 1;
      cfg.attrs = attr; cfg.numAttrs = 1;
      int n = 0;
      e = cudaOccupancyMaxActiveClusters(&n, gemm_pair_kernel, &cfg);
      if (e != cudaSuccess) return e;
      if (n < 1) return cudaErrorInvalidConfiguration;
      g_pair_resident[dev] = n;
    }
    resident = g_pair_resident[dev];
  }
  p.pairs = std::min(resident, p.tiles_m * p.tiles_n);
  FusedLaunch launch(dim3((unsigned)(2 * p.pairs)), kPThreads, kPSmemBytes, stream);     // the cluster of two is the kernel's own attribute
  return cudaLaunchKernelEx(&launch.config, gemm_pair_kernel, ma, mb, mc, p);
}

}  // namespace ago
