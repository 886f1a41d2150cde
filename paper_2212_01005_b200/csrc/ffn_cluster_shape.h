// Tile choice, split and shared-memory layout of the clustered feed-forward kernel (fused_ffn_cluster.cu): host arithmetic only,
// without CUDA, so that its conditions can be checked over whole ranges of shapes on a machine without a device.
#pragma once
#include <algorithm>

namespace ago {
namespace ffn_cluster {

constexpr int kBM = 128;        // rows per cluster
constexpr int kBK = 64;         // reduction elements per ring stage
constexpr int kMaxCS = 4;       // CTAs per cluster
constexpr int kMaxStages = 16;
constexpr int kSmemMax = 227 * 1024 - 1024 - 512;   // ring + slots (alignment slack and barriers apart)
constexpr int kResident[kMaxCS + 1] = {0, 0, 74, 45, 33};   // clusters of 1-CTA-per-SM kernels a B200 keeps resident at once

struct FfnClusterShape {
  int M, K, Hid, N2;
  int CS, NC;              // CTAs per cluster, output columns per CTA (N2 / CS, a multiple of 64, <= 256)
  int T;                   // steps per row block = Hid / BH / CS
  int BH;                  // hidden units per tile: 128, or 64 where 128 would leave SMs without a tile
  int RP;                  // rows kept in shared memory: min(128, M rounded up to 16). The MMAs span 128 rows all the same: rows
                           // past RP are read from whatever follows in shared memory and land in accumulator rows nobody reads
  int stage_bytes, slot_bytes, slots_off, bars_off;
  int J, Tp;               // a row block is split over J clusters, each with Tp = T / J of its steps (J = 1: no split)
  int kblocks;             // K / 64
  int stages;              // ring stages
  int wait_copies;         // the staging of the sums waits for the copies out of this CTA (staging_leaves_ring)
  int w2_off;              // > 0: one step per cluster and everything fits: the step's W2 tiles have stages of their own there
};

// Two warps fill the ring in turn. With two stages or more, the load two before a stage's next one has seen the use before its last one
// over, so that the wait's one bit of parity suffices whichever warp filled it. A single stage holds this many loads: the second
// waits for the first, a third could pass before the second.
constexpr int kLoadsOfOneStage = 2;

// A part's partial sums (64 rows or more) are staged as blocks of 64 columns in two buffers from the start of the ring on. The ring
// itself is free by then. Where the buffers are larger they run into the hidden tiles' slots, which the other CTAs of the cluster may
// still be copying this CTA's tile out of: the kernel then waits until they have used it.
constexpr int kStagedRows = 64;
inline int staging_bytes(const FfnClusterShape& q) {
  return q.J > 1 && q.RP >= kStagedRows ? std::min(2, q.NC / 64) * q.RP * 256 : 0;
}
inline bool staging_leaves_ring(const FfnClusterShape& q) { return staging_bytes(q) > q.stages * q.stage_bytes; }

// Ring, slots and barriers: as many stages as fit. Behind ring and slots lies at least one 128-row operand (the MMAs read 128
// rows from the start of the last tile whatever RP is).
inline int layout(FfnClusterShape* q) {
  q->slot_bytes = q->RP * q->BH * 2;
  const int slots = q->CS * q->slot_bytes, g1 = q->RP * 128 + q->BH * 128, w2 = q->CS * (q->BH / 64) * q->NC * 128;
  q->w2_off = 0;
  // One step per cluster: where the step's W2 tiles fit beside half of the first GEMM's stages, they get memory of their own and
  // are requested at once instead of behind the ring. Not for whole row blocks in tiles of 128: that kernel has stages of 32 KB at
  // compile time and takes every operand through the ring.
  if (!(q->RP == kBM && q->BH == 128) && q->J > 1 && q->Tp == 1 && w2 >= kBM * 128 && (kSmemMax - slots - w2) / g1 >= (q->kblocks + 1) / 2) {
    q->stage_bytes = g1;
    q->stages = std::min(std::min(kMaxStages, q->kblocks), (kSmemMax - slots - w2) / g1);
    q->slots_off = q->stages * g1;
    q->w2_off = q->slots_off + slots;            // behind the slots: what the MMAs read past the rows lies in it
    q->bars_off = q->w2_off + w2;
    q->wait_copies = staging_leaves_ring(*q);
    return q->bars_off + 512 + 1024;
  }
  const int slack = kBM * 128 - q->RP * 128;
  q->stage_bytes = (std::max(g1, q->NC * 128) + 1023) & ~1023;      // 32 KB for whole row blocks and tiles of 128 (NC <= 256)
  q->stages = std::min(kMaxStages, (kSmemMax - slots - slack) / q->stage_bytes);
  q->slots_off = q->stages * q->stage_bytes;
  q->bars_off = q->slots_off + slots + slack;
  q->wait_copies = staging_leaves_ring(*q);
  return q->bars_off + 512 + 1024;
}

// Cluster size, hidden tile and split of the row blocks' hidden tiles over clusters.
inline bool choose_split(FfnClusterShape* q, int row_blocks, const int* resident) {
  // Whole row blocks: among the cluster sizes whose column share fits tensor memory, the least estimated time = rounds of
  // resident clusters x steps per row block x ring stages per step.
  q->CS = 0; q->BH = 128; q->J = 1;
  long best = 0;
  const int htiles = q->Hid / 128;
  for (int cs = 2; cs <= kMaxCS; ++cs) {
    if (q->N2 % cs != 0 || htiles % cs != 0) continue;
    const int nc = q->N2 / cs;
    if (nc % 64 != 0 || nc > 256) continue;
    const long rounds = (row_blocks + resident[cs] - 1) / resident[cs];
    const long cost = rounds * (htiles / cs) * (q->K / kBK + 2 * cs);
    if (q->CS == 0 || cost < best) { q->CS = cs; q->NC = nc; best = cost; }
  }
  if (q->CS == 0) return false;
  q->T = htiles / q->CS;
  if ((long)row_blocks * q->CS < 120) {
    // Few row blocks: one cluster per block of 128 rows leaves most SMs idle, and the hidden dimension is what can fill
    // them. A row block is split over J clusters (J divides its T steps); their outputs meet in an fp32 buffer in device
    // memory, J additions per element instead of one per hidden tile. J = as many parts as still fit one round of
    // resident clusters, each with at least one step. Tiles of 64 hidden units where they put more clusters to work (256 rows of
    // 768 -> 3072: 24 instead of 12, 17.4 -> 13.2 us); otherwise they only stream X twice (512 rows: 18.6 -> 21 us).
    for (int bh = 128; bh >= 64; bh -= 64) {
      const int T = q->Hid / bh / q->CS;
      for (int j = T; j > q->J; --j)
        if (T % j == 0 && (long)row_blocks * j <= resident[q->CS]) { q->BH = bh; q->T = T; q->J = j; break; }
    }
  }
  q->Tp = q->T / q->J;
  return true;
}

// Clusters to launch. Whole row blocks: as many as the device keeps resident, each walks over its share of the blocks. Parts of
// split row blocks: one cluster each, whatever is resident -- the kernel requests a part's W2 tiles once and stages its sums over
// the ring, so a second part has no place in the same cluster; parts do not wait for each other, and J was chosen for one round.
inline int launched_clusters(int row_blocks, int J, int resident) { return J > 1 ? row_blocks * J : std::min(row_blocks, resident); }

}  // namespace ffn_cluster
}  // namespace ago
