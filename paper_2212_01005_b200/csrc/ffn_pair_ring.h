// Ring stages of the paired feed-forward kernel (fused_ffn_pair.cu): what each CTA of a pair loads into them. Without CUDA, so that it
// can be checked on a machine without a device.
#pragma once

namespace ago {
namespace ffn_pair {

constexpr int kFM = 128;          // rows per CTA (256 per cluster)
constexpr int kFK = 64;           // reduction elements per ring stage
constexpr int kFStages = 6;
constexpr int kFStageBytes = 24 * 1024;
constexpr int kXBytes = kFM * kFK * 2, kW1Bytes = kFK * 64 * 2;      // a CTA's rows of X and its half of the tile's W1 columns

// K blocks come in pairs, one barrier per pair that only the leading CTA announces on. An odd number of them leaves the last stage
// without operands, but not without a load: the CTA that does not lead brings W1 rows past the end there (zeros that no product
// reads). Its producer takes part in a stage by its bytes alone; without any, nothing would keep the products from handing the
// stage back a second time before that producer has seen the first, and a wait tells only odd phases from even ones.
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int g1_stage_bytes(int kb, int kblocks, bool leader) { return kb < kblocks ? kXBytes + kW1Bytes : leader ? 0 : kW1Bytes; }
constexpr int g1_stages(int kblocks) { return (kblocks + 1) / 2 * 2; }

}  // namespace ffn_pair
}  // namespace ago
