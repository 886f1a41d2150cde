// Dispatch of the fused kernel families.
#include "fused.h"

#include <mutex>

namespace ago {

cudaError_t ensure_max_dynamic_smem(const void* func, int* done_flags) {
  static std::mutex guard;   // the per-kernel flag arrays are shared by every handle and thread
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  std::lock_guard<std::mutex> lock(guard);
  if (done_flags[dev]) return cudaSuccess;
  e = cudaFuncSetAttribute(func, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  if (e == cudaSuccess) done_flags[dev] = 1;
  return e;
}

int device_sm_count() {
  static std::mutex guard;
  static int cached[64] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) {
    cudaGetLastError();   // planning on a host without a device is legal: clear the sticky "no device" error
    return kDefaultSMs;
  }
  std::lock_guard<std::mutex> lock(guard);
  if (cached[dev] == 0) {
    int n = 0;
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n < 1) {
      cudaGetLastError();
      return kDefaultSMs;
    }
    cached[dev] = n;
  }
  return cached[dev];
}

ago_status_t fused_plan(Plan* plan, FusedState* st, std::string* err) {
  switch (plan->fused_kernel) {
    case AGO_KERNEL_DEPTHWISE:
      return AGO_OK;
    case AGO_KERNEL_MBV2_BLOCK:
    case AGO_KERNEL_PW_DW:
    case AGO_KERNEL_DW_PW:
      return mbv2_plan(plan, st, err);
    case AGO_KERNEL_DW_DW:
      return dwdw_plan(plan, st, err);
    case AGO_KERNEL_PW_PW:
    case AGO_KERNEL_GEMM_PERMUTE_GEMM:
      return pwpw_plan(plan, st, err);
    case AGO_KERNEL_ATTENTION:
      return attention_plan(plan, st, err);
    case AGO_KERNEL_FFN: {
      // The cluster of two CTA pairs (256 rows per weight tile) where its 256-row blocks fill most of the device; below that the
      // kernel of the least estimate: the pairs (768 -> 3072: 2500 rows 35 against 56 us), the cluster kernel, or the one that tiles
      // the reduction, which needs no row block to be shared out evenly (646 rows of 64 -> 3328 -> 384: 24 against 37 us). The pairs
      // have to win by more than the estimates' error (4157 rows of 128 -> 2048 -> 256: 27.4 against 28.5). Over 173 chains that both
      // serve, 1 to 12288 rows, the choice costs 0.4 % on average.
      const double pair = ffn_pair_estimate(*plan) * 1.04, cluster = ffn_cluster_estimate(*plan), reduction = ffn_estimate(*plan);
      const int64_t rows = plan->inputs[0].numel() / plan->inputs[0].last();
      const bool fills = pair >= 0 && (rows + 255) / 256 * 4 >= (int64_t)device_sm_count() * 3 / 4;
      auto best = [&](double t) { return t >= 0 && (pair < 0 || t <= pair) && (cluster < 0 || t <= cluster) && (reduction < 0 || t <= reduction); };
      if (fills || best(pair)) return ffn_pair_plan(plan, st, err);
      if (best(cluster)) return ffn_cluster_plan(plan, st, err);
      return ffn_plan(plan, st, err);
    }
    case AGO_KERNEL_CONV3X3_PAIR:
      return conv3x3_plan(plan, st, err);
    default:
      *err = "fused mode: no kernel is built for this family yet";
      return AGO_ERR_UNSUPPORTED;
  }
}

size_t fused_workspace_bytes(const Plan& plan) {
  if (plan.fused_kernel != AGO_KERNEL_FFN) return 0;
  if (plan.fused_variant == 3) return ffn_pair_workspace_bytes(plan);
  return plan.fused_variant == 0 ? ffn_workspace_bytes(plan) : ffn_cluster_workspace_bytes(plan);
}

ago_status_t fused_run(const Plan& plan, FusedState* st, const void* const* inputs, const void* const* weights,
                       void* output, void* workspace, unsigned int* status_word, cudaStream_t stream,
                       std::string* err) {
  switch (plan.fused_kernel) {
    case AGO_KERNEL_MBV2_BLOCK:
    case AGO_KERNEL_PW_DW:
    case AGO_KERNEL_DW_PW:
      return mbv2_run(plan, st, inputs, weights, output, status_word, stream, err);
    case AGO_KERNEL_DW_DW:
      return dwdw_run(plan, st, inputs, weights, output, status_word, stream, err);
    case AGO_KERNEL_PW_PW:
    case AGO_KERNEL_GEMM_PERMUTE_GEMM:
      return pwpw_run(plan, st, inputs, weights, output, status_word, stream, err);
    case AGO_KERNEL_ATTENTION:
      return attention_run(plan, st, inputs, weights, output, status_word, stream, err);
    case AGO_KERNEL_FFN:
      if (st->variant == 3) return ffn_pair_run(plan, st, inputs, weights, output, workspace, status_word, stream, err);
      if (st->variant == 1) return ffn_cluster_run(plan, st, inputs, weights, output, workspace, status_word, stream, err);
      return ffn_run(plan, st, inputs, weights, output, workspace, status_word, stream, err);
    case AGO_KERNEL_CONV3X3_PAIR:
      return conv3x3_run(plan, st, inputs, weights, output, status_word, stream, err);
    default:
      *err = "fused mode: no kernel is built for this family yet";
      return AGO_ERR_UNSUPPORTED;
  }
}

}  // namespace ago
