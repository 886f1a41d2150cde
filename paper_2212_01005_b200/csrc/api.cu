// C-ABI entry points: handle lifetime, argument checks and the dispatch of one
// run onto the kernels chosen by the planner.
#include <cuda_runtime.h>

#include <cstdio>
#include <cstring>
#include <mutex>
#include <new>
#include <string>

#include "fused.h"
#include "kernels.h"
#include "plan.h"

using namespace ago;

struct ago_subgraph_s {
  Plan plan;
  void* workspace = nullptr;
  size_t workspace_bytes = 0;
  unsigned int* status_word = nullptr;  // device status block (code, wait budget, test hook, spare); allocated at the first run
  int status_device = -1;
  unsigned int wait_budget_us = 0;      // 0: the kernels' default
  unsigned int skip_signal_code = 0;    // test hook, 0: none
  FusedState fused;                     // per-kernel host state (tensor maps, launch geometry)
  std::mutex guard;                     // of everything above that a run changes: runs of one handle may come from several threads
};

namespace {

thread_local ago_status_t g_status = AGO_OK;
thread_local std::string g_msg;

ago_status_t fail(ago_status_t s, const std::string& m) {
  g_status = s;
  g_msg = m;
  return s;
}

ago_status_t cuda_fail(cudaError_t e, const char* what) {
  return fail(AGO_ERR_CUDA, std::string(what) + ": " + cudaGetErrorString(e));
}

constexpr size_t kStatusBlockBytes = 4 * sizeof(unsigned int);   // tc::kStatusWords

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

size_t align256(size_t b) { return (b + 255) & ~size_t(255); }

// Storage of tensors passed between launches: fp32 in PER_OP mode (every
// operator materialises its full-precision result, as the unfused loop nest of
// Section III-A does), the I/O dtype in PER_MINI_SUBGRAPH mode.
int intermediate_dtype(const Plan& p) { return p.mode == AGO_MODE_PER_OP ? AGO_FP32 : p.dtype; }

size_t unfused_workspace(const Plan& p) {
  if (p.stages.size() <= 1) return 0;
  const size_t elems = (size_t)(p.max_intermediate_bytes / elem_bytes(p.dtype));
  bool softmax = false;
  for (const Stage& s : p.stages) softmax = softmax || s.softmax;
  return 2 * align256(elems * (size_t)(softmax ? 4 : elem_bytes(intermediate_dtype(p))));
}

size_t needed_workspace(const Plan& p) {
  if (p.mode == AGO_MODE_FUSED) return fused_workspace_bytes(p);
  return unfused_workspace(p);
}

// Translate ops [first, last] (all element-wise) into an epilogue program.
void make_epilogue(const Plan& p, int first, int last, const void* const* inputs, const void* const* weights,
                   EpiProgram* e) {
  e->n = 0;
  for (int i = first; i <= last; ++i) {
    const OpInfo& o = p.ops[i];
    int k = e->n++;
    e->ptr[k] = nullptr;
    e->f[k] = 0.0f;
    switch (o.op.kind) {
      case AGO_OP_BIAS_ADD: e->code[k] = EPI_BIAS; e->ptr[k] = weights[o.weight]; break;
      case AGO_OP_RELU: e->code[k] = EPI_RELU; break;
      case AGO_OP_RELU6: e->code[k] = EPI_RELU6; break;
      case AGO_OP_GELU_TANH: e->code[k] = EPI_GELU; break;
      case AGO_OP_SCALE: e->code[k] = EPI_SCALE; e->f[k] = o.op.f; break;
      case AGO_OP_ADD_INPUT: e->code[k] = EPI_ADD; e->ptr[k] = inputs[o.op.p[0]]; break;
      default: --e->n; break;
    }
  }
}

cudaError_t launch_complex(const Plan& p, const OpInfo& o, const void* src, int src_dtype, void* dst, int dst_dtype,
                           const void* const* inputs, const void* const* weights, const EpiProgram& epi,
                           bool tuned_depthwise, unsigned int* status, cudaStream_t stream) {
  const int32_t* q = o.op.p;
  if (o.op.kind == AGO_OP_CONV2D && o.depthwise()) {
    DepthwiseArgs a{};
    a.in = src; a.w = weights[o.weight]; a.out = dst;
    a.N = (int)o.in.d[0]; a.H = (int)o.in.d[1]; a.W = (int)o.in.d[2]; a.C = (int)o.in.d[3];
    a.R = q[1]; a.S = q[2]; a.stride = q[3]; a.pad = q[4];
    a.Ho = (int)o.out.d[1]; a.Wo = (int)o.out.d[2];
    a.dtype = p.dtype; a.in_dtype = src_dtype; a.out_dtype = dst_dtype;
    a.epi = epi;
    // the vectorised kernel serves every stage whose input and output are stored in the I/O dtype
    const bool vec_ok = src_dtype == p.dtype && dst_dtype == p.dtype && a.C % (p.dtype == AGO_FP32 ? 4 : 8) == 0;
    return (tuned_depthwise || vec_ok) ? launch_depthwise_fused(a, stream) : launch_depthwise_generic(a, stream);
  }
  GemmArgs g{};
  g.A = src; g.C = dst; g.epi = epi;
  g.a_dtype = src_dtype; g.c_dtype = dst_dtype;
  g.batches = 1; g.heads = 1;
  g.status = status;
  switch (o.op.kind) {
    case AGO_OP_CONV2D: {
      // 3x3 convolutions of equal width with a (bias)(relu) or (bias)(add)(relu) epilogue: tensor-core stage kernel
      if (p.dtype == AGO_BF16 && src_dtype == AGO_BF16 && dst_dtype == AGO_BF16 &&
          conv3x3_tc_supported((int)o.in.d[1], (int)o.in.d[2], (int)o.in.d[3], q[0], q[1], q[2], q[3], q[4])) {
        const float* bias = nullptr; const void* res = nullptr; int relu = 0, k = 0;
        if (k < epi.n && epi.code[k] == EPI_BIAS) bias = static_cast<const float*>(epi.ptr[k++]);
        if (k < epi.n && epi.code[k] == EPI_ADD) res = epi.ptr[k++];
        if (k < epi.n && epi.code[k] == EPI_RELU) { relu = 1; ++k; }
        if (k == epi.n)
          return launch_conv3x3_tc(src, weights[o.weight], bias, res, dst, (int)o.in.d[0], (int)o.in.d[1], (int)o.in.d[2],
                                   (int)o.in.d[3], relu, status, stream);
      }
      g.B = weights[o.weight];
      g.H = (int)o.in.d[1]; g.W = (int)o.in.d[2]; g.Cin = (int)o.in.d[3];
      g.R = q[1]; g.S = q[2]; g.stride = q[3]; g.pad = q[4];
      g.Ho = (int)o.out.d[1]; g.Wo = (int)o.out.d[2];
      g.M = (int)(o.out.d[0] * o.out.d[1] * o.out.d[2]);
      g.N = q[0];
      g.K = g.R * g.S * g.Cin;
      g.a_im2col = 1; g.lda = 0;
      g.b_kmajor = 1; g.ldb = g.K;
      g.ldc = g.N;
      break;
    }
    case AGO_OP_GEMM: {
      g.B = weights[o.weight];
      g.K = (int)o.in.last(); g.N = q[0];
      g.M = (int)(o.in.numel() / g.K);
      g.a_im2col = 0; g.lda = g.K;
      g.b_kmajor = 0; g.ldb = g.N;
      g.ldc = g.N;
      break;
    }
    case AGO_OP_BATCHED_QKT: {
      const int64_t B = o.in.d[0], S = o.in.d[1], E = o.in.d[2];
      const int heads = q[1], hd = q[2];
      g.B = inputs[q[0]];
      g.M = (int)S; g.N = (int)S; g.K = hd;
      g.a_im2col = 0; g.lda = E;
      g.b_kmajor = 1; g.ldb = E;
      g.ldc = S;
      g.batches = (int)(B * heads); g.heads = heads;
      g.a_sb = S * E; g.a_sh = hd; g.b_sb = S * E; g.b_sh = hd;
      g.c_sb = (int64_t)heads * S * S; g.c_sh = S * S;
      break;
    }
    case AGO_OP_BATCHED_PV: {
      const int64_t B = o.in.d[0], S = o.in.d[2];
      const int heads = q[1], hd = q[2];
      const int64_t E = (int64_t)heads * hd;
      g.B = inputs[q[0]];
      g.M = (int)S; g.N = hd; g.K = (int)S;
      g.a_im2col = 0; g.lda = S;
      g.b_kmajor = 0; g.ldb = E;
      g.ldc = E;
      g.batches = (int)(B * heads); g.heads = heads;
      g.a_sb = (int64_t)heads * S * S; g.a_sh = S * S; g.b_sb = S * E; g.b_sh = hd;
      g.c_sb = S * E; g.c_sh = hd;
      break;
    }
    default:
      return cudaErrorInvalidValue;
  }
  if (p.dtype == AGO_BF16 && gemm_pair_supported(g)) return launch_gemm_pair(g, stream);
  if (p.dtype == AGO_BF16 && gemm_tc_supported(g)) return launch_gemm_tc(g, p.dtype, stream);
  return launch_gemm_generic(g, stream);
}

// One launch per stage; intermediates ping-pong between the two halves of `ws`.
ago_status_t run_unfused(ago_subgraph_s* h, const void* const* inputs, const void* const* weights, void* out,
                         void* ws, size_t ws_bytes, unsigned int* status, cudaStream_t stream) {
  const Plan& p = h->plan;
  const size_t need = unfused_workspace(p);
  const int mid = intermediate_dtype(p);
  if (need > 0 && (ws == nullptr || ws_bytes < need))
    return fail(AGO_ERR_WORKSPACE, "workspace missing or smaller than ago_subgraph_workspace_bytes()");
  char* buf[2] = {static_cast<char*>(ws), static_cast<char*>(ws) + need / 2};
  const void* src = inputs[0];
  int src_dtype = p.dtype;
  int flip = 0;
  for (size_t si = 0; si < p.stages.size(); ++si) {
    const Stage& s = p.stages[si];
    const bool last = si + 1 == p.stages.size();
    void* dst = last ? out : static_cast<void*>(buf[flip]);
    // The tensor a row softmax reads stays fp32 in every mode: scores rounded to
    // bf16 before the exponential alone exceed the parity tolerance.
    const bool feeds_softmax = !last && p.stages[si + 1].softmax;
    const int dst_dtype = last ? p.dtype : (feeds_softmax ? AGO_FP32 : mid);
    cudaError_t e;
    if (s.softmax) {
      const Shape& sh = p.ops[s.first].in;
      e = launch_softmax_rows(src, dst, sh.numel() / sh.last(), (int)sh.last(), src_dtype, dst_dtype, stream);
    } else if (s.transpose) {
      const OpInfo& o = p.ops[s.first];
      e = launch_transpose(src, dst, o.in.d, o.in.rank, o.op.p[0], o.op.p[1], src_dtype, dst_dtype, stream);
    } else if (s.complex_index >= 0) {
      EpiProgram epi;
      make_epilogue(p, s.first + 1, s.last, inputs, weights, &epi);
      e = launch_complex(p, p.ops[s.first], src, src_dtype, dst, dst_dtype, inputs, weights, epi, false, status, stream);
    } else {
      EpiProgram epi;
      make_epilogue(p, s.first, s.last, inputs, weights, &epi);
      const Shape& sh = p.ops[s.first].in;
      e = launch_elementwise(src, dst, sh.numel(), (int)sh.last(), p.dtype, src_dtype, dst_dtype, epi, stream);
    }
    if (e != cudaSuccess) return cuda_fail(e, "kernel launch");
    src = dst;
    src_dtype = dst_dtype;
    flip ^= 1;
  }
  return AGO_OK;
}

ago_status_t ensure_status_word(ago_subgraph_s* h) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return cuda_fail(e, "cudaGetDevice");
  if (h->status_word && h->status_device == dev) return AGO_OK;
  if (h->status_word) { cudaFree(h->status_word); h->status_word = nullptr; }
  e = cudaMalloc(&h->status_word, kStatusBlockBytes);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMalloc(status block)");
  const unsigned int init[4] = {0u, h->wait_budget_us, h->skip_signal_code, 0u};
  e = cudaMemcpy(h->status_word, init, sizeof(init), cudaMemcpyHostToDevice);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy(status block)");
  h->status_device = dev;
  return AGO_OK;
}

ago_status_t check_run_args(ago_subgraph_s* h, const void* const* inputs, const void* const* weights,
                            void* const* outputs) {
  if (!h) return fail(AGO_ERR_INVALID_ARG, "handle is NULL");
  if (!inputs || !outputs) return fail(AGO_ERR_INVALID_ARG, "inputs / outputs array is NULL");
  const Plan& p = h->plan;
  if (!p.weight_bytes.empty() && !weights) return fail(AGO_ERR_INVALID_ARG, "weights array is NULL");
  for (int i = 0; i < p.num_inputs; ++i) {
    if (!inputs[i]) return fail(AGO_ERR_INVALID_ARG, "inputs[" + std::to_string(i) + "] is NULL");
    if (!aligned16(inputs[i])) return fail(AGO_ERR_ALIGNMENT, "inputs[" + std::to_string(i) + "] is not 16-byte aligned");
  }
  for (size_t i = 0; i < p.weight_bytes.size(); ++i) {
    if (!weights[i]) return fail(AGO_ERR_INVALID_ARG, "weights[" + std::to_string(i) + "] is NULL");
    if (!aligned16(weights[i])) return fail(AGO_ERR_ALIGNMENT, "weights[" + std::to_string(i) + "] is not 16-byte aligned");
  }
  if (!outputs[0]) return fail(AGO_ERR_INVALID_ARG, "outputs[0] is NULL");
  if (!aligned16(outputs[0])) return fail(AGO_ERR_ALIGNMENT, "outputs[0] is not 16-byte aligned");
  return AGO_OK;
}

}  // namespace

namespace ago {
// Unfused run with an explicitly given workspace and no status word: used by
// the entry point whose scratch is a static device array.
ago_status_t run_unfused_in(ago_subgraph_s* h, const void* const* inputs, const void* const* weights,
                            void* const* outputs, void* ws, size_t ws_bytes, cudaStream_t stream) {
  ago_status_t s = check_run_args(h, inputs, weights, outputs);
  if (s != AGO_OK) return s;
  if (h->plan.mode == AGO_MODE_FUSED)
    return fail(AGO_ERR_UNSUPPORTED, "fused handles keep their intermediates on chip: use ago_subgraph_run");
  const size_t need = unfused_workspace(h->plan);
  if (need > ws_bytes) {
    char buf[160];
    std::snprintf(buf, sizeof(buf), "this subgraph needs %zu bytes of scratch, the built-in array holds %zu", need, ws_bytes);
    return fail(AGO_ERR_WORKSPACE, buf);
  }
  return run_unfused(h, inputs, weights, outputs[0], ws, ws_bytes, nullptr, stream);
}
ago_status_t report_failure(ago_status_t s, const char* msg) { return fail(s, msg); }
}  // namespace ago

namespace {
__global__ void empty_kernel() {
  asm volatile("griddepcontrol.wait;" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}
}  // namespace

extern "C" {

const char* ago_version(void) { return "0.1"; }

ago_status_t ago_launch_empty(int32_t grid, int32_t block, int32_t smem_bytes, void* cuda_stream) {
  if (grid < 1 || grid > 65535 || block < 1 || block > 1024 || smem_bytes < 0 || smem_bytes > 227 * 1024)
    return fail(AGO_ERR_INVALID_ARG, "ago_launch_empty: grid 1..65535, block 1..1024, shared memory 0..227 KB");
  static int smem_opt_in[64] = {};
  cudaError_t e = ago::ensure_max_dynamic_smem(reinterpret_cast<const void*>(empty_kernel), smem_opt_in);
  if (e != cudaSuccess) return cuda_fail(e, "cudaFuncSetAttribute");
  ago::FusedLaunch launch(dim3((unsigned)grid), block, (size_t)smem_bytes, static_cast<cudaStream_t>(cuda_stream));
  e = cudaLaunchKernelEx(&launch.config, empty_kernel);
  if (e != cudaSuccess) return cuda_fail(e, "empty kernel launch");
  return AGO_OK;
}

ago_status_t ago_last_error(const char** msg) {
  if (msg) *msg = g_msg.c_str();
  return g_status;
}

namespace {
// AGO_MODE_AUTO: does fusing this (fusable) chain pay? Not when the intermediates' round trip through device memory
// costs less than about a third of the contractions' tensor-core time: both modes are then bound by the contractions
// (Section VI-B reports the same for pointwise -> pointwise chains). Data-sheet-class constants; only the ratio matters.
bool fusion_pays(const Plan& p) {
  // Feed-forward chains: both ways are estimated, with the kernel that fused_plan chose (768 -> 3072: fused 15.7 against 26 us at 512
  // rows, but 45 against 26 at 3001 and 109 against 91 at 12288; the reduction-tiling kernel 8 against 19 us
  // at 7 rows of 192 -> 1920 -> 256, 77 against 22 at 2215 rows of 64 -> 1920 -> 1024).
  if (p.fused_kernel == AGO_KERNEL_FFN) {
    const double fused = p.fused_variant == 3 ? ffn_pair_estimate(p) : p.fused_variant == 0 ? ffn_estimate(p) : ffn_cluster_estimate(p);
    return fused >= 0.0 && fused <= 0.97 * ffn_unfused_estimate(p);      // a tie: the launches, whose estimate is the closer one
  }
  // Inverted-residual blocks and their pairs: a strip's tile shrinks with the width of the block, and with it what a CTA makes of the
  // weights that it loads. 32 x 31 x 31, 72 -> 144 -> 72 15 against 32 us; 39 x 36 x 36, 160 -> 960 -> 160 717 against 132.
  // (Of 976 shapes the rule has none more than 2 % slower than a library that fuses up to 64 input channels only.)
  if (p.fused_us >= 0.0) return 0.96 * p.fused_us <= conv_unfused_estimate(p);
  const double t_intermediates = (double)p.intermediate_bytes / 6.5e12;
  const double t_tensor = (double)p.flops_tensor / 1.6e15;
  return !(t_tensor > 0.0 && t_intermediates < 0.35 * t_tensor);
}
}  // namespace

ago_subgraph_t ago_subgraph_create(const ago_subgraph_desc_t* desc) {
  if (desc && desc->struct_size == sizeof(ago_subgraph_desc_t) && desc->mode == AGO_MODE_AUTO) {
    ago_subgraph_desc_t d = *desc;
    d.mode = AGO_MODE_FUSED;
    ago_subgraph_t h = ago_subgraph_create(&d);
    if (h && fusion_pays(h->plan)) return h;
    const bool invalid = !h && g_status != AGO_ERR_UNSUPPORTED;   // a malformed chain fails in every mode
    ago_subgraph_destroy(h);
    if (invalid) return nullptr;
    d.mode = AGO_MODE_PER_MINI_SUBGRAPH;
    return ago_subgraph_create(&d);
  }
  ago_subgraph_s* h = new (std::nothrow) ago_subgraph_s();
  if (!h) { fail(AGO_ERR_INVALID_ARG, "out of host memory"); return nullptr; }
  std::string err;
  ago_status_t s = build_plan(desc, &h->plan, &err);
  if (s == AGO_OK && h->plan.mode == AGO_MODE_FUSED) s = fused_plan(&h->plan, &h->fused, &err);
  if (s != AGO_OK) {
    fail(s, err);
    delete h;
    return nullptr;
  }
  g_status = AGO_OK;
  g_msg.clear();
  return h;
}

void ago_subgraph_destroy(ago_subgraph_t h) {
  if (!h) return;
  if (h->status_word) cudaFree(h->status_word);
  delete h;
}

size_t ago_subgraph_workspace_bytes(ago_subgraph_t h) { return h ? needed_workspace(h->plan) : 0; }

ago_status_t ago_subgraph_set_workspace(ago_subgraph_t h, void* dev_ptr, size_t bytes) {
  if (!h) return fail(AGO_ERR_INVALID_ARG, "handle is NULL");
  if (dev_ptr && (reinterpret_cast<uintptr_t>(dev_ptr) & 255u)) return fail(AGO_ERR_ALIGNMENT, "workspace is not 256-byte aligned");
  if (bytes < needed_workspace(h->plan)) return fail(AGO_ERR_WORKSPACE, "workspace smaller than ago_subgraph_workspace_bytes()");
  std::lock_guard<std::mutex> lock(h->guard);
  h->workspace = dev_ptr;
  h->workspace_bytes = bytes;
  ++h->fused.workspace_epoch;   // nothing remembered about the old contents survives an attach
  return AGO_OK;
}

ago_status_t ago_subgraph_run(ago_subgraph_t h, const void* const* inputs, const void* const* weights,
                              void* const* outputs, void* cuda_stream) {
  ago_status_t s = check_run_args(h, inputs, weights, outputs);
  if (s != AGO_OK) return s;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  std::lock_guard<std::mutex> lock(h->guard);
  s = ensure_status_word(h);
  if (s != AGO_OK) return s;
  const Plan& p = h->plan;
  if (p.mode != AGO_MODE_FUSED) return run_unfused(h, inputs, weights, outputs[0], h->workspace, h->workspace_bytes, h->status_word, stream);
  if (p.fused_kernel == AGO_KERNEL_DEPTHWISE) {
    EpiProgram epi;
    make_epilogue(p, 1, (int)p.ops.size() - 1, inputs, weights, &epi);
    if (epi.n != (int)p.ops.size() - 1 || epi.n > kMaxEpi) return fail(AGO_ERR_UNSUPPORTED, "too many simple operators");
    cudaError_t e = launch_complex(p, p.ops[0], inputs[0], p.dtype, outputs[0], p.dtype, inputs, weights, epi, true, h->status_word, stream);
    if (e != cudaSuccess) return cuda_fail(e, "depthwise kernel launch");
    return AGO_OK;
  }
  std::string err;
  if (needed_workspace(p) > 0 && (h->workspace == nullptr || h->workspace_bytes < needed_workspace(p)))
    return fail(AGO_ERR_WORKSPACE, "workspace missing or smaller than ago_subgraph_workspace_bytes()");
  s = fused_run(p, &h->fused, inputs, weights, outputs[0], h->workspace, h->status_word, stream, &err);
  if (s != AGO_OK) return fail(s, err);
  return AGO_OK;
}

ago_status_t ago_subgraph_run_host(ago_subgraph_t h, const void* const* host_inputs, const void* const* weights,
                                   void* const* host_outputs, void* const* dev_inputs, void* const* dev_outputs,
                                   void* cuda_stream) {
  if (!h) return fail(AGO_ERR_INVALID_ARG, "handle is NULL");
  if (!host_inputs || !host_outputs || !dev_inputs || !dev_outputs || !host_outputs[0])
    return fail(AGO_ERR_INVALID_ARG, "NULL array");
  const Plan& p = h->plan;
  cudaStream_t stream = static_cast<cudaStream_t>(cuda_stream);
  for (int i = 0; i < p.num_inputs; ++i) {
    if (!host_inputs[i] || !dev_inputs[i]) return fail(AGO_ERR_INVALID_ARG, "NULL input buffer");
    cudaError_t e = cudaMemcpyAsync(dev_inputs[i], host_inputs[i], (size_t)p.inputs[i].numel() * elem_bytes(p.dtype),
                                    cudaMemcpyHostToDevice, stream);
    if (e != cudaSuccess) return cuda_fail(e, "host-to-device copy");
  }
  ago_status_t s = ago_subgraph_run(h, const_cast<const void* const*>(dev_inputs), weights, dev_outputs, cuda_stream);
  if (s != AGO_OK) return s;
  cudaError_t e = cudaMemcpyAsync(host_outputs[0], dev_outputs[0], (size_t)p.output.numel() * elem_bytes(p.dtype),
                                  cudaMemcpyDeviceToHost, stream);
  if (e != cudaSuccess) return cuda_fail(e, "device-to-host copy");
  return AGO_OK;
}

ago_status_t ago_subgraph_query(ago_subgraph_t h, int32_t what, int64_t* out) {
  if (!h || !out) return fail(AGO_ERR_INVALID_ARG, "NULL argument");
  const Plan& p = h->plan;
  const int idx = (what >> 16) & 0xffff;
  switch (what & 0xffff) {
    case AGO_Q_NUM_WEIGHTS: *out = (int64_t)p.weight_bytes.size(); break;
    case AGO_Q_WEIGHT_BYTES:
      if (idx >= (int)p.weight_bytes.size()) return fail(AGO_ERR_INVALID_ARG, "weight index out of range");
      *out = p.weight_bytes[idx]; break;
    case AGO_Q_OUTPUT_RANK: *out = p.output.rank; break;
    case AGO_Q_OUTPUT_DIM:
      if (idx >= p.output.rank) return fail(AGO_ERR_INVALID_ARG, "dimension index out of range");
      *out = p.output.d[idx]; break;
    case AGO_Q_OUTPUT_BYTES: *out = p.output.numel() * elem_bytes(p.dtype); break;
    case AGO_Q_FLOPS_TENSOR: *out = p.flops_tensor; break;
    case AGO_Q_FLOPS_CUDA: *out = p.flops_cuda; break;
    case AGO_Q_SFU_OPS: *out = p.sfu_ops; break;
    case AGO_Q_IO_BYTES: *out = p.io_bytes; break;
    case AGO_Q_NUM_LINKS: *out = (int64_t)p.link_category.size(); break;
    case AGO_Q_LINK_CATEGORY:
      if (idx >= (int)p.link_category.size()) return fail(AGO_ERR_INVALID_ARG, "link index out of range");
      *out = p.link_category[idx]; break;
    case AGO_Q_NUM_LAUNCHES: *out = p.num_launches; break;
    case AGO_Q_FUSED_KERNEL: *out = p.fused_kernel; break;
    case AGO_Q_INTERMEDIATE_BYTES: *out = p.intermediate_bytes; break;
    case AGO_Q_TILE_ROWS: *out = p.tile_rows; break;
    case AGO_Q_SMEM_BYTES: *out = p.smem_bytes; break;
    case AGO_Q_MODE: *out = p.mode; break;
    case AGO_Q_WORKSPACE_TRAFFIC: *out = p.mode == AGO_MODE_FUSED ? p.workspace_traffic_bytes : 0; break;
    case AGO_Q_FUSED_VARIANT: *out = p.mode == AGO_MODE_FUSED ? p.fused_variant : 0; break;
    default: return fail(AGO_ERR_INVALID_ARG, "unknown query");
  }
  return AGO_OK;
}

ago_status_t ago_subgraph_debug(ago_subgraph_t h, int32_t what, int64_t value) {
  if (!h) return fail(AGO_ERR_INVALID_ARG, "handle is NULL");
  if (value < 0 || value > 0xffffffffll) return fail(AGO_ERR_INVALID_ARG, "ago_subgraph_debug: value out of range");
  std::lock_guard<std::mutex> lock(h->guard);
  if (what == AGO_DEBUG_WAIT_BUDGET_US) h->wait_budget_us = (unsigned int)value;
  else if (what == AGO_DEBUG_SKIP_SIGNAL) h->skip_signal_code = (unsigned int)value;
  else return fail(AGO_ERR_INVALID_ARG, "ago_subgraph_debug: unknown selector");
  if (h->status_word) {   // already on a device: update the block once the work in flight is done
    cudaError_t e = cudaDeviceSynchronize();
    if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceSynchronize");
    const unsigned int words[2] = {h->wait_budget_us, h->skip_signal_code};
    e = cudaMemcpy(h->status_word + 1, words, sizeof(words), cudaMemcpyHostToDevice);
    if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy(status block)");
  }
  return AGO_OK;
}

ago_status_t ago_subgraph_status(ago_subgraph_t h) {
  if (!h) return fail(AGO_ERR_INVALID_ARG, "handle is NULL");
  cudaError_t e = cudaDeviceSynchronize();
  if (e != cudaSuccess) return cuda_fail(e, "cudaDeviceSynchronize");
  std::lock_guard<std::mutex> lock(h->guard);
  if (!h->status_word) return AGO_OK;
  unsigned int w = 0;
  e = cudaMemcpy(&w, h->status_word, sizeof(w), cudaMemcpyDeviceToHost);
  if (e != cudaSuccess) return cuda_fail(e, "cudaMemcpy(status word)");
  if (w != 0) {
    cudaMemset(h->status_word, 0, sizeof(w));
    ++h->fused.workspace_epoch;   // a run that gave up may have left sums and counters behind in the workspace
    char buf[96];
    std::snprintf(buf, sizeof(buf), "a bounded device-side wait expired (code 0x%x)", w);
    return fail(AGO_ERR_TIMEOUT, buf);
  }
  return AGO_OK;
}

}  // extern "C"
