// Fused pair of depthwise convolutions: depthwise 3x3 (pad 1, stride 1) + bias + ReLU6, twice, one kernel
// (the "two depthwise convolutions" subgraph of the micro-benchmark, Section VI-B).
//
// Both operators have no reduction over channels, so the pair is tiled over channels without any recomputation
// (Section III-B, downstream depthwise); the spatial tile of the upstream operator grows by the one-pixel halo of
// the downstream window.
//
// A thread owns one channel pair, SEG output columns and R output rows and streams down the rows with both windows in
// registers: three input rows of SEG + 4 pixels and three intermediate rows of SEG + 2, packed bf16 pairs as they were
// loaded or made (the mixed-precision FMA takes them as they are). One step = the row of the intermediate whose window
// is complete, the request for the next input row (it travels during the second convolution), the output row whose
// window is complete. Nothing passes through shared memory and nothing waits at a barrier. Neighbouring threads are
// neighbouring channel pairs, so a pixel is one 128-byte request of a warp; the SEG + 4 columns that neighbouring
// segments share come from L1.
//
// What bounds it: issue slots (0.69 of them used: 10.5 of 16.2 M warp instructions are the FMAs, 4.4 M go to the integer pipe, which takes
// two cycles each: conversions of the results, clamps, edges, addresses). Per output pair 18 FMAs of the second and
// 18 (SEG + 2) / SEG (R + 2) / R of the first convolution, about 55 instructions in all at 7 columns x 14 rows. The previous
// kernel (input, intermediate and output tiles in shared memory, three barriers per CTA, two CTAs per SM) needed as many
// and ran at half the issue rate: 32 x 56 x 56 x 144 31.7 -> 22.5 us (2.6 TB/s), 3 x 14 x 14 x 128 5.9 -> 2.1 us.
// Measured and not kept: L2 prefetch of the strip (no change), column predicates from a bit mask (23.9 us).
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>

#include "dw_common.cuh"
#include "fused.h"
#include "tc_common.cuh"

namespace ago {

namespace {

using namespace tc;
using namespace dw;

constexpr int kChunk = 16;      // channels come in multiples of 16

struct DwDwParams {
  const __nv_bfloat16* x;
  const __nv_bfloat16* w1;   // [3][3][C]
  const float* b1;
  const __nv_bfloat16* w2;
  const float* b2;
  __nv_bfloat16* out;
  int N, H, W, C;
  int R, strips, nseg, pairs;         // output rows per thread, strips and segments per image, C / 2
  int items;                          // threads with work per image
};

__device__ __forceinline__ uint32_t ldg32_or_zero(const uint8_t* p, bool inside) {
  uint32_t v;
  asm volatile("{\n\t.reg .pred q;\n\tsetp.ne.u32 q, %2, 0;\n\tmov.u32 %0, 0;\n\t@q ld.global.nc.u32 %0, [%1];\n\t}"
               : "=r"(v) : "l"(p), "r"((uint32_t)inside));
  return v;
}

// One output row of a 3x3 window over three rows of packed pairs: OUT values from OUT + 2 columns. The oldest row is used
// up first; after_a() then runs (the request for the row that replaces it).
template <int OUT, class AfterA>
__device__ __forceinline__ void window_row(const uint32_t (&a)[OUT + 2], const uint32_t (&b)[OUT + 2], const uint32_t (&c)[OUT + 2],
                                           const uint32_t (&w)[9], float2 bias, uint32_t (&out)[OUT], AfterA&& after_a) {
  float2 acc[OUT];
#pragma unroll
  for (int j = 0; j < OUT; ++j) {
    acc[j] = fma_pair_from(bias, a[j], w[0]);
    fma_pair(acc[j], a[j + 1], w[1]); fma_pair(acc[j], a[j + 2], w[2]);
  }
  after_a();
#pragma unroll
  for (int j = 0; j < OUT; ++j) {
    fma_pair(acc[j], b[j], w[3]); fma_pair(acc[j], b[j + 1], w[4]); fma_pair(acc[j], b[j + 2], w[5]);
    fma_pair(acc[j], c[j], w[6]); fma_pair(acc[j], c[j + 1], w[7]); fma_pair(acc[j], c[j + 2], w[8]);
    out[j] = relu6_pack(acc[j].x, acc[j].y);
  }
}

// 128 threads, four CTAs per SM: both windows need about 110 registers. CTAs of 256 threads ran the largest case as fast and
// the small ones 0.3 us slower.
constexpr int kThreads = 128;
constexpr int kCtasPerSM = 4;

template <int SEG>
__global__ void __launch_bounds__(kThreads, kCtasPerSM)
dwdw_fused_kernel(const DwDwParams p) {
  // The next grid of the stream starts when this one's CTAs exit (no launch_dependents): CTAs of the next grid that moved in
  // beside this one's landed unevenly on the SMs (33.4 -> 26.7 us at 40 x 45 x 45 x 192).
  grid_dependency_wait();
  const int item = (int)(blockIdx.x * kThreads + threadIdx.x);
  if (item >= p.items) return;
  const int n = blockIdx.y;
  const int q = item / p.pairs, pair = item - q * p.pairs;
  const int strip = q / p.nseg, seg = q - strip * p.nseg;
  const int ho0 = strip * p.R, rows = min(p.R, p.H - ho0), wo0 = seg * SEG;
  const size_t pix = (size_t)p.C * 2, row_bytes = (size_t)p.W * pix;

  uint32_t w1[9], w2[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) {
    w1[k] = __ldg(reinterpret_cast<const uint32_t*>(p.w1 + (size_t)k * p.C) + pair);
    w2[k] = __ldg(reinterpret_cast<const uint32_t*>(p.w2 + (size_t)k * p.C) + pair);
  }
  const float2 bias1 = __ldg(reinterpret_cast<const float2*>(p.b1) + pair);
  const float2 bias2 = __ldg(reinterpret_cast<const float2*>(p.b2) + pair);

  // input row ho0 - 2, from column wo0 - 2 (both may lie outside the image: not dereferenced there)
  const uint8_t* src = reinterpret_cast<const uint8_t*>(p.x) + ((int64_t)n * p.H + ho0 - 2) * (int64_t)row_bytes +
                       ((int64_t)wo0 - 2) * (int64_t)pix + pair * 4;
  uint8_t* dst = reinterpret_cast<uint8_t*>(p.out) + ((int64_t)n * p.H + ho0) * (int64_t)row_bytes + (int64_t)wo0 * (int64_t)pix + pair * 4;
  int hx = ho0 - 2;
  const int cols = p.W - wo0;               // columns of the image from the segment's first on
  auto load_row = [&](uint32_t (&x)[SEG + 4]) {
    const bool hin = (unsigned)hx < (unsigned)p.H;
#pragma unroll
    for (int j = 0; j < SEG + 4; ++j)
      x[j] = ldg32_or_zero(src + j * pix, hin && (j >= 2 || wo0 > 0) && (j < 3 || j < cols + 2));   // wo0 is 0 or >= SEG > 2
    src += row_bytes;
    ++hx;
  };
  uint32_t x[3][SEG + 4], m[3][SEG + 2];
  load_row(x[0]);
  load_row(x[1]);
  load_row(x[2]);
  const int steps = rows + 2;
  // step s makes intermediate row ho0 - 1 + s and, from s = 2 on, output row ho0 + s - 2
  auto step = [&](int s, uint32_t (&xa)[SEG + 4], uint32_t (&xb)[SEG + 4], uint32_t (&xc)[SEG + 4], uint32_t (&ma)[SEG + 2],
                  uint32_t (&mb)[SEG + 2], uint32_t (&mc)[SEG + 2]) {
    window_row<SEG + 2>(xa, xb, xc, w1, bias1, mc, [&] { if (s + 1 < steps) load_row(xa); });
    // the second convolution pads the post-activation tensor: zero outside the image
    if (wo0 == 0) mc[0] = 0u;
    if (cols <= SEG) {
#pragma unroll
      for (int j = 2; j < SEG + 2; ++j) if (j > cols) mc[j] = 0u;
    }
    if ((unsigned)(ho0 - 1 + s) >= (unsigned)p.H) {
#pragma unroll
      for (int j = 0; j < SEG + 2; ++j) mc[j] = 0u;
    }
    if (s >= 2) {
      uint32_t o[SEG];
      window_row<SEG>(ma, mb, mc, w2, bias2, o, [] {});
#pragma unroll
      for (int j = 0; j < SEG; ++j) if (j < 1 || j < cols) *reinterpret_cast<uint32_t*>(dst + j * pix) = o[j];
      dst += row_bytes;
    }
  };
#pragma unroll 1
  for (int s = 0;;) {
    step(s, x[0], x[1], x[2], m[1], m[2], m[0]);
    if (++s == steps) break;
    step(s, x[1], x[2], x[0], m[2], m[0], m[1]);
    if (++s == steps) break;
    step(s, x[2], x[0], x[1], m[0], m[1], m[2]);
    if (++s == steps) break;
  }
}

struct DwDwHost {
  DwDwParams prm;
  int seg = 7;
};

}  // namespace

ago_status_t dwdw_plan(Plan* plan, FusedState* st, std::string* err) {
  const OpInfo& a = plan->ops[0];
  auto* host = new DwDwHost();
  DwDwParams& q = host->prm;
  q = DwDwParams{};
  q.N = (int)a.in.d[0]; q.H = (int)a.in.d[1]; q.W = (int)a.in.d[2]; q.C = (int)a.in.d[3];
  auto bad = [&](const char* m) { *err = std::string("fused depthwise pair: ") + m; delete host; return AGO_ERR_UNSUPPORTED; };
  if (q.C % kChunk != 0) return bad("channels must be a multiple of 16");
  if (q.N > 65535 || q.W > 4096) return bad("batch or width too large");
  q.pairs = q.C / 2;
  // Columns and rows per thread: the halo is amortised over SEG columns and R rows, while the threads should fill the
  // resident slots evenly. Cycles = rounds x steps x the time of a step, which was measured with w warps per scheduler as
  // 200 + 615 w (7 columns) and 150 + 390 w (4 columns): 820 / 540 alone, 2660 / 1710 with four. The estimate meets the
  // measured times of 8 shapes x 15 values of R within 10 %, and its choice is within 5 % of the best of them.
  const long sms = device_sm_count(), cap = sms * kCtasPerSM;
  double best = 0;
  for (int seg : {7, 4}) {
    const int nseg = (q.W + seg - 1) / seg;
    auto step_cycles = [&](long warps) { return seg == 7 ? 200.0 + 615.0 * warps : 150.0 + 390.0 * warps; };
    for (int R = 1; R <= q.H; ++R) {
      const int strips = (q.H + R - 1) / R;
      const long items = (long)q.pairs * nseg * strips;
      if (items > 0x3fffffffL) continue;
      const long ctas = (items + kThreads - 1) / kThreads * q.N, full = ctas / cap, rest = ctas - full * cap;
      const double cost = (R + 2) * (full * step_cycles(kCtasPerSM) + (rest ? step_cycles((rest + sms - 1) / sms) : 0.0));
      if (best == 0 || cost < best) { best = cost; q.R = R; host->seg = seg; q.nseg = nseg; q.strips = strips; q.items = (int)items; }
    }
  }
  if (best == 0) return bad("image too large");
  st->impl = host;
  st->impl_free = [](void* p) { delete static_cast<DwDwHost*>(p); };
  st->tile_rows = q.R; st->grid = (q.items + kThreads - 1) / kThreads * q.N;
  st->smem_bytes = 1024;       // nothing but the 1 KB that is reserved for every CTA
  plan->tile_rows = q.R; plan->smem_bytes = st->smem_bytes;
  return AGO_OK;
}

ago_status_t dwdw_run(const Plan& plan, FusedState* st, const void* const* inputs, const void* const* weights,
                      void* output, unsigned int* status_word, cudaStream_t stream, std::string* err) {
  (void)plan; (void)status_word;
  DwDwHost* host = static_cast<DwDwHost*>(st->impl);
  DwDwParams q = host->prm;
  q.x = static_cast<const __nv_bfloat16*>(inputs[0]);
  q.w1 = static_cast<const __nv_bfloat16*>(weights[0]); q.b1 = static_cast<const float*>(weights[1]);
  q.w2 = static_cast<const __nv_bfloat16*>(weights[2]); q.b2 = static_cast<const float*>(weights[3]);
  q.out = static_cast<__nv_bfloat16*>(output);
  FusedLaunch launch(dim3((unsigned)((q.items + kThreads - 1) / kThreads), (unsigned)q.N), kThreads, 0, stream);
  cudaError_t e = cudaLaunchKernelEx(&launch.config, host->seg == 7 ? dwdw_fused_kernel<7> : dwdw_fused_kernel<4>, q);
  if (e != cudaSuccess) { *err = std::string("fused depthwise pair launch: ") + cudaGetErrorString(e); return AGO_ERR_CUDA; }
  return AGO_OK;
}

}  // namespace ago
