// Depthwise-only mini-subgraph as one kernel: depthwise convolution (no
// reduction over channels, Section III-B) with its simple operators applied
// per element right after the window sum (conventional fusion, Section III-A).
// 3x3 windows with pad 1 (every depthwise stage of the benchmark chains) pass
// along strips of the output, every input column loaded once per strip; the
// other window shapes take one output pixel and one 16-byte channel vector per
// thread and leave the overlap to L1 / L2.
#include <cuda_bf16.h>

#include "fused.h"
#include "kernels.h"
#include "tc_common.cuh"

namespace ago {

namespace {

template <typename T> struct Vec;
template <> struct Vec<float> {
  static constexpr int N = 4;
  __device__ static void load(const void* p, int64_t i, float* v) {
    const float4 t = __ldg(reinterpret_cast<const float4*>(reinterpret_cast<const float*>(p) + i));
    v[0] = t.x; v[1] = t.y; v[2] = t.z; v[3] = t.w;
  }
  __device__ static void store(void* p, int64_t i, const float* v) {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(p) + i) = make_float4(v[0], v[1], v[2], v[3]);
  }
};
template <> struct Vec<__nv_bfloat16> {
  static constexpr int N = 8;
  __device__ static void load(const void* p, int64_t i, float* v) {
    const uint4 t = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const __nv_bfloat16*>(p) + i));
    const uint32_t w[4] = {t.x, t.y, t.z, t.w};
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      v[2 * k] = __uint_as_float(w[k] << 16);
      v[2 * k + 1] = __uint_as_float(w[k] & 0xffff0000u);
    }
  }
  __device__ static void store(void* p, int64_t i, const float* v) {
    uint32_t w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * k], v[2 * k + 1]);
      w[k] = *reinterpret_cast<const uint32_t*>(&h);
    }
    *reinterpret_cast<uint4*>(reinterpret_cast<__nv_bfloat16*>(p) + i) = make_uint4(w[0], w[1], w[2], w[3]);
  }
};

__device__ __forceinline__ float gelu_tanh_f(float v) {
  const float c = 0.7978845608028654f;
  return 0.5f * v * (1.0f + tanhf(c * (v + 0.044715f * v * v * v)));
}

// The epilogue program on one channel vector (fp32), `o` = element offset of the vector in the output.
template <typename VT, int V>   // VT: loads V channels
__device__ __forceinline__ void apply_epilogue(const DepthwiseArgs& a, float* acc, int c0, int64_t o) {
  for (int i = 0; i < a.epi.n; ++i) {
    switch (a.epi.code[i]) {
      case EPI_BIAS: {
        const float* b = reinterpret_cast<const float*>(a.epi.ptr[i]) + c0;
#pragma unroll
        for (int k = 0; k < V; ++k) acc[k] += __ldg(b + k);
        break;
      }
      case EPI_RELU:
#pragma unroll
        for (int k = 0; k < V; ++k) acc[k] = fmaxf(acc[k], 0.0f);
        break;
      case EPI_RELU6:
#pragma unroll
        for (int k = 0; k < V; ++k) acc[k] = fminf(fmaxf(acc[k], 0.0f), 6.0f);
        break;
      case EPI_GELU:
#pragma unroll
        for (int k = 0; k < V; ++k) acc[k] = gelu_tanh_f(acc[k]);
        break;
      case EPI_SCALE:
#pragma unroll
        for (int k = 0; k < V; ++k) acc[k] *= a.epi.f[i];
        break;
      case EPI_ADD: {
        float y[V];
        VT::load(a.epi.ptr[i], o, y);
#pragma unroll
        for (int k = 0; k < V; ++k) acc[k] += y[k];
        break;
      }
    }
  }
}

template <typename T>
__global__ void __launch_bounds__(256) depthwise_vec_kernel(const DepthwiseArgs a, int64_t total_vec) {
  constexpr int V = Vec<T>::N;
  tc::grid_dependency_wait();
  const int64_t gid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (gid >= total_vec) return;
  const int cv = a.C / V;
  const int c0 = (int)(gid % cv) * V;
  int64_t t = gid / cv;
  const int wo = (int)(t % a.Wo); t /= a.Wo;
  const int ho = (int)(t % a.Ho);
  const int64_t n = t / a.Ho;
  float acc[V];
#pragma unroll
  for (int k = 0; k < V; ++k) acc[k] = 0.0f;
  for (int r = 0; r < a.R; ++r) {
    const int h = ho * a.stride + r - a.pad;
    if (h < 0 || h >= a.H) continue;
    for (int s = 0; s < a.S; ++s) {
      const int w = wo * a.stride + s - a.pad;
      if (w < 0 || w >= a.W) continue;
      float x[V], f[V];
      Vec<T>::load(a.in, ((n * a.H + h) * a.W + w) * a.C + c0, x);
      Vec<T>::load(a.w, (int64_t)(r * a.S + s) * a.C + c0, f);
#pragma unroll
      for (int k = 0; k < V; ++k) acc[k] = fmaf(x[k], f[k], acc[k]);
    }
  }
  const int64_t o = gid * V;
  apply_epilogue<Vec<T>, V>(a, acc, c0, o);
  Vec<T>::store(a.out, o, acc);
}

// Four channels of one pixel as stored (pixels and weights), their products added to two pairs of fp32 sums.
template <typename T> struct Quad;
template <> struct Quad<float> {
  typedef ulonglong2 Raw;
  __device__ static void fma(uint64_t (&acc)[2], const Raw& x, const Raw& w) {   // packed pairs: half the instructions
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[0]) : "l"(x.x), "l"(w.x));
    asm("fma.rn.f32x2 %0, %1, %2, %0;" : "+l"(acc[1]) : "l"(x.y), "l"(w.y));
  }
  __device__ static void request(uint32_t dst, const float* src, bool inside) { tc::cp_async_16(dst, src, inside ? 16u : 0u); }
  __device__ static void load(const void* p, int64_t i, float* v) { Vec<float>::load(p, i, v); }
  __device__ static void store(float* p, const float* v) { Vec<float>::store(p, 0, v); }
};
template <> struct Quad<__nv_bfloat16> {
  typedef uint2 Raw;
  __device__ static void fma(uint64_t (&acc)[2], const Raw& x, const Raw& w) {
    // mixed-precision FMAs: the bf16 operands as stored, exact product, fp32 accumulate
    const uint32_t xs[2] = {x.x, x.y}, ws[2] = {w.x, w.y};
#pragma unroll
    for (int k = 0; k < 2; ++k)
      asm("{\n\t.reg .b16 xl, xh, wl, wh;\n\t.reg .f32 a, b;\n\t"
          "mov.b32 {xl, xh}, %1;\n\tmov.b32 {wl, wh}, %2;\n\tmov.b64 {a, b}, %0;\n\t"
          "fma.rn.f32.bf16 a, xl, wl, a;\n\tfma.rn.f32.bf16 b, xh, wh, b;\n\tmov.b64 %0, {a, b};\n\t}"
          : "+l"(acc[k]) : "r"(xs[k]), "r"(ws[k]));
  }
  __device__ static void request(uint32_t dst, const __nv_bfloat16* src, bool inside) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 8, %2;" ::"r"(dst), "l"(src), "r"(inside ? 8u : 0u) : "memory");
  }
  __device__ static void load(const void* p, int64_t i, float* v) {
    const uint2 t = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const __nv_bfloat16*>(p) + i));
    v[0] = tc::bf16_lo(t.x); v[1] = tc::bf16_hi(t.x); v[2] = tc::bf16_lo(t.y); v[3] = tc::bf16_hi(t.y);
  }
  __device__ static void store(__nv_bfloat16* p, const float* v) {
    *reinterpret_cast<uint2*>(p) = make_uint2(tc::pack_bf16x2(v[0], v[1]), tc::pack_bf16x2(v[2], v[3]));
  }
};

struct StripShape {
  int groups;    // groups of four channels per pixel
  int seg;       // output columns per strip
  int segs;      // strips per row block
  int hblocks;   // row blocks per image
  uint32_t items;
  int relu, relu6;   // SIMPLE: the epilogue is [bias] [ReLU | ReLU6]
  const float* bias;
};

constexpr int kStripThreads = 128;
constexpr int kAhead = 2;   // input columns on their way (1: 7% slower on large tensors, 3 or 4: no faster)

// 3x3 window, pad 1, stride STRIDE: thread = (image, block of R output rows, strip of output columns, four channels).
// The input columns of the strip pass by one after the other, each loaded once; a column adds its products to the
// (at most three) output columns whose windows cover it. Weights and sums live in registers, the columns on their way in
// a ring in shared memory that every thread fills and reads for itself: memory latency times bandwidth asks for some 50 KB
// in flight per SM, which the registers of the threads that fit would not hold.
// Bound by memory on large tensors (32 x 56 x 56 x 144, stride 1: fp32 21.9 us, 17.7 at the copy rate, bf16 19.0; with
// windows that slide down in registers and weights fetched for every output 49.0 and 32.3; with the columns on their way
// in registers 30.5 and 23.2), by latency on small ones (8 x 14 x 14 x 192 fp32: 2.3 us, one pixel per thread 4.5).
template <typename T, int STRIDE, int R, bool SIMPLE>
__global__ void __launch_bounds__(kStripThreads) depthwise3x3_strip_kernel(const DepthwiseArgs a, const StripShape q) {
  typedef Quad<T> Q;
  typedef typename Q::Raw Raw;
  constexpr int V = 4;
  constexpr int IN = (R - 1) * STRIDE + 3;   // input rows
  tc::grid_dependency_wait();
  const uint32_t gid = blockIdx.x * (uint32_t)kStripThreads + threadIdx.x;
  if (gid >= q.items) return;
  uint32_t t = gid / (uint32_t)q.groups;
  const int c0 = (int)(gid - t * (uint32_t)q.groups) * V;
  const int sg = (int)(t % (uint32_t)q.segs); t /= (uint32_t)q.segs;
  const int ho0 = (int)(t % (uint32_t)q.hblocks) * R;
  const int64_t n = t / (uint32_t)q.hblocks;
  const int wo0 = sg * q.seg, cols = min(q.seg, a.Wo - wo0), rows = min(R, a.Ho - ho0);
  const int h0 = ho0 * STRIDE - 1;
  const T* src = reinterpret_cast<const T*>(a.in) + (n * a.H + h0) * (int64_t)a.W * a.C + c0;   // row h0 (may lie before the tensor)
  T* dst = reinterpret_cast<T*>(a.out) + ((n * a.Ho + ho0) * (int64_t)a.Wo + wo0) * a.C + c0;
  const int in_pitch = a.W * a.C, out_pitch = a.Wo * a.C;
  Raw w[9];
#pragma unroll
  for (int k = 0; k < 9; ++k) w[k] = __ldg(reinterpret_cast<const Raw*>(reinterpret_cast<const T*>(a.w) + k * a.C + c0));
  float bias[V];
#pragma unroll
  for (int k = 0; k < V; ++k) bias[k] = SIMPLE && q.bias ? __ldg(q.bias + c0 + k) : 0.0f;
  extern __shared__ uint8_t ring_mem[];
  constexpr uint32_t kPiece = sizeof(Raw), kRow = kPiece * kStripThreads, kSlot = kRow * IN;
  const uint32_t ring = tc::smem_u32(ring_mem) + threadIdx.x * kPiece;
  const T* safe = src + a.W * a.C;   // some pixel of this thread's image: address of a copy that only fills with zeros
  auto request = [&](uint32_t slot, int col) {
    const bool in = col >= 0 && col < a.W;
#pragma unroll
    for (int i = 0; i < IN; ++i) {
      const bool ok = in && h0 + i >= 0 && h0 + i < a.H;
      const T* g = ok ? src + (int64_t)i * in_pitch + col * a.C : safe;
      Q::request(ring + slot + i * kRow, g, ok);
    }
  };
  auto fetch = [&](Raw (&x)[IN], uint32_t slot) {
#pragma unroll
    for (int i = 0; i < IN; ++i) x[i] = *reinterpret_cast<const Raw*>(ring_mem + threadIdx.x * kPiece + slot + i * kRow);
  };
  auto add_col = [&](uint64_t (&acc)[R][2], const Raw (&x)[IN], int s) {   // s: the column's place in the window
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int i = 0; i < 3; ++i) Q::fma(acc[r], x[r * STRIDE + i], w[3 * i + s]);
  };
  auto clear = [&](uint64_t (&acc)[R][2]) {
#pragma unroll
    for (int r = 0; r < R; ++r) acc[r][0] = acc[r][1] = 0ull;
  };
  auto finish = [&](uint64_t (&acc)[R][2], int o) {   // output column wo0 + o
#pragma unroll
    for (int r = 0; r < R; ++r)
      if (r < rows) {
        float v[V];
#pragma unroll
        for (int k = 0; k < 2; ++k) asm("mov.b64 {%0, %1}, %2;" : "=f"(v[2 * k]), "=f"(v[2 * k + 1]) : "l"(acc[r][k]));
        T* p = dst + (int64_t)r * out_pitch + o * a.C;
        if (SIMPLE) {
          if (q.bias) {
#pragma unroll
            for (int k = 0; k < V; ++k) v[k] += bias[k];
          }
          if (q.relu6) {
#pragma unroll
            for (int k = 0; k < V; ++k) v[k] = fminf(fmaxf(v[k], 0.0f), 6.0f);
          } else if (q.relu) {
#pragma unroll
            for (int k = 0; k < V; ++k) v[k] = fmaxf(v[k], 0.0f);
          }
        } else {
          apply_epilogue<Q, V>(a, v, c0, p - reinterpret_cast<T*>(a.out));
        }
        Q::store(p, v);
      }
  };
  constexpr uint32_t kRing = (kAhead + 1) * kSlot;
  uint32_t head = 0, tail = 0;   // next slot to fill, slot in use
  auto next = [&](uint32_t& slot) { slot = slot + kSlot == kRing ? 0u : slot + kSlot; };
  const int first = wo0 * STRIDE - 1, n_in = (cols - 1) * STRIDE + 3;
#pragma unroll
  for (int k = 0; k < kAhead; ++k) {
    if (k < n_in) request(head, first + k);
    tc::cp_async_commit();
    next(head);
  }
  auto advance = [&](Raw (&x)[IN], int j) {   // input column j of the strip
    if (j + kAhead < n_in) request(head, first + j + kAhead);
    tc::cp_async_commit();
    next(head);
    asm volatile("cp.async.wait_group %0;" ::"n"(kAhead) : "memory");   // column j has landed
    fetch(x, tail);
    next(tail);
  };
  if (STRIDE == 1) {
    // input column j is tap 2 of output column j - 2, tap 1 of j - 1 and tap 0 of j
    uint64_t acc[3][R][2];
    for (int j0 = 0; j0 < n_in; j0 += 3) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const int j = j0 + k;
        if (j < n_in) {
          Raw x[IN];
          advance(x, j);
          clear(acc[k]);
          add_col(acc[k], x, 0);
          if (j >= 1) add_col(acc[(k + 2) % 3], x, 1);
          if (j >= 2) {
            add_col(acc[(k + 1) % 3], x, 2);
            finish(acc[(k + 1) % 3], j - 2);
          }
        }
      }
    }
  } else {
    // output column o takes input columns 2 o to 2 o + 2; the last of them is the first of the next output column
    uint64_t acc[2][R][2];
    {
      Raw x[IN];
      advance(x, 0);
      clear(acc[0]);
      add_col(acc[0], x, 0);
    }
    for (int j0 = 0; j0 < cols; j0 += 2) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int j = j0 + k;
        if (j < cols) {
          Raw x[IN];
          advance(x, 2 * j + 1);
          add_col(acc[k], x, 1);
          advance(x, 2 * j + 2);
          add_col(acc[k], x, 2);
          clear(acc[k ^ 1]);
          add_col(acc[k ^ 1], x, 0);
          finish(acc[k], j);
        }
      }
    }
  }
}

template <typename T, int STRIDE, int R>
cudaError_t launch_strips(const DepthwiseArgs& a, const StripShape& q, bool simple, cudaStream_t stream) {
  auto kernel = simple ? depthwise3x3_strip_kernel<T, STRIDE, R, true> : depthwise3x3_strip_kernel<T, STRIDE, R, false>;
  constexpr int kSmem = (kAhead + 1) * ((R - 1) * STRIDE + 3) * (int)sizeof(typename Quad<T>::Raw) * kStripThreads;
  static int opt_in[2][64] = {};
  const cudaError_t e = ensure_max_dynamic_smem(reinterpret_cast<const void*>(kernel), opt_in[simple]);
  if (e != cudaSuccess) return e;
  FusedLaunch launch(dim3((q.items + kStripThreads - 1) / kStripThreads), kStripThreads, kSmem, stream);
  return cudaLaunchKernelEx(&launch.config, kernel, a, q);
}
template <typename T, int STRIDE>
cudaError_t launch_strips(const DepthwiseArgs& a, const StripShape& q, int R, bool simple, cudaStream_t stream) {
  return R == 4 ? launch_strips<T, STRIDE, 4>(a, q, simple, stream) : R == 2 ? launch_strips<T, STRIDE, 2>(a, q, simple, stream)
                                                                            : launch_strips<T, STRIDE, 1>(a, q, simple, stream);
}

}  // namespace

cudaError_t launch_depthwise_fused(const DepthwiseArgs& a, cudaStream_t stream) {
  const int V = a.dtype == AGO_FP32 ? 4 : 8;
  if (a.R == 3 && a.S == 3 && a.pad == 1 && (a.stride == 1 || a.stride == 2) && a.C % V == 0 &&
      (int64_t)a.N * a.Ho * a.Wo * (a.C / 4) < (1ll << 31) && (int64_t)a.H * a.W * a.C < (1ll << 31)) {
    StripShape q{};
    int i = 0;
    if (i < a.epi.n && a.epi.code[i] == EPI_BIAS) q.bias = reinterpret_cast<const float*>(a.epi.ptr[i++]);
    if (i < a.epi.n && a.epi.code[i] == EPI_RELU) q.relu = 1, ++i;
    else if (i < a.epi.n && a.epi.code[i] == EPI_RELU6) q.relu6 = 1, ++i;
    const bool simple = i == a.epi.n;
    q.groups = a.C / 4;
    auto split = [&](int rows, int columns) {   // -> threads
      q.segs = (a.Wo + columns - 1) / columns;
      q.seg = (a.Wo + q.segs - 1) / q.segs;
      q.segs = (a.Wo + q.seg - 1) / q.seg;
      q.hblocks = (a.Ho + rows - 1) / rows;
      return (int64_t)a.N * q.hblocks * q.segs * q.groups;
    };
    // The larger a thread's piece, the less of the input is read twice: (R + 2) / R rows, (columns + 2) / columns. The
    // smaller, the shorter the chain of columns a thread walks along and the more threads there are. The largest piece
    // that leaves 240 threads per SM (32 x 28 x 28 x 96, stride 2, fp32: 32256 threads 4.6 us -> 37632 threads 3.0 us;
    // 16 x 28 x 28 x 192: 21504 threads 6.4 us, 37632 threads 4.7 us, 75264 threads 5.1 us), two rows by two columns down to
    // 120 threads per SM, below that one row by two columns.
    const int64_t sms = device_sm_count();
    struct Piece { int rows, columns; int64_t threads; };
    const Piece pieces[] = {{4, 8, 240 * sms}, {4, 4, 240 * sms}, {2, 4, 240 * sms}, {2, 2, 120 * sms}, {1, 2, 0}};
    int R = 1;
    for (const Piece& c : pieces) {
      const int64_t threads = split(c.rows, c.columns);
      R = c.rows; q.items = (uint32_t)threads;
      if (threads >= c.threads) break;
    }
    if (a.dtype == AGO_FP32) return a.stride == 1 ? launch_strips<float, 1>(a, q, R, simple, stream) : launch_strips<float, 2>(a, q, R, simple, stream);
    return a.stride == 1 ? launch_strips<__nv_bfloat16, 1>(a, q, R, simple, stream) : launch_strips<__nv_bfloat16, 2>(a, q, R, simple, stream);
  }
  const int64_t total = (int64_t)a.N * a.Ho * a.Wo * (a.C / V);
  FusedLaunch launch(dim3((unsigned)((total + 255) / 256)), 256, 0, stream);
  return cudaLaunchKernelEx(&launch.config, a.dtype == AGO_FP32 ? depthwise_vec_kernel<float> : depthwise_vec_kernel<__nv_bfloat16>, a, total);
}

}  // namespace ago
