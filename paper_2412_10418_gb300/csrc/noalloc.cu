// noalloc.cu -- cdsl_gemv_noalloc: the weight-streaming GEMM for callers that cannot allocate.
//
// Some callers cannot hand this library a workspace: a host framework whose own caching
// allocator has already reserved the GPU's memory, a real-time loop that must not block on
// cudaMalloc / cudaFree, a runtime that forbids device allocation after start-up. For them this
// entry point is one kernel that needs no scratch in global memory.
//
// What bounds it: HBM, the weights once (R <= 8 rows: at most 16 flops per weight byte). A block
// owns a contiguous range of output rows, even over two blocks per SM, so that no sum crosses
// blocks. Its warps split K: a warp keeps the x values of its 256-wide K step in registers (fp32, as
// given) and streams that step of group after group of output rows, 16 bytes per lane and row,
// the next group's loads in flight while this one's products are summed; packed fp32 FMAs over
// pairs of K values. A group's 16 sums are reduced over the lanes by a transposing butterfly
// and over the warps through shared memory, in a fixed order. The kernel before (split-K blocks
// over 512 K values each, x through shared memory from hi/lo planes that another launch wrote,
// partial sums through global memory) took 45.5 us for 4 rows of 4096 -> 11008 (1.97 TB/s); this
// one takes 22.6 (4.0 TB/s).
#include <cuda.h>

#include <algorithm>

#include "gemm.cuh"
#include "kernels.h"

namespace cdsl {
namespace {

constexpr int kMaxR = 8;
constexpr int kMaxK = 8192;
constexpr int kMaxN = 32768;
constexpr int kThreads = 256, kWarps = kThreads / 32;
constexpr int kStep = 256;            // K values of one 128-bit load per lane
constexpr int kSums = 16;             // sums per group: rows of W x rows of x
constexpr int kBlocks = 2 * kPlanSMs;

__device__ __forceinline__ uint4 ld_stream(const __nv_bfloat16* p) {
  uint4 v;
  asm("ld.global.nc.L1::no_allocate.v4.u32 {%0, %1, %2, %3}, [%4];"
      : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
      : "l"(p));
  return v;
}

// Pairs of fp32 values in one 64-bit register.
__device__ __forceinline__ uint64_t pack2(float lo, float hi) {
  return (uint64_t)__float_as_uint(lo) | ((uint64_t)__float_as_uint(hi) << 32);
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t bf16x2_to_f32x2(uint32_t u) {
  return (uint64_t)(u << 16) | ((uint64_t)(u & 0xffff0000u) << 32);
}

// y[r, n] = sum_k x[r, k] w[n, k], R <= RM rows of x. kw (1, 2, 4 or 8) warps side by side along
// K, the other 8 / kw over the block's groups of 16 / RM rows of W. Dynamic shared memory:
// [groups][kw][16] floats.
template <int RM>
__global__ void __launch_bounds__(kThreads, 2)
    k_gemv_rows(const __nv_bfloat16* __restrict__ w, int N, int K, const float* __restrict__ x,
                int R, float* __restrict__ y, int kw) {
  constexpr int GR = kSums / RM;      // rows of W per group
  extern __shared__ float red[];
  const int n0 = (int)((long long)blockIdx.x * N / gridDim.x);
  const int n1 = (int)((long long)(blockIdx.x + 1) * N / gridDim.x);
  const int groups = (n1 - n0 + GR - 1) / GR;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kwi = warp % kw, rgi = warp / kw, rg = kWarps / kw;
  for (int kb = 0; kb < K; kb += kw * kStep) {
    const int k = kb + kwi * kStep + lane * 8;
    const bool live = k < K;          // K is a multiple of 8
    auto load = [&](int g, uint4 (&v)[GR]) {
#pragma unroll
      for (int i = 0; i < GR; ++i) {
        const int n = n0 + g * GR + i;
        v[i] = live && n < n1 ? ld_stream(w + (size_t)n * K + k) : make_uint4(0u, 0u, 0u, 0u);
      }
    };
    uint4 cur[GR];
    load(rgi, cur);                   // (rows past the range: zero)
    uint64_t xr[RM][4];
#pragma unroll
    for (int r = 0; r < RM; ++r) {
      float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
      if (r < R && live) {
        a = *reinterpret_cast<const float4*>(x + (size_t)r * K + k);
        b = *reinterpret_cast<const float4*>(x + (size_t)r * K + k + 4);
      }
      xr[r][0] = pack2(a.x, a.y);
      xr[r][1] = pack2(a.z, a.w);
      xr[r][2] = pack2(b.x, b.y);
      xr[r][3] = pack2(b.z, b.w);
    }
    for (int g = rgi; g < groups; g += rg) {
      uint4 nxt[GR];
      load(g + rg, nxt);
      uint64_t acc[kSums];
#pragma unroll
      for (int i = 0; i < kSums; ++i) acc[i] = 0ull;
#pragma unroll
      for (int i = 0; i < GR; ++i) {
        const uint32_t q[4] = {cur[i].x, cur[i].y, cur[i].z, cur[i].w};
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const uint64_t wv = bf16x2_to_f32x2(q[c]);
#pragma unroll
          for (int r = 0; r < RM; ++r) acc[i * RM + r] = fma2(wv, xr[r][c], acc[i * RM + r]);
        }
      }
      float s[kSums];
#pragma unroll
      for (int i = 0; i < kSums; ++i)
        s[i] = __uint_as_float((uint32_t)acc[i]) + __uint_as_float((uint32_t)(acc[i] >> 32));
      warp_sums<kSums>(s);            // lane l: the sum of index l / 2 in s[0]
      if ((lane & 1) == 0) {          // this warp's own slot: K steps add up in order
        float* dst = red + ((size_t)g * kw + kwi) * kSums + (lane >> 1);
        *dst = kb == 0 ? s[0] : *dst + s[0];
      }
#pragma unroll
      for (int i = 0; i < GR; ++i) cur[i] = nxt[i];
    }
  }
  __syncthreads();
  const int rows = n1 - n0;
  for (int i = threadIdx.x; i < rows * R; i += kThreads) {
    const int r = i / rows, n = i % rows;
    const float* src = red + (size_t)(n / GR) * kw * kSums + (n % GR) * RM + r;
    float t = 0.f;
    for (int q = 0; q < kw; ++q) t += src[q * kSums];
    y[(size_t)r * N + n0 + n] = t;
  }
}

template <int RM>
void launch_rows(const __nv_bfloat16* w, int N, int K, const float* x, int R, float* y,
                 cudaStream_t s) {
  constexpr int GR = kSums / RM;
  const int blocks = std::min(kBlocks, (N + GR - 1) / GR);
  int kw = 1;   // warps along K: one per K step, up to all of them
  while (kw < kWarps && kw * kStep < K) kw *= 2;
  // at most ceil(N / blocks) rows per block: 108 of them at the largest N, 27.6 KB at 8 rows
  const int groups = ((N + blocks - 1) / blocks + GR - 1) / GR;
  k_gemv_rows<RM><<<blocks, kThreads, (size_t)groups * kw * kSums * sizeof(float), s>>>(
      w, N, K, x, R, y, kw);
}

}  // namespace
}  // namespace cdsl

using namespace cdsl;

extern "C" int32_t cdsl_gemv_noalloc(const void* d_w, int32_t N, int32_t K, const float* d_x,
                                     int32_t R, float* d_y, void* stream) {
  auto aligned = [](const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  if (!d_w || !d_x || !d_y || !aligned(d_w) || !aligned(d_x) || !aligned(d_y)) {
    set_thread_error("cdsl_gemv_noalloc: pointers must be non-NULL and 16-byte aligned");
    return CDSL_EINVAL;
  }
  if (R < 1 || R > kMaxR || K < 8 || K > kMaxK || (K % 8) || N < 1 || N > kMaxN) {
    set_thread_error("cdsl_gemv_noalloc: sizes beyond its limits: need 1 <= R <= 8, "
                     "8 <= K <= 8192 with K % 8 == 0, 1 <= N <= 32768");
    return CDSL_EINVAL;
  }
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  const __nv_bfloat16* w = static_cast<const __nv_bfloat16*>(d_w);
  cudaGetLastError();
  if (R <= 2) launch_rows<2>(w, N, K, d_x, R, d_y, s);
  else if (R <= 4) launch_rows<4>(w, N, K, d_x, R, d_y, s);
  else launch_rows<8>(w, N, K, d_x, R, d_y, s);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) {
    set_thread_error(cudaGetErrorString(e));
    return CDSL_ECUDA;
  }
  return CDSL_OK;
}
