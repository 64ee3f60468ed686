// gemm_simt.cu -- shared-memory tiled GEMM on the CUDA cores, y = x W^T + epilogue.
//
// The general fallback: any row count, float32 or bf16 operands, fp32 accumulation. It is
// the exact-fp32 path of float32 models (tensor cores would round to tf32) and the path for
// shapes the tensor-core and weight-streaming kernels do not cover.
//
// Tile: 128 virtual output rows x 32 activation rows per block of 256 threads, K in steps of
// 32. A thread holds 4 features (lane + 32 i) x 4 rows; W and X stay K-major in shared memory
// (row pitch 36 floats: conflict-free 128-bit reads), so 4 K steps cost 4 reads of W, 4
// broadcast reads of X and 64 FMAs. The next step's operands are loaded into registers while
// the current one is multiplied.
//
// What bounds it: at the sizes of the float32 workload (K of 128 to 688, one to eleven tiles)
// the chain of K steps, each a round trip to memory. A cluster of S blocks therefore shares a
// tile's K range (simt_split: as many as there are steps, at most 8, while the launch stays
// within two blocks per SM); their partial tiles are summed in rank order through distributed
// shared memory, each block finishing a share of the rows. The first step's weights are loaded
// before the previous kernel's results are waited for. Measured: a 16-token request of the
// float32 workload 19.5 -> 3.6 ms against one block per tile, serial over K and over row tiles,
// with a memory round trip per K step (10 to 40 us per projection).
#include <algorithm>

#include "gemm.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace cdsl {
namespace {

constexpr int TV = 128, TR = 32, TK = 32;
constexpr int kPitch = TK + 4;       // floats per row of W and X in shared memory
constexpr int kLd = TV + 4;          // and of the finished tile
constexpr int kSplitMax = 8;

// 4 consecutive K values of a weight or activation row (K and the offset are multiples of 4).
__device__ __forceinline__ float4 ld4(const float* p) {
  return *reinterpret_cast<const float4*>(p);
}
__device__ __forceinline__ float4 ld4(const __nv_bfloat16* p) {
  const uint2 u = *reinterpret_cast<const uint2*>(p);
  return make_float4(__uint_as_float(u.x << 16), __uint_as_float(u.x & 0xffff0000u),
                     __uint_as_float(u.y << 16), __uint_as_float(u.y & 0xffff0000u));
}
__device__ __forceinline__ float4 ld4_act(const float* x, size_t, size_t i) { return ld4(x + i); }
__device__ __forceinline__ float4 ld4_act(const __nv_bfloat16* x, size_t plane, size_t i) {
  const float4 h = ld4(x + i), l = ld4(x + plane + i);
  return make_float4(h.x + l.x, h.y + l.y, h.z + l.z, h.w + l.w);
}

template <typename T>
__global__ void __launch_bounds__(256, 2) k_gemm_simt(const __grid_constant__ GemmArgs a, int S) {
  const LaunchStamp stamp(a.stamp);
  __shared__ __align__(16) float sm[2 * (TV + TR) * kPitch];   // W, X; then the tile [TR][kLd]
  __shared__ float s_rs[TR];
  static_assert(TR * kLd <= (TV + TR) * kPitch, "the tile fits over one stage");
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int t = blockIdx.x / S, rank = blockIdx.x % S;
  const int v0 = t * TV, r0 = blockIdx.y * TR, K = a.K;
  const int rt = min(TR, a.R - r0);
  const int steps = (K + TK - 1) / TK, s0 = rank * steps / S, s1 = (rank + 1) * steps / S;
  const T* xp = reinterpret_cast<const T*>(a.x);
  const size_t plane = (size_t)a.x_plane;
  // this thread stages rows lr + 32 i of W and row lr of X, K values 4 lk .. 4 lk + 3
  const int lr = tid >> 3, lk = (tid & 7) * 4;
  const T* wrow[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) wrow[i] = virtual_row<T>(a, v0 + lr + 32 * i);
  float4 w[4], x;
  auto load_w = [&](int s) {
    const int k = s * TK + lk;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      w[i] = wrow[i] && k < K ? ld4(wrow[i] + k) : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  auto load_x = [&](int s) {
    const int k = s * TK + lk;
    x = lr < rt && k < K ? ld4_act(xp, plane, (size_t)(r0 + lr) * a.ldx + k)
                         : make_float4(0.f, 0.f, 0.f, 0.f);
  };
  if (s0 < s1) load_w(s0);
  pdl_launch_dependents();
  pdl_wait();
  if (s0 < s1) load_x(s0);
  if (a.in_ss) input_row_scales(a, r0, rt, s_rs, tid, 256);
  float acc[4][4];   // [feature lane + 32 i][row 4 warp + j]
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  for (int s = s0; s < s1; ++s) {
    float* Ws = sm + ((s - s0) & 1) * (TV + TR) * kPitch;
    float* Xs = Ws + TV * kPitch;
#pragma unroll
    for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(Ws + (lr + 32 * i) * kPitch + lk) = w[i];
    *reinterpret_cast<float4*>(Xs + lr * kPitch + lk) = x;
    __syncthreads();   // (the other stage's readers passed the previous one)
    if (s + 1 < s1) {
      load_w(s + 1);
      load_x(s + 1);
    }
#pragma unroll
    for (int k = 0; k < TK; k += 4) {
      float4 wv[4], xv[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        wv[i] = *reinterpret_cast<const float4*>(Ws + (lane + 32 * i) * kPitch + k);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        xv[j] = *reinterpret_cast<const float4*>(Xs + (4 * warp + j) * kPitch + k);
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          acc[i][j] = fmaf(wv[i].x, xv[j].x, acc[i][j]);
          acc[i][j] = fmaf(wv[i].y, xv[j].y, acc[i][j]);
          acc[i][j] = fmaf(wv[i].z, xv[j].z, acc[i][j]);
          acc[i][j] = fmaf(wv[i].w, xv[j].w, acc[i][j]);
        }
    }
  }
  __syncthreads();
  float* tile = sm;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) tile[(4 * warp + j) * kLd + lane + 32 * i] = acc[i][j];
  if (S == 1) {
    __syncthreads();
    tile_epilogue<T>(a, v0, r0, rt, tile, kLd, s_rs);
    return;
  }
  // ---- rank r sums rows [r rt / S, (r + 1) rt / S) of the S partial tiles in rank order
  tc::cluster_arrive();
  tc::cluster_wait();
  const int ra = rank * rt / S, rb = (rank + 1) * rt / S;
  float* red = sm + (TV + TR) * kPitch;   // the other stage
  const uint32_t base = tc::smem_u32(tile);
  for (int i = tid; i < (rb - ra) * (TV / 4); i += 256) {
    const int r = i / (TV / 4), v = (i % (TV / 4)) * 4;
    const uint32_t off = ((ra + r) * kLd + v) * 4;
    float4 p[kSplitMax];
#pragma unroll
    for (int q = 0; q < kSplitMax; ++q)
      if (q < S) p[q] = tc::ld_cluster_f32x4(tc::map_cluster_rank(base + off, q));
    float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
    for (int q = 0; q < kSplitMax; ++q)
      if (q < S) {
        sum.x += p[q].x; sum.y += p[q].y; sum.z += p[q].z; sum.w += p[q].w;
      }
    *reinterpret_cast<float4*>(red + r * kLd + v) = sum;
  }
  tc::cluster_arrive();   // this block has read the others' tiles
  __syncthreads();
  if (rb > ra) tile_epilogue<T>(a, v0, r0 + ra, rb - ra, red, kLd, s_rs + ra);
  tc::cluster_wait();     // no block leaves while its tile may still be read
}

// Blocks that share a tile's K range: one per K step while the launch stays within two blocks per
// SM, at most kSplitMax (the portable cluster size).
int simt_split(int K, int blocks) {
  return std::max(1, std::min({kSplitMax, (K + TK - 1) / TK, 2 * kPlanSMs / blocks}));
}

}  // namespace

void launch_gemm_simt(int dtype, const GemmArgs& a, cudaStream_t s) {
  const int tiles = (a.n_virtual + TV - 1) / TV, row_tiles = (a.R + TR - 1) / TR;
  const int S = simt_split(a.K, tiles * row_tiles);
  const dim3 grid(tiles * S, row_tiles);
  if (dtype == CDSL_DTYPE_BF16)
    launch_pdl_cluster(k_gemm_simt<__nv_bfloat16>, grid, dim3(256), 0, S, s, a, S);
  else
    launch_pdl_cluster(k_gemm_simt<float>, grid, dim3(256), 0, S, s, a, S);
}

}  // namespace cdsl
