// gemm_tc.cu -- projection GEMMs of up to kPairRows activation rows on the 5th-generation tensor
// cores (tcgen05 + TMEM + TMA); gemm_pair.cu takes more rows.
//
// Swap-AB: the weights are the M = 128 operand (one tile = 128 virtual output rows, loaded as
// two 64-row TMA boxes so that a tile may draw its halves from different segments: gate/up
// interleave, q/k/v boundaries) and the activation rows are the N operand (N = R rounded up
// to 16, 16..64). Both operands are K-major bf16 in 128-byte-swizzled shared-memory tiles;
// the accumulator lives in TMEM (fp32). The activations come as the hi and lo bf16 planes of
// the split, so each 16-deep K step issues two MMAs into the same accumulator.
//
// Persistent stream-K schedule: a fixed grid of blocks (two per SM when the ring fits in half
// the shared memory) divides the tiles x 64-wide K blocks evenly, so there is no partial last
// wave. With as many tiles as block slots or fewer the same code runs one block per whole tile
// (data-parallel: every segment is a whole tile, no fixup). A block walks its contiguous range
// of (tile, k-block) units; a run of units within one tile is a segment. Warp 0 (one lane)
// streams weights and activations with TMA through a ring of mbarrier-guarded stages; warp 1
// (one lane) issues the MMAs into one of two TMEM accumulators and commits; warps 2-5 drain a
// finished accumulator (TMEM -> registers -> shared memory) while the next segment
// accumulates into the other one. A segment covering a whole tile runs the fused epilogue
// directly; otherwise its partial tile goes to scratch and the last contributing block finishes
// the tile from the partials summed in block order (a deterministic sum).
//
// Cluster split-K (GEMMs with few tiles): a thread-block cluster of S blocks owns one tile and
// block r of it the r-th of S even K ranges. Each block drains its partial tile into shared
// memory; after a cluster barrier every block sums a share of the tile's activation rows over
// the S partials (in block order, through distributed shared memory) and runs the epilogue on
// them. No global partials, no atomics.
//
// Programmatic dependent launch: weights do not depend on the previous kernel, so the TMA
// lane issues the first ring's weight loads before griddepcontrol.wait and the activation
// loads after it; every other dependent access comes after the wait. Every wait on an mbarrier
// is bounded in time; on expiry the block latches CDSL_ETIMEOUT and winds down.
#include <cudaTypedefs.h>

#include <algorithm>

#include "gemm.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace cdsl {
namespace {

constexpr int kMaxStages = 8;
constexpr int kTileLd = 132;     // fp32 epilogue tile row pitch (128 + 4 against bank conflicts)
constexpr int kEpRowsMax = 64;   // activation rows drained per epilogue chunk (at most)
constexpr int kThreads = 192;    // warp 0 TMA, warp 1 MMA, warps 2-5 epilogue
constexpr int kEpThreads = 128;

__host__ __device__ __forceinline__ uint32_t tmem_cols_for(int n_pad) {
  uint32_t c = 32;
  while (c < (uint32_t)n_pad) c <<= 1;
  return c;
}

// Source tensor map and first row of the 64-row half-tile starting at virtual row vstart.
__device__ __forceinline__ void half_source(const GemmArgs& a, int vstart, int* m, int* y) {
  if (a.mode == EPI_SWIGLU) {
    *m = (vstart >> 6) & 1;
    *y = (vstart >> 7) * 64;
    return;
  }
  int base = 0;
  for (int s = 0; s < a.n_seg; ++s) {
    if (vstart < base + a.seg_rows[s] || s == a.n_seg - 1) {
      *m = s;
      *y = vstart - base;
      return;
    }
    base += a.seg_rows[s];
  }
}

// Stream-K partition: block c owns units [start(c), start(c + 1)) (U * C < 2^31, checked on
// the host).
__device__ __forceinline__ int unit_start(int c, int U, int C) { return c * U / C; }
__device__ __forceinline__ int unit_owner(int u, int U, int C) { return ((u + 1) * C - 1) / U; }

constexpr int kMaxContrib = 256;   // contributors to one tile (bounded on the host)
constexpr int kMaxSplit = 8;       // target blocks per tile when tiles are few

// kRegs: the cluster split-K finishes its rows on registers (QKV and residual projections with
// enough rows per block: launch_gemm_tc).
template <bool kRegs>
__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_tc(const __grid_constant__ TcMaps maps, const __grid_constant__ GemmArgs a, TcPlan p,
              float* part, int* tile_cnt) {
  extern __shared__ uint8_t smem_raw[];
  const LaunchStamp stamp(a.stamp);
  __shared__ __align__(8) uint64_t full_bar[kMaxStages];
  __shared__ __align__(8) uint64_t empty_bar[kMaxStages];
  __shared__ __align__(8) uint64_t accf_bar[2];
  __shared__ __align__(8) uint64_t acce_bar[2];
  __shared__ __align__(8) uint64_t drain_bar;   // every MMA this block issued has completed
  __shared__ uint32_t tmem_base;
  __shared__ int s_abort, s_last;
  __shared__ int s_slot_off[kMaxContrib];   // reducer: scratch offset (floats) per contributor
  __shared__ float s_rs[kPairRows];          // input row scales (RMSNorm folded into the GEMM)
  __shared__ QkvRow s_qkv[kRegs ? kPairRows : 1];   // QKV: where this block's rows go

  uint8_t* smem = smem_raw + ((1024 - (tc::smem_u32(smem_raw) & 1023)) & 1023);
  const int NP = p.n_pad, S = p.stages, KBT = p.kb_total;
  const uint32_t stage_bytes = 16384u + 256u * NP;
  const int kEpRows = p.ep_rows;
  float* tileS = reinterpret_cast<float*>(smem + (size_t)S * stage_bytes);  // [ep_rows][kTileLd]
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int c = blockIdx.x, C = gridDim.x;
  const int U = p.tiles * KBT;
  const int SK = p.cluster;   // > 0: cluster split-K, block (tile c / SK, K range c % SK)
  int u0, u1;
  if (SK > 0) {
    const int t = c / SK, r = c % SK;
    u0 = t * KBT + r * KBT / SK;
    u1 = t * KBT + (r + 1) * KBT / SK;
  } else {
    u0 = unit_start(c, U, C);
    u1 = unit_start(c + 1, U, C);
  }
  // hi and lo rows are contiguous in each stage: one MMA with N = 2*NP covers both (the
  // accumulator then holds W.hi in columns [0, NP) and W.lo in [NP, 2NP)).
  const uint32_t acc_cols = tmem_cols_for(2 * NP);

  // TMA producer state (thread 0): unit u0 + i is (t_cur, kb_cur) for the next i to issue
  const int n_units = u1 - u0;
  const int pre = min(S, n_units);
  int t_cur = u0 / KBT, kb_cur = u0 % KBT;
  int n_issued = 0;   // (thread 0) units whose copies were issued
  uint64_t pol = 0;
  auto load_w = [&](int i, int t, int kb) {
    int m0, y0, m1, y1;
    half_source(a, t * 128, &m0, &y0);
    half_source(a, t * 128 + 64, &m1, &y1);
    uint8_t* st = smem + (size_t)(i % S) * stage_bytes;
    tc::tma_load_2d_hint(st, &maps.w[m0], kb * 64, y0, &full_bar[i % S], pol);
    tc::tma_load_2d_hint(st + 8192, &maps.w[m1], kb * 64, y1, &full_bar[i % S], pol);
  };
  auto load_x = [&](int i, int kb) {   // one box of NP rows per plane (the maps' box)
    uint8_t* st = smem + (size_t)(i % S) * stage_bytes;
    tc::tma_load_2d(st + 16384, &maps.xh, kb * 64, 0, &full_bar[i % S]);
    tc::tma_load_2d(st + 16384 + NP * 128, &maps.xl, kb * 64, 0, &full_bar[i % S]);
  };
  if (threadIdx.x == 0) {
    for (int m = 0; m < 3; ++m) tc::tma_prefetch_map(&maps.w[m]);
    tc::tma_prefetch_map(&maps.xh);
    tc::tma_prefetch_map(&maps.xl);
    for (int s = 0; s < S; ++s) {
      tc::mbar_init(&full_bar[s], 1);
      tc::mbar_init(&empty_bar[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&accf_bar[i], 1);
      tc::mbar_init(&acce_bar[i], kEpThreads);
    }
    tc::mbar_init(&drain_bar, 1);
    s_abort = 0;
    tc::fence_mbar_init();
    tc::fence_proxy_async();
    // the first ring's weights do not depend on the previous kernel: issue them while warp 1
    // allocates TMEM
    pol = tc::policy_evict_first();
    for (int i = 0; i < pre; ++i) {
      tc::mbar_expect_tx(&full_bar[i], stage_bytes);
      load_w(i, t_cur, kb_cur);
      if (++kb_cur == KBT) { kb_cur = 0; ++t_cur; }
    }
  }
  if (warp == 1) tc::tmem_alloc(&tmem_base, 2 * acc_cols);
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  pdl_launch_dependents();
  const uint32_t tmem = tmem_base;

  bool gave_up = true;   // (epilogue warps: false once every accumulator has been drained)
  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer
      bool aborted = false;
      int issued = 0;
      pdl_wait();
      {
        int kb = u0 % KBT;
        for (int i = 0; i < pre; ++i) {
          load_x(i, kb);
          if (++kb == KBT) kb = 0;
        }
      }
      issued = pre;
      for (int i = pre; i < n_units; ++i) {
        const int s = i % S, use = i / S;
        if (!tc::mbar_wait(&empty_bar[s], (use - 1) & 1, a.status, a.wait_ns)) {
          aborted = true;
          break;
        }
        tc::mbar_expect_tx(&full_bar[s], stage_bytes);
        load_w(i, t_cur, kb_cur);
        load_x(i, kb_cur);
        if (++kb_cur == KBT) { kb_cur = 0; ++t_cur; }
        ++issued;
      }
      if (aborted) s_abort = 1;
      n_issued = issued;
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---------------- MMA issuer
      const uint32_t idesc = tc::idesc_bf16_f32(128, 2 * NP);
      int seg = 0;
      int u = u0;
      bool ok = true;
      while (u < u1 && ok) {
        const int seg_end = min(u1, (u / KBT + 1) * KBT);
        const int acc = seg & 1;
        if (seg >= 2 &&
            !tc::mbar_wait(&acce_bar[acc], ((seg >> 1) - 1) & 1, a.status, a.wait_ns)) {
          ok = false;
          break;
        }
        tc::tc_fence_after();
        const uint32_t d = tmem + (uint32_t)acc * acc_cols;
        const int seg_begin = u;
        for (; u < seg_end; ++u) {
          const int i = (int)(u - u0), s = i % S, use = i / S;
          if (!tc::mbar_wait(&full_bar[s], use & 1, a.status, a.wait_ns)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const uint32_t sa = tc::smem_u32(smem + (size_t)s * stage_bytes);
          const uint64_t da = tc::desc_sw128(sa);
          const uint64_t dh = tc::desc_sw128(sa + 16384);
          const bool first = (u == seg_begin);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk)   // 4 x K=16 per stage; +32 bytes = +2 in the desc
            tc::umma_bf16(d, da + 2 * kk, dh + 2 * kk, idesc, (first && kk == 0) ? 0u : 1u);
          tc::umma_commit(&empty_bar[s]);
        }
        if (!ok) break;   // an unfinished accumulator is never handed to the epilogue
        tc::umma_commit(&accf_bar[acc]);
        ++seg;
      }
      if (!ok) s_abort = 1;
      // every MMA issued here completes before TMEM is released (fixed limit)
      tc::umma_commit(&drain_bar);
      tc::mbar_wait(&drain_bar, 0, a.status);
    }
  } else {
    // ---------------- epilogue warps 2..5: TMEM lanes 32*(warp % 4) .. +31
    const int etid = threadIdx.x - 64;
    const int quarter = warp & 3;
    pdl_wait();
    int seg = 0;
    int u = u0;
    const int R = min(a.R, NP);
    if constexpr (kRegs) {   // what this block's rows need, while the accumulator fills
      const int ra = (c % SK) * R / SK, rb = (c % SK + 1) * R / SK;
      if (a.in_ss) input_row_scales(a, ra, rb - ra, s_rs, etid, kEpThreads);
      if (a.mode == EPI_QKV) qkv_rows(a, ra, rb - ra, s_qkv, etid, kEpThreads);
      tc::named_barrier(1, kEpThreads);
    } else if (a.in_ss) {   // once per block
      input_row_scales(a, 0, R, s_rs, etid, kEpThreads);
      tc::named_barrier(1, kEpThreads);
    }
    while (u < u1) {
      const int t = u / KBT;
      const int seg_end = min(u1, (t + 1) * KBT);
      const bool whole = (u % KBT) == 0 && seg_end == (t + 1) * KBT;
      const int acc = seg & 1;
      const bool ready = tc::mbar_wait(&accf_bar[acc], (seg >> 1) & 1, a.status, a.wait_ns);
      // the epilogue warps give up together or not at all: named barriers and warp-collective
      // TMEM loads follow
      if (tc::named_barrier_or(1, kEpThreads, !ready)) {
        s_abort = 1;
        break;
      }
      tc::tc_fence_after();
      const uint32_t d = tmem + (uint32_t)acc * acc_cols + ((uint32_t)(quarter * 32) << 16);
      const int slot = (t == u0 / KBT) ? 0 : 1;
      float* my_part = part + ((size_t)(c * 2 + slot) * NP) * 128;
      for (int r0 = 0; r0 < NP; r0 += kEpRows) {
        const int rows = min(kEpRows, NP - r0);
        for (int c0 = 0; c0 < rows; c0 += 16) {
          uint32_t v[16], w[16];
          tc::tmem_ld16_nowait(d + (uint32_t)(r0 + c0), v);
          tc::tmem_ld16_nowait(d + (uint32_t)(NP + r0 + c0), w);
          tc::tmem_wait_ld();
#pragma unroll
          for (int i = 0; i < 16; ++i)
            tileS[(c0 + i) * kTileLd + quarter * 32 + lane] =
                __uint_as_float(v[i]) + __uint_as_float(w[i]);
        }
        // cluster split-K: the partial stays in tileS (ep_rows == NP: one chunk) until the
        // cluster reduction at the end, whose barrier publishes it
        if (kRegs) continue;
        tc::named_barrier(1, kEpThreads);
        const int rt = max(0, min(rows, R - r0));
        if (SK > 0) {
          // (summed and finished at the end)
        } else if (whole) {
          tile_epilogue<__nv_bfloat16>(a, t * 128, r0, rt, tileS, kTileLd, s_rs + r0, etid,
                                       kEpThreads);
        } else {
          for (int i = etid; i < rt * 128; i += kEpThreads) {
            const int r = i >> 7, v = i & 127;
            my_part[(size_t)(r0 + r) * 128 + v] = tileS[r * kTileLd + v];
          }
        }
        tc::named_barrier(1, kEpThreads);
      }
      tc::tc_fence_before();
      tc::mbar_arrive(&acce_bar[acc]);   // accumulator drained: the MMA lane may reuse it
      if (!kRegs && !whole && SK == 0) {
        const int cf = unit_owner(t * KBT, U, C);
        const int cl = unit_owner((t + 1) * KBT - 1, U, C);
        // publish this block's partial and count it (one acquire-release atomic after the
        // barrier)
        tc::named_barrier(1, kEpThreads);
        // the last block to arrive sees every contributor's partial and finishes the tile
        if (etid == 0) s_last = (tc::atom_add_acq_rel_gpu(tile_cnt + t, 1) == cl - cf);
        tc::named_barrier(1, kEpThreads);
        if (s_last) {
          // scratch slot of every contributor: its first segment -> 0, its last -> 1
          for (int j = etid; j <= cl - cf; j += kEpThreads) {
            const int cc = cf + j;
            const int sl = (t == unit_start(cc, U, C) / KBT) ? 0 : 1;
            s_slot_off[j] = (cc * 2 + sl) * NP * 128;
          }
          tc::named_barrier(1, kEpThreads);
          const int ncontrib = cl - cf + 1;
          for (int r0 = 0; r0 < R; r0 += kEpRows) {
            const int rt = min(kEpRows, R - r0);
            // float4 groups: 32 per activation row; all contributors' loads in flight together
            for (int i = etid; i < rt * 32; i += kEpThreads) {
              const int off = (r0 + (i >> 5)) * 128 + (i & 31) * 4;
              float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
              int j = 0;
              for (; j + 4 <= ncontrib; j += 4) {
                float4 v[4];
#pragma unroll
                for (int q = 0; q < 4; ++q)
                  v[q] = __ldcg(reinterpret_cast<const float4*>(part + s_slot_off[j + q] + off));
#pragma unroll
                for (int q = 0; q < 4; ++q) {
                  sum.x += v[q].x; sum.y += v[q].y; sum.z += v[q].z; sum.w += v[q].w;
                }
              }
              for (; j < ncontrib; ++j) {
                const float4 v = __ldcg(reinterpret_cast<const float4*>(part + s_slot_off[j] + off));
                sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
              }
              *reinterpret_cast<float4*>(tileS + (i >> 5) * kTileLd + (i & 31) * 4) = sum;
            }
            tc::named_barrier(1, kEpThreads);
            tile_epilogue<__nv_bfloat16>(a, t * 128, r0, rt, tileS, kTileLd, s_rs + r0, etid,
                                         kEpThreads);
            tc::named_barrier(1, kEpThreads);
          }
          if (etid == 0) tile_cnt[t] = 0;
        }
      }
      u = seg_end;
      ++seg;
    }
    gave_up = u < u1;
  }
  if constexpr (kRegs) {
    // ---- cluster split-K reduction: rank r sums rows [r*R/SK, (r+1)*R/SK) of the SK partial
    //      tiles in rank order (distributed shared memory) and finishes them on registers: a lane
    //      is one output, in QKV both values of a RoPE pair. (Through a summed tile in shared
    //      memory and tile_epilogue it cost two more barriers and, in QKV, the rows' descriptors
    //      and pages after the sums.)
    tc::cluster_arrive();               // this block's partial tile is complete (release)
    tc::cluster_wait();                 // every block's is (acquire)
    // the closing barrier is met as soon as a warp's last sums are read: its second phase runs
    // while the epilogue writes
    bool arrived = false;
    if (warp >= 2 && !gave_up) {
      const int R = min(a.R, NP), r = c % SK, t = c / SK, w = warp & 3;
      const int ra = r * R / SK, rb = (r + 1) * R / SK;
      const uint32_t tile_s = tc::smem_u32(tileS);
      // sums of rows row .. row + NR - 1 of the share at tile columns v0 and v1, eight blocks'
      // loads in flight per row
      auto sums = [&](int row, int v0, int v1, auto& y0, auto& y1) {
        constexpr int NR = sizeof(y0) / sizeof(float);
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          y0[i] = y1[i] = 0.f;
          if (row + i >= rb) continue;   // warp-uniform
          const uint32_t at = tile_s + (uint32_t)((row + i) * kTileLd) * 4;
          for (int q0 = 0; q0 < SK; q0 += 8) {
            float a0[8], a1[8];
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              if (q0 + q >= SK) break;
              const uint32_t src = tc::map_cluster_rank(at, (uint32_t)(q0 + q));
              a0[q] = tc::ld_cluster_f32(src + v0 * 4);
              if (v1 >= 0) a1[q] = tc::ld_cluster_f32(src + v1 * 4);
            }
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              if (q0 + q >= SK) break;
              y0[i] += a0[q];
              if (v1 >= 0) y1[i] += a1[q];
            }
          }
        }
      };
      if (a.mode == EPI_RESID) {   // warp w: features 32 w ..
        for (int row = ra; row < rb; row += 4) {
          float y0[4], y1[4];
          sums(row, w * 32 + lane, -1, y0, y1);
          if (row + 4 >= rb) {
            tc::cluster_arrive();
            arrived = true;
          }
          finish_rows<EPI_RESID, 4>(a, t * 128 + w * 32 + lane, row, rb - row, y0, y1,
                                    s_rs + row - ra, s_qkv);
        }
      } else {   // QKV: warps w and w + 2 share 32 of the tile's 64 pairs, rows two by two
        const int pi = (w & 1) * 32 + lane;
        int v0 = pi, v1 = pi + 64;
        if (a.kv.hd == 64) {   // two heads of 32 pairs per tile
          v0 = pi + (pi & 32);
          v1 = v0 + 32;
        }
        for (int row = ra + (w >> 1) * 2; row < rb; row += 4) {
          float y0[2], y1[2];
          sums(row, v0, v1, y0, y1);
          if (row + 4 >= rb) {
            tc::cluster_arrive();
            arrived = true;
          }
          finish_rows<EPI_QKV, 2>(a, t * 64 + pi, row, rb - row, y0, y1, s_rs + row - ra,
                                  s_qkv + row - ra);
        }
      }
    }
    if (!arrived) tc::cluster_arrive();
    tc::cluster_wait();                 // no block leaves while its tile may still be read
  } else if (SK > 0) {
    // ---- the same with few rows per block: rank r sums rows [r*R/SK, (r+1)*R/SK) of the SK partial
    //      tiles in rank order (distributed shared memory) into a free pipeline stage and runs
    //      the epilogue on them
    // the epilogue warps agree on whether the block gave up (the two named barriers below
    // must be reached by all of them or by none)
    const bool none = warp >= 2 ? tc::named_barrier_or(1, kEpThreads, s_abort != 0) : true;
    tc::cluster_arrive();               // this block's partial tile is complete (release)
    tc::cluster_wait();                 // every block's is (acquire)
    const bool reduce = warp >= 2 && !none;
    const int R = min(a.R, NP), r = c % SK, t = c / SK;
    const int ra = r * R / SK, rb = (r + 1) * R / SK;
    float* red = reinterpret_cast<float*>(smem);   // stage 0 (idle): [rb - ra][kTileLd]
    if (reduce) {
      const int etid = threadIdx.x - 64;
      const uint32_t tile_s = tc::smem_u32(tileS);
      for (int i = etid; i < (rb - ra) * 32; i += kEpThreads) {
        const uint32_t off = ((ra + (i >> 5)) * kTileLd + (i & 31) * 4) * 4;
        float4 sum = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int q = 0; q < SK; ++q) {
          const float4 v = tc::ld_cluster_f32x4(tc::map_cluster_rank(tile_s + off, q));
          sum.x += v.x; sum.y += v.y; sum.z += v.z; sum.w += v.w;
        }
        *reinterpret_cast<float4*>(red + (i >> 5) * kTileLd + (i & 31) * 4) = sum;
      }
    }
    // this block has read the others' tiles (the sums above consumed every load): the
    // barrier's second phase runs while the epilogue writes
    tc::cluster_arrive();
    if (reduce) {
      const int etid = threadIdx.x - 64;
      tc::named_barrier(1, kEpThreads);
      if (rb > ra)
        tile_epilogue<__nv_bfloat16>(a, t * 128, ra, rb - ra, red, kTileLd, s_rs + ra, etid,
                                     kEpThreads);
    }
    tc::cluster_wait();                 // no block leaves while its tile may still be read
  }
  tc::tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && s_abort) {
    // a block that gave up waits for the copies it issued last to land before it leaves (the
    // earlier ones were consumed, so they have landed); fixed limit
    for (int i = max(0, n_issued - S); i < n_issued; ++i)
      tc::mbar_wait(&full_bar[i % S], (i / S) & 1, a.status);
  }
  if (warp == 1) tc::tmem_dealloc(tmem, 2 * acc_cols);
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
size_t g_static_smem = 4096;   // static shared memory of k_gemm_tc (queried at configuration)
int g_max_cluster = 8;         // 16 where non-portable clusters of k_gemm_tc are allowed

}  // namespace

bool tc_supported(const GemmArgs& a) {
  if (a.K % 64 || a.R < 1) return false;
  // 32-bit stream-K unit arithmetic and at most kMaxContrib blocks per tile
  const long long units = (long long)((a.n_virtual + 127) / 128) * (a.K / 64);
  if (a.K / 64 >= kMaxContrib || units * 4 * kPlanSMs >= (1LL << 31)) return false;
  for (int s = 0; s + 1 < a.n_seg; ++s)
    if (a.mode != EPI_SWIGLU && a.seg_rows[s] % 64) return false;
  return true;
}

TcPlan plan_tc(int K, int n_virtual, int R, int n_sm, int force_per_sm, int max_split,
               int cluster) {
  TcPlan p{};
  p.n_pad = (R + 15) / 16 * 16;
  p.tiles = (n_virtual + 127) / 128;
  p.kb_total = K / 64;
  const size_t stage = 16384 + 256 * (size_t)p.n_pad;
  // two blocks per SM when three stages fit in half the shared memory (228 KB per SM, less
  // each block's static part and the 1 KB the runtime reserves per block), else one; the
  // epilogue drains 16 activation rows at a time when that frees room for another stage
  const size_t half = 114 * 1024 - g_static_smem - 1024;
  auto fit = [&](size_t budget, int ep) {
    return (int)std::min<size_t>(kMaxStages, (budget - (size_t)ep * kTileLd * 4 - 1024) / stage);
  };
  int per_sm = 1;
  size_t budget = std::min<size_t>(220 * 1024, 227 * 1024 - g_static_smem);
  const int ep_big = std::min(p.n_pad, kEpRowsMax);
  if (force_per_sm >= 3) {   // more, shallower blocks (measurement aid)
    per_sm = force_per_sm;
    budget = (227 * 1024) / force_per_sm - 1024;
  } else if ((force_per_sm == 2 || force_per_sm == 0) && fit(half, 16) >= 3) {
    per_sm = 2;
    budget = half;
  }
  p.ep_rows = fit(budget, 16) > fit(budget, ep_big) ? 16 : ep_big;
  p.stages = fit(budget, p.ep_rows);
  // at most kMaxSplit blocks share a tile: the fixup then stays cheap next to the streaming
  const long long units = (long long)p.tiles * p.kb_total;
  p.ctas = (int)std::min<long long>(std::min<long long>(units, (long long)per_sm * n_sm),
                                    (long long)p.tiles * (max_split > 0 ? max_split : kMaxSplit));
  // few tiles: a cluster of S <= 12 blocks per tile, all tiles resident at once. Clusters are
  // placed whole within a GPC; on 152 SMs at two blocks each, grids of clusters past ~87 % of
  // the block slots no longer fit in one wave (measured), hence the cap.
  const int cap = per_sm * n_sm * 87 / 100;
  // (the whole partial tile, n_pad rows, stays in shared memory: two stages must still fit)
  const bool tile_fits = fit(budget, p.n_pad) >= 2;
  // Up to 12 blocks per tile while the grid stays within 64 % of the block slots (measured
  // at two blocks per SM, 7B draft down projection 2048 x 5504, 16 tiles: 8.43 us at 12
  // blocks against 9.02 us at 8; larger non-portable clusters or grids lose, e.g. 16 x 16
  // blocks: 14.3 us).
  const int wide = per_sm * n_sm * 64 / 100;
  int S = cluster;
  if (S < 0)
    S = (tile_fits && 2 * p.tiles <= cap)
            ? std::max(std::min(8, cap / p.tiles), std::min(12, wide / p.tiles))
            : 0;
  S = std::min(std::min(S, p.kb_total), g_max_cluster);
  if (S >= 2 && tile_fits) {
    p.cluster = S;
    p.ctas = p.tiles * S;
    p.ep_rows = p.n_pad;   // the whole partial tile stays in shared memory
    p.stages = fit(budget, p.ep_rows);
  } else if (cluster < 0 && max_split == 0 && p.tiles <= per_sm * n_sm &&
             10 * p.tiles >= 9 * n_sm) {
    // about one tile per SM or more, but too many for clusters: one block per whole tile (no
    // split, no fixup). Measured against stream-K over all 304 slots: 38.4 vs 41.2 us (7B
    // gate/up), 46.2 vs 55.2 us (7B LM head), 22.8 vs 25.2 us (draft LM head). The few tile counts
    // between (133 to 136 on 152 SMs) and those above the block slots run stream-K.
    p.ctas = p.tiles;
  }
  p.smem = (size_t)p.stages * stage + (size_t)p.ep_rows * kTileLd * 4 + 1024;
  return p;
}

size_t tc_scratch_floats(const TcPlan& p) {
  return p.cluster ? 0 : (size_t)p.ctas * 2 * p.n_pad * 128;
}

int encode_bf16_map(CUtensorMap* m, const void* base, uint64_t inner, uint64_t outer,
                    uint32_t box_inner, uint32_t box_outer) {
  if (!g_encode) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault,
                                         &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess || !fn)
      return -1;
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  }
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {inner * 2};
  cuuint32_t box[2] = {box_inner, box_outer};
  cuuint32_t estr[2] = {1, 1};
  const CUresult r = g_encode(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims,
                              strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                              CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                              CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? 0 : (int)r;
}

int configure_gemm_tc() {
  auto kernel = k_gemm_tc<true>;   // (the larger static part)
  cudaFuncAttributes fa;
  if (cudaFuncGetAttributes(&fa, kernel) != cudaSuccess) return -1;
  g_static_smem = fa.sharedSizeBytes;
  // plans use at most 220 KB + 1 KB of alignment slack; a block has at most 227 KB in all
  const int dyn = (int)std::min<size_t>(220 * 1024 + 1024, 227 * 1024 - fa.sharedSizeBytes);
  bool nonportable = true;
  int rc = 0;
  for (auto k : {k_gemm_tc<false>, k_gemm_tc<true>}) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) != cudaSuccess)
      nonportable = false;
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, dyn) != cudaSuccess)
      rc = -1;
  }
  cudaGetLastError();
  g_max_cluster = nonportable ? 16 : 8;
  return rc;
}

void launch_gemm_tc(const TcMaps& maps, const GemmArgs& a, const TcPlan& p, float* part,
                    int* tile_cnt, cudaStream_t s) {
  // A cluster's rows are finished on registers where each of its blocks has enough of them: three
  // for QKV (7B verify pass, 20 rows over 5 blocks: 14.8 -> 13.9 us; at two rows, each a round trip
  // of 4-byte remote loads, the small model's requests lose 1.3 %), two for the residual projections
  // (O 11.7 -> 11.1, down 20.2 -> 19.5; the draft's 4 rows over 12 blocks lose: O 4.9 -> 5.6).
  // Gate/up keeps the tile (16 rows over 3 blocks lose 1.5 us a launch).
  const bool regs = p.cluster && ((a.mode == EPI_QKV && a.R >= 3 * p.cluster) ||
                                  (a.mode == EPI_RESID && a.R >= 2 * p.cluster));
  auto kernel = regs ? k_gemm_tc<true> : k_gemm_tc<false>;
  if (p.cluster)
    launch_pdl_cluster(kernel, dim3(p.ctas), dim3(kThreads), p.smem, p.cluster, s, maps, a, p,
                       part, tile_cnt);
  else
    launch_pdl(kernel, dim3(p.ctas), dim3(kThreads), p.smem, s, maps, a, p, part, tile_cnt);
}

}  // namespace cdsl
