// gemm_pair.cu -- projection GEMMs of more than kPairRows activation rows on pairs of SMs
// (tcgen05 cta_group::2).
//
// Swap-AB as in gemm_tc.cu: the weights are the M operand, the activation rows (their hi and
// lo bf16 planes) the N operand. A pair of CTAs works on one tile of 256 weight rows x N
// activation rows (N a multiple of 32, at most 256): each CTA stages its 128 weight rows and
// its half of the N rows of both planes, and one MMA of M = 256 reads both CTAs' shared memory
// and accumulates into both CTAs' TMEM (128 rows x N columns each). QKV and gate/up tiles hold
// two such accumulators, fed from the same activations: a RoPE pair's first and second halves,
// a feature's gate and up rows. The two values an output needs then sit in one thread's
// registers, and no epilogue exchanges values between threads.
//
// What bounds it: above about 100 rows the tensor pipe (hi and lo double the MMA work). A
// 64-wide K block takes 4 N clocks per accumulator; a CTA fetches 16 KB of weights and 128 N
// bytes of activations for it, 48 bytes per clock at N = 256, where one CTA per tile needs 80
// (16 KB + 256 N bytes) and had room for two stages in flight: here it is four or more (three where
// a tile with two accumulators takes 256 rows).
//
// The tensor core truncates when it adds into an fp32 accumulator, so a chain of MMAs shrinks
// the sum: by 1.4e-7 per 64-wide K block, or 6e-8 where the lo plane accumulates apart (planes == 2,
// where TMEM has room), over K = 4096 in one chain 8.8e-6 where the hi/lo split of the activations
// leaves 2.4e-6. A tile's K range is therefore accumulated in chains of at most chain_blocks() blocks,
// into two TMEM accumulator sets in turn; the epilogue warps add each finished chain to fp32 sums in
// their registers (rounded to nearest) while the next one accumulates (k_gemm_pair<.., true>). A K
// range of one chain is finished straight from TMEM (<.., false>). The bound is the rounding error
// of a serial fp32 sum of K products, 1.8e-8 sqrt(K) as measured on the CUDA-core GEMM: 1.1e-6 at
// K = 4096, in chains of 8 blocks, or 12 with lo apart (7e-7). Logits against 64 bits (mean of six seeds;
// the kernels before, which took one chain per tile up to 256 rows and the CUDA cores above): 13B
// slice at 224 rows 1.5e-5 (2.7e-5), 7B slice at 320 rows 1.3e-5 (1.4e-5), small model at 640 rows
// 6.3e-6 (6.4e-6). Gate/up tiles of 129 to 256 rows in one chain of all 80 blocks, which leave TMEM
// no room for a second set, were faster (13B, 224 rows: 90 us against 126) but 2.3e-5 off each.
//
// Schedule (plan_pair): the tiles of a launch are dealt to the pairs in turn (persistent), or,
// with few tiles, a cluster of S pairs splits a tile's K range: the partial tiles go to shared
// memory (the pipeline's stages, idle by then), every CTA of the cluster sums its share of the
// activation rows over the S partials in order through distributed shared memory
// (deterministic) and finishes them. No partial tile goes to global memory.
//
// Warp 0 streams weights and activations with TMA; every copy of a pair signals the leader's
// (even CTA's) stage barrier, which counts both CTAs' bytes. Warp 1 of the leader issues the
// MMAs; the commits arrive on both CTAs' barriers. The other warps drain TMEM (warp w reads lanes
// 32 (w % 4) .. + 31; the warps of the same lanes take groups of columns in turn) and run the
// epilogue on registers: a lane is one feature, so every access of a warp is 32 consecutive
// features.
//
// Programmatic dependent launch and bounded waits as in gemm_tc.cu. A pair one of whose waits
// ran out lands the copies of both its CTAs before either leaves: the leader completes the
// transaction counts of stages that only one of them filled.
#include <algorithm>
#include <cmath>

#include "gemm.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace cdsl {
namespace {

constexpr int kStagesMax = 8;
constexpr int kEpWarps = 16;          // (256 rows, 13B O: 30.1 us with 8, 28.1 with 12, 27.4 with 16)
constexpr int kEpThreads = kEpWarps * 32;
constexpr int kThreads = 64 + kEpThreads;
constexpr int kGroups = kEpWarps / 4;   // warps that share 32 TMEM lanes
constexpr int kChunks = 16 / kGroups;   // groups of 16 columns a warp sums
constexpr int kNMax = 256;
constexpr int kSplitMax = 4;         // pairs per cluster (8 CTAs: the portable cluster size)
constexpr size_t kSmemMax = 216 * 1024;   // dynamic shared memory a plan may use

// 64-wide K blocks per accumulation chain, at most (its truncation against the rounding of a serial
// fp32 sum of K products: see above; 4 where that would ask for fewer). Half as many again with lo
// apart: twice as many keep the bound too, but the small model's short prompts, whose projections of
// up to 128 rows had run in splits of 4 blocks, were 1 % further off than before (logits 6.13e-6
// against 6.07e-6, now 6.05e-6; its first step of 32 prompts 7.64 -> 7.88 ms).
int chain_blocks(int K, int planes) {
  const int one = std::max(4, (int)(0.131 * std::sqrt((double)K)));
  return planes == 2 ? one * 3 / 2 : one;
}

// Accumulators per tile: gate and up, or the two halves of RoPE pairs.
constexpr int accs(int mode) { return mode == EPI_SWIGLU || mode == EPI_QKV ? 2 : 1; }

__host__ __device__ __forceinline__ uint32_t pow2_cols(int n) {
  uint32_t c = 32;
  while (c < (uint32_t)n) c <<= 1;
  return c;
}

// 16 columns of an accumulator, plus those of its lo plane `lo` columns on where it has one.
__device__ __forceinline__ void load_sums(uint32_t taddr, uint32_t lo, float (&v)[16]) {
  tc::tmem_ld16(taddr, v);
  if (lo) {
    float l[16];
    tc::tmem_ld16(taddr + lo, l);
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] += l[i];
  }
}

// finish_rows of 16 rows from c on (of the tile's `rows`, the first of which is r0), kFin at a time.
template <int MODE>
__device__ __forceinline__ void finish_sums(const GemmArgs& a, int L, int r0, int c,
                                            int rows, const float (&v0)[16],
                                            const float (&v1)[16], const float* rs,
                                            const QkvRow* qr) {
  constexpr int kFin = MODE == EPI_QKV || MODE == EPI_RESID ? 8 : 16;
#pragma unroll
  for (int h = 0; h < 16; h += kFin) {
    float y0[kFin], y1[kFin];
#pragma unroll
    for (int i = 0; i < kFin; ++i) {
      y0[i] = v0[h + i];
      y1[i] = v1[h + i];
    }
    finish_rows<MODE, kFin>(a, L, r0 + c + h, rows - c - h, y0, y1, rs + c + h,
                            qr + (MODE == EPI_QKV ? c + h : 0));
  }
}

// kSeg: a tile's K range in several accumulation chains, summed in registers (MT * N <= 256).
template <int MODE, bool kSeg>
__global__ void __launch_bounds__(kThreads, 1)
    k_gemm_pair(const __grid_constant__ TcMaps maps, const __grid_constant__ GemmArgs a,
                const PairPlan p) {
  constexpr int MT = accs(MODE);
  extern __shared__ uint8_t smem_raw[];
  const LaunchStamp stamp(a.stamp);
  __shared__ __align__(8) uint64_t full_bar[kStagesMax];    // leader: both CTAs' copies landed
  __shared__ __align__(8) uint64_t empty_bar[kStagesMax];   // the stage's MMAs have completed
  __shared__ __align__(8) uint64_t accf_bar[2];             // accumulator set complete
  __shared__ __align__(8) uint64_t acce_bar[2];             // leader: drained by both CTAs
  __shared__ __align__(8) uint64_t drain_bar;               // leader: all MMAs completed
  __shared__ __align__(8) uint64_t land_bar;                // odd CTA: the pair's copies landed
  __shared__ uint32_t tmem_base;
  __shared__ int s_abort, s_peer_abort, s_peer_issued;
  __shared__ float s_rs[kNMax];
  __shared__ QkvRow s_qkv[MODE == EPI_QKV ? kNMax : 1];

  uint8_t* smem = smem_raw + ((1024 - (tc::smem_u32(smem_raw) & 1023)) & 1023);
  const int N = p.n, ST = p.stages, KBT = p.kb_total, S = p.split, NT = p.n_tiles;
  const uint32_t stage_bytes = MT * 16384u + 128u * N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = blockIdx.x % (2 * S);        // in the cluster: pair (K split) and half of it
  const int half = rank & 1, q = rank >> 1;
  const uint32_t lead = rank & ~1, peer = rank ^ 1;
  const uint16_t pair_mask = (uint16_t)(3u << lead);
  const int cid = blockIdx.x / (2 * S), CN = gridDim.x / (2 * S);
  const int tiles = p.m_tiles * NT;
  const int kb0 = q * KBT / S, kb1 = (q + 1) * KBT / S, nkb = kb1 - kb0;
  const int my_tiles = cid < tiles ? (tiles - cid + CN - 1) / CN : 0;
  const int nseg = kSeg ? (nkb + p.chain - 1) / p.chain : 1;   // accumulation chains per tile
  const int n_units = my_tiles * nkb;
  const int pre = min(ST, n_units);
  const uint32_t cols = pow2_cols(p.bufs * p.planes * MT * N);
  const uint32_t set = (uint32_t)(p.planes * MT * N);       // columns of an accumulator set and
  const uint32_t lo = (uint32_t)((p.planes - 1) * MT * N);  //   of its lo plane's start

  const uint32_t lead_full = tc::map_cluster_rank(tc::smem_u32(&full_bar[0]), lead);
  uint64_t pol = 0;
  auto load_w = [&](int i, int tm, int kb) {
    uint8_t* st = smem + (size_t)(i % ST) * stage_bytes;
    const uint32_t bar = lead_full + 8u * (uint32_t)(i % ST);
    if constexpr (MODE == EPI_QKV) {
      const int hd = a.kv.hd, hh = hd >> 1, per = 128 / hh;   // heads per CTA
      const int H = a.n_heads, KVH = a.kv.kvh;
#pragma unroll 1
      for (int j = 0; j < per; ++j) {
        const int head = min((tm * 2 + half) * per + j, H + 2 * KVH - 1);   // (past the last:
        const int m = head < H ? 0 : head < H + KVH ? 1 : 2;                //  never stored)
        const int row = (head - (m == 0 ? 0 : m == 1 ? H : H + KVH)) * hd;
        tc::tma_load_2d_pair(st + j * hh * 128, &maps.w[m], kb * 64, row, bar, pol);
        tc::tma_load_2d_pair(st + 16384 + j * hh * 128, &maps.w[m], kb * 64, row + hh, bar, pol);
      }
    } else {
      const int row = tm * 256 + half * 128;
#pragma unroll
      for (int m = 0; m < MT; ++m)
        tc::tma_load_2d_pair(st + 16384 * m, &maps.w[m], kb * 64, row, bar, pol);
    }
  };
  auto load_x = [&](int i, int tn, int kb) {
    uint8_t* st = smem + (size_t)(i % ST) * stage_bytes + MT * 16384;
    const uint32_t bar = lead_full + 8u * (uint32_t)(i % ST);
    const int row = tn * N + half * (N / 2);
    tc::tma_load_2d_pair(st, &maps.xh, kb * 64, row, bar);
    tc::tma_load_2d_pair(st + N * 64, &maps.xl, kb * 64, row, bar);
  };

  if (threadIdx.x == 0) {
    for (int m = 0; m < 3; ++m) tc::tma_prefetch_map(&maps.w[m]);
    tc::tma_prefetch_map(&maps.xh);
    tc::tma_prefetch_map(&maps.xl);
    for (int s = 0; s < ST; ++s) {
      tc::mbar_init(&full_bar[s], 1);
      tc::mbar_init(&empty_bar[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      tc::mbar_init(&accf_bar[i], 1);
      tc::mbar_init(&acce_bar[i], 2 * kEpWarps);
    }
    tc::mbar_init(&drain_bar, 1);
    tc::mbar_init(&land_bar, 1);
    s_abort = s_peer_abort = s_peer_issued = 0;
    tc::fence_mbar_init();
    tc::fence_proxy_async();
  }
  if (warp == 1) tc::tmem_alloc_pair(&tmem_base, cols);
  tc::tc_fence_before();
  __syncthreads();
  tc::cluster_arrive();   // the barriers of every CTA of the cluster are initialized
  tc::cluster_wait();
  tc::tc_fence_after();
  pdl_launch_dependents();
  const uint32_t tmem = tmem_base;
  int n_issued = 0;       // (thread 0) units whose copies were issued

  if (warp == 0) {
    if (lane == 0) {
      // ---------------- TMA producer: the first ring's weights do not depend on the previous
      //                  kernel
      pol = NT == 1 ? tc::policy_evict_first() : tc::policy_evict_normal();
      int tile = cid, kb = kb0;   // next unit's
      for (int i = 0; i < pre; ++i) {
        if (half == 0) tc::mbar_expect_tx(&full_bar[i], 2 * stage_bytes);
        load_w(i, tile / NT, kb);
        if (++kb == kb1) { kb = kb0; tile += CN; }
      }
      pdl_wait();
      {
        int t2 = cid, k2 = kb0;
        for (int i = 0; i < pre; ++i) {
          load_x(i, t2 % NT, k2);
          if (++k2 == kb1) { k2 = kb0; t2 += CN; }
        }
      }
      n_issued = pre;
      for (int i = pre; i < n_units; ++i) {
        const int s = i % ST, use = i / ST;
        if (!tc::mbar_wait(&empty_bar[s], (use - 1) & 1, a.status, a.wait_ns)) {
          s_abort = 1;
          break;
        }
        if (half == 0) tc::mbar_expect_tx(&full_bar[s], 2 * stage_bytes);
        load_w(i, tile / NT, kb);
        load_x(i, tile % NT, kb);
        if (++kb == kb1) { kb = kb0; tile += CN; }
        ++n_issued;
      }
    }
  } else if (warp == 1) {
    if (half == 0 && lane == 0) {
      // ---------------- MMA issuer (the leader's)
      const uint32_t idesc = tc::idesc_bf16_f32(256, N);
      bool ok = true;
      int i = 0;
      for (int g = 0; g < my_tiles * nseg && ok; ++g) {   // accumulation chains, in tile order
        const int buf = g % p.bufs;
        if (g >= p.bufs &&
            !tc::mbar_wait(&acce_bar[buf], (g / p.bufs - 1) & 1, a.status, a.wait_ns)) {
          ok = false;
          break;
        }
        tc::tc_fence_after();
        const uint32_t d = tmem + (uint32_t)buf * set;
        const int seg = g % nseg, len = (seg + 1) * nkb / nseg - seg * nkb / nseg;
        for (int kb = 0; kb < len; ++kb, ++i) {
          const int s = i % ST, use = i / ST;
          if (!tc::mbar_wait(&full_bar[s], use & 1, a.status, a.wait_ns)) {
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const uint32_t sa = tc::smem_u32(smem + (size_t)s * stage_bytes);
          const uint64_t dh = tc::desc_sw128(sa + MT * 16384);
          const uint64_t dl = tc::desc_sw128(sa + MT * 16384 + N * 64);
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {   // K = 16 per MMA: +32 bytes = +2 in the descriptor
#pragma unroll
            for (int m = 0; m < MT; ++m) {
              const uint64_t da = tc::desc_sw128(sa + 16384 * m) + 2 * kk;
              tc::umma_bf16_pair(d + m * N, da, dh + 2 * kk, idesc, (kb | kk) ? 1u : 0u);
              tc::umma_bf16_pair(d + lo + m * N, da, dl + 2 * kk, idesc, (kb | kk | !lo) ? 1u : 0u);
            }
          }
          tc::umma_commit_pair(&empty_bar[s], pair_mask);
        }
        if (!ok) break;   // an unfinished accumulator is never handed to the epilogue
        tc::umma_commit_pair(&accf_bar[buf], pair_mask);
      }
      if (!ok) s_abort = 1;
      // every MMA issued here completes before the pair's TMEM is released (fixed limit)
      tc::umma_commit_pair(&drain_bar, (uint16_t)(1u << rank));
      tc::mbar_wait(&drain_bar, 0, a.status);
    }
  } else {
    // ---------------- epilogue warps
    const int etid = threadIdx.x - 64, quarter = warp & 3, cg = (warp - 2) >> 2;
    const int L = half * 128 + quarter * 32 + lane;
    const uint32_t acce0 = tc::map_cluster_rank(tc::smem_u32(&acce_bar[0]), lead);
    pdl_wait();
    int have = -1;   // N tile whose row scales and destinations are in shared memory
    int g = 0;
    bool ok = true;
    float* const part = reinterpret_cast<float*>(smem) + quarter * 32 + lane;   // (S > 1)
#pragma unroll 1
    for (int tile = cid; tile < tiles; tile += CN) {
      const int tm = tile / NT, tn = tile % NT;
      const int r0 = tn * N, rows = min(N, a.R - r0);
      if (tn != have && (a.in_ss || MODE == EPI_QKV)) {   // while the accumulator fills
        tc::named_barrier(1, kEpThreads);   // the previous tile's readers are done
        if (a.in_ss) input_row_scales(a, r0, rows, s_rs, etid, kEpThreads);
        if (MODE == EPI_QKV) qkv_rows(a, r0, rows, s_qkv, etid, kEpThreads);
        tc::named_barrier(1, kEpThreads);
        have = tn;
      }
      if constexpr (!kSeg) {
        const int buf = g % p.bufs;
        const bool ready = tc::mbar_wait(&accf_bar[buf], (g / p.bufs) & 1, a.status, a.wait_ns);
        if (tc::named_barrier_or(1, kEpThreads, !ready)) {   // all give up together or none does
          s_abort = 1;
          break;
        }
        tc::tc_fence_after();
        const uint32_t d = tmem + (uint32_t)buf * set + ((uint32_t)(quarter * 32) << 16);
        if (S == 1) {
          for (int c = cg * 16; c < rows; c += 16 * kGroups) {
            float y0[16], y1[16];
            load_sums(d + c, lo, y0);
            if constexpr (MT == 2) load_sums(d + N + c, lo, y1);
            finish_sums<MODE>(a, tm * 256 + L, r0, c, rows, y0, MT == 2 ? y1 : y0, s_rs, s_qkv);
          }
        }   // (split K: below, straight from TMEM)
        tc::tc_fence_before();
        __syncwarp();
        if (lane == 0) tc::mbar_arrive_cluster(acce0 + 8u * (uint32_t)buf);
        ++g;
      } else {
        // sums of this warp's column groups: group cg + 4 (j / MT) of accumulator j % MT
        float acc[kChunks][16];
#pragma unroll
        for (int j = 0; j < kChunks; ++j)
#pragma unroll
          for (int i = 0; i < 16; ++i) acc[j][i] = 0.f;
#pragma unroll 1
        for (int seg = 0; seg < nseg; ++seg, ++g) {
          const int buf = g % p.bufs;
          const bool ready =
              tc::mbar_wait(&accf_bar[buf], (g / p.bufs) & 1, a.status, a.wait_ns);
          if (tc::named_barrier_or(1, kEpThreads, !ready)) {
            s_abort = 1;
            ok = false;
            break;
          }
          tc::tc_fence_after();
          const uint32_t d = tmem + (uint32_t)buf * set + ((uint32_t)(quarter * 32) << 16);
#pragma unroll
          for (int j = 0; j < kChunks; ++j) {
            const int c = 16 * (cg + kGroups * (j / MT));
            if (c < rows) {   // warp-uniform
              float v[16];
              load_sums(d + (j % MT) * N + c, lo, v);
#pragma unroll
              for (int i = 0; i < 16; ++i) acc[j][i] += v[i];
            }
          }
          tc::tc_fence_before();
          __syncwarp();
          if (lane == 0) tc::mbar_arrive_cluster(acce0 + 8u * (uint32_t)buf);
        }
        if (!ok) break;
        if (S == 1) {
#pragma unroll
          for (int j = 0; j < kChunks; j += MT) {
            const int c = 16 * (cg + kGroups * (j / MT));
            if (c < rows)
              finish_sums<MODE>(a, tm * 256 + L, r0, c, rows, acc[j], acc[j + MT - 1], s_rs, s_qkv);
          }
        } else {
#pragma unroll
          for (int j = 0; j < kChunks; ++j) {
            const int c = 16 * (cg + kGroups * (j / MT));
            if (c < rows) {
#pragma unroll
              for (int i = 0; i < 16; ++i) part[(size_t)((j % MT) * N + c + i) * 128] = acc[j][i];
            }
          }
        }
      }
    }
  }
  if (S > 1) {
    // ---- split K (one tile per cluster): the partial tiles go to shared memory, [accumulator][row]
    //      [128 features], and CTA q of each half finishes rows [q n / S, (q + 1) n / S) of its 128
    //      weight rows
    const bool gave_up =
        warp >= 2 ? tc::named_barrier_or(1, kEpThreads, s_abort != 0) : true;
    const int quarter = warp & 3, cg = (warp - 2) >> 2;
    const int tm = cid / NT, tn = cid % NT;
    const int r0 = tn * N, rows = min(N, a.R - r0);
    const int L = half * 128 + quarter * 32 + lane;
    const uint32_t mine = tc::smem_u32(smem) + (quarter * 32 + lane) * 4;
    if (!kSeg && !gave_up) {
      float* const part = reinterpret_cast<float*>(smem) + quarter * 32 + lane;
      const uint32_t d = tmem + ((uint32_t)(quarter * 32) << 16);
      tc::tc_fence_after();
      for (int c = cg * 16; c < rows; c += 16 * kGroups) {
#pragma unroll
        for (int m = 0; m < MT; ++m) {
          float y[16];
          load_sums(d + m * N + c, lo, y);
#pragma unroll
          for (int i = 0; i < 16; ++i) part[(size_t)(m * N + c + i) * 128] = y[i];
        }
      }
    }
    tc::cluster_arrive();   // this CTA's partial is complete (release)
    tc::cluster_wait();     // every CTA's is (acquire)
    if (!gave_up) {
      const int ra = q * rows / S, rb = (q + 1) * rows / S;
      for (int c = ra + cg * 8; c < rb; c += 8 * kGroups) {
        float y0[8], y1[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) y0[i] = y1[i] = 0.f;
        for (int s = 0; s < S; ++s) {
          const uint32_t src = tc::map_cluster_rank(mine, (uint32_t)(2 * s + half)) + c * 512;
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const int ci = min(i, rb - 1 - c) * 512;   // (past the share: any row, unused)
            y0[i] += tc::ld_cluster_f32(src + ci);
            if constexpr (MT == 2) y1[i] += tc::ld_cluster_f32(src + N * 512 + ci);
          }
        }
        finish_rows<MODE, 8>(a, tm * 256 + L, r0 + c, min(8, rb - c), y0, y1, s_rs + c,
                             s_qkv + (MODE == EPI_QKV ? c : 0));
      }
    }
  }
  // ---- no CTA leaves while another may still reach its shared memory or its barriers
  tc::tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0) {
    if (half == 1) tc::st_cluster_s32(tc::map_cluster_rank(tc::smem_u32(&s_peer_issued), peer), n_issued);
    if (s_abort) tc::st_cluster_s32(tc::map_cluster_rank(tc::smem_u32(&s_peer_abort), peer), 1);
  }
  tc::cluster_arrive();
  tc::cluster_wait();
  if (threadIdx.x == 0 && (s_abort || s_peer_abort)) {
    // copies in flight land before the pair leaves (the earlier ones were consumed); fixed limit
    if (half == 0) {
      const int mine = n_issued, theirs = s_peer_issued, most = max(mine, theirs);
      for (int i = max(0, most - ST); i < most; ++i) {
        const int s = i % ST;
        if (i >= mine) tc::mbar_expect_tx(&full_bar[s], stage_bytes);          // only the peer's
        else if (i >= theirs) tc::mbar_complete_tx(&full_bar[s], stage_bytes);  // only this one's
        tc::mbar_wait(&full_bar[s], (i / ST) & 1, a.status);
      }
      tc::mbar_arrive_cluster(tc::map_cluster_rank(tc::smem_u32(&land_bar), peer));
    } else {
      tc::mbar_wait(&land_bar, 0, a.status);
    }
  }
  __syncthreads();
  if (warp == 1) tc::tmem_dealloc_pair(tmem, cols);
}

ClusterFit g_fit;   // cluster residency with a plan's largest shared memory (configure_gemm_pair)

template <typename F>
void for_modes(F&& f) {
  f(k_gemm_pair<EPI_STORE, false>);
  f(k_gemm_pair<EPI_STORE, true>);
  f(k_gemm_pair<EPI_RESID, false>);
  f(k_gemm_pair<EPI_RESID, true>);
  f(k_gemm_pair<EPI_SWIGLU, false>);
  f(k_gemm_pair<EPI_SWIGLU, true>);
  f(k_gemm_pair<EPI_QKV, false>);
  f(k_gemm_pair<EPI_QKV, true>);
}

}  // namespace

PairPlan plan_pair(int mode, int K, int n_virtual, int R) {
  const int MT = accs(mode);
  const int m_tiles = (n_virtual + 256 * MT - 1) / (256 * MT), KBT = K / 64;
  PairPlan best{};
  double best_cost = -1;
  const int nt_min = (R + kNMax - 1) / kNMax;
  // (tiles of 128 rows are always among them: two accumulators of more rows may not be allowed)
  const int nt_max = std::max(nt_min + 7, (R + 127) / 128);
  for (int nt = nt_min; nt <= nt_max; ++nt) {
    const int N = ((R + nt - 1) / nt + 31) / 32 * 32;
    if (N > kNMax || (nt > nt_min && N < 32) || (nt - 1) * N >= R) continue;
    const size_t stage = MT * 16384 + 128 * (size_t)N;
    const int tiles = m_tiles * nt;
    for (int S = 1; S <= kSplitMax; ++S) {
      if (S > 1 && S > KBT) continue;
      const int slots = g_fit.active[2 * S];
      if (slots < 1 || (S > 1 && tiles > slots)) continue;
      const int clusters = std::min(tiles, slots);
      const int waves = (tiles + clusters - 1) / clusters;
      // One accumulation chain where that is short enough, its lo plane apart where TMEM has room
      // (rather than a second set), and a second set to fill while one drains where there are
      // several tiles and room for both. Else several chains, which need two sets.
      const int nkb = (KBT + S - 1) / S;
      int planes = 2 * MT * N <= 512 ? 2 : 1, bufs = waves > 1 && 4 * MT * N <= 512 ? 2 : 1;
      const bool seg = nkb > chain_blocks(K, planes);
      if (seg) {
        if (2 * MT * N > 512) continue;
        bufs = 2;
        planes = 4 * MT * N <= 512 ? 2 : 1;
      }
      const int chain = chain_blocks(K, planes);
      const int stages = (int)std::min<size_t>(kStagesMax, (kSmemMax - 1024) / stage);
      if (S > 1 && (size_t)MT * N * 512 > stages * stage) continue;   // its partial tiles reuse them
      // Estimated clocks, fitted to 1,500 measured plans (19 projection shapes, 72 to 1024 rows,
      // chains of up to 16 blocks; with the chains as they are the chosen plan is on average
      // 1.5 % slower than the fastest of its shape and row count, 21 % at most, over 3,027 plans of
      // 24 shapes): a K block costs the MMAs or the fetch of its operands (36
      // bytes per clock and SM, 5,250 in all), the launch at least its weights at 22 bytes per
      // clock and active SM; the last tile's epilogue is never hidden, the earlier ones' only
      // where a second accumulator set fills meanwhile; a split adds the exchange of the
      // partials, each CTA some of the launch.
      const int ctas = clusters * 2 * S;
      const double kb = std::max(4.1 * MT * N, stage * std::max(1 / 36.5, ctas / 5250.0));
      const double ep = 20.0 * MT * N;
      double cost = (double)waves * nkb * kb;
      cost = std::max(cost, 2.0 * n_virtual * K / (22.0 * ctas)) + 33.0 * ctas;
      if (seg) cost += 5500;
      if (S == 1) cost += bufs == 1 ? waves * ep : ep;
      else cost += 260.0 * S + 21.0 * MT * N + 0.2 * ep / S;
      if (best_cost < 0 || cost < best_cost) {
        best_cost = cost;
        best = PairPlan{N, nt, m_tiles, KBT, S, stages, bufs, seg, chain, planes,
                        clusters * 2 * S, (size_t)stages * stage + 1024};
      }
    }
  }
  return best;
}

int configure_gemm_pair() {
  int rc = 0;
  for_modes([&](auto k) {
    if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax) !=
        cudaSuccess)
      rc = -1;
  });
  cudaGetLastError();
  if (rc) return rc;
  fill_cluster_fit(&g_fit, k_gemm_pair<EPI_STORE, false>, kThreads, kSmemMax, 2 * kSplitMax);
  return g_fit.active[2] > 0 ? 0 : -1;
}

int pair_box_rows(int mode, int hd) { return mode == EPI_QKV ? hd / 2 : 128; }

void launch_gemm_pair(const TcMaps& maps, const GemmArgs& a, const PairPlan& p, cudaStream_t s) {
  auto go = [&](auto k) {
    launch_pdl_cluster(k, dim3(p.ctas), dim3(kThreads), p.smem, 2 * p.split, s, maps, a, p);
  };
  switch (a.mode) {
    case EPI_STORE: p.seg ? go(k_gemm_pair<EPI_STORE, true>) : go(k_gemm_pair<EPI_STORE, false>); break;
    case EPI_RESID: p.seg ? go(k_gemm_pair<EPI_RESID, true>) : go(k_gemm_pair<EPI_RESID, false>); break;
    case EPI_SWIGLU:
      p.seg ? go(k_gemm_pair<EPI_SWIGLU, true>) : go(k_gemm_pair<EPI_SWIGLU, false>);
      break;
    default: p.seg ? go(k_gemm_pair<EPI_QKV, true>) : go(k_gemm_pair<EPI_QKV, false>); break;
  }
}

}  // namespace cdsl
