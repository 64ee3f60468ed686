// attention_tc.cu -- attention of the prefill and verify passes of bf16 models on the
// 5th-generation tensor cores (tcgen05 MMA into TMEM).
//
// The pass is split as in attention.cu (attn_layout.cuh): a thread-block cluster of up to 16
// blocks owns one (prompt, KV head, query block), and the chunks of 64 key slots that hold
// keys (prefix positions, then the query block's beam tails) are dealt to its blocks in turn.
// A query block holds up to 128 query vectors -- the MMA's M -- so the 7B verify pass (80
// query vectors per KV head) is one block per chunk and KV head.
//
// Per chunk, with every operand a K-major bf16 tile in 128-byte-swizzled shared memory:
//   S = Q K^T      M = 128 query vectors, N = 64 keys, K = head_dim  -> TMEM columns [0, 64)
//   O += P V       M = 128 query vectors, N = head_dim, K = 64 keys   -> TMEM columns [64, ..)
//                  (three planes: O = P V, added up in registers)
// fp32 inputs from bf16 operands: every fp32 input x is split into planes. Verify passes take two,
// hi = bf16(x) and lo = bf16(x - hi), and each product is hi.hi + hi.lo + lo.hi (lo.lo, about 2^-18
// of the product, is dropped). Prefill passes, whose K/V cache carries every later step and which
// otherwise run in fp32 on the CUDA cores, take three (x to 2^-25) and the six products down to
// lo.hi. Every MMA truncates the sum that it adds to: the small products therefore go first, and in a prefill pass a chunk's P V
// starts anew and is added to fp32 sums in registers, rounded to nearest. Output of 1024 rows at
// 3072 to 4096 keys, against 64 bits: 2.5e-6 of its norm, as of the CUDA-core kernel (nearly all of
// it the rounding of the output to hi and lo planes); with Q and K in two planes and one chain over
// the chunks 9.8e-6, and 2.7e-5 at scores of standard deviation 25 (2.6e-6, CUDA cores 3.2e-6). It
// costs a tenth of the launch: 792 -> 891 us (CUDA cores 2235). The K/V cache stays fp32 in HBM; the
// block converts each chunk while staging it (rows of keys: the score product's K-major B operand,
// and the P V product's MN-major one). Staging is software-pipelined: the next chunk's K rows are
// loaded into registers while this chunk's softmax runs and stored once its P V has completed. Q
// is split once per block, pre-scaled by log2(e) / sqrt(head_dim) (scores in base 2).
//
// What bounds it: the chain of a chunk's phases (loads, conversion, score MMAs, softmax, P V), 6 us
// on eight warps with DRAM and the tensor pipe both below 10 %. Two groups of eight warps work on
// alternate chunks of the block, each with its own K, V and P in shared memory (P over K) and its own
// S, O and softmax state; their partials are added at the end. 13B verify pass (224 rows, 1,100
// keys): 128 us per launch with one group, 112 with two, 108 with V staged by rows as K is (it
// was transposed by 4-byte loads); 176 rows at 4,160 keys 184, 156, 144. Three planes at head_dim
// 128 leave shared memory for one group, and passes with a block per chunk
// (launch_verify) have no use for a second.
//
// Softmax: warps w and w + 4 read TMEM lanes 32(w % 4) .. +31, so each thread owns one query
// vector's row of scores over half the chunk's keys (the two halves exchange their row
// maxima through shared memory; each keeps its own share of the row sum). The running
// reference m is raised only when a chunk's maximum exceeds it by more than kLazy (then O
// and l are rescaled); otherwise p = 2^(s - m) <= e^8, and the final o / l does not
// depend on the reference. The block's partial (m, l, o) are merged across the cluster
// through distributed shared memory as in attention.cu, and the normalized output is written
// as the O projection's hi/lo input.
//
// One thread issues every MMA; tcgen05.commit arrives on an mbarrier that the consumers wait
// on (bounded by the launch's wait limit: on expiry CDSL_ETIMEOUT is latched and the group
// skips its remaining chunks, waits for its own MMAs in flight and still meets every cluster
// barrier).
#include <algorithm>
#include <type_traits>

#include <cooperative_groups.h>

#include "attn_layout.cuh"
#include "kernels.h"
#include "tc_ptx.cuh"

namespace cdsl {
namespace {

namespace cg = cooperative_groups;
using attn::ACH;
using attn::MAXCB;

constexpr int TQB = 128;             // query vectors per block (at most): the MMA's M
constexpr int GTHREADS = 256;        // threads of a group, which works on a chunk at a time
constexpr int TACL = 16;             // blocks per cluster (at most)
constexpr int kIssuer = 128;         // thread of a group that issues its MMAs (warp 4, lane 0)
constexpr float kLazy = 11.5415602f; // raise the softmax reference only past this margin
                                     // (base-2 scores: 8 / ln 2, so p <= e^8)
constexpr float kLog2e = 1.44269504088896341f;

int g_tc_max_cluster = 8;

// NP: planes of Q, K, P and V (2: x = hi + lo; 3: hi + mid + lo, fp32's own precision). NG: groups.
// Each group has its own K, V and P; with two groups or three planes P overwrites K, whose products
// are done by then.
template <int HD, int NP, int NG>
struct TcSmem {
  static constexpr int KB = HD / 64;                        // 64-wide K blocks of Q and K
  static constexpr uint32_t Q_KB = TQB * 128;               // bytes of one K block of Q
  static constexpr uint32_t K_KB = ACH * 128;               // bytes of one K block of K
  static constexpr uint32_t Q_PLANE = KB * Q_KB;            // Q [128][HD] bf16, one plane
  static constexpr uint32_t K_PLANE = KB * K_KB;            // K [64][HD]
  static constexpr uint32_t V_PLANE = K_PLANE;              // V [64][HD]
  static constexpr uint32_t P_PLANE = TQB * 128;            // P [128][64 keys]
  static constexpr uint32_t Q_OFF = 0;
  static constexpr uint32_t K_OFF = Q_OFF + NP * Q_PLANE;
  static constexpr bool ALIAS = NG > 1 || NP > 2;
  static constexpr uint32_t KP = NP * (ALIAS && P_PLANE > K_PLANE ? P_PLANE : K_PLANE);   // K, P
  static constexpr uint32_t V_OFF = K_OFF + KP;
  static constexpr uint32_t P_OFF = ALIAS ? K_OFF : V_OFF + NP * V_PLANE;
  static constexpr uint32_t GROUP = KP + NP * V_PLANE + (ALIAS ? 0 : NP * P_PLANE);   // per group
  static constexpr uint32_t TOTAL = K_OFF + NG * GROUP;
  static constexpr int OP = HD + 4;                         // row pitch of the partial o (floats)
  // partial o [128][OP] fp32 of each group, over everything after the chunks; the block's first
  static_assert(NG * TQB * OP * 4 <= TOTAL, "the partial o fit");
  static constexpr uint32_t O_SIZE = TQB * OP * 4;
  static constexpr uint32_t T_GROUP = 64 + HD;              // TMEM columns of a group: S, O
  static constexpr uint32_t TMEM_COLS = NG * T_GROUP <= 128 ? 128 : NG * T_GROUP <= 256 ? 256 : 512;
  static constexpr size_t bytes = TOTAL + 1024;             // + 1024-byte alignment of the base
};

// 8 fp32 values -> NP planes of 8 bf16 values: x = hi + lo to about 2^-17, with three planes to
// about 2^-25.
template <int NP>
__device__ __forceinline__ void split8(const float (&x)[8], uint4 (&p)[NP]) {
  float r[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) r[i] = x[i];
#pragma unroll
  for (int n = 0; n < NP; ++n) {
    uint32_t u[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const __nv_bfloat16 a = __float2bfloat16_rn(r[2 * i]), b = __float2bfloat16_rn(r[2 * i + 1]);
      u[i] = (uint32_t)__bfloat16_as_ushort(a) | ((uint32_t)__bfloat16_as_ushort(b) << 16);
      r[2 * i] -= __bfloat162float(a);
      r[2 * i + 1] -= __bfloat162float(b);
    }
    p[n] = make_uint4(u[0], u[1], u[2], u[3]);
  }
}

__device__ __forceinline__ void st_shared16(uint8_t* base, uint32_t off, const uint4& v) {
  *reinterpret_cast<uint4*>(base + off) = v;
}

template <int HD, int NP, int NG>
__global__ void __launch_bounds__(NG * GTHREADS, 1) k_attn_tc(AttnArgs a) {
  const LaunchStamp stamp(a.stamp);
  using SM = TcSmem<HD, NP, NG>;
  constexpr int TTHREADS = NG * GTHREADS, TWARPS = TTHREADS / 32;
  constexpr int KB = SM::KB;
  constexpr int DCH = HD / 8;                    // 16-byte bf16 chunks per row of Q and K
  constexpr int K_IT = ACH * DCH / GTHREADS;     // staging items per thread: K and V
                                                 //   (key, 16-byte chunk)
  constexpr int Q_IT = TQB * DCH / TTHREADS;     //   and Q (query vector, chunk)
  extern __shared__ uint8_t smem_raw[];
  uint8_t* sm = smem_raw + ((1024 - (tc::smem_u32(smem_raw) & 1023)) & 1023);
  __shared__ attn::Layout<TQB> L;
  // per group: score / P V products complete, every MMA of it has completed
  __shared__ __align__(8) uint64_t bar_s[NG], bar_o[NG], bar_d[NG];
  __shared__ uint32_t s_tmem;
  __shared__ int s_abort[NG], s_nkeys;
  __shared__ const float* s_kptr[NG][2][ACH];     // K of each key slot of a chunk (V follows); a
                                                  // group's chunks take the buffers in turn
  __shared__ float s_pm[TQB], s_pl[TQB];          // the block's partial (m, l) per query vector
  __shared__ float s_gm[TQB], s_gl[TQB];          // the second group's
  __shared__ float s_mx[NG][2][TQB];              // per half: a chunk's row maxima, then l

  cg::cluster_group cluster = cg::this_cluster();
  const int C = (int)gridDim.x;                   // = cluster size
  const int cx = (int)blockIdx.x;                 // = rank in the cluster
  const int g = blockIdx.y;
  const int n_p = a.n_chunks;
  const int b = a.zmap ? a.zmap[2 * blockIdx.z] : blockIdx.z / a.qb_count;
  const int qb = a.zmap ? a.zmap[2 * blockIdx.z + 1] : blockIdx.z % a.qb_count;
  const int G = a.G, H = a.n_heads;
  const int warp = threadIdx.x >> 5;

  // ---- query vectors and key slots (before the wait: inputs of completed kernels only)
  if (a.rows_late) pdl_wait();
  const int nq = attn::build_layout<TQB, TTHREADS>(L, a, b, qb, cx, C);
  const int nb_chunks = L.nb;                     // chunk_of(L, n_p, cx, C, 0 .. nb_chunks - 1)
  if (a.stamp) attn::count_bytes<TQB, TTHREADS, HD>(L, stamp, qb, cx, nb_chunks, nq, &s_nkeys);
  if (threadIdx.x == 0) {
    for (int q = 0; q < NG; ++q) {
      tc::mbar_init(&bar_s[q], 1);
      tc::mbar_init(&bar_o[q], 1);
      tc::mbar_init(&bar_d[q], 1);
      s_abort[q] = 0;
    }
    tc::fence_mbar_init();
  }
  pdl_wait();                 // q and K/V of the previous kernels are ready
  if (warp == 0) tc::tmem_alloc(&s_tmem, SM::TMEM_COLS);

  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  pdl_launch_dependents();    // (this block has its TMEM before any of the next kernel's)
  const int grp = threadIdx.x / GTHREADS, tid = threadIdx.x % GTHREADS;
  auto group_sync = [&] { tc::named_barrier(1 + grp, GTHREADS); };
  // A group gives up as one: each of its threads brings its own failure to a barrier that ORs them.
  // (From a flag in shared memory read after a barrier, a slow warp could see what a fast one set at
  // its next wait, and the group's warps would then wait at different barriers.)
  bool failed = false;
  auto group_failed = [&] { return failed = tc::named_barrier_or(1 + grp, GTHREADS, failed); };
  const uint32_t tmem = s_tmem + (uint32_t)grp * SM::T_GROUP;
  const uint32_t t_s = tmem, t_o = tmem + 64;      // columns: S [0, 64), O [64, 64 + HD)
  const uint32_t lane_base = (uint32_t)((warp & 3) * 32) << 16;
  const uint32_t sbase = tc::smem_u32(sm);
  uint8_t* const smg = sm + grp * SM::GROUP;       // base of the group's K, V and P
  const uint32_t gbase = sbase + (uint32_t)grp * SM::GROUP;
  const uint32_t idesc_s = tc::idesc_bf16_f32(128, ACH), idesc_o = tc::idesc_bf16_f32(128, HD, true);
  const size_t v_delta_tail = (size_t)a.kv.n_tail_slots * a.kv.kvh * HD;
  const size_t v_delta_pfx = ((size_t)a.kv.kvh << a.kv.page_shift) * HD;
  const int qi = tid & (TQB - 1);                  // softmax: TMEM lane (query vector) and
  const int half = tid / TQB;                      //   half of the chunk's keys
  float m_ref = -INFINITY, l_run = 0.f;
  int nproc = 0;                                    // chunks whose P V has been issued
  // Two planes: O is one chain over the group's chunks in TMEM. Three: every chunk's P V starts
  // anew, and the threads add it to o_sum, rounded to nearest (this half's columns of row qi).
  constexpr bool kChain = NP == 2;
  float o_sum[kChain ? 1 : HD / 32][16];
#pragma unroll
  for (int q = 0; q < (kChain ? 0 : HD / 32); ++q)
#pragma unroll
    for (int e = 0; e < 16; ++e) o_sum[q][e] = 0.f;
  // f(n, m, kb, kk, add) for every product of planes n and m with n + m < NP, the smallest first, of
  // the 16-wide K steps kk of `blocks` 64-wide blocks kb
  auto each_product = [](auto&& f, auto blocks) {
#pragma unroll
    for (int t = NP - 1; t >= 0; --t)
#pragma unroll
      for (int kb = 0; kb < blocks(); ++kb)
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int n = 0; n <= t; ++n) f(n, t - n, kb, kk, t < NP - 1 || (kb | kk | n));
  };
  auto add_o = [&] {   // the finished P V (whole warps)
    if constexpr (!kChain) {
      tc::tc_fence_after();
#pragma unroll
      for (int q = 0; q < HD / 32; ++q) {
        float o[16];
        tc::tmem_ld16(t_o + lane_base + half * (HD / 2) + 16 * q, o);
#pragma unroll
        for (int e = 0; e < 16; ++e) o_sum[q][e] += o[e];
      }
    }
  };

  // Staging is software-pipelined: the group's next K rows (with one group, the V rows too) are
  // loaded from the fp32 cache into registers right after a chunk's score MMAs are issued (in
  // flight during its softmax), and converted and stored once its P V has completed.
  constexpr bool kPreV = NG == 1;
  auto kptrs = [&](int i) {   // the group's threads 0 .. ACH-1: key slot pointers of chunk i
    if (tid < ACH) {
      const int c = attn::chunk_of(L, n_p, cx, C, i);
      const int ks = L.kslot[i * ACH + tid];
      const float* kp = nullptr;
      if (ks >= 0) {
        const int slot = (c * ACH + tid) & ((1 << a.kv.page_shift) - 1);
        kp = c >= n_p ? a.kv.tail + kv_tail_offset(a.kv, a.layer, 0, ks, g)
                      : a.kv.pool + kv_prefix_offset(a.kv, a.layer, ks, 0, g, slot);
      }
      s_kptr[grp][(i / NG) & 1][tid] = kp;
    }
  };
  float4 kr[K_IT][2], vr[K_IT][2];   // raw K and V of the next chunk to stage
  // K or V (v_delta floats behind) rows of chunk i, all loads in flight together (pointers ready)
  auto load_rows = [&](int i, size_t delta, float4 (&x)[K_IT][2]) {
    const float* const* kps = s_kptr[grp][(i / NG) & 1];
#pragma unroll
    for (int u = 0; u < K_IT; ++u) {
      const int idx = tid + u * GTHREADS, j = idx / DCH, dc = idx % DCH;
      const float* kp = kps[j];
      x[u][0] = x[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (kp) {
        x[u][0] = __ldg(reinterpret_cast<const float4*>(kp + delta + dc * 8));
        x[u][1] = __ldg(reinterpret_cast<const float4*>(kp + delta + dc * 8 + 4));
      }
    }
  };
  auto load_k = [&](int i) { load_rows(i, 0, kr); };
  auto load_v = [&](int i) {
    load_rows(i, attn::chunk_of(L, n_p, cx, C, i) >= n_p ? v_delta_tail : v_delta_pfx, vr);
  };
  if (nb_chunks > 0 && nq > 0) {
    // ---- Q once per block: query vector qi is row qi of the A operand (zero rows from nq
    //      on), pre-scaled by log2(e) / sqrt(head_dim) (base-2 scores); and the groups' first
    //      chunks' loads
    if (grp < nb_chunks) kptrs(grp);
    float4 qr[Q_IT][2];
#pragma unroll
    for (int u = 0; u < Q_IT; ++u) {
      const int it = threadIdx.x + u * TTHREADS, qv = it / DCH, dc = it % DCH;
      qr[u][0] = qr[u][1] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (qv < nq) {
        const float* src =
            a.q + (size_t)L.row[qv] * H * HD + (size_t)(g * G + L.gg[qv]) * HD + dc * 8;
        qr[u][0] = *reinterpret_cast<const float4*>(src);
        qr[u][1] = *reinterpret_cast<const float4*>(src + 4);
      }
    }
    __syncthreads();   // the first chunks' pointers
    if (grp < nb_chunks) {
      load_k(grp);
      if (kPreV) load_v(grp);
    }
#pragma unroll
    for (int u = 0; u < Q_IT; ++u) {
      const int it = threadIdx.x + u * TTHREADS, qv = it / DCH, dc = it % DCH;
      const float sc = a.scale * kLog2e;
      const float x[8] = {qr[u][0].x * sc, qr[u][0].y * sc, qr[u][0].z * sc, qr[u][0].w * sc,
                          qr[u][1].x * sc, qr[u][1].y * sc, qr[u][1].z * sc, qr[u][1].w * sc};
      uint4 p[NP];
      split8<NP>(x, p);
      const uint32_t off = SM::Q_OFF + (dc >> 3) * SM::Q_KB + tc::sw128_offset(qv, dc & 7);
#pragma unroll
      for (int n = 0; n < NP; ++n) st_shared16(sm, off + n * SM::Q_PLANE, p[n]);
    }
  }

  if (NG > 1) {   // Q, which both groups' MMAs read, is complete
    tc::fence_proxy_async();
    __syncthreads();
  }
  for (int i = grp; i < nb_chunks && nq > 0; i += NG) {
    const int c = attn::chunk_of(L, n_p, cx, C, i);
    const bool tail = c >= n_p;
    const int t0 = c * ACH;
    if (!kPreV) load_v(i);
    // the group's previous P V has completed: K, V and P may be overwritten
    if (nproc > 0) {
      bool ok = tc::mbar_wait(&bar_o[grp], (nproc - 1) & 1, a.status, a.wait_ns);
      if constexpr (!kChain) ok = __all_sync(0xffffffffu, ok);
      if (!ok) failed = true;
      else add_o();
    }
    if (i + NG < nb_chunks) kptrs(i + NG);
    // ---- stage the chunk: split the loaded K and V into hi/lo and store
#pragma unroll
    for (int u = 0; u < K_IT; ++u) {
      const int idx = tid + u * GTHREADS, j = idx / DCH, dc = idx % DCH;
      const float x[8] = {kr[u][0].x, kr[u][0].y, kr[u][0].z, kr[u][0].w,
                          kr[u][1].x, kr[u][1].y, kr[u][1].z, kr[u][1].w};
      uint4 p[NP];
      split8<NP>(x, p);
      const uint32_t off = SM::K_OFF + (dc >> 3) * SM::K_KB + tc::sw128_offset(j, dc & 7);
#pragma unroll
      for (int n = 0; n < NP; ++n) st_shared16(smg, off + n * SM::K_PLANE, p[n]);
    }
#pragma unroll
    for (int u = 0; u < K_IT; ++u) {
      const int idx = tid + u * GTHREADS, j = idx / DCH, dc = idx % DCH;
      const float x[8] = {vr[u][0].x, vr[u][0].y, vr[u][0].z, vr[u][0].w,
                          vr[u][1].x, vr[u][1].y, vr[u][1].z, vr[u][1].w};
      uint4 p[NP];
      split8<NP>(x, p);
      const uint32_t off = SM::V_OFF + (dc >> 3) * SM::K_KB + tc::sw128_offset(j, dc & 7);
#pragma unroll
      for (int n = 0; n < NP; ++n) st_shared16(smg, off + n * SM::V_PLANE, p[n]);
    }
    tc::fence_proxy_async();
    if (group_failed()) break;
    // ---- S = Q K^T over the head dimension
    if (tid == kIssuer) {
      tc::tc_fence_after();
      each_product(
          [&](int n, int m, int kb, int kk, bool add) {   // K = 16: +32 bytes = +2 in the descriptor
            tc::umma_bf16(
                t_s, tc::desc_sw128(sbase + SM::Q_OFF + n * SM::Q_PLANE + kb * SM::Q_KB) + 2 * kk,
                tc::desc_sw128(gbase + SM::K_OFF + m * SM::K_PLANE + kb * SM::K_KB) + 2 * kk, idesc_s,
                add);
          },
          std::integral_constant<int, KB>());
      tc::umma_commit(&bar_s[grp]);
    }
    if (i + NG < nb_chunks) {   // in flight during this chunk's softmax
      load_k(i + NG);
      if (kPreV) load_v(i + NG);
    }
    // ---- softmax over the chunk: thread t owns TMEM lane qi = t % 128 (a query vector) and
    //      the chunk's keys 32h .. 32h + 31, h = t / 128 (warps w and w + 4 read the same
    //      lanes; tcgen05.ld is warp-collective, so a warp takes every branch as a whole)
    const bool sok = __all_sync(0xffffffffu, tc::mbar_wait(&bar_s[grp], nproc & 1, a.status, a.wait_ns));
    float s[2][16];
    float mx = -INFINITY;
    if (!sok) {
      failed = true;
    } else {
      tc::tc_fence_after();
      uint32_t r[2][16];
#pragma unroll
      for (int q = 0; q < 2; ++q)
        tc::tmem_ld16_nowait(t_s + lane_base + 32 * half + 16 * q, r[q]);
      tc::tmem_wait_ld();
      // prefix chunk: key j is visible below the row's prefix length (one limit per row)
      const int lim = (!tail && qi < nq) ? L.np[qi] - t0 - 32 * half : 0;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          const int j = 32 * half + 16 * q + e;
          const bool vis = tail ? (qi < nq && attn::key_visible(L, qi, i, c, n_p, j))
                                : 16 * q + e < lim;
          s[q][e] = vis ? __uint_as_float(r[q][e]) : -INFINITY;   // masked: 2^(-inf - m) = 0
          mx = fmaxf(mx, s[q][e]);
        }
      s_mx[grp][half][qi] = mx;
    }
    if (group_failed()) break;
    mx = fmaxf(s_mx[grp][0][qi], s_mx[grp][1][qi]);   // the row's maximum, the same in both halves
    {
      // raise the reference where a row's maximum passed it by more than kLazy: its earlier
      // sum and output are rescaled by alpha = exp(m_old - m_new) (both halves decide alike)
      float alpha = 1.f;
      bool rescale_o = false;
      if (mx > -INFINITY && (m_ref == -INFINITY || mx > m_ref + kLazy)) {
        alpha = m_ref == -INFINITY ? 0.f : exp2f(m_ref - mx);
        rescale_o = nproc > 0 && m_ref > -INFINITY;
        l_run *= alpha;
        m_ref = mx;
      }
      // each half rescales its half of the output row's columns, each lane by its own factor
      // (1 where its reference stayed)
      if constexpr (!kChain) {
        if (rescale_o) {
#pragma unroll
          for (int q = 0; q < HD / 32; ++q)
#pragma unroll
            for (int e = 0; e < 16; ++e) o_sum[q][e] *= alpha;
        }
      } else if (__any_sync(0xffffffffu, rescale_o)) {
        const float f = rescale_o ? alpha : 1.f;
#pragma unroll 1
        for (int q = 0; q < HD / 32; ++q) {
          float o[16];
          const uint32_t col = t_o + lane_base + half * (HD / 2) + 16 * q;
          tc::tmem_ld16(col, o);
#pragma unroll
          for (int e = 0; e < 16; ++e) o[e] *= f;
          tc::tmem_st16(col, o);
        }
      }
      float sum = 0.f;
#pragma unroll
      for (int q = 0; q < 2; ++q)
#pragma unroll
        for (int e = 0; e < 16; ++e) {
          s[q][e] = m_ref == -INFINITY ? 0.f : exp2f(s[q][e] - m_ref);
          sum += s[q][e];
        }
      l_run += sum;   // this half's share of the row's sum; the halves are added at the end
      // P row qi: keys 8ch..8ch+7 are 16-byte chunk ch (hi and lo planes); this half writes
      // chunks 4h .. 4h + 3
#pragma unroll
      for (int cc = 0; cc < 4; ++cc) {
        float x[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) x[e] = s[cc >> 1][(cc & 1) * 8 + e];
        uint4 p[NP];
        split8<NP>(x, p);
        const uint32_t off = SM::P_OFF + tc::sw128_offset(qi, 4 * half + cc);
#pragma unroll
        for (int n = 0; n < NP; ++n) st_shared16(smg, off + n * SM::P_PLANE, p[n]);
      }
      tc::fence_proxy_async();
      tc::tc_fence_before();
    }
    group_sync();
    // ---- O = P V over the chunk's 64 keys (kChain: O +=)
    if (tid == kIssuer) {
      tc::tc_fence_after();
      each_product(
          [&](int n, int m, int, int kk, bool add) {   // 16 keys: 2 KB of V
            tc::umma_bf16(t_o, tc::desc_sw128(gbase + SM::P_OFF + n * SM::P_PLANE) + 2 * kk,
                          tc::desc_sw128_mn(gbase + SM::V_OFF + m * SM::V_PLANE, SM::K_KB) + 128 * kk,
                          idesc_o, add || (kChain && nproc));
          },
          std::integral_constant<int, 1>());
      tc::umma_commit(&bar_o[grp]);
    }
    ++nproc;
  }

  // ---- every MMA issued here completes before its operands are overwritten and TMEM is
  //      released (fixed limit, also after a give-up)
  if (tid == kIssuer) {
    tc::umma_commit(&bar_d[grp]);
    tc::mbar_wait(&bar_d[grp], 0, a.status);
  }
  // ---- the block's partial (m, l, o) per query vector into shared memory (o over everything):
  //      each half writes its half of the row's columns; l is the sum of the halves' shares. A
  //      second group leaves its partial there for the first one to add to its own.
  if (failed || (nproc > 0 && !__all_sync(0xffffffffu, tc::mbar_wait(&bar_o[grp], (nproc - 1) & 1,
                                                                     a.status, a.wait_ns))))
    s_abort[grp] = 1;   // (read after the next barrier, no longer written there)
  else if (nproc > 0)
    add_o();
  if (half == 1) s_mx[grp][1][qi] = l_run;
  __syncthreads();
  float* const s_po = reinterpret_cast<float*>(sm);              // [TQB][OP]
  float* const s_go = s_po + SM::O_SIZE / 4;                     // the second group's
  const bool have_o = nproc > 0 && !s_abort[grp];
  if (have_o) tc::tc_fence_after();
  auto each_o = [&](auto&& put) {   // put(column, 16 values) over this half's columns
#pragma unroll(kChain ? 1 : HD / 32)
    for (int q = 0; q < HD / 32; ++q) {
      const int col = half * (HD / 2) + 16 * q;
      float o[16];
#pragma unroll
      for (int e = 0; e < 16; ++e) o[e] = kChain ? 0.f : o_sum[kChain ? 0 : q][e];
      if (kChain && have_o) tc::tmem_ld16(t_o + lane_base + col, o);   // (uniform over the group)
      if (qi < nq) put(col, o);
    }
  };
  if (half == 0) l_run += s_mx[grp][1][qi];
  if (NG > 1 && grp == 1) {
    if (half == 0) {
      s_gm[qi] = have_o ? m_ref : -INFINITY;
      s_gl[qi] = have_o ? l_run : 0.f;
    }
    each_o([&](int col, const float (&o)[16]) {
#pragma unroll
      for (int e = 0; e < 16; e += 4)
        *reinterpret_cast<float4*>(s_go + qi * SM::OP + col + e) =
            make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]);
    });
  }
  if (NG > 1) __syncthreads();
  if (grp == 0) {
    const float m0 = have_o ? m_ref : -INFINITY, m1 = NG > 1 ? s_gm[qi] : -INFINITY;
    const float m = fmaxf(m0, m1);
    const float f0 = m0 > -INFINITY ? exp2f(m0 - m) : 0.f, f1 = m1 > -INFINITY ? exp2f(m1 - m) : 0.f;
    each_o([&](int col, const float (&o)[16]) {
#pragma unroll
      for (int e = 0; e < 16; e += 4) {
        float4 v = make_float4(o[e], o[e + 1], o[e + 2], o[e + 3]);
        if (NG > 1) {
          const float4 w = *reinterpret_cast<const float4*>(s_go + qi * SM::OP + col + e);
          v.x = v.x * f0 + w.x * f1; v.y = v.y * f0 + w.y * f1;
          v.z = v.z * f0 + w.z * f1; v.w = v.w * f0 + w.w * f1;
        }
        *reinterpret_cast<float4*>(s_po + qi * SM::OP + col + e) = v;
      }
    });
    if (half == 0 && qi < nq) {
      s_pm[qi] = m;
      s_pl[qi] = (have_o ? l_run * f0 : 0.f) + (NG > 1 ? s_gl[qi] * f1 : 0.f);
    }
  }
  tc::tc_fence_before();
  cluster.sync();   // every block's partials are visible to the cluster

  // ---- merge: block cx finishes query vectors cx, cx + C, ... (a warp per query vector),
  //      reading the C partials through distributed shared memory, 8 blocks at a time
  constexpr int DPL = HD / 32;
  const int lane = threadIdx.x & 31;
  for (int qv = cx + warp * C; qv < nq; qv += C * TWARPS) {
    float vv[8][DPL];
    auto load_o = [&](int r0) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
#pragma unroll
        for (int c2 = 0; c2 < DPL; ++c2) vv[r][c2] = 0.f;
        if (r0 + r < C) {
          const float* src = cluster.map_shared_rank(s_po, r0 + r) + qv * SM::OP + DPL * lane;
          if constexpr (DPL == 4) {
            const float4 t4 = *reinterpret_cast<const float4*>(src);
            vv[r][0] = t4.x; vv[r][1] = t4.y; vv[r][2] = t4.z; vv[r][3] = t4.w;
          } else {
            const float2 t2 = *reinterpret_cast<const float2*>(src);
            vv[r][0] = t2.x; vv[r][1] = t2.y;
          }
        }
      }
    };
    load_o(0);
    float mr = -INFINITY, lr = 0.f;
    if (lane < C) {
      mr = cluster.map_shared_rank(s_pm, lane)[qv];
      lr = cluster.map_shared_rank(s_pl, lane)[qv];
    }
    const float M = warp_max(mr);
    const float w = (lane < C && mr > -INFINITY) ? exp2f(mr - M) : 0.f;
    const float Lsum = warp_sum(w * lr);
    float acc[DPL];
#pragma unroll
    for (int c2 = 0; c2 < DPL; ++c2) acc[c2] = 0.f;
    for (int r0 = 0; r0 < C; r0 += 8) {
      if (r0 > 0) load_o(r0);
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const float wr = __shfl_sync(0xffffffffu, w, (r0 + r) & 31);
#pragma unroll
        for (int c2 = 0; c2 < DPL; ++c2) acc[c2] = fmaf(wr, vv[r][c2], acc[c2]);
      }
    }
    const float inv = Lsum > 0.f ? 1.0f / Lsum : 0.f;
    __nv_bfloat16* out = reinterpret_cast<__nv_bfloat16*>(a.out);
    const size_t dst = (size_t)L.row[qv] * H * HD + (size_t)(g * G + L.gg[qv]) * HD + DPL * lane;
#pragma unroll
    for (int c2 = 0; c2 < DPL; ++c2) store_act<__nv_bfloat16>(out, a.plane, dst + c2, acc[c2] * inv);
  }
  cluster.sync();   // no block leaves while the others may still read its shared memory
  if (warp == 0) tc::tmem_dealloc(s_tmem, SM::TMEM_COLS);
}

template <int HD, int NP, int NG>
ClusterFit g_tc_fit;   // cluster residency of k_attn_tc<HD, NP, NG> (configure_tc)

template <int HD, int NP, int NG>
int configure_tc() {
  auto k = k_attn_tc<HD, NP, NG>;
  constexpr size_t smem = TcSmem<HD, NP, NG>::bytes;
  if (cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem) != cudaSuccess)
    return -1;
  const bool nonportable =
      cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
  cudaGetLastError();
  fill_cluster_fit(&g_tc_fit<HD, NP, NG>, k, NG * GTHREADS, smem, nonportable ? TACL : 8);
  return nonportable && g_tc_fit<HD, NP, NG>.active[TACL] >= 1 ? 0 : 1;   // 1: portable only
}

template <int HD, int NP, int NG>
void launch_tc(const AttnArgs& a, int n_z, cudaStream_t s) {
  const int chunks = a.n_chunks + a.n_tchunks;
  const ClusterFit& f = g_tc_fit<HD, NP, NG>;
  const int groups = a.kv.kvh * n_z;
  const int cl = a.zmap
                     ? attn_cluster_size_causal(f, g_tc_max_cluster, chunks, groups, a.avg_chunks)
                     : attn_cluster_size(f, g_tc_max_cluster, chunks, groups);
  launch_pdl_cluster(k_attn_tc<HD, NP, NG>, dim3(cl, a.kv.kvh, n_z), dim3(NG * GTHREADS),
                     TcSmem<HD, NP, NG>::bytes, cl, s, a);
}

// A verify pass's cluster that gives every chunk a block of its own has nothing for a second group
// of warps to do but be summed: one group (7B verify pass, 11 chunks in clusters of 11: 17.5 ->
// 17.2 us per launch, the step 5722 -> 5703 us).
template <int HD>
void launch_verify(const AttnArgs& a, int n_z, cudaStream_t s) {
  const int chunks = a.n_chunks + a.n_tchunks;
  if (attn_cluster_size(g_tc_fit<HD, 2, 1>, g_tc_max_cluster, chunks, a.kv.kvh * n_z) >= chunks)
    launch_tc<HD, 2, 1>(a, n_z, s);
  else
    launch_tc<HD, 2, 2>(a, n_z, s);
}

}  // namespace

int attn_tc_qblock(int rows_per_prompt, int G, bool tails) {
  // up to 128 query vectors; with beam tails at most 32 rows meeting in one block (the tail
  // layout runs one lane per row): 32 G vectors (whole rows) when that is smaller; no larger
  // than a prompt's vectors rounded up to whole rows of 16
  const int cap = tails ? std::min(TQB, 32 * G) : TQB;
  const int nq = rows_per_prompt * G;
  return std::max(16, std::min(cap, (nq + 15) / 16 * 16));
}

int configure_attention_tc() {
  int worst = 0;
  for (int r : {configure_tc<128, 2, 2>(), configure_tc<64, 2, 2>(), configure_tc<128, 2, 1>(),
                configure_tc<64, 2, 1>(), configure_tc<128, 3, 1>(), configure_tc<64, 3, 2>()}) {
    if (r < 0) return -1;
    worst = std::max(worst, r);
  }
  g_tc_max_cluster = worst ? 8 : TACL;
  return 0;
}

void launch_attn_tc(const AttnArgs& a, int n_z, cudaStream_t s) {
  // prefill passes with three planes
  if (a.n_tchunks == 0)
    a.kv.hd == 128 ? launch_tc<128, 3, 1>(a, n_z, s) : launch_tc<64, 3, 2>(a, n_z, s);
  else
    a.kv.hd == 128 ? launch_verify<128>(a, n_z, s) : launch_verify<64>(a, n_z, s);
}

}  // namespace cdsl
