// gemm.cuh -- the projection GEMMs of the decoder, y = x W^T, with fused epilogues.
//
// A GEMM runs over a "virtual" weight matrix made of up to three segments so that one launch
// covers the fused projections of a layer:
//   EPI_QKV    : [Wq; Wk; Wv] stacked            -> RoPE on q and k, q to a buffer, k/v to KV
//   EPI_SWIGLU : Wg and Wu interleaved in 64-row blocks (virtual rows 128t..128t+63 are gate
//                rows 64t.., the next 64 the matching up rows) -> silu(g) * u
//   EPI_RESID  : one matrix, h += y (residual stream, fp32)
//   EPI_STORE  : one matrix, fp32 store (logits)
// Output features are processed in tiles of 128 virtual rows; every pair the epilogue needs
// (RoPE's (i, i + hd/2), SwiGLU's (gate_j, up_j)) lies inside one tile.
//
// RMSNorm is folded into the GEMMs: RMSNorm(h) g W^T = rsqrt(mean(h^2) + eps) * ((h . g) W^T),
// the row scale factoring out of the dot product. A RESID epilogue therefore also writes the
// next GEMM's input h . g_next (GEMM-input format) and per 32-feature chunk the partial sums
// of h^2 (and, for the reward head, of w . g . h); the consuming GEMM's epilogue multiplies by
// the row scale computed from those partials in a fixed order (deterministic).
#pragma once

#include "common.cuh"

namespace cdsl {

enum EpiMode : int32_t { EPI_STORE = 0, EPI_RESID = 1, EPI_SWIGLU = 2, EPI_QKV = 3 };

struct GemmArgs {
  const void* w[3];        // segment base pointers, [rows, K] row-major
  int32_t seg_rows[3];     // rows per segment (multiples of 64 except a final ragged one)
  int32_t n_seg;
  int32_t mode;            // EpiMode
  int32_t K;               // input features
  int32_t n_virtual;       // virtual output rows (padded to a multiple of 128 for SWIGLU)
  const void* x;           // activations [R, ldx] (store_act format of the weight dtype)
  int32_t ldx;
  int64_t x_plane;         // elements between the hi and lo planes of x (bf16 models)
  int32_t R;               // activation rows
  // epilogue outputs
  float* out_f32;          // STORE / RESID: [R, ld_out]
  int32_t ld_out;
  void* out_act;           // SWIGLU: [R, ld_act] (store_act format)
  int32_t ld_act;
  int64_t act_plane;       // SWIGLU: plane distance of out_act
  int32_t d_ffn;           // SWIGLU: valid features
  float* q_out;            // QKV: [R, n_heads * hd] fp32 (rotated)
  int32_t n_heads;
  KvStore kv;              // QKV: destination of k, v
  int32_t layer;
  const RowDesc* rows;     // QKV: per-row position and KV destination
  const float2* rope;      // QKV: [pos][hd/2] (cos, sin)
  int32_t* status;         // device status word (bounded waits report CDSL_ETIMEOUT here)
  uint64_t wait_ns;        // limit of the tensor-core kernel's pipeline waits (nanoseconds)
  // input normalization: rows are h . g, scale by rsqrt(sum(in_ss[c][r]) / norm_D + eps)
  const float* in_ss;      // [R][ld_ss] partial sums of squares (norm_D / 32 per row), or nullptr
  int32_t norm_D;
  int32_t ld_ss;           // row stride of the partial-sum arrays (>= D / 32)
  float norm_eps;
  // RESID: next GEMM input and its partial sums
  void* next_x;            // [R, ld_out] GEMM-input format (plane distance act_plane), or nullptr
  const void* next_g;      // [ld_out] gain of the next RMSNorm (weight dtype)
  float* out_ss;           // [R][ld_ss], ld_out / 32 per row
  const float* head_w;     // reward head vector [ld_out] (last target layer only), or nullptr
  float* out_hw;           // [R][ld_ss] partial sums of head_w . g . h
  unsigned long long* stamp;  // in-graph launch timing record (LaunchStamp), or nullptr
};

// Row scale rsqrt(mean(h^2) + eps) from the 32-feature partial sums of row r, by a whole warp:
// lane l sums chunks c = l (mod 32), then the lanes' butterfly. input_row_scales below takes
// the same order, so every consumer of a row derives the same bits.
__device__ __forceinline__ float row_scale(const float* ss, int chunks, int ld, int r, int D,
                                           float eps) {
  float acc = 0.f;
  for (int c = threadIdx.x & 31; c < chunks; c += 32) acc += ss[(size_t)r * ld + c];
  return rsqrtf(warp_sum(acc) / (float)D + eps);
}

// rs[i] = row scale of input row r0 + i for i < n (0 past a.R), computed by `nthr` threads
// (a multiple of 32, tid = 0 .. nthr-1): a warp reads the partials of four rows at a time, a
// row's side by side (the loads wait out a memory round trip before an epilogue may start; with
// the partials of one chunk side by side and lane quads per row the small model's steps took
// 2011 us instead of 1891, its short requests 25.2 ms instead of 23.0). The caller
// synchronizes afterwards.
__device__ __forceinline__ void input_row_scales(const GemmArgs& a, int r0, int n, float* rs,
                                                 int tid, int nthr);

// Pointer to virtual row v of the segmented weight matrix, nullptr for padding rows.
template <typename T>
__device__ __forceinline__ const T* virtual_row(const GemmArgs& a, int v) {
  if (a.mode == EPI_SWIGLU) {
    const int blk = v >> 7, within = v & 127;
    const int row = blk * 64 + (within & 63);
    if (row >= a.d_ffn) return nullptr;
    return reinterpret_cast<const T*>(a.w[within >> 6]) + (size_t)row * a.K;
  }
  int base = 0;
  for (int s = 0; s < a.n_seg; ++s) {
    if (v < base + a.seg_rows[s]) return reinterpret_cast<const T*>(a.w[s]) + (size_t)(v - base) * a.K;
    base += a.seg_rows[s];
  }
  return nullptr;
}

// What the QKV epilogue needs of one activation row: the RoPE position and where the row's k
// and v go (element offset of k, head 0 in the prefix pool or the beam tails). gemm_pair.cu gathers
// these once per row and block (qkv_rows) instead of reading the row descriptor and the page table
// for every feature.
struct QkvRow {
  int32_t pos;
  int32_t where;   // 0: not stored, 1: prefix pool, 2: beam tail
  int64_t base;
};

// rows[i] for activation rows r0 + i, i < n (by `nthr` threads, tid = 0 .. nthr-1; the caller
// synchronizes afterwards).
__device__ __forceinline__ void qkv_rows(const GemmArgs& a, int r0, int n, QkvRow* rows, int tid,
                                         int nthr) {
  const KvStore& kv = a.kv;
  for (int r = tid; r < n; r += nthr) {
    const RowDesc rd = a.rows[r0 + r];
    QkvRow m{rd.pos, 0, 0};
    if (rd.kv_dst >= 0) {
      m.where = 2;
      m.base = (int64_t)kv_tail_offset(kv, a.layer, 0, rd.kv_dst, 0);
    } else if (rd.kv_dst == KV_PREFIX) {
      const int page = kv.page_table[rd.b * kv.max_pages + (rd.pos >> kv.page_shift)];
      if (page >= 0) {
        m.where = 1;
        m.base = (int64_t)kv_prefix_offset(kv, a.layer, page, 0, 0,
                                           rd.pos & ((1 << kv.page_shift) - 1));
      }
    }
    rows[r] = m;
  }
}

__device__ __forceinline__ float silu_f(float g) { return g / (1.0f + expf(-g)); }

// Sum v[i] over the warp's lanes for all i; lane l then holds the sum of index l * NR / 32 in
// v[0] (NR a power of two up to 16: a transposing butterfly, NR shuffles and a few instead of 5 NR).
template <int NR>
__device__ __forceinline__ void warp_sums(float (&v)[NR]) {
  int n = NR;
#pragma unroll
  for (int off = 16; off >= 1; off >>= 1) {
    if (n > 1) {
      const bool upper = (threadIdx.x & off) != 0;
#pragma unroll
      for (int i = 0; i < NR / 2; ++i) {
        if (i < n / 2) {
          const float send = upper ? v[i] : v[i + n / 2];
          const float keep = upper ? v[i + n / 2] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, off);
        }
      }
      n >>= 1;
    } else {
      v[0] += __shfl_xor_sync(0xffffffffu, v[0], off);
    }
  }
}

// Epilogue on registers (the same arithmetic as tile_epilogue's below, which reads a finished tile
// from shared memory: a change to one belongs in both): finish NR activation rows row0 .. row0 + NR - 1 (the first `rows` of them)
// of one output per lane. STORE / RESID: L is the weight row, y0 its sums. SWIGLU: the feature, y0
// its gate and y1 its up sums. QKV: the pair (head, e) = (L / (hd / 2), L % (hd / 2)) over the
// stacked heads, y0 and y1 the sums of dims e and e + hd / 2. rs: row scales of row0 on (a.in_ss),
// qr: QKV row destinations of row0 on. Whole warps call it with 32 consecutive L from a multiple
// of 32; row0 and rows are warp-uniform.
template <int MODE, int NR>
__device__ __forceinline__ void finish_rows(const GemmArgs& a, int L, int row0, int rows,
                                            const float (&y0)[NR], const float (&y1)[NR],
                                            const float* rs, const QkvRow* qr) {
  using T = __nv_bfloat16;
  const int lane = threadIdx.x & 31;
  const bool scaled = a.in_ss != nullptr;
  if constexpr (MODE == EPI_STORE) {
    const int n = L;
    float* const out = a.out_f32 + (size_t)row0 * a.ld_out + n;
    const size_t ld = a.ld_out;
    if (n >= a.n_virtual) return;
#pragma unroll
    for (int i = 0; i < NR; ++i)
      if (i < rows) out[i * ld] = scaled ? y0[i] * rs[i] : y0[i];
  } else if constexpr (MODE == EPI_RESID) {
    const int n = L;
    if (n >= a.n_virtual) return;   // warp-uniform: n_virtual = d_model, a multiple of 64
    const size_t ld = a.ld_out, plane = (size_t)a.act_plane;
    float* const out = a.out_f32 + (size_t)row0 * ld + n;
    T* const nx = reinterpret_cast<T*>(a.next_x);
    T* const nxr = nx + (size_t)row0 * ld + n;
    float h[NR];
#pragma unroll
    for (int i = 0; i < NR; ++i) h[i] = i < rows ? out[i * ld] : 0.f;
    const float g = nx ? to_f32<T>(reinterpret_cast<const T*>(a.next_g)[n]) : 0.f;
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      if (i < rows) {
        h[i] += scaled ? y0[i] * rs[i] : y0[i];
        out[i * ld] = h[i];
        if (nx) store_act<T>(nxr, plane, i * ld, h[i] * g);
      }
    }
    if (a.out_ss) {
      const int i = lane * NR / 32;
      const bool writer = lane % (32 / NR) == 0 && i < rows;
      const size_t at = (size_t)(row0 + i) * a.ld_ss + (n >> 5);
      float s[NR];
#pragma unroll
      for (int q = 0; q < NR; ++q) s[q] = h[q] * h[q];
      warp_sums<NR>(s);
      if (writer) a.out_ss[at] = s[0];
      if (a.head_w) {
        const float gw = a.head_w[n] * g;
#pragma unroll
        for (int q = 0; q < NR; ++q) s[q] = gw * h[q];
        warp_sums<NR>(s);
        if (writer) a.out_hw[at] = s[0];
      }
    }
  } else if constexpr (MODE == EPI_SWIGLU) {
    const int f = L;
    if (f >= a.d_ffn) return;
    const size_t ld = a.ld_act, plane = (size_t)a.act_plane;
    T* const out = reinterpret_cast<T*>(a.out_act) + (size_t)row0 * ld + f;
#pragma unroll
    for (int i = 0; i < NR; ++i) {
      if (i < rows) {
        const float sc = scaled ? rs[i] : 1.f;
        store_act<T>(out, plane, i * ld, silu_f(y0[i] * sc) * (y1[i] * sc));
      }
    }
  } else {   // EPI_QKV: dims e and e + hd / 2 of one head
    const KvStore& kv = a.kv;
    const int hd = kv.hd, half = hd >> 1, H = a.n_heads, KVH = kv.kvh;
    const int head = L / half, e = L % half;
    if (head >= H + 2 * KVH) return;   // warp-uniform: half is 32 or 64
    if (head < H + KVH) {
      float2 cs[NR];
#pragma unroll
      for (int i = 0; i < NR; ++i)
        cs[i] = i < rows ? a.rope[(size_t)qr[i].pos * half + e] : make_float2(1.f, 0.f);
      const int nq = H * hd;
      float* const q = a.q_out + (size_t)row0 * nq + head * hd + e;
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        if (i >= rows) continue;
        const float sc = scaled ? rs[i] : 1.f;
        const float u = y0[i] * sc, v = y1[i] * sc;
        const float ru = u * cs[i].x - v * cs[i].y, rv = v * cs[i].x + u * cs[i].y;
        if (head < H) {
          q[(size_t)i * nq] = ru;
          q[(size_t)i * nq + half] = rv;
        } else if (qr[i].where) {
          float* const d = qr[i].where == 1
                               ? kv.pool + qr[i].base + ((size_t)(head - H) * hd << kv.page_shift)
                               : kv.tail + qr[i].base + (size_t)(head - H) * hd;
          d[e] = ru;
          d[e + half] = rv;
        }
      }
    } else {
      const int vh = head - H - KVH;
#pragma unroll
      for (int i = 0; i < NR; ++i) {
        if (i >= rows || !qr[i].where) continue;
        const float sc = scaled ? rs[i] : 1.f;
        float* const d =
            qr[i].where == 1
                ? kv.pool + qr[i].base + ((size_t)(KVH + vh) * hd << kv.page_shift)
                : kv.tail + qr[i].base + ((size_t)kv.n_tail_slots * KVH + vh) * hd;
        d[e] = y0[i] * sc;
        d[e + half] = y1[i] * sc;
      }
    }
  }
}

// Apply the epilogue (finish_rows is the same on registers) to a finished fp32 tile: tile[r * ldt + v] holds y for activation row
// r0 + r and virtual row v0 + v (v in [0, 128)), for r in [0, rt). s_rs[r] is the input row
// scale of row r0 + r when a.in_ss is set (see input_row_scales). Run by `nthr` threads (a
// multiple of 32; tid = 0 .. nthr-1; all threads of the block by default), which the caller
// synchronizes before and after.
template <typename T>
__device__ void tile_epilogue(const GemmArgs& a, int v0, int r0, int rt, const float* tile,
                              int ldt, const float* s_rs, int tid = -1, int nthr = -1) {
  if (tid < 0) {
    tid = threadIdx.x;
    nthr = blockDim.x;
  }
  // Every field is read once, into registers, before the stores: `a` is reached through a
  // reference (to the kernel parameter), which the compiler must otherwise assume the stores
  // below may alias, re-reading it on every item.
  const int mode = a.mode, R = a.R, nv = a.n_virtual;
  const bool scaled = a.in_ss != nullptr;
  const float* __restrict__ tl = tile;   // shared memory: never aliases the outputs
  if (mode == EPI_STORE) {
    float* __restrict__ const out = a.out_f32;
    const size_t ld = (size_t)a.ld_out;
    for (int idx = tid; idx < rt * 128; idx += nthr) {
      const int r = idx >> 7, v = idx & 127, row = r0 + r, n = v0 + v;
      float y = tl[r * ldt + v];
      if (scaled) y *= s_rs[r];
      if (row < R && n < nv) out[(size_t)row * ld + n] = y;
    }
  } else if (mode == EPI_RESID) {
    float* __restrict__ const out = a.out_f32;
    const size_t ld = (size_t)a.ld_out, plane = (size_t)a.act_plane, ld_ss = (size_t)a.ld_ss;
    T* const next_x = reinterpret_cast<T*>(a.next_x);
    const T* const next_g = reinterpret_cast<const T*>(a.next_g);
    float* const out_ss = a.out_ss;
    const float* const head_w = a.head_w;
    float* const out_hw = a.out_hw;
    // a multiple of 32 items per thread pass: every warp sees 32 features of one row
    for (int idx = tid; idx < rt * 128; idx += nthr) {
      const int r = idx >> 7, v = idx & 127, row = r0 + r, n = v0 + v;
      const bool ok = row < R && n < nv;
      float y = tl[r * ldt + v];
      if (scaled) y *= s_rs[r];
      float hn = 0.f;
      if (ok) {
        float* hp = out + (size_t)row * ld + n;
        hn = *hp + y;
        *hp = hn;
        if (next_x)
          store_act<T>(next_x, plane, (size_t)row * ld + n, hn * to_f32<T>(next_g[n]));
      }
      if (out_ss) {   // warp-uniform
        const float sq = warp_sum(hn * hn);
        float hw = 0.f;
        if (head_w) {
          const float gw = ok ? head_w[n] * to_f32<T>(next_g[n]) : 0.f;
          hw = warp_sum(gw * hn);
        }
        if ((v & 31) == 0 && ok) {
          out_ss[(size_t)row * ld_ss + (n >> 5)] = sq;
          if (head_w) out_hw[(size_t)row * ld_ss + (n >> 5)] = hw;
        }
      }
    }
  } else if (mode == EPI_SWIGLU) {
    T* const out_act = reinterpret_cast<T*>(a.out_act);
    const size_t ld_act = (size_t)a.ld_act, plane = (size_t)a.act_plane;
    const int d_ffn = a.d_ffn, f0 = (v0 >> 7) * 64;
    for (int idx = tid; idx < rt * 64; idx += nthr) {   // gate v, up v + 64
      const int r = idx >> 6, v = idx & 63, row = r0 + r, f = f0 + v;
      if (row >= R || f >= d_ffn) continue;
      float g = tl[r * ldt + v], u = tl[r * ldt + v + 64];
      if (scaled) {
        g *= s_rs[r];
        u *= s_rs[r];
      }
      store_act<T>(out_act, plane, (size_t)row * ld_act + f, silu_f(g) * u);
    }
  } else {   // EPI_QKV
    const KvStore kv = a.kv;
    float* const q_out = a.q_out;
    const RowDesc* const rows = a.rows;
    const float2* const rope = a.rope;
    const int layer = a.layer;
    const int hd = kv.hd, half = hd >> 1;
    const int nq = a.n_heads * hd, nk = kv.kvh * hd;
    for (int idx = tid; idx < rt * 128; idx += nthr) {
      const int r = idx >> 7, v = idx & 127, row = r0 + r, n = v0 + v;
      if (row >= R || n >= nq + 2 * nk) continue;
      float y = tl[r * ldt + v];
      if (scaled) y *= s_rs[r];
      const RowDesc rd = rows[row];
      float val = y;
      const int e = n % hd;  // segments start on head boundaries
      if (n < nq + nk) {     // q or k: rotate-half RoPE with the partner in this tile
        const float2 cs = rope[(size_t)rd.pos * half + (e % half)];
        float other = (e < half) ? tl[r * ldt + v + half] : tl[r * ldt + v - half];
        if (scaled) other *= s_rs[r];
        val = (e < half) ? (y * cs.x - other * cs.y) : (y * cs.x + other * cs.y);
      }
      if (n < nq) {
        q_out[(size_t)row * nq + n] = val;
      } else {
        const int kvsel = (n < nq + nk) ? 0 : 1;
        const int head = (n - nq - kvsel * nk) / hd;
        float* dst = nullptr;
        if (rd.kv_dst >= 0) {
          dst = kv.tail + kv_tail_offset(kv, layer, kvsel, rd.kv_dst, head);
        } else if (rd.kv_dst == KV_PREFIX) {
          const int page = kv.page_table[rd.b * kv.max_pages + (rd.pos >> kv.page_shift)];
          if (page >= 0)
            dst = kv.pool + kv_prefix_offset(kv, layer, page, kvsel, head,
                                             rd.pos & ((1 << kv.page_shift) - 1));
        }
        if (dst) dst[e] = val;
      }
    }
  }
}

__device__ __forceinline__ void input_row_scales(const GemmArgs& a, int r0, int n, float* rs,
                                                 int tid, int nthr) {
  constexpr int kRows = 4;   // rows per warp and pass, their loads in flight together
  const int D = a.norm_D, chunks = D >> 5, R = a.R, lane = tid & 31;
  const float* const ss = a.in_ss;
  const size_t ld = (size_t)a.ld_ss;
  const float eps = a.norm_eps;
  for (int r = (tid >> 5) * kRows; r < n; r += (nthr >> 5) * kRows) {   // warp-uniform
    float acc[kRows];
#pragma unroll
    for (int i = 0; i < kRows; ++i) acc[i] = 0.f;
#pragma unroll 2
    for (int c = lane; c < chunks; c += 32) {
#pragma unroll
      for (int i = 0; i < kRows; ++i)
        if (r + i < n && r0 + r + i < R) acc[i] += ss[(size_t)(r0 + r + i) * ld + c];
    }
#pragma unroll
    for (int i = 0; i < kRows; ++i) acc[i] = warp_sum(acc[i]);
    if (lane < kRows && r + lane < n) {
      float v = acc[0];
#pragma unroll
      for (int i = 1; i < kRows; ++i) v = lane == i ? acc[i] : v;
      rs[r + lane] = r0 + r + lane < R ? rsqrtf(v / (float)D + eps) : 0.f;
    }
  }
}

}  // namespace cdsl
