// CUDA-core kernels of the decode step: row preparation, RMSNorm, row-streaming linear
// (the float32 path and the M<=few GEMV-style projections of the extra heads), RoPE + cache
// store, plain tree attention, argmax, acceptance walk, KV compaction, per-head top-k.
// Templated on the operand type T (float or bf16): operands are rounded to T exactly where
// a tensor-core kernel would consume them; accumulation is float32.
#pragma once
#include <algorithm>

#include "common.cuh"

namespace spec {

// ------------------------------------------------------------------ row preparation
// Embedding row `e` of d elements (or zeros) into the residual stream; 16-byte loads where the type allows.
template <typename T>
__device__ __forceinline__ void embed_row(const T* __restrict__ e, float* __restrict__ x, int d, bool on) {
  if (sizeof(T) == 2 && d % 8 == 0) {
    for (int c8 = threadIdx.x; c8 < (d >> 3); c8 += blockDim.x) {
      const uint4 raw = on ? *reinterpret_cast<const uint4*>(reinterpret_cast<const bf16*>(e) + c8 * 8) : make_uint4(0, 0, 0, 0);
      const __nv_bfloat162* hp = reinterpret_cast<const __nv_bfloat162*>(&raw);
      const float2 f0 = __bfloat1622float2(hp[0]), f1 = __bfloat1622float2(hp[1]), f2 = __bfloat1622float2(hp[2]), f3 = __bfloat1622float2(hp[3]);
      float* dst = x + c8 * 8;
      *reinterpret_cast<float4*>(dst) = make_float4(f0.x, f0.y, f1.x, f1.y);
      *reinterpret_cast<float4*>(dst + 4) = make_float4(f2.x, f2.y, f3.x, f3.y);
    }
  } else {
    for (int c = threadIdx.x; c < d; c += blockDim.x) x[c] = on ? to_f<T>(e[c]) : 0.f;
  }
}

// Verify pass: tree node i of sequence b carries candidate rank[i] of head depth[i]
// (head 0 = the base model's own next token) and sits at position n[b] + depth[i].
template <typename T>
__global__ void prepare_verify_rows(Rows rows, const int* __restrict__ cand, int cand_stride_b, int kmax,
                                    const int* __restrict__ depth, const int* __restrict__ rank, int capacity,
                                    const T* __restrict__ embed, float* __restrict__ x, int d, int vocab,
                                    int* status, unsigned long long* tr) {
  KTrace kt(tr);
  // This kernel lets its dependents start only after its own dependency wait, i.e. after every kernel before it
  // has completed: no kernel of the verification pass begins before the previous step's kernels (its cache
  // compaction above all) are done. The attention kernels rely on that when they fetch keys below the host's
  // lower bound of the committed length ahead of their own dependency wait.
  const int m = blockIdx.x, b = m / rows.R, i = m % rows.R;
  const int dep = depth[i], place = dep * kmax + rank[i];      // (the tree is fixed at set-up)
  pdl_wait();
  pdl_launch_dependents();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  int n = rows.n[b];
  bool ok = (n + rows.R <= capacity);
  if (!ok && threadIdx.x == 0) set_status(status, ST_SEQLEN, 1, b);
  int t = cand[b * cand_stride_b + place];
  if (t < 0 || t >= vocab) { t = 0; if (threadIdx.x == 0 && ok) set_status(status, ST_BOUNDS, 1, m); }
  if (threadIdx.x == 0) {
    rows.tok[m] = t;
    rows.pos[m] = n + dep;
    rows.slot[m] = n + i;
    if (i == 0) rows.cnt[b] = ok ? rows.R : 0;
  }
  embed_row<T>(embed + (size_t)t * d, x + (size_t)m * d, d, true);
}

// Prompt processing: row group v of the pass is prompt tokens [chunk_pos[v], + R) of sequence rows.seq[v].
template <typename T>
__global__ void prepare_prefill_rows(Rows rows, const int* __restrict__ prompt, const int* __restrict__ offsets,
                                     const int* __restrict__ chunk_pos, const T* __restrict__ embed, float* __restrict__ x, int d,
                                     int vocab, int* status) {
  const int m = blockIdx.x, v = m / rows.R, i = m % rows.R, b = rows.seq[v];
  const int start = chunk_pos[v], len = offsets[b + 1] - offsets[b];
  const int p = start + i;
  int t = 0;
  if (p < len) {
    t = prompt[offsets[b] + p];
    if (t < 0 || t >= vocab) { t = 0; if (threadIdx.x == 0) set_status(status, ST_BOUNDS, 2, m); }
  }
  if (threadIdx.x == 0) {
    rows.tok[m] = t;
    rows.pos[m] = p;
    rows.slot[m] = p;
    if (i == 0) {
      const int c = len - start;
      rows.cnt[v] = c < 0 ? 0 : (c > rows.R ? rows.R : c);
      rows.n[v] = start;
    }
  }
  embed_row<T>(embed + (size_t)t * d, x + (size_t)m * d, d, p < len);
}

// After a prefill pass: sequences whose last prompt token is in this pass keep that row's
// final hidden state (float32 and operand type) for the first step's heads and lm_head.
template <typename T>
__global__ void prefill_keep_last(Rows rows, const int* __restrict__ offsets, const int* __restrict__ chunk_pos,
                                  const float* __restrict__ hid, float* __restrict__ h_last,
                                  T* __restrict__ hq_last, int* __restrict__ n_seq, int d) {
  const int v = blockIdx.x, b = rows.seq[v];
  const int len = offsets[b + 1] - offsets[b];
  const int i = len - 1 - chunk_pos[v];
  if (i < 0 || i >= rows.R) return;
  const int m = v * rows.R + i;
  for (int c = threadIdx.x; c < d; c += blockDim.x) {
    float v = hid[(size_t)m * d + c];
    h_last[(size_t)b * d + c] = v;
    hq_last[(size_t)b * d + c] = from_f<T>(v);
  }
  if (threadIdx.x == 0) n_seq[b] = len;
}

// Rows of a pass that are last tokens of prompts, for the rest of the last layer: residual stream and normed operand of row
// end_row[g] of the pass to row g, and the sequence's length.
__global__ void __launch_bounds__(256)
gather_prompt_ends(const int* __restrict__ end_row, const int* __restrict__ end_pos, const float* __restrict__ x, const bf16* __restrict__ u,
                   float* __restrict__ x_end, bf16* __restrict__ u_end, int* __restrict__ n_seq, int d, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  const int g = blockIdx.x;
  const size_t m = end_row[g];
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  for (int c = threadIdx.x; c < (d >> 2); c += blockDim.x) {
    reinterpret_cast<float4*>(x_end + (size_t)g * d)[c] = reinterpret_cast<const float4*>(x + m * d)[c];
    reinterpret_cast<uint2*>(u_end + (size_t)g * d)[c] = reinterpret_cast<const uint2*>(u + m * d)[c];
  }
  if (threadIdx.x == 0) n_seq[g] = end_pos[g] + 1;
}

// Their attention outputs: row end_pos[g] % R of chunk g to row g.
__global__ void __launch_bounds__(256)
gather_attention_ends(const int* __restrict__ end_pos, const bf16* __restrict__ attn, bf16* __restrict__ attn_end, int R, int HD, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  const int g = blockIdx.x;
  const size_t m = (size_t)g * R + end_pos[g] % R;
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  for (int c = threadIdx.x; c < (HD >> 3); c += blockDim.x)
    reinterpret_cast<uint4*>(attn_end + (size_t)g * HD)[c] = reinterpret_cast<const uint4*>(attn + m * HD)[c];
}

// What prompt processing is told by the host, by value: a copy and a memset each for these few hundred ints, and the wait for them, took
// 50 us before the first kernel of a prompt.
constexpr int PS_SEQS = 32, PS_CHUNKS = 96;
struct PrefillSetup {
  int batch, max_batch, chunks;            // sequences, of which the context has room for, chunks of all prompts
  int offsets[PS_SEQS + 1];                // first token of a sequence's prompt
  int page_end[PS_SEQS];                   // of each of max_batch sequences: pages from here on are zero already
  int chunk_seq[PS_CHUNKS], chunk_pos[PS_CHUNKS];
  int ends[6 * PS_SEQS];                   // the tables of PromptEnds, batch entries each
};
struct PrefillTargets {
  int *offsets, *chunk_seq, *chunk_pos, *ends, *status, *gen_cnt, *draws;
  unsigned int *pair_arrive, *item_counter;
  int n_arrive;
};

// Before prompts are processed. The first CTA writes the tables and clears the counters (a wait that ran out may have left some set). All of them: zeros
// in every cache slot that the prompts do not fill, from the page of a sequence's first free slot on, as far as earlier sequences have written
// (attention reads whole tiles of keys; what lies past a sequence's end has weight zero but must be finite). On the 7B shape clearing the whole pool took
// 45 us for a 2048-token prompt and 8 layers, and all free pages 55 us for eight prompts of up to 1024 tokens and 4 layers.
__global__ void __launch_bounds__(256)
prefill_setup(const __grid_constant__ PrefillSetup s, const PrefillTargets to, uint4* __restrict__ pool, int pages_per_seq, int page_size, int pair_vecs, int share) {
  const int tid = threadIdx.x;
  if (to.status && blockIdx.x + blockIdx.y == 0) {
    if (tid < 4) to.status[tid] = 0;
    if (tid == 0) *to.item_counter = 0u;
    for (int i = tid; i < to.n_arrive; i += 256) to.pair_arrive[i] = 0u;
    for (int i = tid; i < s.batch; i += 256) { to.gen_cnt[i] = 0; to.draws[i] = 0; }
    for (int i = tid; i <= s.batch; i += 256) to.offsets[i] = s.offsets[i];
    for (int i = tid; i < s.chunks; i += 256) { to.chunk_seq[i] = s.chunk_seq[i]; to.chunk_pos[i] = s.chunk_pos[i]; }
    for (int i = tid; i < 6 * s.batch; i += 256) to.ends[i] = s.ends[i];
  }
  // grid (sequences times the CTAs that share one's pages, layers * heads); pool page p * max_batch + b is page p of sequence b
  const int b = blockIdx.x / share, len = b < s.batch ? s.offsets[b + 1] - s.offsets[b] : 0, end = s.page_end[b];
  uint4* base = pool + ((size_t)blockIdx.y * pages_per_seq * s.max_batch + b) * pair_vecs;
  for (int p = len / page_size + blockIdx.x % share; p < end; p += share)
    for (int i = tid; i < pair_vecs; i += 256) base[(size_t)p * s.max_batch * pair_vecs + i] = make_uint4(0, 0, 0, 0);
}

// The same for more sequences or chunks than that holds, without the tables: all free pages.
__global__ void __launch_bounds__(256)
clear_free_pages(uint4* __restrict__ pool, const int* __restrict__ offsets, int batch, int pages_per_seq, int max_batch, int page_size,
                 int pair_vecs, int share, unsigned int* __restrict__ item_counter) {
  if (blockIdx.x + blockIdx.y + threadIdx.x == 0) *item_counter = 0u;   // (of attention_umma: an attention that gave up a wait may have left it set)
  // grid (sequences times the CTAs that share one's pages, layers * heads); pool page p * max_batch + b is page p of sequence b
  const int b = blockIdx.x / share, len = b < batch ? offsets[b + 1] - offsets[b] : 0;
  uint4* base = pool + ((size_t)blockIdx.y * pages_per_seq * max_batch + b) * pair_vecs;
  for (int p = len / page_size + blockIdx.x % share; p < pages_per_seq; p += share)
    for (int i = threadIdx.x; i < pair_vecs; i += blockDim.x) base[(size_t)p * max_batch * pair_vecs + i] = make_uint4(0, 0, 0, 0);
}

// ------------------------------------------------------------------ RMSNorm (+ residual)
// u[m] = T(x[m] / rms(x[m]) * g); optionally the unrounded normed row goes to hid (final norm).
template <typename T>
__global__ void rmsnorm_rows(const float* __restrict__ x, const float* __restrict__ gain, float eps, T* __restrict__ u,
                             float* __restrict__ hid, int d, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  int m = blockIdx.x;
  const float* xr = x + (size_t)m * d;
  float ss = 0.f;
  for (int c = threadIdx.x; c < d; c += blockDim.x) {
    const float v = xr[c];
    ss += v * v;
  }
  __shared__ float red[32];
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x < 32) {
    float v = threadIdx.x < (blockDim.x >> 5) ? red[threadIdx.x] : 0.f;
    v = warp_sum(v);
    if (threadIdx.x == 0) red[0] = v;
  }
  __syncthreads();
  float inv = rsqrtf(red[0] / (float)d + eps);
  for (int c = threadIdx.x; c < d; c += blockDim.x) {
    float v = xr[c] * inv * gain[c];
    u[(size_t)m * d + c] = from_f<T>(v);
    if (hid) hid[(size_t)m * d + c] = v;
  }
}

// ------------------------------------------------------------------ row-streaming linear
// y[m][n] = sum_k x[m][k] * W[n][k] for MC rows m at a time; one warp per output n streams
// the weight row once with 16-byte loads. K % 8 == 0.
template <typename T> struct Vec16;
template <> struct Vec16<float> {
  static constexpr int N = 4;
  template <int S> __device__ static void load(const float* p, float (&o)[S]) {
    float4 v = *reinterpret_cast<const float4*>(p);
    o[0] = v.x; o[1] = v.y; o[2] = v.z; o[3] = v.w;
  }
};
template <> struct Vec16<bf16> {
  static constexpr int N = 8;
  template <int S> __device__ static void load(const bf16* p, float (&o)[S]) {
    uint4 v = *reinterpret_cast<const uint4*>(p);
    const __nv_bfloat162* h = reinterpret_cast<const __nv_bfloat162*>(&v);
#pragma unroll
    for (int i = 0; i < 4; ++i) { float2 f = __bfloat1622float2(h[i]); o[2 * i] = f.x; o[2 * i + 1] = f.y; }
  }
};

// A warp computes LR_N outputs of LR_M rows: per step of the inner dimension it fetches LR_N pieces of weight rows and LR_M
// of activation rows and does LR_N * LR_M products with each, and the 32 sums are reduced over the lanes by halving (31
// shuffles; lane l ends up with sum l). Bound by latency at the widths of the float32 configuration, so the first
// weights are fetched before the dependency wait and, where that still leaves the chip half empty, `ks` warps share a
// group of outputs and split the inner dimension. The other warps of a CTA take `ms` groups of rows of the same outputs, which
// then come out of L2 once: at lm_head (32016 x 256, 16 rows) the weights crossing L2 are the bound. What follows the
// projection is done in place of a kernel of its own.
constexpr int LR_N = 4, LR_M = 8, LR_WARPS = 4;
constexpr int LR_PLAIN = 0, LR_SWIGLU = 1, LR_RESIDUAL = 2, LR_ROPE = 3;
template <typename T> struct RowLinear {
  const T* w[3];          // stacked matrices (LR_SWIGLU: gate, up)
  int rows[3];            // their rows
  int group0[3];          // first group of LR_N outputs of each (LR_SWIGLU: groups of LR_N / 2 columns, one range)
  int n_mats;
};

// LR_ROPE (q, k, v): rotate-half RoPE (element i pairs with i + D/2, angle pos * base^(-2i/D)) on q and k in registers; q -> T [M][H*D], k and v -> T into the
// paged cache at the row's slot. A group of q or k is the outputs e, e + 1 and their partners in the other half of the head. A kernel of its own behind the
// projection took 3 us a layer, nearly all of it a launch and two trips to L2 (the row's slot, its page): the projection makes these while its sums are formed.
// A request of the two-layer configuration 2.34 -> 2.25 ms. Which product the rotation fuses is fixed, as that kernel had it.
template <typename T> struct RopeStore {
  Rows rows;
  const float2* cs;       // [position][head_dim / 2] (cos, sin)
  T* q;
  T* pool;
  KVGeom g;
  const int* page_table;
  int layer, H;
};

// Warps that share a group of outputs: as many as have a step of the inner dimension each, while 16 rows (the verification
// pass of a small tree) leave the chip's resident warps, LR_WARPS * 4 an SM, room for them. The number of rows is left out on
// purpose: the split decides the order of a row's sums, and a row's result must not depend on what it is computed with.
// (Choosing by the rows of the call as well gained nothing up to 128 rows: a 24-step request of the two-layer configuration takes
// 3.1 ms either way. From 512 rows a narrow projection is slower for it: 768 x 256 at 512 rows 23 us instead of 16.)
template <typename T> inline int linear_rows_split(int groups, int K) {
  constexpr int RESIDENT = 148 * LR_WARPS * 4, ROW_GROUPS = 16 / LR_M;
  const int steps = K / (32 * Vec16<T>::N), warps = groups * ROW_GROUPS;
  return steps >= 4 && warps * 4 <= RESIDENT ? 4 : (steps >= 2 && warps * 2 <= RESIDENT ? 2 : 1);
}

struct RowLinearShape {
  int ks, ms;
  dim3 grid;
};
template <typename T> inline RowLinearShape linear_rows_shape(int groups, int M, int K) {
  RowLinearShape s;
  const int mg = (M + LR_M - 1) / LR_M;
  s.ks = linear_rows_split<T>(groups, K);
  s.ms = 1;
  while (s.ms * 2 <= LR_WARPS / s.ks && s.ms < mg) s.ms *= 2;
  const int per = LR_WARPS / (s.ks * s.ms);
  s.grid = dim3((groups + per - 1) / per, (mg + s.ms - 1) / s.ms);
  // many outputs: four CTAs per SM walk over the groups, each fetching its next weights ahead
  if (s.ks == 1) s.grid.x = std::min(s.grid.x, std::max(1u, 4u * 148u / s.grid.y));
  return s;
}

template <typename T, int MODE>
__global__ void __launch_bounds__(LR_WARPS * 32, 4)
linear_rows(const T* __restrict__ x, const RowLinear<T> w, float* __restrict__ y, size_t ldy, T* __restrict__ act, int M, int K, int groups, int ks, int ms,
            const RopeStore<T> rs, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  constexpr int VN = Vec16<T>::N;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int kpart = warp % ks, mpart = (warp / ks) % ms;
  const int per = LR_WARPS / (ks * ms), m0 = (blockIdx.y * ms + mpart) * LR_M;
  int g = blockIdx.x * per + warp / (ks * ms);
  // where the current group's outputs are: its matrix, first row there, first column of y
  const T *wa, *wb;
  int N, n0, col0, up = 2;                                     // (a group's outputs: n0, n0 + 1, n0 + up, n0 + up + 1)
  const int D = MODE == LR_ROPE ? rs.g.head_dim : 0, half = D >> 1;
  auto locate = [&](int gg) {
    if (MODE == LR_ROPE) {
      const int mat = gg >= w.group0[2] ? 2 : (gg >= w.group0[1] ? 1 : 0), gi = gg - (mat == 0 ? 0 : (mat == 1 ? w.group0[1] : w.group0[2]));
      wa = wb = mat == 0 ? w.w[0] : (mat == 1 ? w.w[1] : w.w[2]);
      N = mat == 0 ? w.rows[0] : (mat == 1 ? w.rows[1] : w.rows[2]);
      up = mat == 2 ? 2 : half;
      n0 = mat == 2 ? gi * LR_N : gi / (half / 2) * D + gi % (half / 2) * 2;
      col0 = mat;
      return;
    }
    if (MODE == LR_SWIGLU) { wa = w.w[0]; wb = w.w[1]; N = w.rows[0]; n0 = gg * (LR_N / 2); col0 = 0; return; }
    const int mat = w.n_mats > 2 && gg >= w.group0[2] ? 2 : (w.n_mats > 1 && gg >= w.group0[1] ? 1 : 0);
    wa = wb = mat == 0 ? w.w[0] : (mat == 1 ? w.w[1] : w.w[2]);
    N = mat == 0 ? w.rows[0] : (mat == 1 ? w.rows[1] : w.rows[2]);
    n0 = (gg - (mat == 0 ? 0 : (mat == 1 ? w.group0[1] : w.group0[2]))) * LR_N;
    col0 = mat == 0 ? 0 : (mat == 1 ? w.rows[0] : w.rows[0] + w.rows[1]);
  };
  float wv[LR_N][VN], xv[LR_M][VN];
  // (rows past the end of a matrix repeat its last row and are not stored)
  auto load_w = [&](int k) {
#pragma unroll
    for (int j = 0; j < LR_N; ++j) {
      const int n = min(MODE == LR_SWIGLU ? n0 + (j & 1) : (MODE == LR_ROPE ? n0 + (j & 1) + (j >> 1) * up : n0 + j), N - 1);
      Vec16<T>::load((j < 2 ? wa : wb) + (size_t)n * K + k, wv[j]);
    }
  };
  const int k0 = (kpart * 32 + lane) * VN;
  locate(g);
  if (k0 < K) load_w(k0);
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  // LR_ROPE: where this lane's row stands (its sums come last)
  int pos = -1, page = 0, prow = 0;
  if (MODE == LR_ROPE && kpart == 0 && m0 + lane % LR_M < M) {
    const int m = m0 + lane % LR_M, b = m / rs.rows.R;
    if (m - b * rs.rows.R < rs.rows.cnt[b]) {
      const int slot = rs.rows.slot[m];
      pos = rs.rows.pos[m];
      page = rs.page_table[rs.rows.sequence(b) * rs.g.pages_per_seq + slot / rs.g.page_size];
      prow = slot % rs.g.page_size;
    }
  }
  for (;;) {
    float v[LR_N * LR_M];
#pragma unroll
    for (int i = 0; i < LR_N * LR_M; ++i) v[i] = 0.f;
    const int n_this = n0, N_this = N, col_this = col0, up_this = up;
    g += gridDim.x * per;
    const bool more = g < groups;
    for (int k = k0; k < K;) {
#pragma unroll
      for (int i = 0; i < LR_M; ++i) Vec16<T>::load(x + (size_t)min(m0 + i, M - 1) * K + k, xv[i]);
#pragma unroll
      for (int j = 0; j < LR_N; ++j)
#pragma unroll
        for (int i = 0; i < LR_M; ++i)
#pragma unroll
          for (int e = 0; e < VN; ++e) v[j * LR_M + i] = fmaf(wv[j][e], xv[i][e], v[j * LR_M + i]);
      k += ks * 32 * VN;
      if (k < K) load_w(k);
    }
    float2 t = make_float2(1.f, 0.f);
    if (MODE == LR_ROPE && pos >= 0 && col_this < 2) t = rs.cs[(size_t)pos * half + n_this % D + ((lane / LR_M) & 1)];
    // the next group's first weights are on their way while this one's sums are reduced
    if (more) { locate(g); if (k0 < K) load_w(k0); }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const bool hi = (lane & o) != 0;
#pragma unroll
      for (int t = 0; t < o; ++t) {
        const float send = hi ? v[t] : v[t + o], keep = hi ? v[t + o] : v[t];
        v[t] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    if (ks > 1) {                                             // (one group a warp: the loop ends here)
      __shared__ float parts[LR_WARPS][32];
      if (kpart) parts[warp][lane] = v[0];
      __syncthreads();
      if (kpart) return;
      for (int i = 1; i < ks; ++i) v[0] += parts[warp + i][lane];
    }
    const int j = lane / LR_M, m = m0 + lane % LR_M;
    if (MODE == LR_ROPE) {
      const float other = __shfl_xor_sync(0xffffffffu, v[0], 16);
      const int n = n_this + (j & 1) + (j >> 1) * up_this, head = n / D, e = n - head * D;
      if (pos >= 0) {
        const float r = col_this == 2 ? v[0] : (j < 2 ? __fmaf_rn(v[0], t.x, -__fmul_rn(other, t.y)) : __fmaf_rn(v[0], t.x, __fmul_rn(other, t.y)));
        if (col_this == 0) rs.q[(size_t)m * N_this + n] = from_f<T>(r);
        else rs.pool[rs.g.block_offset(page, rs.layer, col_this - 1, head) + (size_t)prow * D + kv_elem<T>(prow, e, D, rs.g.page_size)] = from_f<T>(r);
      }
    } else if (MODE == LR_SWIGLU) {
      const float up = __shfl_xor_sync(0xffffffffu, v[0], 16);
      const int n = n_this + (j & 1);
      if (j < 2 && m < M && n < N_this) act[(size_t)m * N_this + n] = from_f<T>(silu_f(v[0]) * up);
    } else {
      const int n = n_this + j;
      if (m < M && n < N_this) {
        float* dst = y + (size_t)m * ldy + col_this + n;
        if (MODE == LR_RESIDUAL) *dst += v[0];
        else *dst = v[0];
      }
    }
    if (!more || ks > 1) return;
  }
}

// The same sums (bit for bit) where an inner dimension of at most two steps is not split: lm_head of the float32 configurations. A warp keeps the
// activations of its M_ rows in registers through all its groups of N_ outputs and fetches a whole group's weights while it reduces the
// one before; two rows' products are one instruction. linear_rows fetched the activations again for every group (two thirds of its loads) and
// waited for the second step's weights in each. 32016 outputs of 256: 3 rows in a step 9.4 -> 5.3 us, 16 rows 16.5 -> 13.5, 64 rows 55 -> 42. It is
// bound by what 12 warps an SM have under way. Each row's largest in the columns of a CTA goes to best_val / best_idx [M][gridDim.x] where they are
// given: what follows reads those instead of the logits. (Fetching a step's weights as soon as its products are done, not both after them: 14.6 and 45.)
constexpr int LH_STEPS = 2, LH_CTAS = 3;
using f32x2 = unsigned long long;                              // two float32 in a register pair: one instruction does both products
__device__ __forceinline__ f32x2 f32x2_of(float a, float b) { f32x2 r; asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(a), "f"(b)); return r; }
__device__ __forceinline__ void f32x2_parts(f32x2 v, float& a, float& b) { asm("mov.b64 {%0, %1}, %2;" : "=f"(a), "=f"(b) : "l"(v)); }
__device__ __forceinline__ f32x2 fma_f32x2(f32x2 a, f32x2 b, f32x2 c) { f32x2 r; asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c)); return r; }
template <int N_, int M_>
__global__ void __launch_bounds__(LR_WARPS * 32, LH_CTAS)
linear_rows_held(const float* __restrict__ x, const float* __restrict__ w, float* __restrict__ y, size_t ldy, int M, int N, int K, int ms,
                 float* __restrict__ best_val, int* __restrict__ best_idx, unsigned long long* tr) {
  static_assert(N_ * M_ == 32, "a lane a sum");
  KTrace kt(tr);
  pdl_launch_dependents();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int per = LR_WARPS / ms, m0 = (blockIdx.y * ms + warp % ms) * M_, groups = (N + N_ - 1) / N_;
  float4 wv[LH_STEPS][N_];
  f32x2 xv[LH_STEPS][M_ / 2][4];                               // two rows' values of an element side by side
  const int k0 = lane * 4;
  auto load_w = [&](int g) {                                   // (rows past the end repeat the last one and are not stored)
#pragma unroll
    for (int s = 0; s < LH_STEPS; ++s)
#pragma unroll
      for (int j = 0; j < N_; ++j)
        if (k0 + s * 128 < K) wv[s][j] = *reinterpret_cast<const float4*>(w + (size_t)min(g * N_ + j, N - 1) * K + k0 + s * 128);
  };
  int g = blockIdx.x * per + warp / ms;
  if (g < groups) load_w(g);
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  float bv = -INFINITY;
  int bi = 0x7fffffff;
#pragma unroll
  for (int s = 0; s < LH_STEPS; ++s)
#pragma unroll
    for (int i = 0; i < M_ / 2; ++i)
      if (k0 + s * 128 < K) {
        const float4 a = *reinterpret_cast<const float4*>(x + (size_t)min(m0 + 2 * i, M - 1) * K + k0 + s * 128);
        const float4 b = *reinterpret_cast<const float4*>(x + (size_t)min(m0 + 2 * i + 1, M - 1) * K + k0 + s * 128);
        xv[s][i][0] = f32x2_of(a.x, b.x); xv[s][i][1] = f32x2_of(a.y, b.y); xv[s][i][2] = f32x2_of(a.z, b.z); xv[s][i][3] = f32x2_of(a.w, b.w);
      }
  while (g < groups) {
    f32x2 v2[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) v2[i] = 0;
#pragma unroll
    for (int s = 0; s < LH_STEPS; ++s)
      if (k0 + s * 128 < K) {
#pragma unroll
        for (int j = 0; j < N_; ++j) {
          const float e[4] = {wv[s][j].x, wv[s][j].y, wv[s][j].z, wv[s][j].w};
#pragma unroll
          for (int k = 0; k < 4; ++k)
#pragma unroll
            for (int i = 0; i < M_ / 2; ++i) v2[j * (M_ / 2) + i] = fma_f32x2(f32x2_of(e[k], e[k]), xv[s][i][k], v2[j * (M_ / 2) + i]);
        }
      }
    const int n = g * N_ + lane / M_, m = m0 + lane % M_;
    g += gridDim.x * per;
    if (g < groups) load_w(g);
    float v[32];
#pragma unroll
    for (int i = 0; i < 16; ++i) f32x2_parts(v2[i], v[2 * i], v[2 * i + 1]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const bool hi = (lane & o) != 0;
#pragma unroll
      for (int t = 0; t < o; ++t) {
        const float send = hi ? v[t] : v[t + o], keep = hi ? v[t + o] : v[t];
        v[t] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
    }
    if (m < M && n < N) y[(size_t)m * ldy + n] = v[0];
    if (n < N && better(v[0], n, bv, bi)) { bv = v[0]; bi = n; }
  }
  if (!best_val) return;
  __shared__ float sv[LR_WARPS][M_];
  __shared__ int si[LR_WARPS][M_];
#pragma unroll
  for (int o = M_; o < 32; o <<= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
  }
  if (lane < M_) { sv[warp][lane] = bv; si[warp][lane] = bi; }
  __syncthreads();
  const int m = m0 + lane;
  if (warp >= ms || lane >= M_ || m >= M) return;
  for (int k = warp + ms; k < LR_WARPS; k += ms) if (better(sv[k][lane], si[k][lane], bv, bi)) { bv = sv[k][lane]; bi = si[k][lane]; }
  best_val[(size_t)m * gridDim.x + blockIdx.x] = bv;
  best_idx[(size_t)m * gridDim.x + blockIdx.x] = bi;
}
inline bool linear_held(const RowLinearShape& s, int K) { return s.ks == 1 && K <= LH_STEPS * 128; }
// (Up to 4 rows: half the loads a sum; the rows of linear_rows's shape otherwise.) A CTA's columns are every grid.x-th piece of `piece`. Neighbouring pieces
// instead: 3 rows 5.3 -> 6.8 us, 64 rows 42 -> 45.
struct HeldShape { dim3 grid; int cols, ms, piece; };
inline HeldShape linear_held_shape(const RowLinearShape& s, int M, int N) {
  HeldShape h;
  h.cols = M <= 4 ? 8 : 4; h.ms = M <= 4 ? 1 : s.ms;
  h.piece = LR_WARPS / h.ms * h.cols;
  const unsigned y = M <= 4 ? 1u : s.grid.y;
  h.grid = dim3(std::min((unsigned)((N + h.piece - 1) / h.piece), std::max(1u, LH_CTAS * 148u / y)), y);
  return h;
}

// ------------------------------------------------------------------ plain tree attention
// Row i of sequence b sees every cached position < n[b] and row u of the same pass iff bit u of anc[i] is set. A CTA takes
// ROWS query rows of one head and stages tiles of KT keys and values in shared memory (all of them in
// one tile for the contexts of the float32 configuration); within a group of 32 keys a lane owns a key for the scores and
// every 32nd dimension for the values. Two passes over the keys: maximum, then exp / sum / value accumulation with the
// probabilities rounded to T before the product; with one tile the scores stay in registers in between. (With a warp that
// walked the keys one by one out of L2, twice, a 16-node step of the two-layer configuration at 60 positions took 320 us in
// all; with this, the row linear above and their fused steps 138.) Bound by latency: the chain of loads (length, page, keys), then what a
// warp has to do for its row. So where that leaves the CTAs resident at once a row gets AP_WARPS / AP_FEW warps, which share its groups of keys and
// then its dimensions (every sum in the order it has with one warp), and a thread has AP_DEEP key and value loads under way, not one:
// 16 rows of 4 heads at 60 positions 7.5 -> 3.4 us a layer.
constexpr int AP_WARPS = 8, AP_GROUPS = 4;      // at most AP_GROUPS * 32 keys a tile
constexpr int AP_FEW = 2, AP_DEEP = 4;
__host__ __device__ constexpr int attention_plain_tile(int D) { return D <= 64 ? 128 : (D <= 128 ? 64 : 32); }
inline size_t attention_plain_smem(int D) { return ((size_t)2 * attention_plain_tile(D) * (D + 4) + (size_t)AP_WARPS * D) * sizeof(float); }

template <typename T, int EPL, int ROWS>
__global__ void __launch_bounds__(AP_WARPS * 32)
attention_plain(const T* __restrict__ q, T* __restrict__ out, const T* __restrict__ pool, KVGeom g,
                const int* __restrict__ page_table, Rows rows, int layer, int H, float scale, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  extern __shared__ __align__(16) float sm_plain[];
  constexpr int D = EPL * 32, P = D + 4, KT = attention_plain_tile(D), groups = KT / 32, PARTS = AP_WARPS / ROWS;
  float* ks = sm_plain;
  float* vs = ks + KT * P;
  float* qs = vs + KT * P;
  __shared__ long long ko[AP_GROUPS * 32];     // a key's offset in the pool, -1 past the end, and its row in its page
  __shared__ int kr_s[AP_GROUPS * 32];
  __shared__ __align__(16) float ps[ROWS][AP_GROUPS * 32];      // a tile's probabilities, in the operands' type
  __shared__ float pl[PARTS > 1 ? ROWS : 1][AP_GROUPS * 32];    // ... and as they go into the sum
  __shared__ float mx_s[ROWS][PARTS];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, row = warp / PARTS, part = warp % PARTS;
  const int h = blockIdx.x, b = blockIdx.y, i0 = blockIdx.z * ROWS;
  const int kvh = h / (H / g.n_kv_heads);
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  const int* pt = page_table + rows.sequence(b) * g.pages_per_seq;
  const int page0 = pt[min((int)threadIdx.x / g.page_size, g.pages_per_seq - 1)];   // of this thread's key of the first tile (with the loads below)
  const int cnt = rows.cnt[b], n = rows.n[b];
  if (i0 >= cnt) return;
  const int S = n + cnt;
  const int i = i0 + row;
  const bool on = i < cnt;
  const size_t m = (size_t)b * rows.R + i;
  uint32_t a[4];
#pragma unroll
  for (int w = 0; w < 4; ++w) a[w] = on ? rows.anc[i * 4 + w] : 0u;
  if (on) for (int e = part * 32 + lane; e < D; e += PARTS * 32) qs[row * D + e] = to_f<T>(q[m * H * D + h * D + e]);
  // keys [k0, k0 + KT) and, where asked, their values; rows past the end (up to a whole group of 32) are zeros. The
  // divisions by the page size are done once a key; D / 4 lanes (or the warp) then copy a row, AP_DEEP rows under way at a time.
  constexpr int per = D / 4, rpw = per <= 32 ? 32 / per : 1;
  const int sub = per <= 32 ? lane / per : 0, e0 = per <= 32 ? lane - sub * per : lane;
  auto stage = [&](int k0, bool values) {
    const int live = min(KT, (S - k0 + 31) & ~31);
    for (int r = threadIdx.x; r < live; r += AP_WARPS * 32) {
      const int j = k0 + r;
      long long o = -1;
      if (j < S) {
        const int pg = j / g.page_size, prow = j - pg * g.page_size;
        o = (long long)(g.block_offset(k0 ? pt[pg] : page0, layer, 0, kvh) + (size_t)prow * D);
        kr_s[r] = prow;
      }
      ko[r] = o;
    }
    __syncthreads();
    if (sub >= rpw) return;
    for (int c = e0; c < per; c += 32)
      for (int r0 = warp * rpw + sub; r0 < live; r0 += AP_DEEP * AP_WARPS * rpw) {
        float4 kv[AP_DEEP], vv[AP_DEEP];
#pragma unroll
        for (int u = 0; u < AP_DEEP; ++u) {
          const int r = r0 + u * AP_WARPS * rpw;
          kv[u] = vv[u] = make_float4(0.f, 0.f, 0.f, 0.f);
          const long long o = r < live ? ko[r] : -1;
          if (o >= 0) {
            const T* kr = pool + o;
            const T* vr = kr + g.block_elems();
            const int e = kv_elem<T>(kr_s[r], c * 4, D, g.page_size);   // four neighbouring elements stay together
            if (sizeof(T) == 4) {
              kv[u] = *reinterpret_cast<const float4*>(kr + e);
              if (values) vv[u] = *reinterpret_cast<const float4*>(vr + e);
            } else {
              kv[u] = make_float4(to_f<T>(kr[e]), to_f<T>(kr[e + 1]), to_f<T>(kr[e + 2]), to_f<T>(kr[e + 3]));
              if (values) vv[u] = make_float4(to_f<T>(vr[e]), to_f<T>(vr[e + 1]), to_f<T>(vr[e + 2]), to_f<T>(vr[e + 3]));
            }
          }
        }
#pragma unroll
        for (int u = 0; u < AP_DEEP; ++u) {
          const int r = r0 + u * AP_WARPS * rpw;
          if (r < live) {
            *reinterpret_cast<float4*>(ks + r * P + c * 4) = kv[u];
            if (values) *reinterpret_cast<float4*>(vs + r * P + c * 4) = vv[u];
          }
        }
      }
  };
  auto score = [&](int k0, int gr) {
    const int j = k0 + gr * 32 + lane;
    const int u = j - n;                                          // node of this pass, or negative
    const uint32_t word = u < 64 ? (u < 32 ? a[0] : a[1]) : (u < 96 ? a[2] : a[3]);
    const bool vis = on && j < S && (u < 0 || ((word >> (u & 31)) & 1u));
    const float4* kr = reinterpret_cast<const float4*>(ks + (gr * 32 + lane) * P);
    const float4* qr = reinterpret_cast<const float4*>(qs + row * D);
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int e = 0; e < D / 4; ++e) {
      const float4 kv = kr[e], qv = qr[e];
      s.x = fmaf(qv.x, kv.x, s.x); s.y = fmaf(qv.y, kv.y, s.y); s.z = fmaf(qv.z, kv.z, s.z); s.w = fmaf(qv.w, kv.w, s.w);
    }
    return vis ? ((s.x + s.y) + (s.z + s.w)) * scale : -INFINITY;
  };
  const int tiles = (S + KT - 1) / KT;
  constexpr int MINE = (groups + PARTS - 1) / PARTS;              // groups of keys of a tile whose scores are this warp's: part, part + PARTS, ...
  float keep[MINE], mx = -INFINITY;
  for (int t = 0; t < tiles; ++t) {
    __syncthreads();
    stage(t * KT, tiles == 1);
    __syncthreads();
#pragma unroll
    for (int k = 0; k < MINE; ++k) {
      const int gr = part + k * PARTS;
      keep[k] = -INFINITY;
      if (gr < groups && t * KT + gr * 32 < S) keep[k] = score(t * KT, gr);
      mx = fmaxf(mx, keep[k]);
    }
  }
  mx = warp_max(mx);
  if (PARTS > 1) {
    if (lane == 0) mx_s[row][part] = mx;
    __syncthreads();
#pragma unroll
    for (int k = 0; k < PARTS; ++k) mx = fmaxf(mx, mx_s[row][k]);
  }
  constexpr int DIMS = (EPL + PARTS - 1) / PARTS;                 // and the dimensions lane + 32 * (part, part + PARTS, ...) of the values
  float l = 0.f, acc[DIMS];
#pragma unroll
  for (int e = 0; e < DIMS; ++e) acc[e] = 0.f;
  for (int t = 0; t < tiles; ++t) {
    if (tiles > 1) {
      __syncthreads();
      stage(t * KT, true);
      __syncthreads();
    }
#pragma unroll
    for (int k = 0; k < MINE; ++k) {
      const int gr = part + k * PARTS;
      if (gr >= groups || t * KT + gr * 32 >= S) continue;
      const float s = tiles > 1 ? score(t * KT, gr) : keep[k];
      const float p = s == -INFINITY ? 0.f : expf(s - mx);       // (keys a row does not see carry no weight)
      ps[row][gr * 32 + lane] = quant<T>(p);
      if (PARTS > 1) pl[PARTS > 1 ? row : 0][gr * 32 + lane] = p;
      else l += p;
    }
    if (PARTS > 1) __syncthreads();
    else __syncwarp();
#pragma unroll
    for (int gr = 0; gr < groups; ++gr) {
      if (t * KT + gr * 32 >= S) continue;
      if (PARTS > 1) l += pl[PARTS > 1 ? row : 0][gr * 32 + lane];
      if (part >= EPL) continue;
      const float* vr = vs + gr * 32 * P + lane + part * 32;
#pragma unroll
      for (int k4 = 0; k4 < 8; ++k4) {
        const float4 p4 = *reinterpret_cast<const float4*>(&ps[row][gr * 32 + k4 * 4]);
        const float pk[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
        for (int kk = 0; kk < 4; ++kk)
#pragma unroll
          for (int e = 0; e < DIMS; ++e)                         // (a key without weight is left out whatever its values are)
            if (EPL % PARTS == 0 || part + e * PARTS < EPL)
              acc[e] = fmaf(pk[kk], pk[kk] != 0.f ? vr[(k4 * 4 + kk) * P + e * PARTS * 32] : 0.f, acc[e]);
      }
    }
    if (PARTS == 1) __syncwarp();
  }
  if (!on) return;
  const float inv = 1.f / warp_sum(l);
#pragma unroll
  for (int e = 0; e < DIMS; ++e)
    if (part + e * PARTS < EPL) out[m * H * D + h * D + lane + (part + e * PARTS) * 32] = from_f<T>(acc[e] * inv);
}

// ------------------------------------------------------------------ typical acceptance
// Eq. 1: a node passes iff p_base(token | prefix ending at its parent) >
// min(eps, delta * exp(-H(p_base))). One block per row that is some node's parent: it reduces the row's logits
// (softmax at the given temperature, entropy in nats) and decides all the row's children. A thread fetches its
// TYP_CACHE float4 of the row (all of it for vocabularies of up to 32768) before it uses the first and keeps them for
// the second pass; on the 7B shape 6.8 us for 64 nodes. (One block per node and
// two passes over memory before: this kernel and sample_root took 107 us of a step together, now 13.)
constexpr int TYP_THREADS = 1024, TYP_CACHE = 8;
__global__ void __launch_bounds__(TYP_THREADS)
typical_edges(const float* __restrict__ logits, int V, Rows rows, const int* __restrict__ parent,
              float eps, float delta, float inv_temp, int* __restrict__ edge_ok, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  __shared__ float red[32], red2[32];
  const int m = blockIdx.x, b = m / rows.R, u = m % rows.R, tid = threadIdx.x;
  const int warp = tid >> 5, lane = tid & 31;
  // the tree is fixed at set-up: its parents are read before the dependency wait (R <= 128 threads hold a node each)
  const bool child = tid > 0 && tid < rows.R && parent[tid] == u;
  const int any = __syncthreads_or(child);
  pdl_wait();
  if (tid == 0) trace_mark_min(tr, 2);
  const int cnt = rows.cnt[b];
  if (u == 0 && tid == 0 && cnt > 0) edge_ok[m] = 1;
  if (!any || u >= cnt) return;
  const float* z = logits + (size_t)m * V;
  const bool vec = (V & 3) == 0;
  const int v4 = vec ? V >> 2 : 0;
  float4 keep[TYP_CACHE];
#pragma unroll
  for (int k = 0; k < TYP_CACHE; ++k) {
    const int c = tid + k * TYP_THREADS;
    keep[k] = c < v4 ? *reinterpret_cast<const float4*>(z + 4 * c) : make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
  }
  const int rest0 = vec ? 4 * TYP_CACHE * TYP_THREADS : 0;     // elements from here on are read twice
  float mx = -INFINITY;
#pragma unroll
  for (int k = 0; k < TYP_CACHE; ++k)
    mx = fmaxf(fmaxf(mx, fmaxf(keep[k].x * inv_temp, keep[k].y * inv_temp)), fmaxf(keep[k].z * inv_temp, keep[k].w * inv_temp));
  for (int c = rest0 + tid; c < V; c += TYP_THREADS) mx = fmaxf(mx, z[c] * inv_temp);
  mx = warp_max(mx);
  if (lane == 0) red[warp] = mx;
  __syncthreads();
  mx = warp_max(red[lane]);
  __syncthreads();
  float se = 0.f, sez = 0.f;   // sum e, sum e * (z - mx)
  auto add = [&](float x) {
    const float t = x * inv_temp - mx;
    const float e = expf(t);
    se += e;
    sez += e * t;
  };
#pragma unroll
  for (int k = 0; k < TYP_CACHE; ++k)
    if (tid + k * TYP_THREADS < v4) { add(keep[k].x); add(keep[k].y); add(keep[k].z); add(keep[k].w); }
  for (int c = rest0 + tid; c < V; c += TYP_THREADS) add(z[c]);
  se = warp_sum(se);
  sez = warp_sum(sez);
  if (lane == 0) { red[warp] = se; red2[warp] = sez; }
  __syncthreads();
  se = warp_sum(red[lane]);
  sez = warp_sum(red2[lane]);
  if (child && tid < cnt) {
    const float H = logf(se) - sez / se;                        // -sum p log p with p = e / se
    const float thr = fminf(eps, delta * expf(-H));
    const float p = expf(z[rows.tok[b * rows.R + tid]] * inv_temp - mx) / se;
    edge_ok[b * rows.R + tid] = p > thr ? 1 : 0;
  }
}

// ------------------------------------------------------------------ sampled decoding
// Philox-4x32, 10 rounds (Salmon et al., SC 2011): counter c[4], key k[2] -> four 32-bit words.
__device__ __forceinline__ void philox4x32_10(uint32_t (&c)[4], uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int r = 0; r < 10; ++r) {
    if (r) { k0 += 0x9E3779B9u; k1 += 0xBB67AE85u; }
    const uint32_t hi0 = __umulhi(0xD2511F53u, c[0]), lo0 = 0xD2511F53u * c[0];
    const uint32_t hi1 = __umulhi(0xCD9E8D57u, c[2]), lo1 = 0xCD9E8D57u * c[2];
    const uint32_t n0 = hi1 ^ c[1] ^ k0, n2 = hi0 ^ c[3] ^ k1;
    c[0] = n0; c[1] = lo1; c[2] = n2; c[3] = lo0;
  }
}

// Sampled decoding at a temperature (Sec. IV-B: every prompt is also decoded by sampling): the
// token that follows the accepted span is drawn from softmax(logits / temperature) of the last
// accepted node by inverting the cumulative distribution in token order at the uniform
// u = top 24 bits of philox(counter = (draw index, sequence, 0, 0), key = seed) * 2^-24.
// A cluster of SAMPLE_CLUSTER CTAs per sequence; every thread owns a contiguous run of the vocabulary and adds its
// weights in double precision, relative to the row's largest logit (row_max, left by the argmax). Prefix sums over the
// threads of a CTA and over the CTAs (distributed shared memory) give the weight before each run; the one thread whose
// run holds u * total scans it. prefill != 0: the row is the sequence's last prompt position (row b). Bound by the
// double-precision exponentials of 32016 tokens: 4096 threads with 8 each take 6.3 us (one CTA
// of 256 threads with 126 each, reading them twice, and 512 additions by one thread before).
constexpr int SAMPLE_CLUSTER = 8, SAMPLE_THREADS = 512;
__global__ void __cluster_dims__(SAMPLE_CLUSTER, 1, 1) __launch_bounds__(SAMPLE_THREADS)
sample_root(const float* __restrict__ logits, const float* __restrict__ row_max, int V, int R, int K, const int* __restrict__ path,
            const int* __restrict__ count, float temperature, uint32_t seed_lo, uint32_t seed_hi,
            int* __restrict__ draws, int* __restrict__ root_tok, int prefill, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  __shared__ double wsum[SAMPLE_THREADS / 32];
  __shared__ double total_s;                 // weight of this CTA's tokens, read by the whole cluster
  __shared__ int pick_s;                     // rank 0: the drawn token, the last one until a run claims it
  const int b = blockIdx.y, rank = blockIdx.x, tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  int row = b;
  bool on = true;
  if (!prefill) {
    const int len = count[b];
    on = len >= 1;                           // the same for every CTA of the cluster
    if (on) row = b * R + path[b * (K + 1) + len - 1];
  }
  const float* z = logits + (size_t)row * V;
  const double inv_t = 1.0 / (double)temperature;
  const double mx = (double)row_max[row] * inv_t;
  const int runs = SAMPLE_CLUSTER * SAMPLE_THREADS, per = (V + runs - 1) / runs;
  const int run = rank * SAMPLE_THREADS + tid;
  const int c0 = min(V, run * per), c1 = min(V, c0 + per);
  double sum = 0.0;
  if (on) for (int c = c0; c < c1; ++c) sum += exp((double)z[c] * inv_t - mx);
  double incl = sum;                         // inclusive prefix over the warp, then over the CTA
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const double v = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 31) wsum[warp] = incl;
  __syncthreads();
  double before = incl - sum, cta = 0.0;
#pragma unroll
  for (int w = 0; w < SAMPLE_THREADS / 32; ++w) {
    if (w < warp) before += wsum[w];
    cta += wsum[w];
  }
  if (tid == 0) { total_s = cta; if (rank == 0) pick_s = V - 1; }
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  double total = 0.0;
#pragma unroll
  for (int r = 0; r < SAMPLE_CLUSTER; ++r) {
    uint32_t remote;
    double v;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(&total_s)), "r"(r));
    asm volatile("ld.shared::cluster.f64 %0, [%1];" : "=d"(v) : "r"(remote) : "memory");
    if (r < rank) before += v;
    total += v;
  }
  uint32_t ctr[4] = {(uint32_t)draws[b], (uint32_t)b, 0u, 0u};
  philox4x32_10(ctr, seed_lo, seed_hi);
  const double u = (double)(ctr[0] >> 8) * (1.0 / 16777216.0);
  const double target = u * total;
  // The first run whose end passes the target holds the token: of every warp the lowest such run is scanned and the
  // lowest token wins (should rounding keep all runs below the target, the last token is the answer).
  const unsigned past = __ballot_sync(0xffffffffu, on && c0 < c1 && before + sum > target);
  if (past && lane == __ffs(past) - 1) {
    double acc = before;
    int pick = c1 - 1;
    for (int c = c0; c < c1; ++c) {
      acc += exp((double)z[c] * inv_t - mx);
      if (acc > target) { pick = c; break; }
    }
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(&pick_s)), "r"(0));
    asm volatile("red.relaxed.cluster.shared::cluster.min.s32 [%0], %1;" ::"r"(remote), "r"(pick) : "memory");
  }
  __syncwarp();
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  if (on && rank == 0 && tid == 0) { root_tok[b] = pick_s; draws[b] += 1; }
}

// ------------------------------------------------------------------ bounded-wait self test
// One warp waits on an mbarrier that nothing will ever complete, with the given time limit: the wait
// gives up, records ST_TIMEOUT with where = 99 in the status word and the kernel returns normally.
__global__ void wait_probe(int* status, unsigned long long limit_ns) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
    mbar_wait(&bar, 0, status, 99, limit_ns);
  }
}

// ------------------------------------------------------------------ acceptance walk
struct AcceptArgs {
  Rows rows;
  const int* pidx;             // [row] argmax of the base logits
  const int *parent, *depth;   // tree arrays [R]
  const int* edge_ok;          // typical mode: per-row pass flag; NULL = greedy token match
  int K, frag_token, d, mode;  // mode 0 = verify step, 1 = prefill (row b is sequence b)
  const int* status;           // mode 1: the status word, which goes to host_status in pinned host memory
  int* host_status;
  const float* hid;            // [rows][d]
  int *am, *path, *count, *out_tok, *n_old, *root_tok;
  float* h_last;
  bf16* hq_last;               // optional bf16 copy of h_last (operand of the extra heads' GEMM)
  int *gen_log, *gen_cnt, gen_cap;
};

// One block per sequence: takes the nodes' argmax, walks the tree (a node is accepted iff its parent is and its
// token is the argmax at the parent, or its Eq. 1 flag is set), takes the deepest accepted node
// (lowest index on ties), applies the fragment-integrity rule, and publishes the step's result
// and the next step's state.
__global__ void __launch_bounds__(256) accept_kernel(AcceptArgs a, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  const int b = blockIdx.x, R = a.rows.R;
  __shared__ int am_s[SPEC_MAX_NODES], tok_s[SPEC_MAX_NODES], par_s[SPEC_MAX_NODES], dep_s[SPEC_MAX_NODES];
  __shared__ int edge_s[SPEC_MAX_NODES];
  __shared__ int last_s, len_s, best_s;
  if (a.mode == 1) {
    if (threadIdx.x == 0) {
      a.am[b] = a.root_tok[b] = a.pidx[b];
      a.gen_cnt[b] = 0;
    }
    if (b == 0 && threadIdx.x < 4) a.host_status[threadIdx.x] = a.status[threadIdx.x];
    return;
  }
  const int cnt = a.rows.cnt[b], m0 = b * R;
  for (int i = threadIdx.x; i < cnt; i += blockDim.x) {
    am_s[i] = a.am[m0 + i] = a.pidx[m0 + i];
    tok_s[i] = a.rows.tok[m0 + i];
    par_s[i] = a.parent[i];
    dep_s[i] = a.depth[i];
    if (a.edge_ok) edge_s[i] = a.edge_ok[m0 + i];
  }
  if (threadIdx.x == 0) best_s = SPEC_MAX_NODES - 1;            // the root
  __syncthreads();
  // a thread per node walks up to the root (at most K + 1 steps): the node is accepted iff every edge on the way passes; the
  // deepest accepted node wins, the lowest index among equals
  for (int v = threadIdx.x; v < cnt; v += blockDim.x) {
    bool ok = true;
    for (int u = v; u > 0 && ok; u = par_s[u]) ok = a.edge_ok ? edge_s[u] != 0 : tok_s[u] == am_s[par_s[u]];
    if (ok) atomicMax(&best_s, dep_s[v] * SPEC_MAX_NODES + (SPEC_MAX_NODES - 1 - v));
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    int len = 0, last = 0;
    for (int j = 0; j <= a.K; ++j) a.path[b * (a.K + 1) + j] = -1;
    if (cnt > 0) {
      const int best = SPEC_MAX_NODES - 1 - best_s % SPEC_MAX_NODES;
      len = dep_s[best] + 1;
      int path[SPEC_MAX_HEADS + 1];
      for (int u = best; u >= 0; u = par_s[u]) path[dep_s[u]] = u;
      if (a.frag_token >= 0) {
        int keep = 1;
        for (int j = 0; j < len; ++j) if (tok_s[path[j]] == a.frag_token) keep = j + 1;
        len = keep;
      }
      int n = a.rows.n[b], gc = a.gen_cnt[b];
      for (int j = 0; j < len; ++j) {
        int t = tok_s[path[j]];
        a.path[b * (a.K + 1) + j] = path[j];
        a.out_tok[b * (a.K + 1) + j] = t;
        if (gc + j < a.gen_cap) a.gen_log[(size_t)b * a.gen_cap + gc + j] = t;
      }
      last = path[len - 1];
      a.n_old[b] = n;
      a.rows.n[b] = n + len;
      a.gen_cnt[b] = gc + len;
      a.root_tok[b] = am_s[last];
    }
    a.count[b] = len;
    last_s = last; len_s = len;
  }
  __syncthreads();
  if (len_s > 0) {
    // the accepted node's hidden row feeds the next step's heads (d % 4 == 0); four groups per
    // thread are loaded before the first store, so the copy is one trip to L2 for most widths
    const float4* src = reinterpret_cast<const float4*>(a.hid + (size_t)(m0 + last_s) * a.d);
    float4* dst = reinterpret_cast<float4*>(a.h_last + (size_t)b * a.d);
    const int n4 = a.d >> 2;
    for (int c0 = threadIdx.x; c0 < n4; c0 += 4 * blockDim.x) {
      float4 v[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int c = c0 + k * blockDim.x;
        v[k] = c < n4 ? src[c] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int c = c0 + k * blockDim.x;
        if (c >= n4) continue;
        dst[c] = v[k];
        if (a.hq_last) {
          __nv_bfloat162 lo = __floats2bfloat162_rn(v[k].x, v[k].y), hi = __floats2bfloat162_rn(v[k].z, v[k].w);
          uint2 pk;
          pk.x = *reinterpret_cast<uint32_t*>(&lo);
          pk.y = *reinterpret_cast<uint32_t*>(&hi);
          *reinterpret_cast<uint2*>(a.hq_last + (size_t)b * a.d + c * 4) = pk;
        }
      }
    }
  }
}

// ------------------------------------------------------------------ KV compaction
// Moves the accepted path's K/V rows from slot n_old + path[j] to slot n_old + j, for every
// layer and KV head. path[j] >= j and strictly increasing, so no row is overwritten that a later j still reads, and
// the rows a CTA moves may all be fetched before the first is stored: the kernel is one chain of dependent loads long
// (path, page, row), whatever the path's length. A thread moves 16 bytes (a chunk of eight 16-bit or four 32-bit elements,
// which the cache layout keeps together) of one row in COMPACT_HEADS neighbouring heads; rows beyond the block's share
// follow in further rounds, in order. On the 7B shape 6.2 -> 2.1 us a step (one row after the other, two bytes a thread).
// The step's result block also goes to pinned host memory from here, which saves a copy behind the step's last kernel.
constexpr int COMPACT_HEADS = 4;
template <typename T>
__global__ void __launch_bounds__(128)
compact_kv(T* __restrict__ pool, KVGeom g, const int* __restrict__ page_table,
           const int* __restrict__ path, const int* __restrict__ count,
           const int* __restrict__ n_old, int K, const int* __restrict__ result, int* __restrict__ host_result, int n_result,
           unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  constexpr int EPC = 16 / sizeof(T);
  const int groups = (g.n_kv_heads + COMPACT_HEADS - 1) / COMPACT_HEADS;
  const int b = blockIdx.y, blk = blockIdx.x;              // (layer*2 + kv) * groups + group of heads
  const int head0 = blk % groups * COMPACT_HEADS, lk = blk / groups;
  const int D = g.head_dim, per = D / EPC;                 // chunks of a row
  const int rows = per >= 128 ? 1 : 128 / per;             // rows a round moves
  const int j0 = threadIdx.x / per, c0 = threadIdx.x - j0 * per;
  const int* pt = page_table + b * g.pages_per_seq;
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  if (blockIdx.x + blockIdx.y == 0)
    for (int i = threadIdx.x; i < n_result; i += 128) host_result[i] = result[i];
  const int len = count[b], n0 = n_old[b];
  const size_t head_stride = g.pool_pages() * 2 * g.block_elems();
  for (int j1 = 0; j1 < len; j1 += rows) {
    const int j = j1 + j0;
    T* to = nullptr;
    uint4 v[COMPACT_HEADS];
    if (j0 < rows && j < len) {
      const int node = path[b * (K + 1) + j], src = n0 + node, dst = n0 + j;
      if (node != j) {
        const int sr = src % g.page_size, dr = dst % g.page_size;
        const T* s = pool + g.block_offset(pt[src / g.page_size], lk >> 1, lk & 1, head0) + (size_t)sr * D + kv_elem<T>(sr, c0 * EPC, D, g.page_size);
        to = pool + g.block_offset(pt[dst / g.page_size], lk >> 1, lk & 1, head0) + (size_t)dr * D + kv_elem<T>(dr, c0 * EPC, D, g.page_size);
#pragma unroll
        for (int h = 0; h < COMPACT_HEADS; ++h)
          if (head0 + h < g.n_kv_heads) v[h] = *reinterpret_cast<const uint4*>(s + h * head_stride);
      }
    }
    __syncthreads();                                       // the round's rows have been read
    if (to) {
#pragma unroll
      for (int h = 0; h < COMPACT_HEADS; ++h)
        if (head0 + h < g.n_kv_heads) *reinterpret_cast<uint4*>(to + h * head_stride) = v[h];
    }
  }
}

// ------------------------------------------------------------------ extra decoding heads
// r[b][k] = T(h + SiLU(W_k h + b_k)), h = T(h_last[b]). One warp per output element row i of
// head k; MC sequences at a time.
template <typename T, int MC>
__global__ void medusa_resblock(const float* __restrict__ h_last, const T* const* __restrict__ Wk,
                                const T* const* __restrict__ bk, T* __restrict__ r, int B, int K, int d,
                                unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  constexpr int VN = Vec16<T>::N;
  int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int row = blockIdx.x * (blockDim.x >> 5) + warp;   // k * d + i
  int b0 = blockIdx.y * MC;
  if (row >= K * d) return;
  int k = row / d, i = row % d;
  const T* wr = Wk[k] + (size_t)i * d;
  float acc[MC];
#pragma unroll
  for (int j = 0; j < MC; ++j) acc[j] = 0.f;
  for (int c = lane * VN; c < d; c += 32 * VN) {
    float wv[8];
    Vec16<T>::load(wr + c, wv);
#pragma unroll
    for (int j = 0; j < MC; ++j) {
      if (b0 + j < B) {
        const float* hr = h_last + (size_t)(b0 + j) * d + c;
#pragma unroll
        for (int e = 0; e < VN; ++e) acc[j] = fmaf(wv[e], quant<T>(hr[e]), acc[j]);
      }
    }
  }
#pragma unroll
  for (int j = 0; j < MC; ++j) {
    float v = warp_sum(acc[j]);
    if (lane == 0 && b0 + j < B) {
      float h = quant<T>(h_last[(size_t)(b0 + j) * d + i]);
      r[((size_t)(b0 + j) * K + k) * d + i] = from_f<T>(h + silu_f(v + to_f<T>(bk[k][i])));
    }
  }
}

// Top-k of `n` pairs (v[c], ix[c]) (ix == nullptr: index base + c) in shared memory by a CTA of 256 threads, ordered (value
// desc, index asc): the first kmax <= 16 go to emit(rank, value, index), absent ones as (-inf, 0x7fffffff). NaN never
// wins. `v` and `ix` are scratch afterwards. Called by all threads.
// Selection instead of kmax rounds of a block-wide argmax (two barriers each): the kmax-th largest of the maxima of 64
// groups of four threads is a lower bound of the kmax-th largest value, only a few times kmax values reach it, and those
// are ranked against each other. Where more than TOPK_CAP reach it (many equal values), the rounds do the work. For the four
// heads of a batch-1 7B step this and fewer, wider slices took the kernel from 26 to 10 us, for 64 rows from 183 to 32 us.
constexpr int TOPK_CAP = 256;
template <typename Emit>
__device__ __forceinline__ void block_topk(float* v, int* ix, int base, int n, int kmax, Emit emit) {
  __shared__ float gv[64], cv[TOPK_CAP];
  __shared__ int gi[64], ci[TOPK_CAP];
  __shared__ float tau_v;
  __shared__ int tau_i, count;
  const int tid = threadIdx.x;
  constexpr int NONE = 0x7fffffff;
  float bv = -INFINITY; int bi = NONE;
  for (int c = tid; c < n; c += 256) {
    const float x = v[c]; const int i = ix ? ix[c] : base + c;
    if (better(x, i, bv, bi)) { bv = x; bi = i; }
  }
#pragma unroll
  for (int o = 1; o <= 2; o <<= 1) {
    const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    if (better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
  }
  if ((tid & 3) == 0) { gv[tid >> 2] = bv; gi[tid >> 2] = bi; }
  if (tid == 0) { tau_v = -INFINITY; tau_i = NONE - 1; count = 0; }   // fewer than kmax groups hold a value: all values pass
  __syncthreads();
  if (tid < 64 && gi[tid] != NONE) {
    const float x = gv[tid]; const int i = gi[tid];
    int rank = 0;
#pragma unroll 16
    for (int j = 0; j < 64; ++j) rank += better(gv[j], gi[j], x, i) ? 1 : 0;
    if (rank == kmax - 1) { tau_v = x; tau_i = i; }
  }
  __syncthreads();
  const float tv = tau_v; const int ti = tau_i;
  for (int c = tid; c < n; c += 256) {
    const float x = v[c]; const int i = ix ? ix[c] : base + c;
    if (x >= tv && i != NONE && !better(tv, ti, x, i)) {
      const int at = atomicAdd(&count, 1);
      if (at < TOPK_CAP) { cv[at] = x; ci[at] = i; }
    }
  }
  __syncthreads();
  const int nc = count;
  if (nc <= TOPK_CAP) {
    if (tid < nc) {
      const float x = cv[tid]; const int i = ci[tid];
      int rank = 0;
      for (int j = 0; j < nc; ++j) rank += better(cv[j], ci[j], x, i) ? 1 : 0;
      if (rank < kmax) emit(rank, x, i);
    }
    if (tid >= nc && tid < kmax) emit(tid, -INFINITY, NONE);
    return;
  }
  // many equal values: kmax rounds of a block-wide argmax, the owner of the winner taking it out (a value taken out is NaN)
  const int warp = tid >> 5;
  for (int t = 0; t < kmax; ++t) {
    bv = -INFINITY; bi = NONE;
    int bc = -1;
    for (int c = tid; c < n; c += 256) {
      const float x = v[c]; const int i = ix ? ix[c] : base + c;
      if (better(x, i, bv, bi)) { bv = x; bi = i; bc = c; }
    }
    const float mv = bv; const int mi = bi;
    warp_argmax(bv, bi);
    if ((tid & 31) == 0) { cv[warp] = bv; ci[warp] = bi; }
    __syncthreads();
    bv = cv[0]; bi = ci[0];
    for (int w = 1; w < 8; ++w) if (better(cv[w], ci[w], bv, bi)) { bv = cv[w]; bi = ci[w]; }
    if (bc >= 0 && mi == bi && mv == bv) v[bc] = __int_as_float(0x7fc00000);
    if (tid == 0) emit(t, bv, bi);
    __syncthreads();
  }
}

// Merges the partial lists of one (sequence, head) row into cand[b][k+1][0..kmax) and applies
// the override table; the row of head 0 of each sequence also writes cand[b][0][0] = root.
// The row's nblocks * kmax candidates sit in shared memory (ms: nblocks * kmax * 8 bytes). Called by all threads of a
// CTA of 256; the lists are read around L1 (another CTA of the same launch may have written them).
__device__ __forceinline__ void topk_merge_row(const float* pk_val, const int* pk_idx, int nblocks, int row, int K, int kmax,
                                               const int* __restrict__ root_tok, const int* __restrict__ cand_override,
                                               int* __restrict__ cand, float* ms) {
  const int b = row / K, k = row % K;
  const int total = nblocks * kmax;
  float* v = ms;
  int* ix = reinterpret_cast<int*>(ms + total);
  for (int c = threadIdx.x; c < total; c += blockDim.x) {
    const size_t o = (size_t)row * total + c;          // lists of a row are contiguous: [row][block][kmax]
    v[c] = __ldcg(pk_val + o);
    ix[c] = __ldcg(pk_idx + o);
  }
  __syncthreads();
  int* out = cand + ((size_t)b * (K + 1) + k + 1) * kmax;
  block_topk(v, ix, 0, total, kmax, [&](int t, float, int i) {
    const int ovr = cand_override ? cand_override[((size_t)b * K + k) * kmax + t] : -1;
    const int tokv = ovr >= 0 ? ovr : i;
    out[t] = (tokv == 0x7fffffff) ? 0 : tokv;
  });
  if (k == 0 && threadIdx.x == 0) cand[(size_t)b * (K + 1) * kmax] = root_tok[b];
}

}  // namespace spec
