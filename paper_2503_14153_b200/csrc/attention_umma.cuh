// Tree-masked attention on the 5th-generation tensor cores (tcgen05, accumulators in tensor memory) for
// passes over long contexts, for batched passes and for prompt processing.
//
// A CTA owns one head, ROWS = 64 or 128 query rows and one split of the keys, and walks its keys in tiles of 128.
// With 128 rows (prompt chunks, trees of more than 64 nodes) a thread of a softmax group owns a row of the tile. Taking
// 128 rows at a time instead of two CTAs of 64, each reading the keys, shortens a layer's attention over a 2048-token
// prompt (16 chunks, 32 heads) from 146 to 118 us. What follows describes 64 rows.
// Where there are more (row group, head) items than SMs, a CTA takes one after another, the longest first, the next free one by a
// counter: the query rows (TMA) and the first key tiles of the next item are on their way, and its first scores computed, while the
// softmax warps finish the last one, and tensor memory and barriers are set up once. What remains exposed of an item is the merge
// of its streams. A CTA an item spent about 10 us around 8 tiles of 1.4: with this and the merge below, 16 sequences of 64 rows at
// 128..2048 keys 81 -> 70 us a layer (K and V alone take 44; 76 while an item's last P V waited behind the next one's first scores), eight ragged prompts through 4 layers 5.30 -> 5.02 ms; one
// sequence of 8192 keys 33.6 -> 32.8.
// A warp can read only the 32 tensor-memory lanes of
// its own SM quarter, and lane = MMA row, so to put all four quarters to work the 64 query rows are given
// twice to the 128-row MMA: rows 0..63 ("low stream") take care of keys 0..63 of every tile, rows 64..127
// (the same queries again, "high stream") of keys 64..127.
//   S = Q K^T      A = Q (twice), B = the tile's K slabs exactly as the cache holds them (K-major, 128-byte
//                  swizzle): both streams get the row's 128 scores, each thread reads its 64;
//   P = exp2(scale * S - ref) under the tree mask, rounded to bf16 into shared memory as a block-diagonal
//       operand: row r < 64 fills keys 0..63 and leaves 64..127 zero, row r + 64 the other way round;
//   O += P V       A = P, B = the tile's V slabs as the cache holds them (MN-major), accumulating in tensor
//                  memory: rows 0..63 collect the low keys' contribution, rows 64..127 the high keys'.
// `ref` is a stream's running reference: it is raised (and the stream's O row and sum rescaled, O by a
// load / multiply / store of its tensor-memory row) only when a tile's maximum exceeds it by more than 2^8,
// which after the first tile almost never happens. Two groups of four warps take alternate tiles, each with
// its own score buffer and O accumulator (4 x 128 = all 512 tensor-memory columns): while one group
// exponentiates, the tensor cores work for the other. A producer warp brings a tile's four 16 KB slabs
// (K / V x dims 0..63 / 64..127) with four 5-dimensional TMA loads straight out of the page pool -- the
// library places page p of sequence b at pool page p * max_batch + b and keeps the pages of a (layer, head)
// side by side, so a sequence's pages are a strided dimension of the tensor map --; one thread issues all
// MMAs. Of the four streams of a row (two groups x two key halves) the groups' two sit in the same tensor-memory
// lane, so each thread adds them straight from both accumulators; the key halves hand over their raw sums, 16 dims at a
// time, through the blocks of the P operands that are free between items (staging all four streams took 135 KB of shared memory, the next
// item's tiles among it, and 2.3 us). The key
// splits of a (sequence, head) form one thread-block cluster, split s owning tiles s, s + cluster
// size, ... (which tiles does not depend on the length, so the first two can be asked for before the
// dependency wait when they lie below the host's lower bound of the committed length): each CTA leaves its
// merged partial in its own shared memory, and after a cluster barrier every CTA finishes a share of the
// rows, reading all the partials through distributed shared memory -- no partial sums in HBM. Every mbarrier wait is bounded; a CTA whose wait ran out still joins the cluster barriers, so its
// peers do not wait for it.
#pragma once
#include <cuda.h>

#include "attention_tc.cuh"
#include "common.cuh"
#include "gemm_cluster.cuh"

namespace spec {

constexpr int AU_KT = 128;        // keys per tile
constexpr int AU_THREADS = 320;   // warps 0..3: softmax group 0; warps 4..7: group 1; warp 8: producer; warp 9: MMA
constexpr float AU_RESCALE_LOG2 = 8.f;   // a stream's reference is raised when a tile's maximum exceeds it by more than this
constexpr int AU_MAX_CLUSTER = 8; // most key splits (portable cluster size)
constexpr int AU_EXP = 132;       // floats per staged output row: head_dim + 4 (16-byte aligned rows, banks shifted by 4)

__host__ __device__ inline size_t attention_umma_smem() {
  return 1024 /*alignment*/ + 32768 /*Q, twice*/ + 2 * 32768 /*P*/ + 2 * 65536 /*K/V stages*/ + 512 /*barriers, items*/;
}

__device__ __forceinline__ void tma_load_5d(void* smem_dst, const void* tmap, int c0, int c1, int c2, int c3, int c4, uint64_t* bar) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4, %5, %6, %7}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(tmap), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}
// 128-byte-swizzle descriptor with explicit leading / stride byte offsets (MN-major operands use both).
__device__ __forceinline__ uint64_t make_sw128_desc(uint32_t smem_addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((smem_addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(lbo >> 4) << 16;
  d |= (uint64_t)(sbo >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}
__device__ __forceinline__ void tmem_st32(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x32.b32 [%0], "
      "{%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31,%32};"
      ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]), "r"(r[9]), "r"(r[10]),
        "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]), "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]),
        "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]), "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}
__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ float2 dsmem_ld2(uint32_t addr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void fence_proxy_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

constexpr int AU_ITEMS = 8;       // announced (row group, head) items a CTA can have in hand (its roles are at most six items apart)

__device__ __forceinline__ float exp2_fast(float x) {        // (results below 2^-126 are zero; the others are exp2f's)
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
// Barrier of the eight softmax warps, and the same telling whether `v` holds in all of their threads.
__device__ __forceinline__ void softmax_bar() { asm volatile("bar.sync 1, 256;" ::: "memory"); }
__device__ __forceinline__ bool softmax_and(bool v) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.and.pred q, 2, 256, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"((uint32_t)v) : "memory");
  return r != 0;
}

template <int HD, int ROWS>
__global__ void __launch_bounds__(AU_THREADS, 1)
attention_umma(const __grid_constant__ CUtensorMap tm_kv, const __grid_constant__ CUtensorMap tm_q, const AttnTcArgs a, unsigned long long* tr) {
  static_assert(HD == 128, "two 64-dim slabs per row");
  static_assert(ROWS == 64 || ROWS == 128, "query rows per CTA");
  KTrace kt(tr);
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* sm = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  uint8_t* q_s = sm;                          // 2 slabs x [128 rows][128 B] (64 rows: rows 64.. repeat rows 0..63)
  uint8_t* p_s = sm + 32768;                  // [2 buffers] x 2 slabs x [128 rows][128 B]; slab h = keys [64 h, +64) of the tile
  uint8_t* kv_s = sm + 32768 + 65536;         // [2 stages] x (K slab 0, K slab 1, V slab 0, V slab 1) x [128 keys][128 B]
  uint64_t* bars = reinterpret_cast<uint64_t*>(kv_s + 2 * 65536);
  uint64_t* k_full = bars;                    // [2] K slabs of a stage have landed
  uint64_t* k_empty = bars + 2;               // [2] ... have been read by the tile's score MMAs
  uint64_t* v_full = bars + 4;                // [2]
  uint64_t* v_empty = bars + 6;               // [2] ... by the tile's P V MMAs
  uint64_t* s_full = bars + 8;                // [2] scores of a tile are in tensor memory
  uint64_t* p_full = bars + 10;               // [2] P operand written (the group's four warps)
  uint64_t* o_done = bars + 12;               // [2] P V of a tile has been added to the group's accumulator
  uint64_t* q_full = bars + 14;               // an item's query rows have landed
  uint64_t* q_empty = bars + 15;              // ... have been read by its score MMAs
  uint64_t* item_full = bars + 16;            // [AU_ITEMS] an item is announced
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 16 + AU_ITEMS);
  int4* items = reinterpret_cast<int4*>(bars + 18 + AU_ITEMS);   // [AU_ITEMS] (row group or -1: no more, head, committed length, rows)

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int H = a.H, R = a.rows.R, n_items = H * a.rows.B;
  const int sp = blockIdx.y, ncl = (int)gridDim.y;             // key split = rank in the cluster; split sp owns tiles sp, sp + ncl, ...
  // Items are (row group, head) pairs, the longest sequences first (the host sorts by its bounds of the lengths). With one split
  // a CTA begins with the item of its number and takes the next free one, by a counter, when it is through.
  const int item0 = ncl == 1 ? (int)blockIdx.x : (int)(blockIdx.z * H + blockIdx.x);
  auto group_of = [&](int item) { const int zb = item / H; return a.rows.B <= ATTN_MAX_SEQS ? (int)a.order[zb] : zb; };
  auto tiles_of = [&](int n, int cnt) -> int {
    if (cnt <= 0 && n < 0) return -n;                          // (see announce)
    const int total = cnt > 0 ? (n + cnt + AU_KT - 1) / AU_KT : 0;
    return sp < total ? (total - sp + ncl - 1) / ncl : 0;
  };
  // ---- producer's loads of tile t of an item, the T-th of the CTA: two K slabs and two V slabs, K one tile ahead of V (K is
  // released by the score MMAs, long before the tile's V is released by the P V MMAs) ----
  auto load_half = [&](int T, int t, int seq, int lh, int v, uint64_t* fullb, uint64_t* emptyb, int where) -> bool {
    const int st = T & 1;
    if (T >= 2 && !mbar_wait(&emptyb[st], ((T >> 1) - 1) & 1, a.status, where)) return false;
    uint8_t* dst = kv_s + st * 65536 + v * 32768;
    mbar_expect_tx(&fullb[st], 32768);
    const int page0 = (sp + t * ncl) * (AU_KT / 16);
    tma_load_5d(dst, &tm_kv, 0, 32 * v, seq, page0, lh, &fullb[st]);       // slab rows of a page's pair: K dims 0..63, K 64..127, V, V
    tma_load_5d(dst + 16384, &tm_kv, 0, 32 * v + 16, seq, page0, lh, &fullb[st]);
    return true;
  };
  auto kv_head = [&](int h) { return a.layer * a.g.n_kv_heads + h / (H / a.g.n_kv_heads); };
  auto load_k = [&](int T, int t, int seq, int lh) { return load_half(T, t, seq, lh, 0, k_full, k_empty, 50); };
  auto load_v = [&](int T, int t, int seq, int lh) { return load_half(T, t, seq, lh, 1, v_full, v_empty, 56); };
  // The producer thread sets up the barriers itself and at once asks for its first two tiles where they lie
  // wholly below the host's lower bound of the committed length: those keys were written by earlier steps (no
  // kernel of this step starts before the kernels of the step before it have completed), so the loads need not
  // wait for the kernel before this one, and which tiles a split owns does not depend on the length.
  int pre = 0;                                                 // tiles whose loads went out before the dependency wait
  if (threadIdx.x == 8 * 32) {
    for (int i = 0; i < 16 + AU_ITEMS; ++i) mbar_init(&bars[i], (i == 10 || i == 11) ? 4 : 1);
    mbar_fence_init();
    const int z = group_of(item0), n_lo = z < ATTN_MAX_SEQS ? a.n_lo[z] : 0;
    if ((sp + 1) * AU_KT <= n_lo) {
      const int seq = a.rows.sequence(z), lh = kv_head(item0 % H);
      load_k(0, 0, seq, lh);
      pre = 1;
      if ((sp + ncl + 1) * AU_KT <= n_lo) { load_k(1, 1, seq, lh); pre = 2; }
      load_v(0, 0, seq, lh);
    }
  }
  if (warp == 9) { tmem_alloc(tmem_slot, 512); tmem_relinquish(); }
  // with 64 rows the P operands' off-diagonal blocks stay zero for the whole kernel
  if (ROWS == 64) {
    for (int c = threadIdx.x; c < 65536 / 16; c += AU_THREADS) reinterpret_cast<uint4*>(p_s)[c] = make_uint4(0, 0, 0, 0);
    fence_proxy_async_smem();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  // Dependents may start only now: this CTA holds all of the SM's tensor memory, and a dependent kernel's CTA
  // that took some first would wait for this grid while this CTA waited for its columns.
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);

  // ---- cluster of key splits: what a CTA leaves for its peers, in the stages (all its tiles have been read by then) ----
  float* ex = reinterpret_cast<float*>(kv_s);                  // [ROWS][AU_EXP]
  float* cml = ex + ROWS * AU_EXP;                             // [ROWS] (reference, sum)

  if (warp == 8) {
    pre = __shfl_sync(0xffffffffu, pre, 0);                    // (counted by its first thread above)
    if (elect_one()) {
      int T = 0, q_items = 0;
      // (a group that turns out to have no rows although the loads of its first tiles are out, an error of the pass, goes through all
      // roles with these tiles and no row that sees a key or is stored: the stages stay in step, and the CTA's further items are computed)
      auto announce = [&](int k, int it) -> int4 {
        int4 v = make_int4(-1, 0, 0, 0);
        if (it < n_items) {
          v.x = group_of(it); v.y = it % H;
          v.z = a.rows.n[v.x]; v.w = a.rows.cnt[v.x];
          if (k == 0 && v.w <= 0 && pre > 0) v.z = -pre;
        }
        items[k % AU_ITEMS] = v;
        mbar_arrive(&item_full[k % AU_ITEMS]);
        return v;
      };
      int4 cur = announce(0, item0);
      bool ok = true;
      for (int k = 0; cur.x >= 0 && ok; ++k) {
        const int nt = tiles_of(cur.z, cur.w), seq = a.rows.sequence(cur.x), lh = kv_head(cur.y);
        if (k) pre = 0;
        int4 next = make_int4(-1, 0, 0, 0);
        // the next item: from the counter, which the last to ask puts back to zero
        auto ask = [&]() {
          int it = n_items;
          if (ncl == 1)
            do {
              const unsigned int got = atomicAdd(a.arrive, 1u);
              if (got == (unsigned)(n_items - 1)) *a.arrive = 0u;
              it = (int)(gridDim.x + got);
            } while (it < n_items && a.rows.cnt[group_of(it)] <= 0);     // (a group without rows has nothing to do)
          next = announce(k + 1, it);
        };
        if (nt == 0) {
          ask();                                               // a group without rows, or a split without tiles
        } else {
          if (q_items > 0 && !mbar_wait(q_empty, (q_items - 1) & 1, a.status, 53)) { ok = false; break; }
          ++q_items;
          // the query rows (with 64 of them each at r and at r + 64). Rows beyond the group's count bring whatever is there: a
          // row's scores and output depend on no other row, and theirs are not stored.
          mbar_expect_tx(q_full, 32768);
#pragma unroll
          for (int j = 0; j < 4; ++j)
            tma_load_2d(q_s + (j & 1) * 16384 + (j >> 1) * 8192, &tm_q, cur.y * HD + (j & 1) * 64, cur.x * R + (ROWS == 128 ? (j >> 1) * 64 : 0), q_full);
          if (pre < 1) ok = load_k(T, 0, seq, lh);
          if (ok && pre < 2 && nt > 1) ok = load_k(T + 1, 1, seq, lh);
          if (ok && pre < 1) ok = load_v(T, 0, seq, lh);
          // (asking takes two trips to L2, in which this thread issues no loads: not before the second tile's are out)
          if (nt == 1) ask();
          for (int t = 1; t < nt && ok; ++t) {
            if (t + 1 < nt) ok = load_k(T + t + 1, t + 1, seq, lh);
            if (ok) ok = load_v(T + t, t, seq, lh);
            if (t == 1) ask();
          }
          T += nt;
        }
        cur = next;
      }
    }
  } else if (warp == 9) {
    if (elect_one()) {
      // ---- MMA issuer. Order within an item S(0), S(1), then PV(t), S(t + 2) for t = 0, 1, ...: the scores of the next two tiles are
      // always out before a group's probabilities are awaited, and no MMA waits behind a load it does not need (an item's last P V
      // does not wait for the next item's queries; its first scores are computed while the softmax warps merge) ----
      const uint32_t idesc_s = make_idesc_bf16(128, AU_KT);                  // A and B K-major
      const uint32_t idesc_o = make_idesc_bf16(128, HD) | (1u << 16);        // B (V) MN-major
      const uint32_t q_addr = smem_u32(q_s);
      bool ok = true;
      int T0 = 0, q_items = 0;                                               // tiles and items with tiles so far
      for (int k = 0; ok; ++k) {
        if (!mbar_wait(&item_full[k % AU_ITEMS], (k / AU_ITEMS) & 1, a.status, 60)) break;
        const int4 v = items[k % AU_ITEMS];
        if (v.x < 0) break;
        const int nt = tiles_of(v.z, v.w);
        auto mma_s = [&](int t) -> bool {
          const int T = T0 + t, bf = T & 1;
          if (t == 0 && !mbar_wait(q_full, q_items & 1, a.status, 61)) return false;
          if (!mbar_wait(&k_full[bf], (T >> 1) & 1, a.status, 51)) return false;
          tc_fence_after();
          const uint32_t d_addr = tmem + (uint32_t)(bf * 128);
          const uint32_t k_addr = smem_u32(kv_s + bf * 65536);
#pragma unroll
          for (int j = 0; j < HD / 16; ++j) {                                 // k-steps of 16 dims
            const uint64_t ad = make_kmajor_sw128_desc(q_addr + (j >> 2) * 16384) + 2 * (j & 3);
            const uint64_t bd = make_kmajor_sw128_desc(k_addr + (j >> 2) * 16384) + 2 * (j & 3);
            tc_mma_f16(d_addr, ad, bd, idesc_s, j > 0 ? 1u : 0u);
          }
          tc_commit(&s_full[bf]);
          tc_commit(&k_empty[bf]);
          if (t == nt - 1) tc_commit(q_empty);
          return true;
        };
        if (nt > 0) ok = mma_s(0);
        if (ok && nt > 1) ok = mma_s(1);
        if (ok && k == 0) trace_mark_max(tr, 3);
        for (int t = 0; t < nt && ok; ++t) {
          const int T = T0 + t, bf = T & 1;
          if (!mbar_wait(&p_full[bf], (T >> 1) & 1, a.status, 52) || !mbar_wait(&v_full[bf], (T >> 1) & 1, a.status, 57)) { ok = false; break; }
          tc_fence_after();
          const uint32_t d_addr = tmem + 256u + (uint32_t)(bf * 128);          // the group's accumulator
          const uint32_t p_addr = smem_u32(p_s + bf * 32768), v_addr = smem_u32(kv_s + bf * 65536 + 32768);
#pragma unroll
          for (int j = 0; j < AU_KT / 16; ++j) {                              // k-steps of 16 keys
            const uint64_t ad = make_kmajor_sw128_desc(p_addr + (j >> 2) * 16384) + 2 * (j & 3);
            const uint64_t bd = make_sw128_desc(v_addr + j * 2048, 16384, 1024);
            tc_mma_f16(d_addr, ad, bd, idesc_o, (t >= 2 || j > 0) ? 1u : 0u);   // a group's first tile of an item starts its accumulator
          }
          tc_commit(&o_done[bf]);
          tc_commit(&v_empty[bf]);
          if (t + 2 < nt) ok = mma_s(t + 2);
        }
        T0 += nt;
        if (nt > 0) ++q_items;
      }
    }
  } else {
    // ---- softmax groups: every second tile; a thread = one query row (64 rows: and one half of every tile's keys) ----
    const int grp = warp >> 2;                                 // softmax group of warps 0..3 / 4..7
    const int q4 = warp & 3;                                   // SM quarter = tensor-memory lanes [32 q4, +32)
    const int mrow = q4 * 32 + lane;                           // this thread's MMA row (tensor-memory lane)
    const int qrow = mrow & (ROWS - 1);                        // its query row
    const int kh = ROWS == 64 ? mrow >> 6 : 0;                 // 64 rows: its key half of every tile
    const uint32_t lane_base = (uint32_t)(q4 * 32) << 16;
    int T0 = 0;                                                // the CTA's tiles before this item
    for (int k = 0;; ++k) {
      bool ok = mbar_wait(&item_full[k % AU_ITEMS], (k / AU_ITEMS) & 1, a.status, 62);
      const volatile int* item = reinterpret_cast<const volatile int*>(items + k % AU_ITEMS);
      if (!softmax_and(ok) || item[0] < 0) break;              // (the same in all 256 threads)
      const int n = item[2], nt = tiles_of(n, item[3]);
      float m_ref = -INFINITY, l_run = 0.f;
      int my_tiles = 0;
      uint32_t anc[4];
#pragma unroll
      for (int w = 0; w < 4; ++w) anc[w] = qrow < item[3] ? __ldg(a.rows.anc + qrow * 4 + w) : 0u;
      // Raises the stream's reference to the tile's maximum `tmax` (unscaled) where it has to and returns what the sums so far
      // are multiplied by; the group's previous tile must be through the tensor cores by then (its P operand and
      // accumulator are reused), which is awaited here.
      auto raise_reference = [&](float tmax, int t, int T) -> float {
        tmax *= a.scale_log2;
        // raise the reference only when it is too low by more than 2^AU_RESCALE_LOG2 (or not set yet)
        const bool raise = tmax > m_ref + AU_RESCALE_LOG2 || (m_ref == -INFINITY && tmax > -INFINITY);
        const float m_new = raise ? tmax : m_ref;
        const float alpha = raise ? exp2f(m_ref - m_new) : 1.f;   // 0 the first time
        if (t >= 2 && !mbar_wait(&o_done[grp], ((T >> 1) - 1) & 1, a.status, 55)) { ok = false; return 1.f; }
        if (__any_sync(0xffffffffu, raise && my_tiles > 0)) {
          // rescale this lane's accumulator row (other lanes of the warp multiply by one)
          tc_fence_after();
          const uint32_t o_addr = tmem + lane_base + 256u + (uint32_t)(grp * 128);
#pragma unroll 1
          for (int c = 0; c < 4; ++c) {
            uint32_t r[32];
            tmem_ld32(o_addr + c * 32, r);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) * alpha);
            tmem_st32(o_addr + c * 32, r);
          }
          tmem_st_wait();
        }
        m_ref = m_new;
        return alpha;
      };
      for (int t = (T0 ^ grp) & 1; t < nt; t += 2) {
        const int bf = grp;
        if (!mbar_wait(&s_full[bf], ((T0 + t) >> 1) & 1, a.status, 54)) { ok = false; break; }
        tc_fence_after();
        if constexpr (ROWS == 128) {
          // a thread has all 128 keys of the tile: 32 scores at a time, read out of tensor memory once for the maximum and
          // once for the probabilities (128 of them would not stay in registers)
          const uint32_t s_addr = tmem + lane_base + (uint32_t)(bf * 128);
          const int k0 = (sp + t * ncl) * AU_KT;
          uint32_t vis[4] = {0xffffffffu, 0xffffffffu, 0xffffffffu, 0xffffffffu};
          const bool whole = k0 + AU_KT <= n;                     // no tree row, nothing past the end
          if (!whole) {
            const unsigned long long v0 = attn_vis64(anc, k0, n), v1 = attn_vis64(anc, k0 + 64, n);
            vis[0] = (uint32_t)v0; vis[1] = (uint32_t)(v0 >> 32); vis[2] = (uint32_t)v1; vis[3] = (uint32_t)(v1 >> 32);
          }
          float tmax = -INFINITY;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t r[32];
            tmem_ld32(s_addr + c * 32, r);
            tmem_ld_wait();
            if (whole) {
#pragma unroll
              for (int j = 0; j < 32; ++j) tmax = fmaxf(tmax, __uint_as_float(r[j]));
            } else {
#pragma unroll
              for (int j = 0; j < 32; ++j) if ((vis[c] >> j) & 1u) tmax = fmaxf(tmax, __uint_as_float(r[j]));
            }
          }
          const float alpha = raise_reference(tmax, t, T0 + t);
          if (!ok) break;
          const float base = (m_ref == -INFINITY) ? 0.f : m_ref;
          l_run *= alpha;
          uint8_t* p_row = p_s + bf * 32768 + mrow * 128;
          float l0 = 0.f, l1 = 0.f;
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            uint32_t r[32], pk[16];
            tmem_ld32(s_addr + c * 32, r);
            tmem_ld_wait();
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              float p0 = exp2_fast(fmaf(__uint_as_float(r[j]), a.scale_log2, -base));
              float p1 = exp2_fast(fmaf(__uint_as_float(r[j + 1]), a.scale_log2, -base));
              if (!whole) {
                if (!((vis[c] >> j) & 1u)) p0 = 0.f;
                if (!((vis[c] >> (j + 1)) & 1u)) p1 = 0.f;
              }
              l0 += p0; l1 += p1;
              pk[j >> 1] = pack_bf16(p0, p1);
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              const int ch = (c & 1) * 4 + g;
              *reinterpret_cast<uint4*>(p_row + (c >> 1) * 16384 + ((ch ^ (mrow & 7)) << 4)) =
                  make_uint4(pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
            }
          }
          l_run += l0 + l1;
        } else {
          const uint32_t s_addr = tmem + lane_base + (uint32_t)(bf * 128 + kh * 64);
          const int k0 = (sp + t * ncl) * AU_KT + kh * 64;       // first key of this thread's half
          uint32_t r0[32], r1[32];
          tmem_ld32(s_addr, r0);
          tmem_ld32(s_addr + 32, r1);
          uint32_t vis0 = 0xffffffffu, vis1 = 0xffffffffu;
          if (k0 + 64 > n) {                                      // the half reaches into the tree rows or past the end
            const unsigned long long v = attn_vis64(anc, k0, n);
            vis0 = (uint32_t)v; vis1 = (uint32_t)(v >> 32);
          }
          tmem_ld_wait();
          float tmax = -INFINITY;
          if ((vis0 & vis1) == 0xffffffffu) {
#pragma unroll
            for (int j = 0; j < 32; ++j) tmax = fmaxf(tmax, fmaxf(__uint_as_float(r0[j]), __uint_as_float(r1[j])));
          } else {
#pragma unroll
            for (int j = 0; j < 32; ++j) {
              if ((vis0 >> j) & 1u) tmax = fmaxf(tmax, __uint_as_float(r0[j]));
              if ((vis1 >> j) & 1u) tmax = fmaxf(tmax, __uint_as_float(r1[j]));
            }
          }
          const float alpha = raise_reference(tmax, t, T0 + t);
          if (!ok) break;
          l_run *= alpha;
          const float base = (m_ref == -INFINITY) ? 0.f : m_ref;
          // probabilities of this thread's 64 keys, rounded to bf16, into row `mrow` of slab `kh` of the P operand
          float l0 = 0.f, l1 = 0.f;
          uint8_t* p_row = p_s + bf * 32768 + kh * 16384 + mrow * 128;
#pragma unroll
          for (int c = 0; c < 2; ++c) {
            const uint32_t (&r)[32] = c ? r1 : r0;
            const uint32_t vc = c ? vis1 : vis0;
            uint32_t pk[16];
#pragma unroll
            for (int j = 0; j < 32; j += 2) {
              float p0 = exp2_fast(fmaf(__uint_as_float(r[j]), a.scale_log2, -base));
              float p1 = exp2_fast(fmaf(__uint_as_float(r[j + 1]), a.scale_log2, -base));
              if (!((vc >> j) & 1u)) p0 = 0.f;
              if (!((vc >> (j + 1)) & 1u)) p1 = 0.f;
              l0 += p0; l1 += p1;
              pk[j >> 1] = pack_bf16(p0, p1);
            }
#pragma unroll
            for (int g = 0; g < 4; ++g) {
              const int ch = c * 4 + g;
              *reinterpret_cast<uint4*>(p_row + ((ch ^ (mrow & 7)) << 4)) = make_uint4(pk[4 * g], pk[4 * g + 1], pk[4 * g + 2], pk[4 * g + 3]);
            }
          }
          l_run += l0 + l1;
        }
        ++my_tiles;
        fence_proxy_async_smem();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(&p_full[bf]);
      }
      // the group's last tile must be through the tensor cores before its accumulator is read
      const int t_last = nt - 1 - ((T0 + nt - 1 - grp) & 1);   // (negative: the group has none)
      if (ok && t_last >= 0 && !mbar_wait(&o_done[grp], ((T0 + t_last) >> 1) & 1, a.status, 58)) ok = false;
      // ---- the streams of a query row are merged: the two groups' (each thread reads both accumulators of its tensor-memory lane), with
      // 64 rows also the two key halves', which sit in lanes 64 apart, through the diagonal blocks of the P operands (the others stay
      // zero). The order of the sums is that of the tiles: the group of the item's first tile before the other group, in each the low keys
      // before the high ones, whichever group that is and wherever in the CTA's row of items the item stands ----
      // (opaque: the addresses made from them would otherwise be kept in registers through the tiles' loop)
      const int z = item[0], h = item[1], cnt = item[3];       // (read again: registers)
      int mrow_ = mrow, qrow_ = qrow;
      asm volatile("" : "+r"(mrow_), "+r"(qrow_));
      auto ml = [&](int g) { return reinterpret_cast<float2*>(p_s + g * 32768); };   // [128 lanes] (reference, sum), in the group's own P operand
      ml(grp)[mrow_] = ok && t_last >= 0 ? make_float2(m_ref, l_run) : make_float2(-INFINITY, 0.f);
      tc_fence_before();
      if (!softmax_and(ok)) break;                             // both groups' sums are there and their accumulators complete
      tc_fence_after();
      const int kh_ = ROWS == 64 ? mrow_ >> 6 : 0, first = T0 & 1;                                // group of the item's first tile
      constexpr int STREAMS = ROWS == 64 ? 4 : 2;
      float2 st[STREAMS];
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const float2 own = ml(first ^ k)[mrow_];
        if (ROWS == 64) {
          const float2 other = ml(first ^ k)[mrow_ ^ 64];
          st[2 * k] = kh_ ? other : own;
          st[STREAMS == 4 ? 2 * k + 1 : 0] = kh_ ? own : other;
        } else {
          st[k] = own;
        }
      }
      float mm = st[0].x;
#pragma unroll
      for (int k = 1; k < STREAMS; ++k) mm = fmaxf(mm, st[k].x);
      const float base = mm == -INFINITY ? 0.f : mm;
      float wt[STREAMS], L = 0.f;
#pragma unroll
      for (int k = 0; k < STREAMS; ++k) { wt[k] = exp2f(st[k].x - base); L = __fmaf_rn(wt[k], st[k].y, L); }
      // (16 dims at a time, and nothing spilled: with all of the SM's shared memory in use there is hardly any L1 to spill to)
      auto raw16 = [&](int k, int d, uint32_t (&r)[16]) {      // dims [d, +16) of this lane in the k-th group's accumulator
        tmem_ld16(tmem + lane_base + 256u + (uint32_t)((first ^ k) * 128 + d), r);
        tmem_ld_wait();
      };
      auto emit16 = [&](int d, const float (&v)[16]) {         // ... to the output, or to the cluster's exchange
        if (ncl > 1) {
#pragma unroll
          for (int j = 0; j < 16; j += 4)
            *reinterpret_cast<float4*>(ex + (size_t)qrow_ * AU_EXP + d + j) = make_float4(v[j], v[j + 1], v[j + 2], v[j + 3]);
        } else if (qrow_ < cnt) {
          const float inv = 1.f / L;
          uint4* dst = reinterpret_cast<uint4*>(a.out + ((size_t)z * R + qrow_) * H * HD + h * HD + d);
#pragma unroll
          for (int j = 0; j < 2; ++j)
            dst[j] = make_uint4(pack_bf16(v[8 * j] * inv, v[8 * j + 1] * inv), pack_bf16(v[8 * j + 2] * inv, v[8 * j + 3] * inv),
                                pack_bf16(v[8 * j + 4] * inv, v[8 * j + 5] * inv), pack_bf16(v[8 * j + 6] * inv, v[8 * j + 7] * inv));
        }
      };
      if constexpr (ROWS == 128) {
#pragma unroll 1
        for (int d = grp * 64; d < grp * 64 + 64; d += 16) {
          float v[16] = {};
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (nt <= k) break;                                // (a group without a tile has no accumulator)
            uint32_t r[16];
            raw16(k, d, r);
#pragma unroll
            for (int j = 0; j < 16; ++j) v[j] = __fmaf_rn(wt[k], __uint_as_float(r[j]), v[j]);
          }
          emit16(d, v);
        }
      } else {
        // the thread of key half kh finishes dims [32 kh_, +32) of the group's 64 and hands over what it has of the other 32, 16 at a time
        softmax_bar();                                         // (the sums have been read: they lie in two of the blocks)
        auto at = [&](int half, int c) {                       // 16-byte chunk c of this row in the block for the threads of `half`
          return reinterpret_cast<float4*>(p_s + grp * 32768 + half * (16384 + 8192) + qrow_ * 128 + ((c ^ (qrow_ & 7)) << 4));
        };
        auto rows_bar = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(3 + grp * 2 + ((mrow_ >> 5) & 1)) : "memory"); };   // the two warps of these rows and this group
#pragma unroll 1
        for (int i = 0; i < 2; ++i) {
          if (i) rows_bar();                                   // the first 16 have been read
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (nt <= k) break;                                // (a group without a tile has no accumulator)
            uint32_t r[16];
            raw16(k, grp * 64 + (kh_ ^ 1) * 32 + i * 16, r);
#pragma unroll
            for (int j = 0; j < 4; ++j) *reinterpret_cast<uint4*>(at(kh_ ^ 1, k * 4 + j)) = make_uint4(r[4 * j], r[4 * j + 1], r[4 * j + 2], r[4 * j + 3]);
          }
          rows_bar();
          float v[16] = {};
#pragma unroll
          for (int k = 0; k < 2; ++k) {
            if (nt <= k) break;
            uint32_t r[16];
            raw16(k, grp * 64 + kh_ * 32 + i * 16, r);
            const float w_lo = wt[(2 * k) % STREAMS], w_hi = wt[(2 * k + 1) % STREAMS];
#pragma unroll
            for (int j = 0; j < 4; ++j) {
              const float4 o4 = *at(kh_, k * 4 + j);
              const float o[4] = {o4.x, o4.y, o4.z, o4.w};
#pragma unroll
              for (int i4 = 0; i4 < 4; ++i4) {
                const float own = __uint_as_float(r[4 * j + i4]);
                v[4 * j + i4] = __fmaf_rn(w_hi, kh_ ? own : o[i4], __fmaf_rn(w_lo, kh_ ? o[i4] : own, v[4 * j + i4]));
              }
            }
          }
          emit16(grp * 64 + kh_ * 32 + i * 16, v);
        }
      }
      if (ncl > 1 && grp == 0 && kh == 0) *reinterpret_cast<float2*>(cml + qrow * 2) = make_float2(mm, L);
      tc_fence_before();
      softmax_bar();                                           // the accumulators and P operands may be written again
      T0 += nt;
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 9) { tc_fence_after(); tmem_dealloc(tmem, 512); }
  if (ncl == 1) return;
  __syncwarp();
  cluster_sync_all();
  const int z = group_of(item0), h = item0 % H, cnt = a.rows.cnt[z];
  // ---- the cluster's partials: CTA `rank` finishes rows [rank * rpc, +rpc) from everybody's shared memory ----
  {
    const int rank = (int)cluster_ctarank();
    const int rpc = (ROWS + ncl - 1) / ncl;
    const uint32_t ex_local = smem_u32(ex), cml_local = smem_u32(cml);
    uint32_t ex_r[AU_MAX_CLUSTER], cml_r[AU_MAX_CLUSTER];
#pragma unroll
    for (int s2 = 0; s2 < AU_MAX_CLUSTER; ++s2) {
      ex_r[s2] = dsmem_addr(ex_local, (uint32_t)min(s2, ncl - 1));
      cml_r[s2] = dsmem_addr(cml_local, (uint32_t)min(s2, ncl - 1));
    }
    for (int it = threadIdx.x; it < rpc * (HD / 4); it += AU_THREADS) {
      const int row = rank * rpc + it / (HD / 4), d = (it % (HD / 4)) * 4;
      if (row >= ROWS || row >= cnt) continue;
      float2 mlv[AU_MAX_CLUSTER];
      float4 ov[AU_MAX_CLUSTER];
#pragma unroll
      for (int s2 = 0; s2 < AU_MAX_CLUSTER; ++s2) {
        mlv[s2] = make_float2(-INFINITY, 0.f);
        ov[s2] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (s2 < ncl) {
          mlv[s2] = dsmem_ld2(cml_r[s2] + (uint32_t)(row * 8));
          ov[s2] = dsmem_ld4(ex_r[s2] + (uint32_t)((row * AU_EXP + d) * 4));
        }
      }
      float mm = -INFINITY;
#pragma unroll
      for (int s2 = 0; s2 < AU_MAX_CLUSTER; ++s2) mm = fmaxf(mm, mlv[s2].x);
      float L = 0.f;
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int s2 = 0; s2 < AU_MAX_CLUSTER; ++s2) {
        const float w = exp2f(mlv[s2].x - mm);                 // a valid row sees itself: mm is finite
        L += w * mlv[s2].y;
        acc.x += w * ov[s2].x; acc.y += w * ov[s2].y; acc.z += w * ov[s2].z; acc.w += w * ov[s2].w;
      }
      const float inv = 1.f / L;
      const size_t m = (size_t)z * R + row;
      *reinterpret_cast<uint2*>(a.out + m * H * HD + h * HD + d) =
          make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
    }
  }
  // nobody leaves while a peer may still read its shared memory (the values read are in registers by then: nothing to publish)
  __syncwarp();
  cluster_arrive_relaxed();
  cluster_wait();
}

}  // namespace spec
