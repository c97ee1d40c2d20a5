// bf16 linear for passes of many rows (batched verification, prompt processing), where the projections are
// compute-bound: y = x W^T on the 5th-generation tensor cores, two SMs per output tile, with the element-wise step
// that follows the projection applied in the epilogue.
//
// Operands are swapped as in gemm_stream (weight rows are the MMA's M). A cluster of two CTAs owns an output tile
// of [256 weight rows] x [NT activation rows] and issues tcgen05.mma.cta_group::2 (M 256, N NT): each CTA holds
// the accumulator of its own 128 weight rows and brings in those 128 weight rows and half of the activation rows.
// Why pairs: a 64-wide K chunk of a 128 x 256 tile in one CTA writes 48 KB into shared memory and reads 48 KB out
// of it in the 512 cycles its MMAs take at full rate, 192 bytes per cycle where an SM moves 128; the pair's chunk
// is 32 KB in and 32 KB out per CTA, 128 bytes per cycle. Two accumulators of NT tensor-memory columns alternate, so
// that the epilogue of one tile runs under the MMAs of the next. Persistent: cluster c takes tiles
// c, c + clusters, ...; tile = weight pair * m_tiles + activation tile, so the clusters that share weights run side
// by side and the weights cross HBM once. Where there are tiles for less than half of the clusters (a 256-row pass has
// 16 tiles of an output projection for 74 clusters), every tile's K chunks are dealt to `parts` clusters: each leaves float32
// partial sums, and the CTA of a tile that arrives last (arrival counter, nobody waits) adds them in order, so that the sum
// does not depend on who that is, and does the tile's epilogue. (Dealing the last wave's tiles to all clusters where whole
// tiles leave some of them idle does not pay: the clusters share the L2's bandwidth, so that fewer of them run faster; at 2048
// rows the output and down projections took 184 us instead of 120.)
//
// The work of a launch is a list of items: tiles of `tile_rows` activation rows (256, or fewer where that fills the waves better or gives a narrow
// projection to more clusters), of which those from cut_first on, the last wave's, may be cut into slices. The host chooses by a model of the
// kernel's time (plan_pair); an element's inner dimension runs through in the same order whatever the rows of its item. Fewer rows a stage leave
// room for more stages: 16 rows, the last tokens of prompts, have eleven.
//
// Modes:
//  * GP_PLAIN     float32 sums to out[m][ld] (columns below n_cols only). The only mode whose sums are results as they stand:
//                 the two halves of the inner dimension go to the two accumulators and are added in registers, because the error
//                 of a running sum in the tensor cores grows with its length (K 4096: 4.4e-6 of the result in one accumulator,
//                 2.1e-6 in two halves; the weight streamer, which cuts about every other tile, 3.9e-6 at M = 1008). The first
//                 half is taken out of tensor memory under the MMAs of the second, and both accumulators are given back
//                 before the stores, so that the next tile's MMAs run under them: 112 us instead of 114 at M = 1008, N = 11008,
//                 K = 4096; 98 instead of 94 at M = 2048, K = 1024, where the stores take longer than the MMAs.
//  * GP_RESIDUAL  x[m][n] += sum, in place (output and down projections)
//  * GP_SWIGLU    act[m][n] = bf16(SiLU(gate) * up): a CTA's 128 weight rows are 64 rows of the gate and the same 64
//                 rows of the up matrix
//  * GP_ROPE      stacked q, k, v: rotates q and k, writes bf16 q rows and the cache rows
// In the last two modes an output needs two weight rows of the tile, which sit in different tensor-memory lanes: the
// threads swap halves of their activation rows through 16 KB of shared memory, 16 rows at a time.
//
// Measured on the 7B shape at M = 1024 (inside a step, launch to end, per layer), against a kernel with 128 x 256 tiles per
// CTA that wrote float32 sums for separate glue kernels: gate+up 175 -> 141 us (1.31 PFLOP/s) and the 33 us SwiGLU kernel
// gone, q/k/v 107 -> 91 us and the 23 us RoPE / store kernel gone, output 41 -> 39, down 92 -> 84 us; a step of 16
// sequences through 8 layers 5.58 -> 4.56 ms.
//
// A tile's epilogue runs under the next tile's MMAs, but the last one of a CTA does not: with eight epilogue warps the time from
// the last MMA to the end of the kernel was 10.0 us for q/k/v, 11.4 for the output, 10.3 for the gate+up and 13.8 for the down projection
// (M = 1024), with sixteen, in half as long strides, it is 7.0, 7.0, 7.1 and 7.1; a step of 16 sequences through 8 layers 4.14 -> 4.04 ms.
//
// Warp roles (both CTAs): warp 0 feeds a ring of 32 KB stages (TMA, completing on the leader CTA's barrier), warp
// 1 of the leader issues the MMAs, warps 2..17 drain: four warps per SM quarter, one for each quarter of the tile's
// activation rows. Every wait is bounded; a CTA whose wait ran out still takes part in the closing cluster barrier.
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "gemm_cluster.cuh"
#include "gemm_stream.cuh"

namespace spec {

constexpr int GP_PLAIN = 0, GP_RESIDUAL = 1, GP_SWIGLU = 2, GP_ROPE = 3;
// How a launch's sums are made: GP_WHOLE, an element's inner dimension in one run (GP_PLAIN: in halves); GP_SHARED, a tile's chunks on several clusters;
// GP_RUNS, in the runs and in the order in which the projections of up to 128 rows add it up, a run an accumulator: a prompt of two chunks in one
// pass over the weights, with the sums of the two passes that it took.
constexpr int GP_WHOLE = 0, GP_SHARED = 1, GP_RUNS = 2;
constexpr int GP_EPI = 512, GP_THREADS = 64 + GP_EPI;   // producer, MMA issuer, sixteen epilogue warps (four per SM quarter)
constexpr int GP_QUARTERS = 4;                          // parts of a tile's activation rows that the epilogue warps share out

struct PairGemmParams {
  int M, KC;                                // activation rows, K / 64
  int n_mats;
  int mat_tile0[GS_MAX_MATS + 1];           // first 128-row weight tile of each stacked matrix
  int n_tiles, w_pairs, m_tiles;            // weight tiles (all matrices), pairs of them, activation tiles
  int tile_rows;                            // activation rows of a tile: a multiple of 16, at most NT (parts > 1: NT)
  int cut_first, cut;                       // tiles from cut_first on are done as `cut` slices of tile_rows / cut activation rows each (a multiple of 16)
  int stages;                               // of the ring
  int runs, run_bufs;                       // GP_RUNS: accumulators of an item, at most, and items whose accumulators tensor memory holds (1 or 2)
  SegMap seg;                               // GP_RUNS, GP_SWIGLU: how the weight streamer deals the stacked gate and up tiles' chunks out
  int plan_tiles;                           // host: tiles of the launch whose sharing (parts) this one follows, 0: its own
  int parts;                                // clusters that share a tile's K chunks (1: tiles are whole)
  float* part;                              // parts > 1: [tile][part][CTA of the pair][NT][128] float32
  unsigned int* arrive;                     // parts > 1: [tile][CTA of the pair], zero between launches
  int packed;                               // 1: the tensor maps view pre-tiled images, 0: row-major matrices
  int n_cols;                               // GP_PLAIN: columns stored; GP_RESIDUAL / GP_SWIGLU: weight rows of one matrix
  size_t ld;                                // GP_PLAIN: row pitch of out
  int* clear;                               // GP_PLAIN: four ints set to zero, or nullptr
  float* best_val;                          // GP_PLAIN: [4 * n_tiles][M] each row's largest of 32 columns and its column (value descending, column
  int* best_idx;                            // ascending), or nullptr; out may then be nullptr
  float* out;                               // GP_PLAIN: sums; GP_RESIDUAL: residual stream [M][n_cols]
  bf16* act;                                // GP_SWIGLU: [M][n_cols]
  // GP_ROPE
  int kind0;                                // what the first matrix is: 0 q, 1 k (a prompt's last layer projects k and v alone)
  int q_chunk;                              // > 0: row m's query goes to row m * q_chunk + position % q_chunk of q (the last rows of prompts)
  int H, layer;
  Rows rows;
  const float2* cs;                         // [position][head_dim / 2] (cos, sin)
  bf16* q;                                  // [M][H * head_dim]
  bf16* pool;
  KVGeom g;
  const int* page_table;
  int* status;
  unsigned long long* trace;
};

template <int NT> struct PairCfg {
  static constexpr int BK = 64;
  static constexpr int A_BYTES = 128 * BK * 2;
  static constexpr int B_BYTES = (NT / 2) * BK * 2;
  static constexpr int RING_BYTES = 6 * (A_BYTES + B_BYTES);
  static constexpr int MAX_STAGES = 11;
  static __host__ __device__ constexpr int stage_bytes(int rows) { return A_BYTES + rows / 2 * BK * 2; }
  static __host__ __device__ constexpr int stages(int rows) { return RING_BYTES / stage_bytes(rows) < MAX_STAGES ? RING_BYTES / stage_bytes(rows) : MAX_STAGES; }
  static constexpr int EX_COLS = 8;                               // activation rows swapped in one direction at a time
  static constexpr int EX_BYTES = GP_QUARTERS * 2 * 64 * EX_COLS * 4;       // [part][direction][column][64 pairs] float32
  static constexpr int META_BYTES = NT * 16;                      // GP_ROPE: (cache offset, position, swizzle row) of a row
  static constexpr int SMEM_BYTES = RING_BYTES + EX_BYTES + META_BYTES + 1024 /*alignment slack*/ + 256 /*barriers*/;
  static constexpr int TMEM_COLS = 2 * NT;
};

// ---- cta_group::2 forms ----
__device__ __forceinline__ void tmem_alloc2(uint32_t* smem_dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(smem_dst)), "r"(ncols) : "memory");
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc2(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_mma_f16_pair(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc, uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n\t}"
      ::"r"(tmem_d), "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrives on the barrier at this offset in both CTAs once all MMAs issued so far by this thread are complete.
__device__ __forceinline__ void tc_commit_pair(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %1;"
               ::"r"(smem_u32(bar)), "h"((uint16_t)3) : "memory");
}
// 2D tiled TMA load into this CTA's shared memory that completes on a barrier of either CTA of the pair.
__device__ __forceinline__ void tma_load_2d_pair(void* smem_dst, const void* tmap, int x, int y, uint32_t cluster_bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes.cta_group::2 [%0], [%1, {%3, %4}], [%2];"
      ::"r"(smem_u32(smem_dst)), "l"(tmap), "r"(cluster_bar), "r"(x), "r"(y)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t cluster_bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(cluster_bar) : "memory");
}
// Barrier of one part's four epilogue warps; epilogue_bar, epilogue_and: of all sixteen, telling whether `v` holds in all of their threads.
__device__ __forceinline__ void group_bar(int id) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }
__device__ __forceinline__ void epilogue_bar() { asm volatile("bar.sync 6, %0;" ::"n"(GP_EPI) : "memory"); }
__device__ __forceinline__ bool epilogue_and(bool v) {
  uint32_t r;
  asm volatile("{\n\t.reg .pred p, q;\n\tsetp.ne.b32 p, %1, 0;\n\tbar.red.and.pred q, 7, %2, p;\n\tselp.b32 %0, 1, 0, q;\n\t}"
               : "=r"(r) : "r"((uint32_t)v), "n"(GP_EPI) : "memory");
  return r != 0;
}

struct PairTmaps {
  CUtensorMap a[GS_MAX_MATS];
  CUtensorMap b, b_cut;                     // boxes of half a tile's and half a slice's activation rows
};

struct PairRowMeta {
  long long kv;      // element offset of the row's slot within its (layer, head) K|V blocks; -1: row not in use
  int pos, prow;
};

template <int MODE, int NT, int FORM>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(GP_THREADS, 1)
gemm_pair(const __grid_constant__ PairTmaps tm, const PairGemmParams p) {
  using Cfg = PairCfg<NT>;
  constexpr bool SPLIT = FORM == GP_SHARED, RUNS = FORM == GP_RUNS;
  const int stages = p.stages, stage_bytes = Cfg::stage_bytes(p.tile_rows);
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* tiles = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  float* exch = reinterpret_cast<float*>(tiles + Cfg::RING_BYTES);
  PairRowMeta* meta = reinterpret_cast<PairRowMeta*>(tiles + Cfg::RING_BYTES + Cfg::EX_BYTES);
  uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + Cfg::RING_BYTES + Cfg::EX_BYTES + Cfg::META_BYTES);
  uint64_t* full = bars;                    // leader's: both CTAs' operands of a stage have landed
  uint64_t* empty = bars + Cfg::MAX_STAGES;          // each CTA's: the stage has been read
  uint64_t* acc_full = bars + 2 * Cfg::MAX_STAGES;   // each CTA's
  uint64_t* acc_empty = bars + 2 * Cfg::MAX_STAGES + 2;   // leader's: drained by the sixteen warps of both CTAs
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * Cfg::MAX_STAGES + 4);
  volatile uint32_t* last_slot = reinterpret_cast<volatile uint32_t*>(bars + 2 * Cfg::MAX_STAGES + 5);   // this CTA completes a split tile

  KTrace kt(p.trace);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int cl = blockIdx.x >> 1, ncl = gridDim.x >> 1;
  const int KC = p.KC;
  // this cluster's work: tiles cl, cl + ncl, ..., or with parts > 1 one part of one tile
  const int total_tiles = p.w_pairs * p.m_tiles, parts = SPLIT ? p.parts : 1;
  const int items = SPLIT ? total_tiles * parts : p.cut_first + (total_tiles - p.cut_first) * p.cut;
  const int my_tiles = cl < items ? (SPLIT ? 1 : (items - 1 - cl) / ncl + 1) : 0;
  const int k_lo = SPLIT ? cl % parts * KC / parts : 0, k_hi = SPLIT ? (cl % parts + 1) * KC / parts : KC;
  static_assert(MODE != GP_PLAIN || FORM == GP_WHOLE, "plain sums are results as they stand, in halves");
  // GP_RUNS: number of runs of a weight pair's tiles and first chunk of the r-th
  auto runs_of = [&](int wp) { return MODE == GP_SWIGLU ? p.seg.nseg(wp) : p.runs; };
  auto run_start = [&](int wp, int r) { return MODE == GP_SWIGLU ? (r ? p.seg.lo(p.seg.owner(wp * KC) + r) - wp * KC : 0) : r * KC / p.runs; };
  const int halves = MODE == GP_PLAIN && KC > 1 ? 2 : 1;    // accumulators a tile's inner dimension is cut into
  // this cluster's i-th item: weight pair, first activation row and rows
  struct Item { int tau, wp, row0, rows; };
  auto item_of = [&](int i) {
    Item v;
    int sub = 0;
    v.tau = SPLIT ? cl / parts : cl + i * ncl;
    v.rows = SPLIT ? NT : p.tile_rows;
    if (!SPLIT && v.tau >= p.cut_first) {
      const int s = v.tau - p.cut_first;
      v.rows = p.tile_rows / p.cut;
      v.tau = p.cut_first + s / p.cut;
      sub = s % p.cut;
    }
    v.wp = v.tau / p.m_tiles;
    v.row0 = (v.tau - v.wp * p.m_tiles) * (SPLIT ? NT : p.tile_rows) + sub * v.rows;
    return v;
  };

  pdl_launch_dependents();

  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(&acc_full[0], 1); mbar_init(&acc_full[1], 1);
    mbar_init(&acc_empty[0], 2 * GP_EPI / 32); mbar_init(&acc_empty[1], 2 * GP_EPI / 32);
    mbar_fence_init();
    for (int i = 0; i < p.n_mats; ++i) tma_prefetch_desc(&tm.a[i]);
    tma_prefetch_desc(&tm.b);
    if (!SPLIT && p.cut_first < total_tiles) tma_prefetch_desc(&tm.b_cut);
  }
  if (warp == 1) tmem_alloc2(tmem_slot, Cfg::TMEM_COLS);
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                       // the peer's barriers are set up
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // weight tile of this CTA in pair wp (a last odd tile is computed twice and stored once)
  auto mat_of = [&](int nt) {
    int mat = 0;
#pragma unroll
    for (int i = 1; i < GS_MAX_MATS; ++i)
      if (i < p.n_mats && nt >= p.mat_tile0[i]) mat = i;
    return mat;
  };

  if (warp == 0) {
    if (elect_one()) {
      // ---- producer: this CTA's weight rows and its half of the activation rows ----
      struct At { int i, kc, wp, row0, rows; };
      auto at_tile = [&](At& a) {
        const Item v = item_of(a.i);
        a.wp = v.wp; a.row0 = v.row0; a.rows = v.rows;
      };
      auto next = [&](At& a) { if (++a.kc == k_hi) { a.kc = k_lo; ++a.i; at_tile(a); } };
      auto expect = [&](const At& a, int st) { if (rank == 0) mbar_expect_tx(&full[st], 2 * (Cfg::A_BYTES + a.rows / 2 * Cfg::BK * 2)); };
      auto load_a = [&](uint8_t* dst, const At& a, uint32_t bar) {
        if (MODE == GP_SWIGLU) {
          const int row = (p.packed ? (a.wp * KC + a.kc) * 128 : a.wp * 128) + rank * 64, x = p.packed ? 0 : a.kc * Cfg::BK;
          tma_load_2d_pair(dst, &tm.a[0], x, row, bar);
          tma_load_2d_pair(dst + Cfg::A_BYTES / 2, &tm.a[1], x, row, bar);
        } else {
          const int nt = min(2 * a.wp + rank, p.n_tiles - 1), mat = mat_of(nt), t = nt - p.mat_tile0[mat];
          tma_load_2d_pair(dst, &tm.a[mat], p.packed ? 0 : a.kc * Cfg::BK, p.packed ? (t * KC + a.kc) * 128 : t * 128, bar);
        }
      };
      auto load_b = [&](uint8_t* dst, const At& a, uint32_t bar) {
        tma_load_2d_pair(dst, SPLIT || a.rows == p.tile_rows ? &tm.b : &tm.b_cut, a.kc * Cfg::BK, a.row0 + rank * (a.rows / 2), bar);
      };
      const int n_units = my_tiles * (k_hi - k_lo);
      const int n_pre = n_units < stages ? n_units : stages;
      const uint32_t full0 = dsmem_addr(smem_u32(full), 0);            // the leader's barriers
      At a{0, k_lo, 0, 0, 0};
      at_tile(a);
      At b = a;
      // weights do not depend on the kernel before this one
      for (int i = 0; i < n_pre; ++i, next(a)) {
        expect(a, i);
        load_a(tiles + i * stage_bytes, a, full0 + 8 * i);
      }
      pdl_wait();
      for (int i = 0; i < n_pre; ++i, next(b)) load_b(tiles + i * stage_bytes + Cfg::A_BYTES, b, full0 + 8 * i);
      bool ok = true;
      int issued = n_pre, st = 0;
      uint32_t ph = 0;
      for (; issued < n_units; ++issued, next(a)) {
        if (!mbar_wait(&empty[st], ph, p.status, 40)) { ok = false; break; }
        uint8_t* dst = tiles + st * stage_bytes;
        expect(a, st);
        load_a(dst, a, full0 + 8 * st);
        load_b(dst + Cfg::A_BYTES, a, full0 + 8 * st);
        if (++st == stages) { st = 0; ph ^= 1; }
      }
      if (!ok && rank == 0) {
        for (int i = issued > stages ? issued - stages : 0; i < issued; ++i)
          mbar_wait(&full[i % stages], (i / stages) & 1, p.status, 43);
      }
    }
  } else if (warp == 1) {
    if (rank == 0 && elect_one()) {
      // ---- MMA issuer of the pair ----
      const uint64_t adesc0 = make_kmajor_sw128_desc(smem_u32(tiles)), bdesc0 = make_kmajor_sw128_desc(smem_u32(tiles) + Cfg::A_BYTES);
      bool ok = true;
      int st = 0;
      uint32_t ph = 0;
      for (int i = 0; RUNS && i < my_tiles && ok; ++i) {
        const int buf = p.run_bufs == 2 ? i & 1 : 0, use = p.run_bufs == 2 ? i >> 1 : i;
        if (!mbar_wait(&acc_empty[buf], (use & 1) ^ 1, p.status, 44)) { ok = false; break; }
        tc_fence_after();
        const Item item = item_of(i);
        const uint32_t idesc = make_idesc_bf16(256, item.rows);
        const int nr = runs_of(item.wp);
        for (int r = 0; r < nr && ok; ++r) {
          const uint32_t d_addr = tmem_base + (uint32_t)((buf * p.runs + r) * p.tile_rows);
          const int k_first = run_start(item.wp, r), k_end = r + 1 < nr ? run_start(item.wp, r + 1) : KC;
          for (int kc = k_first; kc < k_end; ++kc) {
            if (!mbar_wait(&full[st], ph, p.status, 41)) { ok = false; break; }
            if (i == 0 && kc == 0) trace_mark_min(p.trace, 2);
            tc_fence_after();
            const uint64_t adesc = adesc0 + (uint64_t)(st * (stage_bytes >> 4)), bdesc = bdesc0 + (uint64_t)(st * (stage_bytes >> 4));
#pragma unroll
            for (int k = 0; k < Cfg::BK / 16; ++k)
              tc_mma_f16_pair(d_addr, adesc + 2 * k, bdesc + 2 * k, idesc, (kc > k_first || k > 0) ? 1u : 0u);
            tc_commit_pair(&empty[st]);
            if (++st == stages) { st = 0; ph ^= 1; }
          }
        }
        if (ok) tc_commit_pair(&acc_full[buf]);
      }
      for (int i = 0; !RUNS && i < my_tiles * halves && ok; ++i) {   // (accumulator fills: tiles, or halves of tiles in turn)
        const int buf = i & 1;
        if (!mbar_wait(&acc_empty[buf], ((i >> 1) & 1) ^ 1, p.status, 44)) { ok = false; break; }
        tc_fence_after();
        const uint32_t d_addr = tmem_base + (uint32_t)(buf * NT), idesc = make_idesc_bf16(256, item_of(halves == 2 ? i >> 1 : i).rows);
        const int mid = (k_lo + k_hi) >> 1;
        const int k_first = halves == 2 && buf ? mid : k_lo, k_end = halves == 2 && !buf ? mid : k_hi;
        for (int kc = k_first; kc < k_end; ++kc) {
          if (!mbar_wait(&full[st], ph, p.status, 41)) { ok = false; break; }
          if (i == 0 && kc == k_lo) trace_mark_min(p.trace, 2);
          tc_fence_after();
          const uint64_t adesc = adesc0 + (uint64_t)(st * (stage_bytes >> 4)), bdesc = bdesc0 + (uint64_t)(st * (stage_bytes >> 4));
#pragma unroll
          for (int k = 0; k < Cfg::BK / 16; ++k)
            tc_mma_f16_pair(d_addr, adesc + 2 * k, bdesc + 2 * k, idesc, (kc > k_first || k > 0) ? 1u : 0u);
          tc_commit_pair(&empty[st]);
          if (++st == stages) { st = 0; ph ^= 1; }
        }
        if (!ok) break;
        tc_commit_pair(&acc_full[buf]);
      }
      trace_mark_max(p.trace, 3);
    }
  } else {
    // ---- epilogue: warp w may touch tensor-memory lanes [32 (w % 4), +32); warps 2..5 take the first quarter of the
    // item's 16-row groups, warps 6..9 the second, ... ----
    constexpr int HC = NT / GP_QUARTERS;                      // rows of a quarter of the largest tile
    const int q = warp & 3, hf = (warp - 2) >> 2;
    const int wl = q * 32 + lane;                             // weight row within the CTA's 128
    const uint32_t acc_empty0 = dsmem_addr(smem_u32(acc_empty), 0);
    pdl_wait();
    if (MODE == GP_PLAIN && p.clear && blockIdx.x == 0 && threadIdx.x < 68) p.clear[threadIdx.x - 64] = 0;
    for (int i = 0; i < my_tiles; ++i) {
      // the accumulator that completes the tile (GP_RUNS: the accumulators' place)
      const int buf = RUNS ? (p.run_bufs == 2 ? i & 1 : 0) : (halves == 2 ? 1 : i & 1);
      const uint32_t acc_ph = RUNS ? (p.run_bufs == 2 ? i >> 1 : i) & 1 : (halves == 2 ? i & 1 : (i >> 1) & 1);
      const Item item = item_of(i);
      const int tau = item.tau, wp = item.wp, groups = item.rows >> 4;
      const int g0 = hf * groups / GP_QUARTERS, ng = (hf + 1) * groups / GP_QUARTERS - g0;   // this warp's 16-row groups
      const int nt = 2 * wp + rank;
      const int m0 = item.row0 + g0 * 16;                     // this warp's first activation row
      const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)((RUNS ? buf * p.runs * p.tile_rows : buf * NT) + g0 * 16);
      const int nr = RUNS ? runs_of(wp) : 1;
      constexpr bool split = SPLIT;
      // (what the epilogue needs besides the sums is fetched while the tile's MMAs run)
      // GP_RESIDUAL: old values of the first rows
      float xo[16];
      const int rcol = nt * 128 + wl;
      const bool ron = MODE == GP_RESIDUAL && nt < p.n_tiles && rcol < p.n_cols;
      auto fetch_x = [&](int g, float (&v)[16]) {
        const float* src = p.out + (size_t)(m0 + g * 16) * p.n_cols + rcol;
        const int live = ron ? p.M - m0 - g * 16 : 0;
#pragma unroll
        for (int j = 0; j < 16; ++j) {                         // (a running pointer: registers)
          v[j] = j < live ? *src : 0.f;
          src += p.n_cols;
        }
      };
      if (MODE == GP_RESIDUAL && !split && ng > 0) fetch_x(0, xo);
      // GP_ROPE: the rows' positions and cache slots
      PairRowMeta* mrow = meta + hf * HC;                     // (a place of its own: the other quarters may be behind, on another item)
      if (MODE == GP_ROPE) {
        const int e = threadIdx.x - 64 - hf * 128;
        group_bar(1 + hf);                                     // everybody is through with the previous tile's rows
        if (e < ng * 16) {
          PairRowMeta v{-1, 0, 0};
          const int m = m0 + e;
          if (m < p.M) {
            const int b = m / p.rows.R, ri = m - b * p.rows.R;
            if (ri < p.rows.cnt[b]) {
              const int slot = p.rows.slot[m];
              const int page = p.page_table[p.rows.sequence(b) * p.g.pages_per_seq + slot / p.g.page_size];
              v.prow = slot % p.g.page_size;
              v.pos = p.rows.pos[m];
              v.kv = (long long)page * 2 * (long long)p.g.block_elems() + (long long)v.prow * p.g.head_dim;
            }
          }
          mrow[e] = v;
        }
        group_bar(1 + hf);
      }
      // GP_PLAIN: the sums over the first half of the inner dimension, kept in registers
      float first[MODE == GP_PLAIN ? HC : 1];
      if constexpr (MODE == GP_PLAIN) {
#pragma unroll
        for (int j = 0; j < HC; ++j) first[j] = 0.f;
        if (halves == 2) {
          if (!epilogue_and(mbar_wait(&acc_full[0], acc_ph, p.status, 42))) break;
          tc_fence_after();
          // (all of a quarter's HC columns, also where the item has fewer: they are this CTA's, and rows that are not its own are not stored)
          uint32_t r[HC / 32][32];
#pragma unroll
          for (int g = 0; g < HC / 32; ++g) tmem_ld32(taddr - NT + g * 32, r[g]);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < HC; ++j) first[j] = __uint_as_float(r[j / 32][j % 32]);
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(acc_empty0);
        }
      }
      // (all warps give up when one of them does: barriers follow)
      if (!epilogue_and(mbar_wait(&acc_full[buf], acc_ph, p.status, 42))) break;
      tc_fence_after();
      // partial sums of this warp's rows, part k at parts_at + k * PART
      constexpr size_t PART = (size_t)2 * NT * 128;
      const float* parts_at = p.part + ((size_t)tau * parts * 2 + rank) * (NT * 128) + (size_t)hf * HC * 128 + wl;
      if (split) {
        float* mine = const_cast<float*>(parts_at) + (cl % parts) * PART;
#pragma unroll 1
        for (int g = 0; g < HC / 32; ++g) {
          uint32_t r[32];
          tmem_ld32(taddr + g * 32, r);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 32; ++j) __stcg(mine + (g * 32 + j) * 128, __uint_as_float(r[j]));
        }
        tc_fence_before();
        __threadfence();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8 * buf);
        epilogue_bar();        // every warp's part precedes the arrival
        if (threadIdx.x == 64) {
          unsigned int* ctr = p.arrive + 2 * tau + rank;
          const bool last = atomicAdd(ctr, 1u) == (unsigned)(parts - 1);
          if (last) *ctr = 0u;
          *last_slot = last;
        }
        epilogue_bar();
        const bool last = *last_slot != 0;
        epilogue_bar();        // everybody has read it
        if (!last) continue;
        __threadfence();
        if (MODE == GP_RESIDUAL) fetch_x(0, xo);
      }
      // sums of this thread's weight row for activation rows [g * 16, +16) of the warp's quarter
      auto acc = [&](int g, uint32_t (&r)[16]) {
        if (!split) {
          tmem_ld16(taddr + g * 16, r);
          tmem_ld_wait();
          if constexpr (RUNS) {
            for (int k = 1; k < nr; ++k) {
              uint32_t more[16];
              tmem_ld16(taddr + k * p.tile_rows + g * 16, more);
              tmem_ld_wait();
#pragma unroll
              for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(more[j]));
            }
          }
          return;
        }
        const float* src = parts_at + g * 16 * 128;
        float v[16];
#pragma unroll
        for (int j = 0; j < 16; ++j) v[j] = __ldcg(src + j * 128);
        for (int k = 1; k < parts; ++k) {
          src += PART;
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] += __ldcg(src + j * 128);
        }
#pragma unroll
        for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(v[j]);
      };
      if constexpr (MODE == GP_PLAIN) {
        const int col = nt * 128 + wl;
        float* dst = p.out + (size_t)m0 * p.ld + col;
        const bool on = nt < p.n_tiles && col < p.n_cols;
#pragma unroll
        for (int g = 0; g < HC / 16; ++g) {                    // (16 columns at a time: registers)
          uint32_t r[16];
          tmem_ld16(taddr + g * 16, r);
          tmem_ld_wait();
#pragma unroll
          for (int j = 0; j < 16; ++j) first[g * 16 + j] += __uint_as_float(r[j]);
        }
        // (given back before the stores: the next tile's MMAs run under them)
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8 * buf);
        const int live = on && p.out ? min(p.M - m0, ng * 16) : 0;
#pragma unroll
        for (int j = 0; j < HC; ++j) {                         // (a running pointer: separate addresses cost 2-3 us a tile)
          if (j < live) *dst = first[j];
          dst += p.ld;
        }
        if (p.best_val) {
          // 32 rows at a time, halved over the lanes (46 shuffles; 64 warp-wide reductions took longer than the tile's MMAs): lane l
          // ends with row l and the lane its largest came from. Columns that are not there count as NaN, which never wins.
#pragma unroll
          for (int j = 0; j < HC; j += 32) {
            int from[16];
            auto wins = [](float v, int i, float ov, int oi) { return better(v, i, ov, oi) || (ov != ov && v == v); };
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              const bool hi = (lane & 16) != 0;
              float lo_v = on ? first[j + i] : __int_as_float(0x7fc00000), hi_v = on ? first[j + i + 16] : __int_as_float(0x7fc00000);
              const float keep = hi ? hi_v : lo_v, got = __shfl_xor_sync(0xffffffffu, hi ? lo_v : hi_v, 16);
              const bool take = wins(got, lane ^ 16, keep, lane);
              first[j + i] = take ? got : keep;
              from[i] = take ? lane ^ 16 : lane;
            }
#pragma unroll
            for (int o = 8; o > 0; o >>= 1) {
              const bool hi = (lane & o) != 0;
#pragma unroll
              for (int i = 0; i < o; ++i) {
                const float keep = hi ? first[j + i + o] : first[j + i];
                const int keep_f = hi ? from[i + o] : from[i];
                const float got = __shfl_xor_sync(0xffffffffu, hi ? first[j + i] : first[j + i + o], o);
                const int got_f = __shfl_xor_sync(0xffffffffu, hi ? from[i] : from[i + o], o);
                const bool take = wins(got, got_f, keep, keep_f);
                first[j + i] = take ? got : keep;
                from[i] = take ? got_f : keep_f;
              }
            }
            const int m = m0 + j + lane;
            const float best = first[j];
            if (nt < p.n_tiles && m < p.M && j + lane < ng * 16) {
              p.best_val[(size_t)(nt * 4 + q) * p.M + m] = best == best ? best : -INFINITY;
              p.best_idx[(size_t)(nt * 4 + q) * p.M + m] = best == best ? nt * 128 + q * 32 + from[0] : 0x7fffffff;
            }
          }
        }
        continue;
      } else if constexpr (MODE == GP_RESIDUAL) {
        // old values of the next 16 rows are fetched while 16 rows are finished
#pragma unroll 1
        for (int g = 0; g < ng; ++g) {
          uint32_t r[16];
          float next[16];
          if (g + 1 < ng) fetch_x(g + 1, next);
          acc(g, r);
          float* dst = p.out + (size_t)(m0 + g * 16) * p.n_cols + rcol;
          const int live = ron ? p.M - m0 - g * 16 : 0;
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            if (j < live) *dst = xo[j] + __uint_as_float(r[j]);
            dst += p.n_cols;
          }
#pragma unroll
          for (int j = 0; j < 16; ++j) xo[j] = next[j];
        }
      } else {
        // outputs that need two weight rows of the tile: row pairs (lower, upper) = (gate, up) or a rotation pair
        const int D = p.g.head_dim;
        const int nt_c = min(nt, p.n_tiles - 1);
        const int mat = MODE == GP_ROPE ? mat_of(nt_c) : 0;
        const int hp = MODE == GP_ROPE ? D >> 1 : 64;           // distance between the rows of a pair
        const bool lower = (wl & hp) == 0;
        const int pr = hp == 64 ? (wl & 63) : ((wl & 31) | ((wl >> 6) << 5));   // pair 0..63
        float* ex_lo = exch + hf * (2 * 64 * Cfg::EX_COLS);      // written by the lower rows' threads
        float* ex_up = ex_lo + 64 * Cfg::EX_COLS;
        if (MODE == GP_SWIGLU) {
          const int col = nt * 64 + pr;
          const bool on = col < p.n_cols;
#pragma unroll 1
          for (int g = 0; g < ng; ++g) {
            uint32_t r[16];
            acc(g, r);
            if (g) group_bar(1 + hf);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              if (lower) ex_lo[j * 64 + pr] = __uint_as_float(r[8 + j]);
              else ex_up[j * 64 + pr] = __uint_as_float(r[j]);
            }
            group_bar(1 + hf);
            const int mb = m0 + g * 16 + (lower ? 0 : 8);
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const float gt = lower ? __uint_as_float(r[j]) : ex_lo[j * 64 + pr];
              const float up = lower ? ex_up[j * 64 + pr] : __uint_as_float(r[8 + j]);
              if (on && mb + j < p.M) p.act[(size_t)(mb + j) * p.n_cols + col] = __float2bfloat16_rn(silu_f(gt) * up);
            }
          }
          group_bar(1 + hf);
        } else {
          const int kind = mat + p.kind0;                        // 0 q, 1 k, 2 v
          const int n_rows_mat = (kind == 0 ? p.H : p.g.n_kv_heads) * D;
          const int row = (nt_c - p.mat_tile0[mat]) * 128 + wl;  // weight row within its matrix
          const bool on = nt < p.n_tiles && row < n_rows_mat;
          const int head = row / D, dim = row - head * D;
          const int half = D >> 1;
          const size_t lh = ((size_t)p.layer * p.g.n_kv_heads + head) * p.g.pool_pages() * 2 * p.g.block_elems();
          if (kind == 2) {
            bf16* dst = p.pool + lh + p.g.block_elems();
#pragma unroll 1
            for (int g = 0; g < ng; ++g) {
              uint32_t r[16];
              acc(g, r);
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const PairRowMeta v = mrow[g * 16 + j];
                if (on && v.kv >= 0) dst[v.kv + kv_elem<bf16>(v.prow, dim, D, p.g.page_size)] = __float2bfloat16_rn(__uint_as_float(r[j]));
              }
            }
          } else {
            const int di = dim & (half - 1);                     // the pair's place in its head
#pragma unroll 1
            for (int g = 0; g < ng; ++g) {
              uint32_t r[16];
              const int jb = g * 16 + (lower ? 0 : 8);
              float2 t[8];
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const PairRowMeta v = mrow[jb + j];
                t[j] = p.cs[(size_t)v.pos * half + di];          // (position 0 for rows not in use)
              }
              acc(g, r);
              if (g) group_bar(1 + hf);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                if (lower) ex_lo[j * 64 + pr] = __uint_as_float(r[8 + j]);
                else ex_up[j * 64 + pr] = __uint_as_float(r[j]);
              }
              group_bar(1 + hf);
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const PairRowMeta v = mrow[jb + j];
                if (!on || v.kv < 0) continue;
                const float a = lower ? __uint_as_float(r[j]) : ex_lo[j * 64 + pr];
                const float c = lower ? ex_up[j * 64 + pr] : __uint_as_float(r[8 + j]);
                                // (the rounding of the other kernels that rotate: one product rounded, the other fused into the sum)
                const bf16 lo = __float2bfloat16_rn(__fmaf_rn(a, t[j].x, -__fmul_rn(c, t[j].y)));
                const bf16 hi = __float2bfloat16_rn(__fmaf_rn(c, t[j].x, __fmul_rn(a, t[j].y)));
                if (kind == 0) {
                  const int m = m0 + jb + j;
                  bf16* dst = p.q + (size_t)(p.q_chunk ? m * p.q_chunk + v.pos % p.q_chunk : m) * p.H * D + head * D + di;
                  dst[0] = lo;
                  dst[half] = hi;
                } else {
                  bf16* dst = p.pool + lh + v.kv;
                  dst[kv_elem<bf16>(v.prow, di, D, p.g.page_size)] = lo;
                  dst[kv_elem<bf16>(v.prow, di + half, D, p.g.page_size)] = hi;
                }
              }
            }
            group_bar(1 + hf);
          }
        }
      }
      if (split) continue;                                    // (its accumulator was given back above)
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster(acc_empty0 + 8 * buf);
    }
  }

  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                       // nobody leaves while the pair's MMAs, copies or arrivals may still reach it
  if (warp == 1) { tc_fence_after(); tmem_dealloc2(tmem_base, Cfg::TMEM_COLS); }
}

}  // namespace spec
