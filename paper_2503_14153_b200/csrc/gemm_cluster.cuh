// Weight-streaming bf16 linear whose split-K partial sums never leave the chip: the CTAs that
// share an output tile form a thread-block cluster and exchange their float32 accumulators through
// distributed shared memory, so the kernel writes finished results and the element-wise step that
// used to follow in a kernel of its own runs in the epilogue.
//
// The exchange: once its MMAs are complete a CTA announces that its ring is free (cluster barrier, arrive only), puts its
// accumulators into its own shared memory, a block of columns (or rows) per CTA that finishes them, and when every ring of
// the cluster is free (the barrier's wait) sends each block with one bulk copy that completes on the receiver's mbarrier.
// A CTA exits only after everybody has received (another arrive / wait pair, under the finishing work). Only the pass's
// rows travel, not the MT rows of the MMA.
// The tail, last MMA to the end of the kernel, is what bounds these kernels beside the weight stream. On the 7B shape with 64
// rows it was 7.1 us for gate+up, 3.6 and 3.5 for the output and down projections and 2.8 for q/k/v with four epilogue warps that sent
// single values with remote stores (q/k/v: read them), and is 4.1, 2.5, 2.9 and 1.6; a layer 96.4 -> 93.2 us. In-kernel
// timestamps of gate+up: draining 2.0 -> 0.7 us and finishing 3.0 -> 1.2 with eight warps; 0.5 us for each barrier.cluster.arrive with release
// semantics where nothing has to be published (now .relaxed); the copies themselves, 48 KB out of the middle CTA with two CTAs an
// SM, 1.7 us.
//
// Four modes (operands swapped as in gemm_stream: 128 weight rows are the MMA's M, the MT activation
// rows its N; MT covers all rows of the pass):
//  * GC_RESIDUAL (output and down projections): a cluster of 8 CTAs per 128-row weight tile, CTA r
//    streaming the r-th eighth of the K chunks. CTA r owns output columns [16 r, 16 r + 16) of the
//    tile: it adds the eight parts in rank order, adds the residual stream x in place (old values
//    fetched during the exchange) and leaves the sum of squares of its piece of every row (the RMSNorm
//    that follows needs the row's mean square) in ss_part[m][tile * 8 + r].
//  * GC_SWIGLU (gate and up projections): a cluster of 3 CTAs per pair (gate tile t, up tile t); the
//    2 KC units of the pair are cut into three equal runs, so CTA 0 holds a gate part, CTA 1 a gate
//    and an up part (two accumulators) and CTA 2 an up part. Each CTA finishes a share of the tile's columns (48, 32 and 48):
//    gate = G0 + G1, up = U1 + U2, act = bf16(SiLU(gate) * up).
//  * GC_PLAIN (a projection by itself; lm_head): a cluster of 1 to 8 per tile, CTA r streaming the r-th part of the K chunks, its
//    first half into one accumulator and its second into another (the error of a running sum grows with its
//    length), and finishing a block of rows: float32 sums, and where asked each row's largest in the tile.
//  * GC_ROPE (query, key and value projections, stacked): a cluster of 2 CTAs per 128-row tile of the
//    stacked matrices, each streaming half of the K chunks (96 pairs on the 7B shape: all co-resident, which
//    96 clusters of 3 are not). A tile holds whole heads (head_dim 64 or
//    128), so after the exchange the cluster rotates the query / key pairs (i, i + head_dim / 2) by the
//    row's position, writes the bf16 query rows and puts the bf16 key and value rows into the paged cache
//    at the row's slot; each CTA takes half of the activation rows.
// Sums are added in a fixed order: results are bit-reproducible. Every wait is bounded; a CTA whose
// wait ran out still sends its blocks and arrives at the cluster barriers, so its cluster mates never wait for it.
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "gemm_stream.cuh"

namespace spec {

constexpr int GC_RESIDUAL = 0, GC_SWIGLU = 1, GC_ROPE = 2, GC_PLAIN = 3;
constexpr int GC_THREADS = 320, GC_EPI = GC_THREADS - 64;     // producer, MMA issuer, eight epilogue warps (two per SM quarter)
constexpr int GC_RES_CLUSTER = 8, GC_GLU_CLUSTER = 3, GC_ROPE_CLUSTER = 2;

struct ClusterGemmParams {
  int M, K, KC;                 // activation rows (<= MT), inner size, K / 64
  int stages;                   // of the ring: ClusterCfg<MT>::FEWEST_STAGES to MAX_STAGES (see cluster_stages)
  int N;                        // weight rows of one matrix (output columns)
  const uint8_t* packed[3];     // pre-tiled images (GC_RESIDUAL: [0]; GC_SWIGLU: gate, up; GC_ROPE: q, k, v) or nullptr -> tensor maps a[i]
  float* x;                     // GC_RESIDUAL: [M][N] float32 residual stream, updated in place
  float* ss_part;               // GC_RESIDUAL: [M][ceil(N/128) * 8] sums of squares of the updated pieces, or nullptr
  bf16* act;                    // GC_SWIGLU: [M][N] bf16
  // GC_PLAIN: sums to y[M][ldy], columns below N (y may be nullptr), and of every row's sums in this tile the largest and its column (value
  // descending, column ascending) to best_val / best_idx [M][tiles] (may be nullptr); clear: four ints set to zero, or nullptr
  float* y;
  size_t ldy;
  float* best_val;
  int* best_idx;
  int* clear;
  // GC_ROPE: tiles [0, tile0[1]) belong to q, [tile0[1], tile0[2]) to k, the rest to v
  int tile0[3];
  int tile_first;               // first tile of the launch (a prompt's last layer may take k and v alone)
  int H;                        // query heads
  int layer;
  Rows rows;
  const float2* cs;             // [position][head_dim / 2] (cos, sin)
  bf16* q;                      // [M][H * head_dim]
  bf16* pool;                   // paged KV cache
  KVGeom g;
  const int* page_table;
  int* status;
  unsigned long long* trace;
};

template <int MT> struct ClusterCfg {
  static constexpr int BK = 64;
  static constexpr int A_BYTES = 128 * BK * 2;
  static constexpr int B_BYTES = MT * BK * 2;
  static constexpr int STAGE_BYTES = A_BYTES + B_BYTES;
  static constexpr int STAGES = (MT <= 32) ? 5 : (MT == 64 ? 4 : 3);      // two CTAs an SM
  static constexpr int FEWEST_STAGES = MT == 16 ? 4 : STAGES;             // three (GC_RESIDUAL)
  static constexpr int EXTRA_BYTES = 1024 /*alignment slack*/ + 256 /*barriers*/;
  static constexpr int MAX_STAGES = (227 * 1024 - EXTRA_BYTES) / STAGE_BYTES < 12 ? (227 * 1024 - EXTRA_BYTES) / STAGE_BYTES : 12;   // one CTA an SM
  static constexpr int smem_bytes(int stages) { return stages * STAGE_BYTES + EXTRA_BYTES; }
};

// Clusters of `size` CTAs that the chip holds at one CTA an SM (cudaOccupancyMaxActiveClusters): a cluster lies within a group of neighbouring SMs, so
// 15 clusters of eight fit, not 18.
constexpr int CLUSTERS_ALONE[9] = {0, 148, 74, 45, 33, 26, 22, 15, 15};

// Stages of a launch of `tiles` clusters of `cluster` CTAs with at most `units` K chunks each. Where all clusters fit at one CTA an SM (the projections
// of narrow models: at d_model 1024 q/k/v has 24 CTAs of 8 chunks, gate+up 66 of 11) a CTA gets a stage for every
// chunk as far as shared memory goes, so that all of its weights are under way before the dependency wait and the chain behind it is
// activation tiles, MMAs and the exchange: a 64-row step of six layers of d_model 1024 284 -> 263 us. The others get the ring of which two fit an SM:
// with the deep one the last clusters run when the first ones are through (eight layers of 64 rows, d_model 2048, ffn 6144, down in 16 clusters of
// eight: 468 us with the deep ring, 399 with the shallow one).
// The output and down projections of up to 16 rows in more clusters than that, with short runs (wo of the 7B shape: 32 clusters of 8 CTAs, 8 chunks
// each), have a ring of which three fit an SM: the attention before wo has 32 CTAs, and with two an SM a few clusters did not find room beside those and
// began when it ended: wo 9.9 -> 7.5 us. (With 64 rows attention has 128 CTAs and three stages cost more than they give: 10.1 -> 10.8.)
template <int MT, int MODE> inline int cluster_stages(int tiles, int cluster, int units) {
  using Cfg = ClusterCfg<MT>;
  if (tiles > CLUSTERS_ALONE[cluster]) return MODE == GC_RESIDUAL && MT == 16 && tiles * cluster > 148 && units <= 8 ? Cfg::FEWEST_STAGES : Cfg::STAGES;
  return units <= Cfg::STAGES ? Cfg::STAGES : (units < Cfg::MAX_STAGES ? units : Cfg::MAX_STAGES);
}

__device__ __forceinline__ uint32_t cluster_ctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ uint32_t cluster_nctarank() {
  uint32_t r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ void cluster_sync_all() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_arrive_relaxed() { asm volatile("barrier.cluster.arrive.relaxed.aligned;" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire.aligned;" ::: "memory"); }
__device__ __forceinline__ uint32_t dsmem_addr(uint32_t local_smem_addr, uint32_t rank) {
  uint32_t a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(local_smem_addr), "r"(rank));
  return a;
}
__device__ __forceinline__ float4 dsmem_ld4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void dsmem_st(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory");
}
// Bulk copy from this CTA's shared memory into another CTA's, completing on that CTA's barrier (16-byte aligned, size
// a multiple of 16).
__device__ __forceinline__ void bulk_push(uint32_t dst_cluster, const void* src, uint32_t bytes, uint32_t bar_cluster) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst_cluster), "r"(smem_u32(src)), "r"(bytes), "r"(bar_cluster) : "memory");
}
// Generic-proxy writes to shared memory become visible to bulk copies that read it.
__device__ __forceinline__ void fence_smem_async() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }
__device__ __forceinline__ void add4(float4& a, const float4& b) { a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w; }

__device__ __forceinline__ uint32_t pack_bf16x2(float lo, float hi) {
  __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<uint32_t*>(&v);
}

// Which product of a sum is rounded and which is fused into it is spelled out: left to the compiler it went with the code around it, and the
// bf16 operands made from the results, and the tokens in the end, with it. (The instances of few rows differ from the others only so
// that every number of rows keeps the rounding that it has had.)
template <int MT> __device__ __forceinline__ float sum_sq(const float4& v) {
  const float xy = MT <= 32 ? __fmaf_rn(v.y, v.y, __fmul_rn(v.x, v.x)) : __fmaf_rn(v.x, v.x, __fmul_rn(v.y, v.y));
  return __fmaf_rn(v.w, v.w, __fmaf_rn(v.z, v.z, xy));
}
__device__ __forceinline__ float rotate_lo(float a, float c, float co, float si) { return __fmaf_rn(a, co, -__fmul_rn(c, si)); }
template <int MT> __device__ __forceinline__ float rotate_hi(float a, float c, float co, float si) {
  return MT == 16 ? __fmaf_rn(a, si, __fmul_rn(c, co)) : __fmaf_rn(c, co, __fmul_rn(a, si));
}

// Rows of one accumulator (or of a stretch of its columns) at `taddr`, in groups of 16 of which the two epilogue warps of an SM quarter take every
// second one: put(row, value) in the thread that owns the weight row, for rows below M.
// With `second` > 0 the accumulator that many columns further on is added. One group's code for all of them: a kernel runs through
// this once, and unrolled over the groups, with a pointer chosen for every row, it waited for its instructions: staging q/k/v of 64 rows took
// 1.3 us and of 69 rows 3.7 (now 0.6 and 0.7), a step of 69 rows on six layers of d_model 1024 333 us (now 312), and the code of the whole
// epilogue had lm_head's registers spilled.
template <typename F>
__device__ __forceinline__ void tmem_rows(uint32_t taddr, int hf, int M, F&& put, int second = 0) {
#pragma unroll 1
  for (int m0 = hf * 16; m0 < M; m0 += 32) {                 // (the same in the whole warp)
    uint32_t r[16];
    tmem_ld16(taddr + m0, r);
    tmem_ld_wait();
    if (second) {
      uint32_t r2[16];
      tmem_ld16(taddr + second + m0, r2);
      tmem_ld_wait();
#pragma unroll
      for (int j = 0; j < 16; ++j) r[j] = __float_as_uint(__uint_as_float(r[j]) + __uint_as_float(r2[j]));
    }
#pragma unroll
    for (int j = 0; j < 16; ++j)
      if (m0 + j < M) put(m0 + j, __uint_as_float(r[j]));
  }
}

// One run of K chunks of one weight tile, accumulated into one tensor-memory buffer.
struct GcSeg {
  int mat, kc0, kc1;
};

template <int MT, int MODE>
__global__ void __launch_bounds__(GC_THREADS, 2)
gemm_cluster(const __grid_constant__ StreamTmaps tm, const ClusterGemmParams p) {
  using Cfg = ClusterCfg<MT>;
  const int stages = p.stages, ring_bytes = stages * Cfg::STAGE_BYTES;
  const int mma_n = (p.M + 15) & ~15;                        // the MMA's N: only rows that are there are fetched
  const uint32_t stage_tx = Cfg::A_BYTES + mma_n * Cfg::BK * 2;
  constexpr bool PLAIN = MODE == GC_PLAIN;
  const int CS = PLAIN ? (int)cluster_nctarank() : (MODE == GC_RESIDUAL ? GC_RES_CLUSTER : (MODE == GC_SWIGLU ? GC_GLU_CLUSTER : GC_ROPE_CLUSTER));
  constexpr int TMEM_COLS = (MODE == GC_SWIGLU || PLAIN ? 2 : 1) * MT < 32 ? 32 : (MODE == GC_SWIGLU || PLAIN ? 2 : 1) * MT;   // 32 to 256
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* tiles = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  uint64_t* bars = reinterpret_cast<uint64_t*>(tiles + ring_bytes);
  uint64_t* full = bars;
  uint64_t* empty = bars + stages;
  uint64_t* acc_full = bars + 2 * stages;
  uint64_t* part_full = bars + 2 * stages + 1;               // the other CTAs' parts of this CTA's outputs have landed
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bars + 2 * stages + 2);
  float* staging = reinterpret_cast<float*>(tiles);          // reuses the ring once every MMA is complete

  KTrace kt(p.trace);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = (int)cluster_ctarank();
  const int t = blockIdx.x / CS + (MODE == GC_ROPE ? p.tile_first : 0);   // weight tile (GC_SWIGLU: tile pair; GC_ROPE: of the stacked q, k, v)
  const int KC = p.KC;
  int rope_mat = 0;
  if (MODE == GC_ROPE) rope_mat = t >= p.tile0[2] ? 2 : (t >= p.tile0[1] ? 1 : 0);
  const int t_in_mat = MODE == GC_ROPE ? t - p.tile0[rope_mat] : t;

  // this CTA's runs
  GcSeg seg[2];
  int nseg = 0;
  if (PLAIN) {
    const int k0 = rank * KC / CS, k1 = (rank + 1) * KC / CS, mid = (k0 + k1 + 1) >> 1;
    seg[nseg++] = GcSeg{0, k0, mid};
    if (mid < k1) seg[nseg++] = GcSeg{0, mid, k1};
  } else if (MODE != GC_SWIGLU) {
    seg[0] = GcSeg{rope_mat, rank * KC / CS, (rank + 1) * KC / CS};
    nseg = 1;
  } else {
    const int u_lo = rank * 2 * KC / CS, u_hi = (rank + 1) * 2 * KC / CS;
    if (u_lo < KC) seg[nseg++] = GcSeg{0, u_lo, u_hi < KC ? u_hi : KC};
    if (u_hi > KC) seg[nseg++] = GcSeg{1, u_lo > KC ? u_lo - KC : 0, u_hi - KC};
  }
  const int n_units = (seg[0].kc1 - seg[0].kc0) + (nseg > 1 ? seg[1].kc1 - seg[1].kc0 : 0);

  // ---- layout of the exchange, in the ring: `in`, the parts of this CTA's outputs, then `out`, what it sends ----
  constexpr int LEAST_BYTES = (MODE == GC_RESIDUAL ? Cfg::FEWEST_STAGES : Cfg::STAGES) * Cfg::STAGE_BYTES;   // of a ring
  const int M = p.M;
  // GC_ROPE: CTA 0 finishes activation rows [0, r_half), CTA 1 the rest
  const int r_half = (M + 1) / 2, r_row0 = rank * r_half, r_rows = MODE == GC_ROPE ? (rank ? M - r_half : r_half) : 0;
  // GC_SWIGLU: the tile's columns in groups of 16, of which CTA 0 finishes 0..2, CTA 1 3 and 4, CTA 2 5..7
  constexpr int GLU_FIRST[4] = {0, 3, 5, 8};
  const int glu_g0 = GLU_FIRST[rank % 3], glu_ng = GLU_FIRST[rank % 3 + 1] - glu_g0;
  // GC_PLAIN: more than 64 rows in two rounds, because the ring does not hold all of them staged and arriving at once
  constexpr int ROUNDS = PLAIN && MT > 64 ? 2 : 1, RT = ROUNDS == 2 ? 64 : MT;
  const int rr = ROUNDS == 2 ? (M + 31) / 32 * 16 : M;       // rows of a round (at most RT)
  // GC_RESIDUAL: rows that travel as bulk copies; the ring of MT = 128 has no room for the staged copy of all rows beside the
  // arriving ones when there are more than about 100, and the others are sent straight from tensor memory
  const int S = MODE == GC_RESIDUAL ? min(M, (ring_bytes - GC_RES_CLUSTER * M * 64) / ((GC_RES_CLUSTER - 1) * 64) - 1) : rr;
  // GC_PLAIN: CTA r finishes the r-th block of rows of a round
  const int rb = PLAIN ? (rr + CS - 1) / CS : 0;
  const int in_pitch = MODE == GC_RESIDUAL ? M * 16 : (rr | 1) * 16;       // floats of a group of 16 columns (odd: banks)
  const int out_pitch = (S | 1) * 16;
  float* in = staging;
  float* out = staging + (MODE == GC_RESIDUAL ? GC_RES_CLUSTER * in_pitch : MODE == GC_SWIGLU ? 4 * glu_ng * in_pitch : PLAIN ? CS * rb * 128 : 2 * r_rows * 128);
  static_assert(!PLAIN || LEAST_BYTES >= (2 * RT + 8) * 512, "a round's rows staged, and eight parts of this CTA's block");
  static_assert(MODE != GC_RESIDUAL || LEAST_BYTES >= GC_RES_CLUSTER * MT * 64 + (GC_RES_CLUSTER - 1) * 64 * 17, "in, and 16 rows of out");
  static_assert(MODE != GC_SWIGLU || LEAST_BYTES >= (4 * 3 + 5) * (RT | 1) * 64, "CTA 0 and 2: four parts of three groups, five groups to send");
  static_assert(MODE != GC_SWIGLU || LEAST_BYTES >= (4 * 2 + 2 * 6) * (RT | 1) * 64, "CTA 1: four parts of two groups, six groups of two accumulators");
  static_assert(MODE != GC_ROPE || LEAST_BYTES >= 3 * ((MT + 1) / 2) * 512, "own and arriving rows, rows to send");
  // bytes that arrive in a round of `rows` rows
  auto in_bytes = [&](int rows) -> uint32_t {
    return MODE == GC_RESIDUAL ? (GC_RES_CLUSTER - 1) * S * 64 : MODE == GC_SWIGLU ? (rank == 1 ? 2 : 3) * glu_ng * rows * 64 : PLAIN ? (CS - 1) * max(0, min(rb, rows - rank * rb)) * 512 : r_rows * 512;
  };

  pdl_launch_dependents();

  if (threadIdx.x == 0) {
    for (int i = 0; i < stages; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(acc_full, 1);
    mbar_init(part_full, 1);
    mbar_fence_init();
    mbar_expect_tx(part_full, in_bytes(rr));                 // (the first copy comes after the first cluster barrier)
    for (int i = 0; i < (MODE == GC_RESIDUAL || PLAIN ? 1 : (MODE == GC_ROPE ? 3 : 2)); ++i) if (!p.packed[i]) tma_prefetch_desc(&tm.a[i]);
    tma_prefetch_desc(&tm.b);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, TMEM_COLS); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;

  // unit i of this CTA -> (segment, K chunk)
  auto unit = [&](int i, int& s, int& kc) {
    const int n0 = seg[0].kc1 - seg[0].kc0;
    if (i < n0) { s = 0; kc = seg[0].kc0 + i; } else { s = 1; kc = seg[1].kc0 + (i - n0); }
  };

  // GC_RESIDUAL: a finishing thread's items (row, group of four columns) and their old values
  constexpr int X_PER = MODE == GC_RESIDUAL ? (MT * 4 + GC_EPI - 1) / GC_EPI : 1;
  float4 xo[X_PER];
  bool x_on[X_PER];

  // GC_ROPE: what a finishing thread needs to know about its items (row bookkeeping, cos / sin, destination) is
  // fetched by the epilogue warps while the MMAs run, not after the cluster barrier
  constexpr int R_ROWS_MAX = (MT + GC_ROPE_CLUSTER - 1) / GC_ROPE_CLUSTER, R_ITEMS = R_ROWS_MAX * 16;
  constexpr int R_PER = MODE == GC_ROPE ? (R_ITEMS + GC_EPI - 1) / GC_EPI : 1;
  bool r_on[R_PER];
  int r_mrow[R_PER], r_lo_c[R_PER];
  float4 r_cs01[R_PER], r_cs23[R_PER];
  bf16* r_dst[R_PER];
  auto rope_meta = [&]() {
    constexpr int PER = R_PER;
    const int e = threadIdx.x - 64;
    const int D = p.g.head_dim, half = D >> 1, gph = half >> 2;       // pair groups per head
    const int n_rows_mat = rope_mat == 0 ? p.H * D : p.g.n_kv_heads * D;
    bool (&on)[R_PER] = r_on;
    int (&mrow)[R_PER] = r_mrow, (&lo_c)[R_PER] = r_lo_c;
    float4 (&cs01)[R_PER] = r_cs01, (&cs23)[R_PER] = r_cs23;
    bf16* (&dst)[R_PER] = r_dst;
#pragma unroll
      for (int k = 0; k < PER; ++k) {
        const int it = e + GC_EPI * k, ml = it >> 4, pg = it & 15;
        const int m = r_row0 + ml;
        const int hh = pg / gph, g = pg % gph;
        lo_c[k] = hh * D + 4 * g;
        mrow[k] = ml;
        const int row_lo = t_in_mat * 128 + lo_c[k];                      // weight row within its matrix
        on[k] = ml < r_rows && row_lo < n_rows_mat;
        cs01[k] = cs23[k] = make_float4(1.f, 0.f, 1.f, 0.f);
        dst[k] = nullptr;
        if (on[k]) {
          const int b = m / p.rows.R, ri = m % p.rows.R;
          on[k] = ri < p.rows.cnt[b];
          const int head = row_lo / D, i = 4 * g;
          if (rope_mat < 2) {
            const float2* c = p.cs + (size_t)p.rows.pos[m] * half + i;
            cs01[k] = *reinterpret_cast<const float4*>(c);
            cs23[k] = *reinterpret_cast<const float4*>(c + 2);
          }
          if (rope_mat == 0) {
            dst[k] = p.q + (size_t)m * p.H * D + head * D + i;
          } else {
            const int slot = p.rows.slot[m];
            const int page = p.page_table[p.rows.sequence(b) * p.g.pages_per_seq + slot / p.g.page_size], prow = slot % p.g.page_size;
            // (a group of four lies inside one 16-byte chunk of the row: the chunk swizzle keeps it contiguous)
            dst[k] = p.pool + p.g.block_offset(page, p.layer, rope_mat - 1, head) + (size_t)prow * D + kv_elem<bf16>(prow, i, D, p.g.page_size);
            lo_c[k] |= (kv_elem<bf16>(prow, i + half, D, p.g.page_size) - kv_elem<bf16>(prow, i, D, p.g.page_size)) << 16;   // distance to the upper half's group
          }
        }
      }
  };

  if (warp == 0) {
    if (elect_one()) {
      // ---- producer: weights before the dependency wait, activation tiles after it ----
      const uint64_t wpol = l2_policy_evict_first();
      const int n_pre = n_units < stages ? n_units : stages;
      auto load_a = [&](uint8_t* dst, int s, int kc, uint64_t* bar) {
        const int mat = seg[s].mat;
        if (p.packed[mat])
          bulk_load_1d_hint(dst, p.packed[mat] + ((size_t)t_in_mat * KC + kc) * Cfg::A_BYTES, Cfg::A_BYTES, bar, wpol);
        else
          tma_load_2d_hint(dst, &tm.a[mat], kc * Cfg::BK, t_in_mat * 128, bar, wpol);
      };
      for (int i = 0; i < n_pre; ++i) {
        int s, kc;
        unit(i, s, kc);
        mbar_expect_tx(&full[i], stage_tx);
        load_a(tiles + i * Cfg::STAGE_BYTES, s, kc, &full[i]);
      }
      pdl_wait();
      for (int i = 0; i < n_pre; ++i) {
        int s, kc;
        unit(i, s, kc);
        tma_load_2d(tiles + i * Cfg::STAGE_BYTES + Cfg::A_BYTES, &tm.b, kc * Cfg::BK, 0, &full[i]);
      }
      bool ok = true;
      int issued = n_pre, st = 0;
      uint32_t ph = 0;                                       // (a ring that is refilled has been filled once)
      for (; issued < n_units; ++issued) {
        if (!mbar_wait(&empty[st], ph, p.status, 30)) { ok = false; break; }
        int s, kc;
        unit(issued, s, kc);
        uint8_t* a = tiles + st * Cfg::STAGE_BYTES;
        mbar_expect_tx(&full[st], stage_tx);
        load_a(a, s, kc, &full[st]);
        tma_load_2d(a + Cfg::A_BYTES, &tm.b, kc * Cfg::BK, 0, &full[st]);
        if (++st == stages) { st = 0; ph ^= 1; }
      }
      if (!ok) {
        for (int i = issued > stages ? issued - stages : 0; i < issued; ++i)
          mbar_wait(&full[i % stages], (i / stages) & 1, p.status, 33);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      // ---- MMA issuer: one accumulator per run ----
      const uint32_t idesc = make_idesc_bf16(128, mma_n);
      bool ok = true;
      int done = 0, st = 0;
      uint32_t ph = 0;
      const uint64_t adesc0 = make_kmajor_sw128_desc(smem_u32(tiles)), bdesc0 = make_kmajor_sw128_desc(smem_u32(tiles) + Cfg::A_BYTES);
      for (int s = 0; s < nseg && ok; ++s) {
        const uint32_t d_addr = tmem_base + (uint32_t)(s * MT);
        const int n = seg[s].kc1 - seg[s].kc0;
        for (int v = 0; v < n; ++v, ++done) {
          if (!mbar_wait(&full[st], ph, p.status, 31)) { ok = false; break; }
          if (done == 0) trace_mark_min(p.trace, 2);
          tc_fence_after();
          const uint64_t adesc = adesc0 + (uint64_t)(st * (Cfg::STAGE_BYTES >> 4)), bdesc = bdesc0 + (uint64_t)(st * (Cfg::STAGE_BYTES >> 4));
#pragma unroll
          for (int k = 0; k < Cfg::BK / 16; ++k)
            tc_mma_f16(d_addr, adesc + 2 * k, bdesc + 2 * k, idesc, (v > 0 || k > 0) ? 1u : 0u);
          if (done + stages < n_units) tc_commit(&empty[st]);     // (a stage that is not filled again needs no announcement)
          if (++st == stages) { st = 0; ph ^= 1; }
        }
      }
      if (ok) tc_commit(acc_full);         // arrives once every MMA above is complete (and has read its operands)
      trace_mark_max(p.trace, 3);
    }
  } else {
    // ---- epilogue: what it needs besides the sums is fetched while the MMAs run ----
    pdl_wait();
    if (MODE == GC_ROPE) rope_meta();
    if (PLAIN && p.clear && blockIdx.x == 0 && threadIdx.x < 68) p.clear[threadIdx.x - 64] = 0;
    if (MODE == GC_RESIDUAL) {
#pragma unroll
      for (int k = 0; k < X_PER; ++k) {
        const int it = (int)threadIdx.x - 64 + GC_EPI * k, m = it >> 2, col = t * 128 + rank * 16 + (it & 3) * 4;
        x_on[k] = m < M && col < p.N;
        xo[k] = x_on[k] ? *reinterpret_cast<const float4*>(p.x + (size_t)m * p.N + col) : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
    mbar_wait(acc_full, 0, p.status, 32);
  }

  // ---- exchange: this CTA's MMAs are complete, its ring is free. Its accumulators go to shared memory (`out`, or `in` where
  // the columns are its own) while the others finish theirs ----
  const int e = (int)threadIdx.x - 64;                       // epilogue thread
  const bool epi = warp >= 2;
  const int q = warp & 3, hf = warp >= 6 ? 1 : 0, w = q * 32 + lane;   // its tensor-memory lane = weight row of the tile
  const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16);
  const int grp = w >> 4;                                    // its group of 16 columns
#pragma unroll 1
  for (int rd = 0; rd < ROUNDS; ++rd) {
    const int m0 = rd * rr, Mr = min(rr, M - m0);            // rows of this round
    __syncwarp();
    if (rd == 0) {
      if (warp == 0) cluster_arrive();                       // (its first thread has set up the barrier the copies complete on)
      else cluster_arrive_relaxed();                         // (a ring is free once its MMAs are complete; nothing else to publish)
    } else {
      // everybody has received the first round (so `out` may be overwritten) and is through with it (`in`)
      if (epi) {
        asm volatile("bar.sync 5, %0;" ::"n"(GC_EPI) : "memory");
        if (e == 0) mbar_expect_tx(part_full, in_bytes(Mr));
        __syncwarp();
      }
      if (warp == 2) cluster_arrive();
      else cluster_arrive_relaxed();
      cluster_wait();
    }
    if (epi) {
      tc_fence_after();
      if (MODE == GC_RESIDUAL) {
        const bool own = grp == rank;
        float* dst = (own ? in + rank * in_pitch : out + (grp - (grp > rank)) * out_pitch) + (w & 15);
        const int rows = own ? M : S;
        tmem_rows(taddr, hf, M, [&](int m, float v) { if (MT < 128 || m < rows) dst[m * 16] = v; });
      } else if (MODE == GC_SWIGLU) {
        const bool own = grp >= glu_g0 && grp < glu_g0 + glu_ng;
        for (int s = 0; s < nseg; ++s) {
          const int slot = seg[s].mat == 0 ? rank : rank + 1;  // gate parts of CTA 0 and 1, up parts of CTA 1 and 2
          float* dst = (own ? in + (slot * glu_ng + grp - glu_g0) * in_pitch
                            : out + (s * (8 - glu_ng) + (grp < glu_g0 ? grp : grp - glu_ng)) * out_pitch) + (w & 15);
          tmem_rows(taddr + (uint32_t)(s * MT + m0), hf, Mr, [&](int m, float v) { dst[m * 16] = v; });
        }
      } else if (PLAIN) {
        // rows of this CTA's block to its place in `in`, all others to `out`; the two halves of the run are added here
        const int own0 = rank * rb, to_out = (int)(out - in);  // (block `rank` of `in` starts at row rank * rb)
        tmem_rows(taddr + (uint32_t)m0, hf, Mr, [&](int m, float v) { in[((unsigned)(m - own0) < (unsigned)rb ? 0 : to_out) + m * 128 + w] = v; }, nseg > 1 ? MT : 0);
      } else {
        // the other CTA's rows to `out`, its own beside the place where the other's part arrives; both [warp][row][32 columns]
        const int mine = (r_rows * 4 + q * r_rows - r_row0) * 32 + lane;
        const int theirs = (int)(out - in) + (q * (M - r_rows) - (rank ? 0 : r_half)) * 32 + lane;
        const int below = rank ? theirs : mine, above = rank ? mine : theirs;      // where the rows below r_half and the others go
        tmem_rows(taddr, hf, M, [&](int m, float v) { in[(m < r_half ? below : above) + m * 32] = v; });
      }
      tc_fence_before();
      fence_smem_async();
      asm volatile("bar.sync %0, 64;" ::"r"(1 + q) : "memory");   // the two warps of a quarter have staged its columns
    }
    if (rd == 0) cluster_wait();                             // every ring of the cluster is free
    if (PLAIN && CS > 1 && epi) {
      asm volatile("bar.sync 6, %0;" ::"n"(GC_EPI) : "memory");   // all columns are staged
      if (warp == 2 && lane < CS && lane != rank) {
        const int rows = min(rb, Mr - lane * rb);
        if (rows > 0)
          bulk_push(dsmem_addr(smem_u32(in + (size_t)rank * rb * 128), (uint32_t)lane), out + (size_t)lane * rb * 128, rows * 512, dsmem_addr(smem_u32(part_full), (uint32_t)lane));
      }
    }
    if (!PLAIN && epi && hf == 0) {
      // the first of a quarter's warps sends its columns
      if (MODE == GC_ROPE) {
        const int n = M - r_rows;                            // (all four warps' blocks lie in the other CTA's `in`)
        if (lane == 0 && n > 0)
          bulk_push(dsmem_addr(smem_u32(in + q * n * 32), (uint32_t)(rank ^ 1)), out + q * n * 32, n * 128, dsmem_addr(smem_u32(part_full), (uint32_t)(rank ^ 1)));
      } else if ((lane & 15) == 0) {
        const int to = MODE == GC_RESIDUAL ? grp : (grp < GLU_FIRST[1] ? 0 : (grp < GLU_FIRST[2] ? 1 : 2));
        if (to != rank) {
          const uint32_t bar = dsmem_addr(smem_u32(part_full), (uint32_t)to), there = dsmem_addr(smem_u32(in), (uint32_t)to);
          if (MODE == GC_RESIDUAL) {
            bulk_push(there + (uint32_t)(rank * in_pitch * 4), out + (grp - (grp > rank)) * out_pitch, S * 64, bar);
          } else {
            const int g0 = GLU_FIRST[to], ng = GLU_FIRST[to + 1] - g0;
            for (int s = 0; s < nseg; ++s) {
              const int slot = seg[s].mat == 0 ? rank : rank + 1;
              bulk_push(there + (uint32_t)((slot * ng + grp - g0) * in_pitch * 4), out + (s * (8 - glu_ng) + (grp < glu_g0 ? grp : grp - glu_ng)) * out_pitch,
                        Mr * 64, bar);
            }
          }
        }
      }
    }
    if (MODE == GC_RESIDUAL && S < M) {                                    // (the same in every CTA of the cluster)
      if (epi) {
        const uint32_t dst = dsmem_addr(smem_u32(in + rank * in_pitch + (w & 15)), (uint32_t)grp);
        tmem_rows(taddr, hf, M, [&](int m, float v) { if (m >= S && grp != rank) dsmem_st(dst + (uint32_t)(m * 64), v); });
        tc_fence_before();
      }
      __syncwarp();
      cluster_sync_all();
    }
    if (epi) {
      asm volatile("bar.sync 5, %0;" ::"n"(GC_EPI) : "memory");   // the own parts, written by the other warps
      mbar_wait(part_full, rd, p.status, 34);
    }
    __syncwarp();
    if (rd == ROUNDS - 1) cluster_arrive_relaxed();          // this CTA reads nobody's shared memory but its own from here on

    if (epi) {
      if (MODE == GC_RESIDUAL) {
        // the eight parts of columns [16 rank, +16) in rank order, the residual stream in place and the sums of squares
#pragma unroll
        for (int k = 0; k < X_PER; ++k) {
          const int it = e + GC_EPI * k, m = it >> 2, c4 = it & 3;
          float ss = 0.f;
          if (m < M) {
            float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
            const float* src = in + m * 16 + c4 * 4;
#pragma unroll
            for (int rr = 0; rr < CS; ++rr) add4(acc, *reinterpret_cast<const float4*>(src + rr * in_pitch));
            add4(xo[k], acc);
            if (x_on[k]) {
              ss = sum_sq<MT>(xo[k]);
              *reinterpret_cast<float4*>(p.x + (size_t)m * p.N + t * 128 + rank * 16 + c4 * 4) = xo[k];
            }
          }
          if (p.ss_part) {
            // the four column groups of a row sit in four neighbouring lanes
            ss += __shfl_xor_sync(0xffffffffu, ss, 1);
            ss += __shfl_xor_sync(0xffffffffu, ss, 2);
            if (c4 == 0 && m < M) p.ss_part[(size_t)m * (((p.N + 127) >> 7) * CS) + t * CS + rank] = ss;
          }
        }
      } else if (PLAIN) {
        // a warp has a row: 128 columns of it in every part, added in rank order
        const int rows = min(rb, Mr - rank * rb), n0 = t * 128 + lane * 4;
        const bool vec = (p.ldy & 3) == 0 && (reinterpret_cast<uintptr_t>(p.y) & 15) == 0 && n0 + 4 <= p.N;
        const int tiles_n = (p.N + 127) >> 7;
        constexpr int U = MT > 64 ? 2 : 4, STEP = GC_EPI / 32; // rows in flight a warp
        for (int i0 = warp - 2; i0 < rows; i0 += U * STEP) {
          float4 a[U];
#pragma unroll
          for (int k = 0; k < U; ++k) a[k] = *reinterpret_cast<const float4*>(in + min(i0 + k * STEP, rows - 1) * 128 + lane * 4);
          for (int r = 1; r < CS; ++r)
#pragma unroll
            for (int k = 0; k < U; ++k) add4(a[k], *reinterpret_cast<const float4*>(in + ((size_t)r * rb + min(i0 + k * STEP, rows - 1)) * 128 + lane * 4));
#pragma unroll
          for (int k = 0; k < U; ++k) {
            const int i = i0 + k * STEP, m = m0 + rank * rb + i;
            if (i >= rows) continue;
            const float v[4] = {a[k].x, a[k].y, a[k].z, a[k].w};
            if (p.y) {
              float* dst = p.y + (size_t)m * p.ldy + n0;
              if (vec) *reinterpret_cast<float4*>(dst) = a[k];
              else
                for (int j = 0; j < 4; ++j) if (n0 + j < p.N) dst[j] = v[j];
            }
            if (p.best_val) {
              float bv = -INFINITY;
              int bi = 0x7fffffff;
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (n0 + j < p.N && better(v[j], n0 + j, bv, bi)) { bv = v[j]; bi = n0 + j; }
              warp_argmax(bv, bi);
              if (lane == 0) { p.best_val[(size_t)m * tiles_n + t] = bv; p.best_idx[(size_t)m * tiles_n + t] = bi; }
            }
          }
        }
      } else if (MODE == GC_SWIGLU) {
        const int gpr = glu_ng * 4;                            // groups of four columns per row: 12 or 8
        constexpr int PER = (RT * 12 + GC_EPI - 1) / GC_EPI;
        const int part = glu_ng * in_pitch;
        float4 ga[PER], ua[PER];
#pragma unroll
        for (int k = 0; k < PER; ++k) {
          const int it = min(e + GC_EPI * k, Mr * gpr - 1), m = glu_ng == 3 ? it / 12 : it >> 3, w4 = it - m * gpr;
          const float* src = in + (w4 >> 2) * in_pitch + m * 16 + (w4 & 3) * 4;
          ga[k] = *reinterpret_cast<const float4*>(src);
          ua[k] = *reinterpret_cast<const float4*>(src + 2 * part);
          add4(ga[k], *reinterpret_cast<const float4*>(src + part));
          add4(ua[k], *reinterpret_cast<const float4*>(src + 3 * part));
        }
#pragma unroll
        for (int k = 0; k < PER; ++k) {
          const int it = e + GC_EPI * k, m = glu_ng == 3 ? it / 12 : it >> 3, w4 = it - m * gpr;
          const int col = t * 128 + glu_g0 * 16 + 4 * w4;
          uint2 o;
          o.x = pack_bf16x2(silu_f(ga[k].x) * ua[k].x, silu_f(ga[k].y) * ua[k].y);
          o.y = pack_bf16x2(silu_f(ga[k].z) * ua[k].z, silu_f(ga[k].w) * ua[k].w);
          if (m < Mr && col < p.N) *reinterpret_cast<uint2*>(p.act + (size_t)(m0 + m) * p.N + col) = o;
        }
      } else {
        // the tile holds 128 / D whole heads; an item is (row, group of four rotation pairs): columns [lo, lo + 4) and
        // [lo + D/2, lo + D/2 + 4) of one head
        const int half = p.g.head_dim >> 1;
        const float* first = rank ? in : in + (size_t)r_rows * 128;         // CTA 0's part, then CTA 1's
        const float* second = rank ? in + (size_t)r_rows * 128 : in;
#pragma unroll
        for (int k = 0; k < R_PER; ++k) {
          if (!r_on[k]) continue;
          const int lo = r_lo_c[k] & 0xffff, hi = lo + half;
          const int o_lo = ((lo >> 5) * r_rows + r_mrow[k]) * 32 + (lo & 31), o_hi = ((hi >> 5) * r_rows + r_mrow[k]) * 32 + (hi & 31);
          float4 a = *reinterpret_cast<const float4*>(first + o_lo), c = *reinterpret_cast<const float4*>(first + o_hi);
          add4(a, *reinterpret_cast<const float4*>(second + o_lo));
          add4(c, *reinterpret_cast<const float4*>(second + o_hi));
          const float4 t01 = r_cs01[k], t23 = r_cs23[k];
          uint2 lo_o, hi_o;
          if (rope_mat < 2) {
            lo_o.x = pack_bf16x2(rotate_lo(a.x, c.x, t01.x, t01.y), rotate_lo(a.y, c.y, t01.z, t01.w));
            lo_o.y = pack_bf16x2(rotate_lo(a.z, c.z, t23.x, t23.y), rotate_lo(a.w, c.w, t23.z, t23.w));
            hi_o.x = pack_bf16x2(rotate_hi<MT>(a.x, c.x, t01.x, t01.y), rotate_hi<MT>(a.y, c.y, t01.z, t01.w));
            hi_o.y = pack_bf16x2(rotate_hi<MT>(a.z, c.z, t23.x, t23.y), rotate_hi<MT>(a.w, c.w, t23.z, t23.w));
          } else {
            lo_o.x = pack_bf16x2(a.x, a.y); lo_o.y = pack_bf16x2(a.z, a.w);
            hi_o.x = pack_bf16x2(c.x, c.y); hi_o.y = pack_bf16x2(c.z, c.w);
          }
          const int up = rope_mat == 0 ? half : (r_lo_c[k] >> 16);
          *reinterpret_cast<uint2*>(r_dst[k]) = lo_o;
          *reinterpret_cast<uint2*>(r_dst[k] + up) = hi_o;
        }
      }
    }
  }
  // nobody leaves while a copy out of its shared memory may still be on its way
  __syncwarp();
  cluster_wait();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, TMEM_COLS);
}

}  // namespace spec
