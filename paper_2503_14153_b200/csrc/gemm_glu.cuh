// Gate and up projections with their SwiGLU for passes of 65 to 128 rows over a narrow model: act = bf16(SiLU(x Wg^T) * (x Wu^T)).
//
// The weight streamer cuts the K chunks of every 128-row weight tile of such a launch into the same `cs` runs, each summed on its own and
// added in order, and a second kernel takes the partial sums out of memory again. Here the CTAs of a (gate tile, up tile) pair are a
// cluster: CTA r sums run r of both tiles into two accumulators, an activation tile serving both, and finishes a block of rows with the
// others' parts, which arrive in its shared memory. The sums are the streamer's, bit for bit: same runs, added in the same order.
// At most one CTA an SM; the whole run's weights are asked for before the dependency wait as far as the ring of four 48 KB
// stages goes. What bounds it is the chain activation tile -> MMAs -> exchange (see gemm_cluster.cuh) -> finish.
// Six layers of d_model 1024, 2 x 22 tiles in clusters of 6, 69 rows: 13.0 -> 8.9 us a layer, a step 312 -> 282; 7 of the 8.9 us are the wait for the
// kernel before, the first activation tile, the exchange and the finish.
//
// Epilogue: sixteen warps, in every SM quarter one for the even and one for the odd 16-row groups of each accumulator. More than GLU_ROUND rows
// go in two rounds, because shared memory does not hold all of them staged and arriving at once.
#pragma once
#include <cuda.h>

#include "common.cuh"
#include "gemm_cluster.cuh"
#include "gemm_stream.cuh"

namespace spec {

constexpr int GLU_EPI = 512, GLU_THREADS = 64 + GLU_EPI;     // producer, MMA issuer, sixteen epilogue warps
constexpr int GLU_MAX_CLUSTER = 8, GLU_MAX_STAGES = 4, GLU_STAGE_BYTES = 3 * 16384, GLU_ROUND = 96;

struct GluGemmParams {
  int M, KC, N;                 // activation rows (65..128), K / 64, columns of one matrix
  int stages;
  const uint8_t* packed[2];     // pre-tiled gate and up images or nullptr -> tensor maps a[0], a[1]
  bf16* act;                    // [M][N]
  int* status;
  unsigned long long* trace;
};

__host__ __device__ inline int glu_round_rows(int M) { return M <= GLU_ROUND ? M : (M + 31) / 32 * 16; }
// Shared memory of a launch: the ring, or what the exchange puts in its place (a round's rows of both matrices staged, and a block of them from every
// CTA), whichever is larger.
inline int glu_smem_bytes(int M, int cs, int stages) {
  const int rr = glu_round_rows(M), rb = (rr + cs - 1) / cs;
  const int exchange = (rr + cs * rb) * 1024, ring = stages * GLU_STAGE_BYTES;
  return (exchange > ring ? exchange : ring) + 1024 /*alignment slack*/ + 256 /*barriers*/;
}

__global__ void __launch_bounds__(GLU_THREADS, 1)
gemm_glu(const __grid_constant__ StreamTmaps tm, const GluGemmParams p) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* bar_area = smem_raw + (((raw + 127u) & ~127u) - raw);       // 128 bytes, then the ring on the next 1024-byte boundary
  uint8_t* tiles = smem_raw + (((raw + 128u + 127u + 1023u) & ~1023u) - raw);
  uint64_t* full = reinterpret_cast<uint64_t*>(bar_area);
  uint64_t* empty = full + GLU_MAX_STAGES;
  uint64_t* acc_full = full + 2 * GLU_MAX_STAGES;
  uint64_t* part_full = acc_full + 1;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(part_full + 1);
  float* staging = reinterpret_cast<float*>(tiles);

  KTrace kt(p.trace);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int cs = (int)cluster_nctarank(), rank = (int)cluster_ctarank();
  const int t = blockIdx.x / cs, KC = p.KC, M = p.M, stages = p.stages;
  const int k0 = rank * KC / cs, n_units = (rank + 1) * KC / cs - k0;
  const int mma_n = (M + 15) & ~15;
  const uint32_t stage_tx = 2 * 16384 + mma_n * 128;
  const int rr = glu_round_rows(M), rounds = rr < M ? 2 : 1, rb = (rr + cs - 1) / cs;
  float* out = staging;                                      // [matrix][row of the round][128 columns]
  float* in = staging + 2 * rr * 128;                        // [CTA][matrix][row of this CTA's block][128 columns]
  auto block_rows = [&](int r, int rows) { return max(0, min(rb, rows - r * rb)); };
  auto in_bytes = [&](int rows) -> uint32_t { return (uint32_t)((cs - 1) * block_rows(rank, rows) * 1024); };

  if (threadIdx.x == 0) {
    for (int i = 0; i < GLU_MAX_STAGES; ++i) { mbar_init(&full[i], 1); mbar_init(&empty[i], 1); }
    mbar_init(acc_full, 1);
    mbar_init(part_full, 1);
    mbar_fence_init();
    mbar_expect_tx(part_full, in_bytes(rr));                 // (the first copy comes after the first cluster barrier)
    for (int i = 0; i < 2; ++i) if (!p.packed[i]) tma_prefetch_desc(&tm.a[i]);
    tma_prefetch_desc(&tm.b);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, 256); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  pdl_launch_dependents();                                   // (this CTA has its tensor memory)
  const uint32_t tmem_base = *tmem_slot;

  if (warp == 0) {
    if (elect_one()) {
      // ---- producer: weights before the dependency wait, activation tiles after it ----
      const uint64_t wpol = l2_policy_evict_first();
      const int n_pre = n_units < stages ? n_units : stages;
      auto load_w = [&](uint8_t* dst, int kc, uint64_t* bar) {
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (p.packed[i]) bulk_load_1d_hint(dst + i * 16384, p.packed[i] + ((size_t)t * KC + kc) * 16384, 16384, bar, wpol);
          else tma_load_2d_hint(dst + i * 16384, &tm.a[i], kc * 64, t * 128, bar, wpol);
        }
      };
      for (int i = 0; i < n_pre; ++i) {
        mbar_expect_tx(&full[i], stage_tx);
        load_w(tiles + i * GLU_STAGE_BYTES, k0 + i, &full[i]);
      }
      pdl_wait();
      for (int i = 0; i < n_pre; ++i) tma_load_2d(tiles + i * GLU_STAGE_BYTES + 32768, &tm.b, (k0 + i) * 64, 0, &full[i]);
      bool ok = true;
      int issued = n_pre, st = 0;
      uint32_t ph = 0;
      for (; issued < n_units; ++issued) {
        if (!mbar_wait(&empty[st], ph, p.status, 70)) { ok = false; break; }
        uint8_t* dst = tiles + st * GLU_STAGE_BYTES;
        mbar_expect_tx(&full[st], stage_tx);
        load_w(dst, k0 + issued, &full[st]);
        tma_load_2d(dst + 32768, &tm.b, (k0 + issued) * 64, 0, &full[st]);
        if (++st == stages) { st = 0; ph ^= 1; }
      }
      if (!ok) {
        // give the copies already in flight a bounded time to land
        for (int i = issued > stages ? issued - stages : 0; i < issued; ++i)
          mbar_wait(&full[i % stages], (i / stages) & 1, p.status, 73);
      }
    }
  } else if (warp == 1) {
    if (elect_one()) {
      // ---- MMA issuer: gate sums in tensor-memory columns [0, 128), up sums in [128, 256) ----
      const uint32_t idesc = make_idesc_bf16(128, mma_n);
      const uint64_t desc0 = make_kmajor_sw128_desc(smem_u32(tiles));
      bool ok = true;
      int st = 0;
      uint32_t ph = 0;
      for (int v = 0; v < n_units; ++v) {
        if (!mbar_wait(&full[st], ph, p.status, 71)) { ok = false; break; }
        if (v == 0) trace_mark_min(p.trace, 2);
        tc_fence_after();
        const uint64_t g = desc0 + (uint64_t)(st * (GLU_STAGE_BYTES >> 4)), u = g + (16384 >> 4), b = u + (16384 >> 4);
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          tc_mma_f16(tmem_base, g + 2 * k, b + 2 * k, idesc, (v > 0 || k > 0) ? 1u : 0u);
          tc_mma_f16(tmem_base + 128, u + 2 * k, b + 2 * k, idesc, (v > 0 || k > 0) ? 1u : 0u);
        }
        if (v + stages < n_units) tc_commit(&empty[st]);     // (a stage that is not filled again needs no announcement)
        if (++st == stages) { st = 0; ph ^= 1; }
      }
      if (ok) tc_commit(acc_full);
      trace_mark_max(p.trace, 3);
    }
  } else {
    pdl_wait();
    mbar_wait(acc_full, 0, p.status, 72);
  }

  // ---- exchange: this CTA's MMAs are complete, its ring is free (see gemm_cluster) ----
  const bool epi = warp >= 2;
  const int e = (int)threadIdx.x - 64, q = warp & 3, set = (warp - 2) >> 2, mat = set & 1, hf = set >> 1;
  const int w = q * 32 + lane;                               // its tensor-memory lane = weight row of the tile
  const uint32_t taddr = tmem_base + ((uint32_t)(q * 32) << 16) + (uint32_t)(mat * 128);
#pragma unroll 1
  for (int rd = 0; rd < rounds; ++rd) {
    const int m0 = rd * rr, Mr = min(rr, M - m0);            // rows of this round
    __syncwarp();
    if (rd == 0) {
      if (warp == 0) cluster_arrive();                       // (its first thread has set up the barrier the copies complete on)
      else cluster_arrive_relaxed();
    } else {
      // everybody has received the first round (so `out` may be overwritten) and is through with it (`in`)
      if (epi) {
        asm volatile("bar.sync 5, %0;" ::"n"(GLU_EPI) : "memory");
        if (e == 0) mbar_expect_tx(part_full, in_bytes(Mr));
        __syncwarp();
      }
      if (warp == 2) cluster_arrive();
      else cluster_arrive_relaxed();
      cluster_wait();
    }
    if (epi) {
      tc_fence_after();
      float* dst = out + mat * rr * 128 + w;
      tmem_rows(taddr + (uint32_t)m0, hf, Mr, [&](int m, float v) { dst[m * 128] = v; });
      tc_fence_before();
      fence_smem_async();
      asm volatile("bar.sync 5, %0;" ::"n"(GLU_EPI) : "memory");       // all columns are staged
    }
    if (rd == 0) cluster_wait();                             // every ring of the cluster is free
    if (warp == 2 && lane < 2 * cs && (lane >> 1) != rank) {
      const int to = lane >> 1, i = lane & 1, rows = block_rows(to, Mr);
      if (rows > 0)
        bulk_push(dsmem_addr(smem_u32(in + (size_t)(2 * rank + i) * rb * 128), (uint32_t)to), out + (size_t)(i * rr + to * rb) * 128, rows * 512,
                  dsmem_addr(smem_u32(part_full), (uint32_t)to));
    }
    if (epi) mbar_wait(part_full, rd, p.status, 74);
    __syncwarp();
    if (rd == rounds - 1) cluster_arrive_relaxed();          // this CTA reads nobody's shared memory but its own from here on
    if (epi) {
      // a warp has a row: 128 columns of it in every part, added in the order of the runs
      const int rows = block_rows(rank, Mr), col = t * 128 + lane * 4;
      for (int i = warp - 2; i < rows; i += GLU_EPI / 32) {
        const float* own = out + (size_t)(rank * rb + i) * 128 + lane * 4;
        const float* src = in + i * 128 + lane * 4;
        float4 g = make_float4(0.f, 0.f, 0.f, 0.f), u = g;
        for (int r = 0; r < cs; ++r) {
          const float4 gr = *reinterpret_cast<const float4*>(r == rank ? own : src + (size_t)(2 * r) * rb * 128);
          const float4 ur = *reinterpret_cast<const float4*>(r == rank ? own + rr * 128 : src + (size_t)(2 * r + 1) * rb * 128);
          if (r == 0) { g = gr; u = ur; } else { add4(g, gr); add4(u, ur); }
        }
        uint2 o;
        o.x = pack_bf16x2(silu_f(g.x) * u.x, silu_f(g.y) * u.y);
        o.y = pack_bf16x2(silu_f(g.z) * u.z, silu_f(g.w) * u.w);
        if (col < p.N) *reinterpret_cast<uint2*>(p.act + (size_t)(m0 + rank * rb + i) * p.N + col) = o;
      }
    }
  }
  // nobody leaves while a copy out of its shared memory may still be on its way
  __syncwarp();
  cluster_wait();
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem_base, 256);
}

}  // namespace spec
