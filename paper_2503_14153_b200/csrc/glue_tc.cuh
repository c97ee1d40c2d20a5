// Glue kernels of the bf16 verification forward: they consume the float32 partial sums the
// weight-streaming GEMM leaves (adding a tile's slots in CTA order), apply the element-wise
// step of the layer (residual + RMSNorm, RoPE + cache store, SwiGLU) and write the bf16
// operand of the next GEMM. All are vectorised (16-byte accesses), take part in programmatic
// dependent launch (trigger at entry, wait before the first dependent access) and keep the
// rounding points of the reference path: float32 until the operand is rounded to bf16.
#pragma once
#include "common.cuh"
#include "gemm_cluster.cuh"
#include "gemm_stream.cuh"
#include "kernels_simple.cuh"

namespace spec {

// Partial sums of one GEMM launch: part[slot][m][ld], padded column space (tile nt = columns
// [128 nt, 128 nt + 128)).
struct PartView {
  const float* part;
  size_t slot_stride;
  int ld;
  SegMap seg;                  // how the GEMM dealt its units: gives the slots of a tile
  int mt_shift;                // log2 of the activation rows per tile
  int single;                  // 1: every tile is one finished slot (gemm_pair's plain sums, the float32 logits): read it directly
};

constexpr int PV_UNROLL = 12;

// Sum over the slots of the tile that holds padded columns [colp, colp+4) of row m.
__device__ __forceinline__ float4 part_sum4(const PartView& pv, int m, int colp) {
  const int ns = pv.seg.nseg((colp >> 7) * pv.seg.m_tiles + (m >> pv.mt_shift));
  const float* src = pv.part + (size_t)m * pv.ld + colp;
  float4 v[PV_UNROLL];
#pragma unroll
  for (int s = 0; s < PV_UNROLL; ++s)
    v[s] = (s < ns) ? __ldcg(reinterpret_cast<const float4*>(src + (size_t)s * pv.slot_stride)) : make_float4(0.f, 0.f, 0.f, 0.f);
  float4 a = v[0];
#pragma unroll
  for (int s = 1; s < PV_UNROLL; ++s)
    if (s < ns) { a.x += v[s].x; a.y += v[s].y; a.z += v[s].z; a.w += v[s].w; }
  for (int s = PV_UNROLL; s < ns; ++s) {
    float4 w = __ldcg(reinterpret_cast<const float4*>(src + (size_t)s * pv.slot_stride));
    a.x += w.x; a.y += w.y; a.z += w.z; a.w += w.w;
  }
  return a;
}

// The same for a view of finished sums (pv.single).
__device__ __forceinline__ float4 part_one4(const PartView& pv, int m, int colp) {
  return __ldcg(reinterpret_cast<const float4*>(pv.part + (size_t)m * pv.ld + colp));
}

__device__ __forceinline__ uint2 pack4_bf16(float a, float b, float c, float d) {
  __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
  uint2 r;
  r.x = *reinterpret_cast<uint32_t*>(&lo);
  r.y = *reinterpret_cast<uint32_t*>(&hi);
  return r;
}

// ------------------------------------------------------------------ residual + RMSNorm
// x[m] += sum of the partial slots (when pv.part != nullptr); u[m] = bf16(x / rms(x) * g);
// optionally the unrounded normed row goes to hid. A cluster of NORM_CLUSTER CTAs (on
// neighbouring SMs) shares a row, each with its own slice of the columns, so that one SM does
// not have to pull a whole row's partial sums through its load queues; the slices' sums of
// squares are exchanged through distributed shared memory and added in rank order. Every
// thread issues all its loads at once (one trip to L2) and keeps its values in registers; the
// gains do not depend on the previous kernel and are fetched before the dependency wait.
// d % 4 == 0; grid (rows, NORM_CLUSTER).
constexpr int NORM_THREADS = 512;
constexpr int NORM_CLUSTER = 2;
constexpr int NORM_CACHE = 2;   // float4 values a thread keeps between the two passes

__global__ void __cluster_dims__(1, NORM_CLUSTER, 1) __launch_bounds__(NORM_THREADS)
norm_reduce_tc(float* __restrict__ x, const PartView pv, const float* __restrict__ gain, float eps,
               bf16* __restrict__ u, float* __restrict__ hid, int d, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  const int m = blockIdx.x, rank = blockIdx.y;
  float* xr = x + (size_t)m * d;
  const int n4 = d >> 2;
  const int per = (n4 + NORM_CLUSTER - 1) / NORM_CLUSTER;
  const int c_lo = rank * per, c_hi = min(n4, c_lo + per);
  float4 gk[NORM_CACHE];
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) {
    const int c4 = c_lo + threadIdx.x + k * NORM_THREADS;
    gk[k] = c4 < c_hi ? *reinterpret_cast<const float4*>(gain + c4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  float4 keep[NORM_CACHE];
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) {
    const int c4 = c_lo + threadIdx.x + k * NORM_THREADS;
    if (c4 < c_hi) {
      float4 v = *reinterpret_cast<const float4*>(xr + c4 * 4);
      if (pv.part) {
        const float4 a = part_sum4(pv, m, c4 * 4);
        v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
        *reinterpret_cast<float4*>(xr + c4 * 4) = v;
      }
      keep[k] = v;
      ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    }
  }
  for (int c4 = c_lo + threadIdx.x + NORM_CACHE * NORM_THREADS; c4 < c_hi; c4 += NORM_THREADS) {
    float4 v = *reinterpret_cast<const float4*>(xr + c4 * 4);
    if (pv.part) {
      const float4 a = part_sum4(pv, m, c4 * 4);
      v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
      *reinterpret_cast<float4*>(xr + c4 * 4) = v;
    }
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
  __shared__ float red[32];
  __shared__ float slice_ss;
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < (NORM_THREADS >> 5); ++w) t += red[w];
    slice_ss = t;
  }
  // exchange the slices' sums through distributed shared memory (cluster barrier: release / acquire)
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  float tot = 0.f;
#pragma unroll
  for (int r = 0; r < NORM_CLUSTER; ++r) {
    uint32_t remote;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(remote) : "r"(smem_u32(&slice_ss)), "r"(r));
    float v;
    asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(remote) : "memory");
    tot += v;                                           // rank order: the same sum in every CTA
  }
  // nobody may leave (and give up its shared memory) before every CTA has read it
  asm volatile("barrier.cluster.arrive.release.aligned;\n\tbarrier.cluster.wait.acquire.aligned;" ::: "memory");
  const float inv = rsqrtf(tot / (float)d + eps);
  auto emit = [&](int c4, const float4& v, const float4& g) {
    const float4 o = make_float4(v.x * inv * g.x, v.y * inv * g.y, v.z * inv * g.z, v.w * inv * g.w);
    *reinterpret_cast<uint2*>(u + (size_t)m * d + c4 * 4) = pack4_bf16(o.x, o.y, o.z, o.w);
    if (hid) *reinterpret_cast<float4*>(hid + (size_t)m * d + c4 * 4) = o;
  };
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) {
    const int c4 = c_lo + threadIdx.x + k * NORM_THREADS;
    if (c4 < c_hi) emit(c4, keep[k], gk[k]);
  }
  for (int c4 = c_lo + threadIdx.x + NORM_CACHE * NORM_THREADS; c4 < c_hi; c4 += NORM_THREADS)
    emit(c4, *reinterpret_cast<const float4*>(xr + c4 * 4), *reinterpret_cast<const float4*>(gain + c4 * 4));
}

// RMSNorm of rows whose sums of squares already exist in pieces (the residual cluster epilogue leaves
// ss_part[m][n_ss], the sum of squares of every 16-column piece of row m): u[m] = bf16(x / rms(x) * g).
// gridDim.y plain CTAs share a row, each adding all the row's pieces itself in a fixed order (the same sum in
// every CTA), so nothing is exchanged between CTAs. One trip to L2 per thread.
__global__ void __launch_bounds__(NORM_THREADS)
norm_scaled_tc(const float* __restrict__ x, const float* __restrict__ ss_part, int n_ss, const float* __restrict__ gain,
               float eps, bf16* __restrict__ u, float* __restrict__ hid, int d, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  const int m = blockIdx.x;
  const float* xr = x + (size_t)m * d;
  const int n4 = d >> 2;
  const int per = (n4 + (int)gridDim.y - 1) / (int)gridDim.y;
  const int c_lo = blockIdx.y * per, c_hi = min(n4, c_lo + per);
  float4 gk[NORM_CACHE];
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) {
    const int c4 = c_lo + threadIdx.x + k * NORM_THREADS;
    gk[k] = c4 < c_hi ? *reinterpret_cast<const float4*>(gain + c4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  float4 keep[NORM_CACHE];
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) {
    const int c4 = c_lo + threadIdx.x + k * NORM_THREADS;
    keep[k] = c4 < c_hi ? *reinterpret_cast<const float4*>(xr + c4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  float ss = 0.f;
  for (int i = threadIdx.x; i < n_ss; i += NORM_THREADS) ss += __ldcg(ss_part + (size_t)m * n_ss + i);
  __shared__ float red[NORM_THREADS / 32];
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < NORM_THREADS / 32; ++w) tot += red[w];
  const float inv = rsqrtf(tot / (float)d + eps);
  auto emit = [&](int c4, const float4& v, const float4& g) {
    const float4 o = make_float4(v.x * inv * g.x, v.y * inv * g.y, v.z * inv * g.z, v.w * inv * g.w);
    *reinterpret_cast<uint2*>(u + (size_t)m * d + c4 * 4) = pack4_bf16(o.x, o.y, o.z, o.w);
    if (hid) *reinterpret_cast<float4*>(hid + (size_t)m * d + c4 * 4) = o;
  };
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) {
    const int c4 = c_lo + threadIdx.x + k * NORM_THREADS;
    if (c4 < c_hi) emit(c4, keep[k], gk[k]);
  }
  for (int c4 = c_lo + threadIdx.x + NORM_CACHE * NORM_THREADS; c4 < c_hi; c4 += NORM_THREADS)
    emit(c4, *reinterpret_cast<const float4*>(xr + c4 * 4), *reinterpret_cast<const float4*>(gain + c4 * 4));
}

// The same sums where no projection has left the pieces' (a prompt of two chunks in one pass): a CTA a row makes them out of x, as the residual epilogue
// of 128 rows does, and adds them as norm_scaled_tc does. d % 16 == 0, at most NORM_PIECES pieces.
constexpr int NORM_PIECES = 1024;
__global__ void __launch_bounds__(NORM_THREADS)
norm_pieces_tc(const float* __restrict__ x, const float* __restrict__ gain, float eps, bf16* __restrict__ u, int d, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  const int m = blockIdx.x, n4 = d >> 2;
  const float* xr = x + (size_t)m * d;
  float4 gk[NORM_CACHE], keep[NORM_CACHE];
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) {
    const int c4 = threadIdx.x + k * NORM_THREADS;
    gk[k] = c4 < n4 ? *reinterpret_cast<const float4*>(gain + c4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  __shared__ float pieces[NORM_PIECES], red[NORM_THREADS / 32];
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) {
    const int c4 = threadIdx.x + k * NORM_THREADS;
    keep[k] = c4 < n4 ? *reinterpret_cast<const float4*>(xr + c4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  // (the four column groups of a piece sit in four neighbouring lanes; n4 is a multiple of four)
  auto piece = [&](int c4, const float4& v) {
    float ss = sum_sq<128>(v);
    ss += __shfl_xor_sync(0xffffffffu, ss, 1);
    ss += __shfl_xor_sync(0xffffffffu, ss, 2);
    if ((threadIdx.x & 3) == 0 && c4 < n4) pieces[c4 >> 2] = ss;
  };
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) piece(threadIdx.x + k * NORM_THREADS, keep[k]);
  for (int c0 = NORM_CACHE * NORM_THREADS; c0 < n4; c0 += NORM_THREADS) {
    const int c4 = c0 + threadIdx.x;
    piece(c4, c4 < n4 ? *reinterpret_cast<const float4*>(xr + c4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f));
  }
  __syncthreads();
  float ss = 0.f;
  for (int i = threadIdx.x; i < (n4 >> 2); i += NORM_THREADS) ss += pieces[i];
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  float tot = 0.f;
#pragma unroll
  for (int w = 0; w < NORM_THREADS / 32; ++w) tot += red[w];
  const float inv = rsqrtf(tot / (float)d + eps);
  auto emit = [&](int c4, const float4& v, const float4& g) {
    *reinterpret_cast<uint2*>(u + (size_t)m * d + c4 * 4) = pack4_bf16(v.x * inv * g.x, v.y * inv * g.y, v.z * inv * g.z, v.w * inv * g.w);
  };
#pragma unroll
  for (int k = 0; k < NORM_CACHE; ++k) {
    const int c4 = threadIdx.x + k * NORM_THREADS;
    if (c4 < n4) emit(c4, keep[k], gk[k]);
  }
  for (int c4 = threadIdx.x + NORM_CACHE * NORM_THREADS; c4 < n4; c4 += NORM_THREADS)
    emit(c4, *reinterpret_cast<const float4*>(xr + c4 * 4), *reinterpret_cast<const float4*>(gain + c4 * 4));
}

// The same operation for passes of many rows (batched verification, prompt processing): one CTA of
// NORMW_THREADS per row, no cluster. With hundreds of rows the kernel is bound by bandwidth, not by the
// latency of one row, so what counts is loads in flight: a thread fetches all its pieces of x and of the
// partial sums before it uses the first (NORMW_CACHE float4 each; rows longer than that loop), and, where no sums are to be added (PARTS false: the
// projections of many rows update x themselves), 40 registers instead of 101 let five CTAs share an SM (1024 rows of 4096: 9.9 -> 7.3 us, 2048: 14.0 -> 12.1; 896 of 1024: 5.7 -> 4.6)
constexpr int NORMW_THREADS = 256;
constexpr int NORMW_CACHE = 4;

template <bool PARTS>
__global__ void __launch_bounds__(NORMW_THREADS, PARTS ? 1 : 5)
norm_rows_wide(float* __restrict__ x, const PartView pv, const float* __restrict__ gain, float eps,
               bf16* __restrict__ u, float* __restrict__ hid, int d, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  const int m = blockIdx.x;
  float* xr = x + (size_t)m * d;
  const int n4 = d >> 2;
  float4 gk[NORMW_CACHE];
#pragma unroll
  for (int k = 0; k < NORMW_CACHE; ++k) {
    const int c4 = threadIdx.x + k * NORMW_THREADS;
    gk[k] = c4 < n4 ? *reinterpret_cast<const float4*>(gain + c4 * 4) : make_float4(0.f, 0.f, 0.f, 0.f);
  }
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  float4 keep[NORMW_CACHE], add[NORMW_CACHE];
#pragma unroll
  for (int k = 0; k < NORMW_CACHE; ++k) {
    const int c4 = threadIdx.x + k * NORMW_THREADS;
    keep[k] = add[k] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (c4 < n4) {
      keep[k] = *reinterpret_cast<const float4*>(xr + c4 * 4);
      if (PARTS && pv.part) add[k] = part_sum4(pv, m, c4 * 4);
    }
  }
  float ss = 0.f;
#pragma unroll
  for (int k = 0; k < NORMW_CACHE; ++k) {
    const int c4 = threadIdx.x + k * NORMW_THREADS;
    if (c4 < n4) {
      float4& v = keep[k];
      if (PARTS && pv.part) {
        v.x += add[k].x; v.y += add[k].y; v.z += add[k].z; v.w += add[k].w;
        *reinterpret_cast<float4*>(xr + c4 * 4) = v;
      }
      ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
    }
  }
  for (int c4 = threadIdx.x + NORMW_CACHE * NORMW_THREADS; c4 < n4; c4 += NORMW_THREADS) {
    float4 v = *reinterpret_cast<const float4*>(xr + c4 * 4);
    if (PARTS && pv.part) {
      const float4 a = part_sum4(pv, m, c4 * 4);
      v.x += a.x; v.y += a.y; v.z += a.z; v.w += a.w;
      *reinterpret_cast<float4*>(xr + c4 * 4) = v;
    }
    ss += v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w;
  }
  __shared__ float red[NORMW_THREADS / 32];
  __shared__ float row_ss;
  ss = warp_sum(ss);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = ss;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
#pragma unroll
    for (int w = 0; w < NORMW_THREADS / 32; ++w) t += red[w];
    row_ss = t;
  }
  __syncthreads();
  const float inv = rsqrtf(row_ss / (float)d + eps);
  auto emit = [&](int c4, const float4& v, const float4& g) {
    const float4 o = make_float4(v.x * inv * g.x, v.y * inv * g.y, v.z * inv * g.z, v.w * inv * g.w);
    *reinterpret_cast<uint2*>(u + (size_t)m * d + c4 * 4) = pack4_bf16(o.x, o.y, o.z, o.w);
    if (hid) *reinterpret_cast<float4*>(hid + (size_t)m * d + c4 * 4) = o;
  };
#pragma unroll
  for (int k = 0; k < NORMW_CACHE; ++k) {
    const int c4 = threadIdx.x + k * NORMW_THREADS;
    if (c4 < n4) emit(c4, keep[k], gk[k]);
  }
  for (int c4 = threadIdx.x + NORMW_CACHE * NORMW_THREADS; c4 < n4; c4 += NORMW_THREADS)
    emit(c4, *reinterpret_cast<const float4*>(xr + c4 * 4), *reinterpret_cast<const float4*>(gain + c4 * 4));
}

// ------------------------------------------------------------------ RoPE + cache store
// Sums the QKV partial slots, rotates q and k (rotate-half pairs (e, e + D/2), table
// cs[pos][e] = (cos, sin)), writes q as bf16 [M][H*D] and k, v as bf16 into the paged cache at
// the row's slot. qp0 / kp0 / vp0: first padded column of the q / k / v matrix in the partials.
// gridDim.y CTAs share a row; D % 8 == 0.
__global__ void __launch_bounds__(256)
rope_store_tc(const PartView pv, int qp0, int kp0, int vp0, Rows rows, const float2* __restrict__ cs,
              bf16* __restrict__ q, bf16* __restrict__ pool, KVGeom g, const int* __restrict__ page_table,
              int layer, int H, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  const int m = blockIdx.x, b = m / rows.R, i = m % rows.R;
  const int D = g.head_dim, half = D >> 1, Hkv = g.n_kv_heads;
  const int q4 = half >> 2;                       // float4 groups per half head
  const int n_rot = (H + Hkv) * q4, n_v = Hkv * (D >> 2);
  const int tid = blockIdx.y * blockDim.x + threadIdx.x, nthr = gridDim.y * blockDim.x;
  // row bookkeeping and partial sums are independent loads: issue them together
  const int cnt = rows.cnt[b], pos = rows.pos[m], slot = rows.slot[m];
  // item -> first padded column of its group of four (rotated items also take the group half a head further)
  auto item_col = [&](int it) {
    if (it < n_rot) {
      const int head = it / q4, e = (it % q4) * 4;
      return (head < H ? qp0 + head * D : kp0 + (head - H) * D) + e;
    }
    const int iv = it - n_rot;
    return vp0 + (iv / (D >> 2)) * D + (iv % (D >> 2)) * 4;
  };
  auto finish = [&](int it, const float4& a, const float4& c) {
    if (i >= cnt) return;
    if (it < n_rot) {
      const int head = it / q4, e = (it % q4) * 4;
      const float4 t01 = *reinterpret_cast<const float4*>(cs + (size_t)pos * half + e);
      const float4 t23 = *reinterpret_cast<const float4*>(cs + (size_t)pos * half + e + 2);
      const uint2 lo = pack4_bf16(a.x * t01.x - c.x * t01.y, a.y * t01.z - c.y * t01.w, a.z * t23.x - c.z * t23.y, a.w * t23.z - c.w * t23.w);
      const uint2 hi = pack4_bf16(c.x * t01.x + a.x * t01.y, c.y * t01.z + a.y * t01.w, c.z * t23.x + a.z * t23.y, c.w * t23.z + a.w * t23.w);
      if (head < H) {
        bf16* dst = q + (size_t)m * H * D + head * D + e;
        *reinterpret_cast<uint2*>(dst) = lo;
        *reinterpret_cast<uint2*>(dst + half) = hi;
      } else {
        const int page = page_table[rows.sequence(b) * g.pages_per_seq + slot / g.page_size], prow = slot % g.page_size;
        bf16* dst = pool + g.block_offset(page, layer, 0, head - H) + (size_t)prow * D;
        *reinterpret_cast<uint2*>(dst + kv_elem<bf16>(prow, e, D, g.page_size)) = lo;
        *reinterpret_cast<uint2*>(dst + kv_elem<bf16>(prow, e + half, D, g.page_size)) = hi;
      }
    } else {
      const int iv = it - n_rot;
      const int kh = iv / (D >> 2), e = (iv % (D >> 2)) * 4;
      const int page = page_table[rows.sequence(b) * g.pages_per_seq + slot / g.page_size], prow = slot % g.page_size;
      bf16* dst = pool + g.block_offset(page, layer, 1, kh) + (size_t)prow * D;
      *reinterpret_cast<uint2*>(dst + kv_elem<bf16>(prow, e, D, g.page_size)) = pack4_bf16(a.x, a.y, a.z, a.w);
    }
  };
  for (int it = tid; it < n_rot + n_v; it += nthr) {
    const int colp = item_col(it);
    const float4 a = part_sum4(pv, m, colp);
    const float4 c = it < n_rot ? part_sum4(pv, m, colp + half) : make_float4(0.f, 0.f, 0.f, 0.f);
    finish(it, a, c);
  }
}

// ------------------------------------------------------------------ SwiGLU
// act[m][f] = bf16(SiLU(gate) * up), gate / up = sums of the partial slots of the gate and up
// matrices (padded columns gp0 + f and up0 + f). F % 4 == 0. Bound by L2. ROWS = SWIGLU_ROWS, where no tile has more than two slots (7B shape): a
// thread has four columns of that many rows, fetches all their slots before it uses the first and finds the tile's slots, which takes
// divisions, once; 128 rows of 2 x 11008 take 5.3 us behind the projection (12.5 with an item a thread after the other). ROWS = 1: more slots.
constexpr int SWIGLU_ROWS = 4;                               // (divides the activation tiles of the streamer)
template <int ROWS>
__global__ void __launch_bounds__(256)
swiglu_reduce_tc(const PartView pv, int gp0, int up0, bf16* __restrict__ act, int M, int F, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  const int f = (int)(blockIdx.x * 256 + threadIdx.x) * 4, m0 = (int)blockIdx.y * ROWS;
  const int mt = m0 >> pv.mt_shift;
  const int ns_g = f < F && ROWS > 1 ? pv.seg.nseg(((gp0 + f) >> 7) * pv.seg.m_tiles + mt) : 0;
  const int ns_u = f < F && ROWS > 1 ? pv.seg.nseg(((up0 + f) >> 7) * pv.seg.m_tiles + mt) : 0;
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  if (f >= F) return;
  auto emit = [&](int m, const float4& gt, const float4& up) {
    *reinterpret_cast<uint2*>(act + (size_t)m * F + f) =
        pack4_bf16(silu_f(gt.x) * up.x, silu_f(gt.y) * up.y, silu_f(gt.z) * up.z, silu_f(gt.w) * up.w);
  };
  if constexpr (ROWS > 1) {
    const float* src = pv.part + (size_t)m0 * pv.ld + f;
    float4 g[ROWS], u[ROWS], g1[ROWS], u1[ROWS];
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      if (m0 + r >= M) continue;
      const float* row = src + (size_t)r * pv.ld;
      g[r] = __ldcg(reinterpret_cast<const float4*>(row + gp0));
      u[r] = __ldcg(reinterpret_cast<const float4*>(row + up0));
      if (ns_g > 1) g1[r] = __ldcg(reinterpret_cast<const float4*>(row + gp0 + pv.slot_stride));
      if (ns_u > 1) u1[r] = __ldcg(reinterpret_cast<const float4*>(row + up0 + pv.slot_stride));
    }
#pragma unroll
    for (int r = 0; r < ROWS; ++r) {
      if (m0 + r >= M) continue;
      if (ns_g > 1) { g[r].x += g1[r].x; g[r].y += g1[r].y; g[r].z += g1[r].z; g[r].w += g1[r].w; }
      if (ns_u > 1) { u[r].x += u1[r].x; u[r].y += u1[r].y; u[r].z += u1[r].z; u[r].w += u1[r].w; }
      emit(m0 + r, g[r], u[r]);
    }
  } else {
    emit(m0, part_sum4(pv, m0, gp0 + f), part_sum4(pv, m0, up0 + f));
  }
}

// ------------------------------------------------------------------ extra decoding heads
// r[b*K + k0 + kk][i] = bf16(h + SiLU(z + bias_k[i])), z = sum of the partial slots of head
// matrix kk of this launch group (padded columns kk * dpad + i), h = hq_last[b][i] (already
// bf16). grid (B * nk, CTAs per row).
__global__ void __launch_bounds__(256)
medusa_act_tc(const PartView pv, int dpad, const bf16* __restrict__ hq_last, const bf16* const* __restrict__ bias,
              bf16* __restrict__ r, int K, int k0, int nk, int d, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  const int b = blockIdx.x / nk, kk = blockIdx.x % nk, k = k0 + kk;
  const bf16* bk = bias[k];
  for (int c4 = blockIdx.y * blockDim.x + threadIdx.x; c4 < (d >> 2); c4 += gridDim.y * blockDim.x) {
    const int i = c4 * 4;
    const float4 z = part_sum4(pv, b, kk * dpad + i);
    const uint2 hraw = *reinterpret_cast<const uint2*>(hq_last + (size_t)b * d + i);
    const uint2 braw = *reinterpret_cast<const uint2*>(bk + i);
    const __nv_bfloat162* hp = reinterpret_cast<const __nv_bfloat162*>(&hraw);
    const __nv_bfloat162* bp = reinterpret_cast<const __nv_bfloat162*>(&braw);
    const float2 h01 = __bfloat1622float2(hp[0]), h23 = __bfloat1622float2(hp[1]);
    const float2 b01 = __bfloat1622float2(bp[0]), b23 = __bfloat1622float2(bp[1]);
    *reinterpret_cast<uint2*>(r + ((size_t)b * K + k) * d + i) =
        pack4_bf16(h01.x + silu_f(z.x + b01.x), h01.y + silu_f(z.y + b01.y), h23.x + silu_f(z.z + b23.x), h23.y + silu_f(z.w + b23.y));
  }
}

// lm_head consumers of the GEMM's partial sums. argmax_partials_tc: row m, vocabulary slice
// blockIdx.y of gridDim.y: logits = sum of the slots (written out when `logits` is given), the
// slice's best (value desc, index asc) goes to pval / pidx [m][gridDim.y]. The CTA of a row that
// arrives last (arrive[m], zero between launches) picks the row's best among the slices' and writes
// pval2[m] / pidx2[m]: the order (value desc, index asc) is total, so the result does not depend on
// who arrives last, and no finishing kernel is needed.
__global__ void __launch_bounds__(256)
argmax_partials_tc(const PartView pv, int V, float* __restrict__ logits, float* __restrict__ pval, int* __restrict__ pidx,
                   unsigned int* __restrict__ arrive, float* __restrict__ pval2, int* __restrict__ pidx2,
                   unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  const int m = blockIdx.x, nsl = gridDim.y;
  const bool vec = (pv.ld & 3) == 0;                           // (rows of any length come from the float32 path only)
  const int v4 = (V + 3) >> 2;
  const int per = (v4 + nsl - 1) / nsl;
  const int c_lo = blockIdx.y * per, c_hi = min(v4, c_lo + per);
  float bv = -INFINITY; int bi = 0x7fffffff;
  auto take = [&](int c4, const float4& a) {
    const float z[4] = {a.x, a.y, a.z, a.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = c4 * 4 + j;
      if (n < V) {
        if (logits) logits[(size_t)m * V + n] = z[j];
        if (better(z[j], n, bv, bi)) { bv = z[j]; bi = n; }
      }
    }
  };
  if (pv.single && !vec) {
    const float* z = pv.part + (size_t)m * pv.ld;
    for (int n = c_lo * 4 + threadIdx.x; n < min(V, c_hi * 4); n += blockDim.x)
      if (better(__ldcg(z + n), n, bv, bi)) { bv = __ldcg(z + n); bi = n; }
  } else if (pv.single) {
    // passes of many rows (finished sums, 131 MB at 1024 rows): bound by bandwidth, so a thread keeps four loads in flight
    constexpr int U = 4;
    for (int c0 = c_lo + threadIdx.x; c0 < c_hi; c0 += U * blockDim.x) {
      float4 a[U];
#pragma unroll
      for (int k = 0; k < U; ++k) if (c0 + k * (int)blockDim.x < c_hi) a[k] = part_one4(pv, m, (c0 + k * (int)blockDim.x) * 4);
#pragma unroll
      for (int k = 0; k < U; ++k) if (c0 + k * (int)blockDim.x < c_hi) take(c0 + k * (int)blockDim.x, a[k]);
    }
  } else {
    for (int c4 = c_lo + threadIdx.x; c4 < c_hi; c4 += blockDim.x) take(c4, part_sum4(pv, m, c4 * 4));
  }
  __shared__ float sv[8];
  __shared__ int si[8];
  warp_argmax(bv, bi);
  if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = bv; si[threadIdx.x >> 5] = bi; }
  __syncthreads();
  __shared__ int last_s;
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) if (better(sv[w], si[w], bv, bi)) { bv = sv[w]; bi = si[w]; }
    pval[(size_t)m * nsl + blockIdx.y] = bv;
    pidx[(size_t)m * nsl + blockIdx.y] = bi;
    __threadfence();
    const unsigned int old = atomicAdd(arrive + m, 1u);
    last_s = old == (unsigned int)(nsl - 1);
    if (last_s) arrive[m] = 0u;
  }
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  bv = -INFINITY; bi = 0x7fffffff;
  for (int t = threadIdx.x; t < nsl; t += blockDim.x) {
    const float v = __ldcg(pval + (size_t)m * nsl + t); const int i = __ldcg(pidx + (size_t)m * nsl + t);
    if (better(v, i, bv, bi)) { bv = v; bi = i; }
  }
  __syncthreads();                                           // sv / si are reused
  warp_argmax(bv, bi);
  if ((threadIdx.x & 31) == 0) { sv[threadIdx.x >> 5] = bv; si[threadIdx.x >> 5] = bi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int w = 1; w < (int)(blockDim.x >> 5); ++w) if (better(sv[w], si[w], bv, bi)) { bv = sv[w]; bi = si[w]; }
    pval2[m] = bv;
    pidx2[m] = bi;
  }
}

// The best (value desc, index asc) of every row among its tiles' [M][tiles], a warp a row.
__global__ void __launch_bounds__(256)
argmax_tiles(const float* __restrict__ val, const int* __restrict__ idx, int M, int tiles, float* __restrict__ pval2, int* __restrict__ pidx2,
             unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  const int m = blockIdx.x * 8 + (threadIdx.x >> 5), lane = threadIdx.x & 31;
  if (m >= M) return;
  float bv = -INFINITY;
  int bi = 0x7fffffff;
#pragma unroll 8
  for (int t = lane; t < tiles; t += 32) {
    const float v = __ldcg(val + (size_t)m * tiles + t);
    const int i = __ldcg(idx + (size_t)m * tiles + t);
    if (better(v, i, bv, bi)) { bv = v; bi = i; }
  }
  warp_argmax(bv, bi);
  if (lane == 0) { pval2[m] = bv; pidx2[m] = bi; }
}

// The same among slots [slots][M] (passes of many rows): a CTA takes 32 rows, its warps every 32nd slot.
__global__ void __launch_bounds__(1024)
argmax_slots(const float* __restrict__ val, const int* __restrict__ idx, int M, int slots, float* __restrict__ pval2, int* __restrict__ pidx2,
             unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  __shared__ float sv[32][33];
  __shared__ int si[32][33];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, m = blockIdx.x * 32 + lane;
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  float bv = -INFINITY;
  int bi = 0x7fffffff;
  if (m < M) {
#pragma unroll 8
    for (int t = warp; t < slots; t += 32) {
      const float v = __ldcg(val + (size_t)t * M + m);
      const int i = __ldcg(idx + (size_t)t * M + m);
      if (better(v, i, bv, bi)) { bv = v; bi = i; }
    }
  }
  sv[warp][lane] = bv; si[warp][lane] = bi;
  __syncthreads();
  bv = sv[lane][warp]; bi = si[lane][warp];                  // (row `warp` of the 32)
  warp_argmax(bv, bi);
  const int row = blockIdx.x * 32 + warp;
  if (lane == 0 && row < M) { pval2[row] = bv; pidx2[row] = bi; }
}

// Per-head top-k straight from the partial sums of the heads' lm_head GEMM (no materialised logits): each
// row's kmax best (value desc, index asc) of this block's slice of the vocabulary go to the partial lists
// pk_val / pk_idx [row][block][kmax]; grid (slices, rows), the view's first row being row `row0` of the lists. The CTA of a row that arrives last (arrive[row],
// zero between launches) merges the row's lists itself (topk_merge_row: the result does not depend on who
// that is). Dynamic shared memory: the larger of slice * 4 and gridDim.x * kmax * 8 bytes.
__global__ void __launch_bounds__(256)
topk_slices_tc(const PartView pv, int V, int row0, int slice, int kmax, float* pk_val, int* pk_idx,
               unsigned int* __restrict__ arrive, int K, const int* __restrict__ root_tok,
               const int* __restrict__ cand_override, int* __restrict__ cand, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  pdl_wait();
  if (threadIdx.x == 0) trace_mark_min(tr, 2);
  extern __shared__ float zs[];
  const int row = row0 + blockIdx.y, n0 = blockIdx.x * slice, n1 = min(n0 + slice, V);    // slice % 4 == 0
  for (int c4 = threadIdx.x; c4 * 4 < n1 - n0; c4 += blockDim.x) {
    const float4 a = part_sum4(pv, blockIdx.y, n0 + c4 * 4);
    zs[c4 * 4] = a.x; zs[c4 * 4 + 1] = a.y; zs[c4 * 4 + 2] = a.z; zs[c4 * 4 + 3] = a.w;
  }
  __syncthreads();
  const size_t list = ((size_t)row * gridDim.x + blockIdx.x) * kmax;
  block_topk(zs, nullptr, n0, n1 - n0, kmax, [&](int t, float v, int i) { pk_val[list + t] = v; pk_idx[list + t] = i; });
  __threadfence();                                           // every writer's list entries, before the arrival below
  __syncthreads();
  __shared__ int last_s;
  if (threadIdx.x == 0) {
    const unsigned int old = atomicAdd(arrive + row, 1u);
    last_s = old == gridDim.x - 1;
    if (last_s) arrive[row] = 0u;
  }
  __syncthreads();
  if (!last_s) return;
  __threadfence();
  topk_merge_row(pk_val, pk_idx, (int)gridDim.x, row, K, kmax, root_tok, cand_override, cand, zs);
}

// Per-head top-k where the projection left each row's largest in every tile of 128 tokens (float32: of `tile` tokens, every tiles-th
// piece of `piece`; best_val / best_idx [row][tiles]) beside the logits: the
// kmax best lie in tiles whose largest is among the kmax best of those, so a CTA a row reads the maxima and a dozen tiles instead of the vocabulary.
// Of the maxima of up to 64 groups of tiles (kmax or more of them) the kmax-th largest is a bound that kmax values reach; what reaches it in the tiles that do is
// ranked (order: value descending, index ascending; NaN never wins). Where more than TOPK_CAP values reach it (many equal ones), kmax
// rounds over those tiles decide. 4 heads over 32016 tokens: 9.6 us of topk_slices_tc -> 4.1; 64 rows: 22.3 -> 5.2; 3 float32
// heads 8.6 -> 4.1.
constexpr int TOPK_MAX_TILES = 512;                          // (and at least kmax)
__global__ void __launch_bounds__(256)
topk_tiles(const float* __restrict__ z, int ldz, const float* __restrict__ best_val, const int* __restrict__ best_idx, int tiles, int tile, int piece, int V, int kmax, int K,
           const int* __restrict__ root_tok, const int* __restrict__ cand_override, int* __restrict__ cand, unsigned long long* tr) {
  KTrace kt(tr);
  pdl_launch_dependents();
  constexpr int NONE = 0x7fffffff, PER = TOPK_MAX_TILES / 256;
  __shared__ float gv[64], cv[TOPK_CAP];
  __shared__ int gi[64], ci[TOPK_CAP], list[TOPK_MAX_TILES];
  __shared__ float tau_v;
  __shared__ int tau_i, n_list, count;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row = blockIdx.x, b = row / K, k = row % K;
  int* out = cand + ((size_t)b * (K + 1) + k + 1) * kmax;
  const int* ovr = cand_override ? cand_override + ((size_t)b * K + k) * kmax : nullptr;
  auto emit = [&](int t, int i) {
    const int o = ovr ? ovr[t] : -1, tok = o >= 0 ? o : i;
    out[t] = tok == NONE ? 0 : tok;
  };
  if (tid == 0) { tau_v = -INFINITY; tau_i = NONE - 1; n_list = count = 0; }   // fewer than kmax groups hold a value: all values pass
  pdl_wait();
  if (tid == 0) trace_mark_min(tr, 2);
  if (k == 0 && tid == 0) cand[(size_t)b * (K + 1) * kmax] = root_tok[b];
  float tv[PER];
  int ti[PER];
  float bv = -INFINITY; int bi = NONE;
#pragma unroll
  for (int j = 0; j < PER; ++j) {
    const int t = tid + j * 256;
    tv[j] = t < tiles ? __ldcg(best_val + (size_t)row * tiles + t) : -INFINITY;
    ti[j] = t < tiles ? __ldcg(best_idx + (size_t)row * tiles + t) : NONE;
    if (better(tv[j], ti[j], bv, bi)) { bv = tv[j]; bi = ti[j]; }
  }
  if (tiles <= 64) {
    if (tid < 64) { gv[tid] = bv; gi[tid] = bi; }            // (a group a tile)
  } else {
#pragma unroll
    for (int o = 1; o <= 2; o <<= 1) {
      const float ov = __shfl_xor_sync(0xffffffffu, bv, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (better(ov, oi, bv, bi)) { bv = ov; bi = oi; }
    }
    if ((tid & 3) == 0) { gv[tid >> 2] = bv; gi[tid >> 2] = bi; }
  }
  __syncthreads();
  if (tid < 64 && gi[tid] != NONE) {
    const float x = gv[tid]; const int i = gi[tid];
    int rank = 0;
#pragma unroll 16
    for (int j = 0; j < 64; ++j) rank += better(gv[j], gi[j], x, i) ? 1 : 0;
    if (rank == kmax - 1) { tau_v = x; tau_i = i; }
  }
  __syncthreads();
  const float bound = tau_v; const int bound_i = tau_i;
  auto reaches = [&](float x, int i) { return x >= bound && i != NONE && !better(bound, bound_i, x, i); };
#pragma unroll
  for (int j = 0; j < PER; ++j)
    if (reaches(tv[j], ti[j])) list[atomicAdd(&n_list, 1)] = tid + j * 256;
  __syncthreads();
  const int nl = n_list;
  const float* zr = z + (size_t)row * ldz;
  auto token = [&](int t, int c) { return (c / piece * tiles + t) * piece + c % piece; };
  for (int l = warp; l < nl; l += 8)
    for (int c = lane * 4; c < tile; c += 128) {
      const int n0 = token(list[l], c);
      float x[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) x[j] = -INFINITY;
      if (n0 < ldz) { const float4 v = __ldcg(reinterpret_cast<const float4*>(zr + n0)); x[0] = v.x; x[1] = v.y; x[2] = v.z; x[3] = v.w; }   // (ldz % 4 == piece % 4 == 0)
#pragma unroll
      for (int j = 0; j < 4; ++j)
        if (n0 + j < V && reaches(x[j], n0 + j)) {
          const int at = atomicAdd(&count, 1);
          if (at < TOPK_CAP) { cv[at] = x[j]; ci[at] = n0 + j; }
        }
    }
  __syncthreads();
  const int nc = count;
  if (nc <= TOPK_CAP) {
    if (tid < nc) {
      const float x = cv[tid]; const int i = ci[tid];
      int rank = 0;
      for (int j = 0; j < nc; ++j) rank += better(cv[j], ci[j], x, i) ? 1 : 0;
      if (rank < kmax) emit(rank, i);
    }
    if (tid >= nc && tid < kmax) emit(tid, NONE);
    return;
  }
  // many equal values: kmax rounds, each the best below the one before
  float pv = INFINITY; int pi = -1;
  for (int t = 0; t < kmax; ++t) {
    bv = -INFINITY; bi = NONE;
    for (int c = tid; c < nl * tile; c += 256) {
      const int n = token(list[c / tile], c % tile);
      if (n >= V) continue;
      const float x = __ldcg(zr + n);
      if (better(pv, pi, x, n) && better(x, n, bv, bi)) { bv = x; bi = n; }
    }
    warp_argmax(bv, bi);
    __syncthreads();                                         // (cv / ci of the round before have been read)
    if (lane == 0) { cv[warp] = bv; ci[warp] = bi; }
    __syncthreads();
    bv = cv[0]; bi = ci[0];
    for (int w = 1; w < 8; ++w) if (better(cv[w], ci[w], bv, bi)) { bv = cv[w]; bi = ci[w]; }
    if (tid == 0) emit(t, bi);
    pv = bv; pi = bi;
  }
}

// y[m][n] = sum of the partial slots (logical columns of a single matrix): the stand-alone linear. clear: four ints set to zero, or nullptr.
__global__ void __launch_bounds__(256)
part_sum_rows(const PartView pv, float* __restrict__ y, int M, int N, int* __restrict__ clear) {
  pdl_launch_dependents();
  pdl_wait();
  if (clear && blockIdx.x == 0 && threadIdx.x < 4) clear[threadIdx.x] = 0;
  const int n4 = (N + 3) >> 2;
  const size_t total = (size_t)M * n4;
  for (size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x; idx < total; idx += (size_t)gridDim.x * blockDim.x) {
    const int m = (int)(idx / n4), n = (int)(idx % n4) * 4;
    const float4 a = part_sum4(pv, m, n);
    const float v[4] = {a.x, a.y, a.z, a.w};
    for (int j = 0; j < 4 && n + j < N; ++j) y[(size_t)m * N + n + j] = v[j];
  }
}

}  // namespace spec
