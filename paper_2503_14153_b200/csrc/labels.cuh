// Syntax-enriched training labels (Sec. III-C): Labels[i][s] = L0[s + i] (padded with [PAD]
// past the end); per column the last [FRAG] along the head axis is found and every label
// beyond it becomes [IGNORE] (a column without a marker keeps only row 0). HBM-bound: the
// sequence is read once through a shared-memory window of blockDim.x + num_heads tokens and
// the (num_heads + 1) x seq_len matrix is written once, each row coalesced.
#pragma once
#include <stdint.h>

namespace spec {

constexpr int LABEL_THREADS = 256;
constexpr int LABEL_MAX_HEADS = 64;

__global__ void __launch_bounds__(LABEL_THREADS)
build_labels_kernel(const int32_t* __restrict__ tokens, int seq_len, int num_heads, int32_t frag, int32_t pad,
                    int32_t ignore, int32_t* __restrict__ labels) {
  __shared__ int32_t win[LABEL_THREADS + LABEL_MAX_HEADS];
  const int seq = blockIdx.y;
  const int s0 = blockIdx.x * LABEL_THREADS;
  const int32_t* l0 = tokens + (size_t)seq * seq_len;
  for (int c = threadIdx.x; c < LABEL_THREADS + num_heads; c += LABEL_THREADS) {
    const int s = s0 + c;
    win[c] = s < seq_len ? l0[s] : pad;
  }
  __syncthreads();
  const int s = s0 + threadIdx.x;
  if (s >= seq_len) return;
  int last = 0;
  for (int i = 0; i <= num_heads; ++i)
    if (win[threadIdx.x + i] == frag) last = i;
  int32_t* out = labels + (size_t)seq * (num_heads + 1) * seq_len + s;
  for (int i = 0; i <= num_heads; ++i) out[(size_t)i * seq_len] = i <= last ? win[threadIdx.x + i] : ignore;
}

// The same where the rows of the matrix are 16-byte aligned (seq_len a multiple of four, an aligned matrix): a thread has four neighbouring columns and
// writes 16 bytes a row. 256 x 2048, ten heads: 8.1 -> 6.8 us out of a cold L2 (rows that are not aligned take four scattered stores in this
// form: 8.2 -> 11.0, so they keep the other).
constexpr int LABEL_VEC_THREADS = 128, LABEL_VEC_COLS = 4 * LABEL_VEC_THREADS;
__global__ void __launch_bounds__(LABEL_VEC_THREADS)
build_labels_vec(const int32_t* __restrict__ tokens, int seq_len, int num_heads, int32_t frag, int32_t pad, int32_t ignore, int32_t* __restrict__ labels) {
  __shared__ int32_t win[LABEL_VEC_COLS + LABEL_MAX_HEADS + 4];
  const int seq = blockIdx.y, s0 = blockIdx.x * LABEL_VEC_COLS;
  const int32_t* l0 = tokens + (size_t)seq * seq_len;
  for (int c = threadIdx.x; c < LABEL_VEC_COLS + num_heads + 4; c += LABEL_VEC_THREADS) win[c] = s0 + c < seq_len ? l0[s0 + c] : pad;
  __syncthreads();
  const int c0 = threadIdx.x * 4, s = s0 + c0;
  if (s >= seq_len) return;
  int last[4] = {0, 0, 0, 0};
  for (int i = 0; i < num_heads + 4; ++i) {
    if (win[c0 + i] != frag) continue;                       // (in row i - j of column j)
#pragma unroll
    for (int j = 0; j < 4; ++j)
      if (i >= j && i - j <= num_heads) last[j] = i - j;
  }
  int32_t* out = labels + (size_t)seq * (num_heads + 1) * seq_len + s;
  int4 v = make_int4(win[c0], win[c0 + 1], win[c0 + 2], win[c0 + 3]);
  for (int i = 0; i <= num_heads; ++i) {
    *reinterpret_cast<int4*>(out) = make_int4(i <= last[0] ? v.x : ignore, i <= last[1] ? v.y : ignore, i <= last[2] ? v.z : ignore, i <= last[3] ? v.w : ignore);
    out += seq_len;
    v = make_int4(v.y, v.z, v.w, win[c0 + i + 4]);
  }
}

}  // namespace spec
