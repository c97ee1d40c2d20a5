// C ABI of the draft-and-verify decode loop: context set-up, workspace carving, the
// per-step kernel schedule and the debug taps. All device work is enqueued on the caller's
// stream (a step is recorded once on a stream of the library's own and replayed on the caller's);
// every device buffer lies in the caller's workspace.
#include "../../include/spec_decode.h"

#include <cuda.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdio.h>
#include <stdlib.h>
#include <string.h>

#include <algorithm>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <vector>

#include "attention_tc.cuh"
#include "attention_umma.cuh"
#include "common.cuh"
#include "gemm_cluster.cuh"
#include "gemm_glu.cuh"
#include "gemm_stream.cuh"
#include "gemm_pair.cuh"
#include "glue_tc.cuh"
#include "kernels_simple.cuh"
#include "labels.cuh"

using namespace spec;

namespace {

thread_local std::string g_create_error = "no error";

constexpr int PREFILL_ROWS = 128;   // rows of one chunk of a prompt (a chunk's causal mask is one ancestor set per row)
// Chunks a prompt-processing pass takes at most on the tensor-core path: 18 chunks = 2304 rows = 9 activation tiles, with
// which the tiles of all four projections of the 7B shape fill the 74 CTA pairs to 95-97% of whole waves (16 chunks: 86-93%).
// A 2048-token prompt through 8 layers of that shape: 17.6 ms at 128 rows a pass, 7.1 ms in one; eight ragged prompts of
// 128..1024 tokens through 4 layers: 14.2 ms in passes of one chunk a prompt (mostly padding at the end), 7.5 ms (both with every
// layer computed whole; they take 6.2 and 6.0 ms since the last one goes on with the prompts' last rows).
constexpr int PREFILL_CHUNKS = 18;
constexpr int TRACE_CAP = 1024;     // launches of one step the timeline can hold
constexpr int SM_SLOTS = 296;       // 148 SMs x 2 co-resident GEMM CTAs
constexpr int N_COPY_EVERY = 4;         // enqueue-only steps between two copies of the committed lengths to the host
constexpr int MAX_STEPS_AHEAD = 8;      // enqueue-only steps the host may run ahead of the device
constexpr int ATTN_ROWS_WARPS = 6;      // warps of the CTA-per-16-rows attention kernel
constexpr int ATTN_SPLIT_TILES = 8;       // fewest KV tiles a split of attention_tc gets (2..8 measured alike)
constexpr int ATTN_STAGES = 4;          // tiles attention_tc has in flight
constexpr int ATTN_SINGLE_TILES = 12;   // contexts of at most this many 64-key tiles use one KV split
constexpr int ATTN_LONG_KEYS = 2048;    // default context length from which passes of more than 32 rows use the shared-K/V kernel

constexpr int GP_NT = 256;              // activation rows per tile of the many-row projection kernel
constexpr int GP_MAX_CLUSTERS = SM_SLOTS / 4;   // its clusters: two CTAs each, one CTA per SM
constexpr int GP_SPLIT_KC = 64;         // see pair_parts
constexpr size_t GP_PART_FLOATS = (size_t)GP_MAX_CLUSTERS * 2 * GP_NT * 128;   // a part of a tile per cluster
constexpr int GP_ARRIVE = GP_MAX_CLUSTERS;   // at most half as many shared tiles as clusters, two CTAs each

inline size_t round_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// bf16 row-major [rows][cols] matrix, box = box_rows x 64 columns (128 bytes), 128-byte swizzle. With `image` the
// matrix is a pre-tiled image seen as rows of 64 columns: its bytes are in shared-memory order already, no swizzle.
bool make_tmap(CUtensorMap* tm, const void* ptr, uint64_t rows, uint64_t cols, uint32_t box_rows, bool image = false) {
  EncodeTiledFn fn = get_encode_fn();
  if (!fn) return false;
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(tm, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, image ? CU_TENSOR_MAP_SWIZZLE_NONE : CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

struct Bump {
  uint8_t* base;
  size_t off = 0;
  explicit Bump(void* b) : base(static_cast<uint8_t*>(b)) {}
  template <typename T> T* take(size_t count, size_t align = 256) {
    off = round_up(off, align);
    T* p = base ? reinterpret_cast<T*>(base + off) : nullptr;
    off += count * sizeof(T);
    return p;
  }
};

int mt_for_rows(int M) {
  if (M <= 16) return 16;
  if (M <= 32) return 32;
  if (M <= 64) return 64;
  return 128;
}

// Launch with or without the programmatic-dependent-launch attribute.
template <typename... Params, typename... Args>
cudaError_t launch_k(bool pdl, void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t st, Args&&... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = block; cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

// One launch of the weight-streaming GEMM: shapes, the dealing of units to CTAs and the view
// of its partial sums.
struct GemmPlan {
  StreamGemmParams p;
  int MT, grid;
};

bool plan_gemm(int M, int K, int n_mats, const int* rows, int g_max, GemmPlan* out) {
  if (M < 1 || K < 64 || K % 64 || n_mats < 1 || n_mats > GS_MAX_MATS || g_max < 1) return false;
  GemmPlan& g = *out;
  g = GemmPlan{};
  StreamGemmParams& p = g.p;
  g.MT = mt_for_rows(M);
  p.M = M; p.K = K; p.n_mats = n_mats;
  int tiles = 0, col = 0;
  for (int i = 0; i < n_mats; ++i) {
    if (rows[i] < 1) return false;
    p.mat_tile0[i] = tiles; p.mat_rows[i] = rows[i]; p.mat_col0[i] = col;
    tiles += (rows[i] + 127) / 128;
    col += rows[i];
  }
  for (int i = n_mats; i <= GS_MAX_MATS; ++i) p.mat_tile0[i] = tiles;
  p.n_tiles = tiles;
  p.seg.KC = K / 64;
  p.seg.m_tiles = (M + g.MT - 1) / g.MT;
  long long total = (long long)tiles * p.seg.m_tiles * p.seg.KC;
  if (total > 0x3fffffff || (total + 1) * (long long)g_max >= 0x7fffffffLL) return false;
  p.seg.total = (int)total;
  g.grid = (int)std::min<long long>(g_max, total);
  p.seg.G = g.grid;
  return true;
}

// Upper bound of the partial-sum slots a tile can have when the units go to at most g_max CTAs.
int plan_slot_bound(const GemmPlan& g) {
  const SegMap& s = g.p.seg;
  return (int)(((long long)s.KC * s.G) / s.total) + 2;
}

size_t plan_part_floats(const GemmPlan& g) { return (size_t)plan_slot_bound(g) * g.p.M * g.p.n_tiles * 128; }

// The shared-memory attribute of a kernel is per device: it is set on every launch's device the first time
// that device is seen (indexed by the device ordinal), not once per process.
constexpr int kAttrDevices = 64;
inline bool* attr_flag(bool (&flags)[kAttrDevices]) {
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kAttrDevices) dev = 0;
  return &flags[dev];
}

template <int MT, int DEEP>
cudaError_t launch_gs_mt(cudaStream_t st, bool pdl, int grid, const StreamTmaps& tm, const StreamGemmParams& p) {
  static bool attr_set_dev[kAttrDevices] = {};
  bool& attr_set = *attr_flag(attr_set_dev);
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(gemm_stream<MT, DEEP>, cudaFuncAttributeMaxDynamicSharedMemorySize, StreamCfg<MT, DEEP>::SMEM_BYTES);
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  return launch_k(pdl, gemm_stream<MT, DEEP>, dim3(grid), dim3(192), (size_t)StreamCfg<MT, DEEP>::SMEM_BYTES, st, tm, p);
}
// Grids of at most one CTA per SM get the deep ring (one resident CTA must keep the SM's share
// of the memory pipe full by itself).
cudaError_t launch_gs(cudaStream_t st, bool pdl, const GemmPlan& g, const StreamTmaps& tm) {
  const bool deep = g.grid <= SM_SLOTS / 2;
  switch (g.MT) {
    case 16: return deep ? launch_gs_mt<16, 1>(st, pdl, g.grid, tm, g.p) : launch_gs_mt<16, 0>(st, pdl, g.grid, tm, g.p);
    case 32: return deep ? launch_gs_mt<32, 1>(st, pdl, g.grid, tm, g.p) : launch_gs_mt<32, 0>(st, pdl, g.grid, tm, g.p);
    case 64: return deep ? launch_gs_mt<64, 1>(st, pdl, g.grid, tm, g.p) : launch_gs_mt<64, 0>(st, pdl, g.grid, tm, g.p);
    default: return deep ? launch_gs_mt<128, 1>(st, pdl, g.grid, tm, g.p) : launch_gs_mt<128, 0>(st, pdl, g.grid, tm, g.p);
  }
}

// The launch of gemm_cluster<MT, MODE> over `tiles` clusters of `cluster` CTAs with a ring of `stages`.
struct ClusterLaunch {
  cudaLaunchConfig_t cfg{};
  cudaLaunchAttribute at[2];
  ClusterLaunch(cudaStream_t st, bool pdl, int tiles, int cluster, size_t smem) {
    cfg.gridDim = dim3(tiles * cluster); cfg.blockDim = dim3(GC_THREADS); cfg.dynamicSmemBytes = smem; cfg.stream = st;
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = cluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = pdl ? 2 : 1;
  }
};
template <int MT, int MODE> cudaError_t allow_deepest_ring() {
  return cudaFuncSetAttribute(gemm_cluster<MT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, ClusterCfg<MT>::smem_bytes(ClusterCfg<MT>::MAX_STAGES));
}
template <int MODE> int cluster_units(int KC, int cluster) { return ((MODE == GC_SWIGLU ? 2 : 1) * KC + cluster - 1) / cluster; }   // K chunks of a CTA, at most

template <int MT, int MODE>
cudaError_t launch_gc_mt(cudaStream_t st, bool pdl, int tiles, int cluster, const StreamTmaps& tm, ClusterGemmParams p, bool* attr_set) {
  if (!*attr_set) {
    cudaError_t e = allow_deepest_ring<MT, MODE>();
    if (e != cudaSuccess) return e;
    *attr_set = true;
  }
  p.stages = cluster_stages<MT, MODE>(tiles, cluster, cluster_units<MODE>(p.KC, cluster));
  ClusterLaunch l(st, pdl, tiles, cluster, (size_t)ClusterCfg<MT>::smem_bytes(p.stages));
  return cudaLaunchKernelEx(&l.cfg, gemm_cluster<MT, MODE>, tm, p);
}

// Stages that such a launch takes, and the clusters of it that the device holds at once at one CTA an SM. (At two an SM the runtime does not tell: for
// kernels with tensor memory it answers one CTA an SM whatever their shared memory.)
template <int MT, int MODE>
cudaError_t cluster_residency(int tiles, int cluster, int KC, int* out) {
  cudaError_t e = allow_deepest_ring<MT, MODE>();
  if (e != cudaSuccess) return e;
  out[0] = cluster_stages<MT, MODE>(tiles, cluster, cluster_units<MODE>(KC, cluster));
  ClusterLaunch l(nullptr, false, tiles, cluster, (size_t)ClusterCfg<MT>::smem_bytes(ClusterCfg<MT>::MAX_STAGES));
  return cudaOccupancyMaxActiveClusters(&out[1], gemm_cluster<MT, MODE>, &l.cfg);
}

// CTAs that share each tile of a GC_PLAIN launch: as many as let all clusters be resident at once (96 KB of shared memory a CTA) and have
// two K chunks each; 0: more tiles than CTAs fit, the weight streamer deals them out evenly.
int plain_cluster(int tiles, int KC, int max_ctas) {
  constexpr int size[] = {8, 6, 4, 3, 2, 1}, most[] = {33, 45, 71, 93, 148, SM_SLOTS};
  for (int i = 0; i < 6; ++i)
    if (tiles <= most[i] && 2 * size[i] <= std::max(KC, 2) && (long long)tiles * size[i] <= max_ctas) return size[i];
  return 0;
}

cudaError_t launch_gc_plain(cudaStream_t st, bool pdl, int tiles, int cluster, const StreamTmaps& tm, const ClusterGemmParams& p) {
  static bool set[4][kAttrDevices] = {};
  switch (mt_for_rows(p.M)) {
    case 16: return launch_gc_mt<16, GC_PLAIN>(st, pdl, tiles, cluster, tm, p, attr_flag(set[0]));
    case 32: return launch_gc_mt<32, GC_PLAIN>(st, pdl, tiles, cluster, tm, p, attr_flag(set[1]));
    case 64: return launch_gc_mt<64, GC_PLAIN>(st, pdl, tiles, cluster, tm, p, attr_flag(set[2]));
    default: return launch_gc_mt<128, GC_PLAIN>(st, pdl, tiles, cluster, tm, p, attr_flag(set[3]));
  }
}

PartView plan_view(const GemmPlan& g) {
  PartView v{};
  v.part = g.p.part; v.slot_stride = g.p.slot_stride; v.ld = g.p.n_tiles * 128; v.seg = g.p.seg;
  v.mt_shift = g.MT == 16 ? 4 : (g.MT == 32 ? 5 : (g.MT == 64 ? 6 : 7));
  return v;
}

}  // namespace

struct spec_ctx {
  spec_config cfg;
  cudaStream_t stream;
  int T, K, kmax, B;                   // tree nodes, heads, candidates per head, current batch
  bool tc;                             // bf16 tensor-core path
  size_t esz;                          // operand element size
  int Mcap, cap, pages_per_seq, gen_cap, nsplit_attn, n_argmax, topk_slice, topk_blocks;
  bool qkv_fused, keep_logits;
  bool packed = false;                 // linear weights are pre-tiled images (SPEC_FLAG_PACKED_WEIGHTS)
  bool pdl = true;                     // programmatic dependent launch between the kernels of a step
  int gemm_ctas = 288;                 // persistent CTAs of the weight-streaming GEMM (measured best; at most SM_SLOTS)
  int l2_prefetch = 0;
  bool gc_attr_set[11] = {};            // per context (and so per device): shared-memory attribute of each gemm_cluster instance set
  int long_attn_keys = ATTN_LONG_KEYS; // SPEC_OPT_LONG_ATTN_KEYS (0 = never)
  bool attn_umma = true;               // SPEC_OPT_ATTN_UMMA: the long-context kernel is the tcgen05 one (head_dim 128)
  CUtensorMap tm_kv;                   // 5-D view of the page pool for its TMA loads
  bool tm_kv_ok = false;
  bool wide_gemm = true;               // SPEC_OPT_WIDE_GEMM: passes of more than 128 rows use the two-SM kernel (gemm_pair)
  int cluster_epilogue = 7;            // SPEC_OPT_CLUSTER_EPILOGUE: which projections finish their split-K sums inside a cluster
                                       // (bits: 1 output/down, 2 gate+up, 4 q/k/v)
  int small_gemm_ctas = 288;           // CTAs of GEMMs with at most 48 weight tiles (Wo, down); 288 since the weights are pre-tiled (192 before)
  std::vector<int> h_parent, h_depth, h_rank;
  std::vector<int> n_hi, n_lo;         // host upper / lower bounds of the committed lengths
  std::vector<int> written;            // [max_batch] cache slots from here on hold zeros (nothing is known of a new workspace)
  std::vector<const void*> wq, wk, wv, wo, wg, wu, wd, mw, mb;
  std::vector<const float*> an, fn;
  const void *embed, *lm_head;
  const float* final_norm;
  KVGeom geom;
  // device buffers (workspace)
  int *d_n, *d_cnt, *d_n_old, *d_root, *d_count, *d_path, *d_out_tok, *d_gen_cnt, *d_gen_log, *d_cand, *d_cand_ov;
  int *d_tok, *d_pos, *d_slot, *d_am, *d_edge, *d_parent, *d_depth, *d_rank, *d_page_table, *d_prompt, *d_offsets;
  int *d_result;                       // [4 + B * (K + 3)]: d_status, d_n, d_count, d_out_tok
  int* h_result = nullptr;             // the same in pinned host memory, written by the step's last kernel
  int* h_result_dev = nullptr;         // its device address
  int *d_status, *d_pidx, *d_pk_idx, *d_draws;
  int head_rows;                       // rows of the heads' logits computed at a time (without tensor cores)
  int chunk_cap;                       // prompt chunks the row buffers hold in one pass
  int *d_chunk_seq, *d_chunk_pos, *d_chunk_n, *d_chunk_cnt;   // [max_batch * ceil(max_seq / 128)]: sequence and first token; [chunk_cap]
  uint32_t *d_anc_tree, *d_anc_chain;
  const void **d_mw, **d_mb;
  float *d_x, *d_hid, *d_h_last, *d_part, *d_logits, *d_pval, *d_part_o, *d_part_ml, *d_pk_val;
  float* d_ss_part = nullptr;          // [128 rows][d / 128 tiles x 8]: sums of squares the residual cluster epilogue leaves
  float2* d_rope;
  void *d_u, *d_q, *d_attn, *d_act, *d_hq, *d_hq_last, *d_r, *d_pool;
  size_t part_floats;
  std::map<std::tuple<const void*, uint64_t, uint64_t, uint32_t, bool>, CUtensorMap> tmaps;
  long long launches = 0;
  // optional device timeline of the last step: four stamps per launch (see KTrace)
  bool trace_on = false;
  unsigned long long* d_trace = nullptr;
  unsigned int* d_attn_arrive = nullptr;
  unsigned int* d_pair_arrive = nullptr;  // [GP_ARRIVE] arrival counters of the shared tiles, zero between launches
  unsigned int* d_row_arrive = nullptr;   // [Mcap] arrival counters of the per-row finishing steps, zero between launches
  float* d_pval2 = nullptr;            // finished per-row argmax (tensor-core path)
  int* d_pidx2 = nullptr;
  int trace_n = 0;
  std::vector<std::string> trace_names;
  std::vector<unsigned long long> trace_init;
  unsigned long long* next_trace(const char* name) {
    if (!trace_on || trace_n >= TRACE_CAP) return nullptr;
    trace_names.push_back(name);
    return d_trace + 4 * (size_t)(trace_n++);
  }
  // CUDA-graph replay of the step's kernel sequence: one instantiated graph per (override given?)
  // variant, valid while the sequences stay below the length bound its attention launches were
  // planned for and no option changed (epoch)
  bool graph_on = true;
  bool capturing = false;
  cudaStream_t cap_stream = nullptr;
  struct StepGraph {
    cudaGraphExec_t exec = nullptr;
    unsigned long long epoch = 0;
    int B = 0;
    long long n_launches = 0;
    std::vector<int> n_hi_plan, n_lo_plan;
    unsigned long long prefills = 0;   // the prompts it was recorded or last checked for
    std::vector<int> order;            // sequences, longest first, where the recorded attention hands its CTAs out in that order
  };
  StepGraph step_graph[2];
  unsigned long long graph_epoch = 1;
  unsigned long long prefills = 0;
  long long graph_captures = 0;
  bool prefilled = false;
  // timing: phase boundaries of the last step; optional per-launch timing of one kernel kind
  cudaEvent_t phase_ev[6] = {nullptr, nullptr, nullptr, nullptr, nullptr, nullptr};
  // enqueue-only steps: the committed lengths are copied to pinned host memory now and then, so
  // the host's bounds on them stay tight without a synchronisation
  int* h_n_pinned = nullptr;           // [max_batch], behind h_result
  cudaEvent_t n_ev = nullptr;
  bool n_copy_pending = false;
  int n_copy_steps_after = 0;          // steps enqueued after the pending copy
  int steps_since_n_copy = 0;          // enqueue-only steps since the last copy was issued
  bool phase_valid = false;
  bool phase_timing = false;           // SPEC_OPT_PHASE_TIMING
  int profile_kind = 0;                 // SPEC_PROFILE_*
  std::vector<cudaEvent_t> prof_ev;     // pairs, reused every step
  int prof_used = 0;
  double prof_ms = 0.0;
  long long prof_launches = 0;
  std::string err = "no error";

  int fail(int code, const std::string& msg) { err = msg; return code; }
  const CUtensorMap* tmap(const void* p, uint64_t rows, uint64_t cols, uint32_t box_rows, bool image = false) {
    auto key = std::make_tuple(p, rows, cols, box_rows, image);
    auto it = tmaps.find(key);
    if (it != tmaps.end()) return &it->second;
    CUtensorMap tm;
    if (!make_tmap(&tm, p, rows, cols, box_rows, image)) return nullptr;
    return &tmaps.emplace(key, tm).first->second;
  }
};

namespace {

bool validate_tree(const spec_config* cfg, const spec_tree* tree, int* kmax_out, std::string* why) {
  int T = tree->n_nodes;
  if (T < 1 || T > SPEC_MAX_NODES || !tree->parent || !tree->depth || !tree->rank) { *why = "n_nodes out of range or null arrays"; return false; }
  if (tree->parent[0] != -1 || tree->depth[0] != 0 || tree->rank[0] != 0) { *why = "node 0 must be the root"; return false; }
  int kmax = 1;
  for (int v = 1; v < T; ++v) {
    int p = tree->parent[v];
    if (p < 0 || p >= v) { *why = "parent must precede child"; return false; }
    if (tree->depth[v] != tree->depth[p] + 1 || tree->depth[v] > cfg->n_medusa) { *why = "bad depth"; return false; }
    if (tree->rank[v] < 0 || tree->rank[v] >= SPEC_MAX_TOPK) { *why = "bad rank"; return false; }
    for (int u = 1; u < v; ++u)
      if (tree->parent[u] == p && tree->rank[u] == tree->rank[v]) { *why = "siblings share a rank"; return false; }
    if (tree->rank[v] + 1 > kmax) kmax = tree->rank[v] + 1;
  }
  *kmax_out = kmax;
  return true;
}

bool validate_config(const spec_config* c, std::string* why) {
  if (c->n_layers < 1 || c->d_model < 8 || c->n_heads < 1 || c->n_kv_heads < 1 || c->head_dim < 32 ||
      c->d_ffn < 8 || c->vocab < 2 || c->max_batch < 1 || c->max_seq < 1 || c->page_size < 1) { *why = "non-positive size"; return false; }
  if (c->dtype != 0 && c->dtype != 1) { *why = "dtype must be 0 or 1"; return false; }
  if (c->n_heads % c->n_kv_heads) { *why = "n_heads must be a multiple of n_kv_heads"; return false; }
  if (c->head_dim % 32 || c->head_dim > 256) { *why = "head_dim must be a multiple of 32, <= 256"; return false; }
  if (c->d_model % 8 || c->d_ffn % 8 || (c->n_heads * c->head_dim) % 8) { *why = "widths must be multiples of 8"; return false; }
  if (c->n_medusa < 0 || c->n_medusa > SPEC_MAX_HEADS) { *why = "n_medusa out of range"; return false; }
  if (c->accept_mode != 0 && c->accept_mode != 1) { *why = "accept_mode must be 0 or 1"; return false; }
  if (c->sampling != 0 && c->sampling != 1) { *why = "sampling must be 0 or 1"; return false; }
  if (c->sampling && (c->accept_mode != 1 || !(c->temperature > 0.f))) { *why = "sampled decoding needs accept_mode 1 and a positive temperature"; return false; }
  bool tc = c->dtype == 1 && !(c->flags & SPEC_FLAG_SIMPLE_KERNELS);
  if ((c->flags & SPEC_FLAG_PACKED_WEIGHTS) && !tc) { *why = "pre-tiled weights need the bf16 tensor-core path"; return false; }
  if (tc) {
    if (c->d_model % 64 || c->d_ffn % 64 || (c->n_heads * c->head_dim) % 64) { *why = "bf16 path needs widths that are multiples of 64"; return false; }
    if (c->head_dim != 64 && c->head_dim != 128) { *why = "bf16 path needs head_dim 64 or 128"; return false; }
    if (c->page_size != 16) { *why = "bf16 path needs page_size 16"; return false; }
    if (c->d_model < 128 || c->d_ffn < 128 || c->vocab < 128 || c->n_kv_heads * c->head_dim < 128) { *why = "bf16 path needs every weight matrix to have at least 128 rows"; return false; }
  } else if (c->dtype == 1 && c->head_dim % 64) { *why = "bf16 cache needs head_dim multiple of 64"; return false; }
  return true;
}

// KV splits of an attention launch over `groups` row groups: as many as fit beside each other, at most `most`.
int attn_splits(int most, int n_heads, int groups) { return std::max(1, std::min(most, (SM_SLOTS / 2) / (n_heads * groups))); }

int max_prompt_chunks(const spec_config& f) { return f.max_batch * (int)((f.max_seq + PREFILL_ROWS - 1) / PREFILL_ROWS); }   // of the longest prompts
// Chunks a prompt-processing pass takes where the workspace has room for them.
int full_chunk_cap(const spec_ctx* c) {
  return c->tc ? std::max(c->cfg.max_batch, std::min(PREFILL_CHUNKS, max_prompt_chunks(c->cfg))) : c->cfg.max_batch;
}

// Floats of the row maxima that a float32 projection [M, K] x [N, K] leaves (RowBest), 0 where it leaves none.
size_t held_best_floats(int M, int N, int K) {
  const RowLinearShape sh = linear_rows_shape<float>((N + LR_N - 1) / LR_N, M, K);
  return linear_held(sh, K) ? 2 * (size_t)M * linear_held_shape(sh, M, N).grid.x : 0;
}

// Lays the workspace out; with base == nullptr only measures it. chunk_cap: prompt chunks of a pass, at least one a sequence;
// share_tiles: with scratch for the partial sums of gemm_pair's shared tiles even if no other use asks for that much.
size_t carve(spec_ctx* c, void* base, int chunk_cap, bool share_tiles) {
  const spec_config& f = c->cfg;
  Bump b(base);
  int B = f.max_batch, T = c->T, K = c->K, d = f.d_model, F = f.d_ffn, V = f.vocab;
  int HD = f.n_heads * f.head_dim;
  const int max_chunks = max_prompt_chunks(f);
  c->chunk_cap = chunk_cap;
  // a workspace with less than full room: buffers that are never in use at the same time share their place
  const bool spare = chunk_cap < full_chunk_cap(c) || !share_tiles;
  c->Mcap = (int)round_up((size_t)std::max(B * std::max(T, PREFILL_ROWS), c->chunk_cap * PREFILL_ROWS), 128);
  c->cap = (int)round_up((size_t)f.max_seq + T, f.page_size);
  if (64 % f.page_size == 0) c->cap = (int)round_up(c->cap, 64);   // whole 64-key attention tiles
  c->pages_per_seq = c->cap / f.page_size;
  c->gen_cap = f.max_seq + K + 1;
  c->n_argmax = 8;                // argmax partials per row (vocabulary slices)
  c->topk_slice = ((V + SM_SLOTS - 1) / SM_SLOTS + 3) / 4 * 4;
  c->topk_blocks = (V + c->topk_slice - 1) / c->topk_slice;
  c->nsplit_attn = c->tc ? std::max(1, std::min(16, (SM_SLOTS / 2) / (f.n_heads * B))) : 1;   // most KV splits a launch may use
  int Mlog = (int)round_up((size_t)B * T, 16);
  c->keep_logits = !c->tc || (f.flags & SPEC_FLAG_KEEP_LOGITS) || f.accept_mode == 1;
  size_t M = c->Mcap;

  // what a step hands to the host lies side by side, so that its last kernel writes it to host memory in one go: status word,
  // committed lengths, counts, emitted tokens
  c->d_result = b.take<int>(4 + (size_t)B * (2 + K + 1));
  c->d_status = c->d_result; c->d_n = c->d_result + 4; c->d_count = c->d_n + B; c->d_out_tok = c->d_count + B;
  c->d_trace = b.take<unsigned long long>((size_t)TRACE_CAP * 4);
  c->d_attn_arrive = b.take<unsigned int>((size_t)c->chunk_cap * f.n_heads * 2);
  // (the projections' shared tiles and the selections' rows are never counted at the same time: a kernel touches its counters
  // after its dependency wait and leaves them at zero)
  static_assert(GP_ARRIVE <= PREFILL_ROWS, "Mcap is at least PREFILL_ROWS");
  c->d_row_arrive = b.take<unsigned int>(c->Mcap);
  c->d_pair_arrive = spare ? c->d_row_arrive : b.take<unsigned int>(GP_ARRIVE);
  c->d_pval2 = b.take<float>(c->Mcap); c->d_pidx2 = b.take<int>(c->Mcap);
  c->d_draws = b.take<int>(B);
  c->d_cnt = b.take<int>(B); c->d_n_old = b.take<int>(B); c->d_root = b.take<int>(B);
  c->d_path = b.take<int>((size_t)B * (K + 1));
  c->d_gen_cnt = b.take<int>(B);
  // (the log of generated tokens is empty while prompts are processed: in a small workspace the chunks' bookkeeping lies there)
  c->d_gen_log = b.take<int>(std::max((size_t)B * c->gen_cap, 2 * (size_t)max_chunks + 2 * (size_t)chunk_cap));
  if (spare) {
    c->d_chunk_seq = c->d_gen_log; c->d_chunk_pos = c->d_chunk_seq + max_chunks;
    c->d_chunk_n = c->d_chunk_pos + max_chunks; c->d_chunk_cnt = c->d_chunk_n + chunk_cap;
  }
  c->d_cand = b.take<int>((size_t)B * (K + 1) * c->kmax); c->d_cand_ov = b.take<int>((size_t)B * (K ? K : 1) * c->kmax);
  c->d_tok = b.take<int>(M); c->d_pos = b.take<int>(M); c->d_slot = b.take<int>(M); c->d_am = b.take<int>(M);
  c->d_edge = b.take<int>(M);
  c->d_parent = b.take<int>(SPEC_MAX_NODES); c->d_depth = b.take<int>(SPEC_MAX_NODES); c->d_rank = b.take<int>(SPEC_MAX_NODES);
  c->d_anc_tree = b.take<uint32_t>(SPEC_MAX_NODES * 4); c->d_anc_chain = b.take<uint32_t>(PREFILL_ROWS * 4);
  c->d_page_table = b.take<int>((size_t)B * c->pages_per_seq);
  if (!spare) {
    c->d_chunk_seq = b.take<int>(max_chunks); c->d_chunk_pos = b.take<int>(max_chunks);
    c->d_chunk_n = b.take<int>(c->chunk_cap); c->d_chunk_cnt = b.take<int>(c->chunk_cap);
  }
  c->d_prompt = b.take<int>((size_t)B * f.max_seq); c->d_offsets = b.take<int>(B + 1);
  c->d_mw = b.take<const void*>(SPEC_MAX_HEADS); c->d_mb = b.take<const void*>(SPEC_MAX_HEADS);
  c->d_x = b.take<float>(M * d, 1024); c->d_hid = b.take<float>(M * d, 1024); c->d_h_last = b.take<float>((size_t)B * d);
  // split-K / plain projection outputs
  size_t pf = 0;
  {
    int Ms[3] = {B * T, B * PREFILL_ROWS, B};
    for (int i = 0; i < 3; ++i) {
      size_t m = Ms[i];
      if (c->tc) {
        int KD = f.n_kv_heads * f.head_dim;
        int r_qkv[3] = {HD, KD, KD}, r_o[1] = {d}, r_gu[2] = {F, F}, r_dn[1] = {d};
        GemmPlan g;
        if (plan_gemm((int)m, d, 3, r_qkv, SM_SLOTS, &g)) pf = std::max(pf, plan_part_floats(g));
        if (plan_gemm((int)m, HD, 1, r_o, SM_SLOTS, &g)) pf = std::max(pf, plan_part_floats(g));
        if (plan_gemm((int)m, d, 2, r_gu, SM_SLOTS, &g)) pf = std::max(pf, plan_part_floats(g));
        if (plan_gemm((int)m, F, 1, r_dn, SM_SLOTS, &g)) pf = std::max(pf, plan_part_floats(g));
        int r_lm[1] = {V};
        if (plan_gemm((int)m, d, 1, r_lm, SM_SLOTS, &g)) pf = std::max(pf, plan_part_floats(g));
        int r_hd[GS_MAX_MATS] = {d, d, d, d};
        if (plan_gemm((int)m, d, GS_MAX_MATS, r_hd, SM_SLOTS, &g)) pf = std::max(pf, plan_part_floats(g));
      }
    }
    // (float32: each row's largest out of lm_head, whatever the number of rows)
    if (f.dtype == 0)
      for (int m = 1; m <= B * std::max(T, K); ++m) pf = std::max(pf, held_best_floats(m, V, d));
  }
  // (split tiles of the many-row projections leave their partial sums here too)
  if (share_tiles && c->tc && c->Mcap > 128 && std::max(d, std::max(HD, F)) >= 64 * GP_SPLIT_KC) pf = std::max(pf, GP_PART_FLOATS);
  c->part_floats = pf;
  c->d_part = b.take<float>(pf, 1024);
  // (without tensor cores the heads' logits lie here too, `head_rows` at a time: they are used up before the verification pass
  // writes its own)
  c->d_logits = c->keep_logits ? b.take<float>((size_t)Mlog * V, 1024) : nullptr;
  c->head_rows = (int)std::min((size_t)B * K, (size_t)Mlog * V / round_up(V, 4));
  c->d_pval = b.take<float>((size_t)c->n_argmax * M, 1024); c->d_pidx = b.take<int>((size_t)c->n_argmax * M, 1024);
  // partial outputs of the KV splits: rows times splits, over the passes that use more than one split
  size_t split_rows = (size_t)c->nsplit_attn * B * std::max(T, PREFILL_ROWS);
  for (int g = 1; g <= c->chunk_cap; ++g)
    split_rows = std::max(split_rows, (size_t)attn_splits(c->nsplit_attn, f.n_heads, g) * g * PREFILL_ROWS);
  c->d_part_o = c->tc ? b.take<float>(split_rows * HD, 1024) : nullptr;
  c->d_part_ml = c->tc ? b.take<float>(split_rows * f.n_heads * 2) : nullptr;
  c->d_ss_part = c->tc ? b.take<float>((size_t)128 * ((d + 127) / 128) * GC_RES_CLUSTER) : nullptr;
  c->d_pk_val = b.take<float>((size_t)c->topk_blocks * B * (K ? K : 1) * c->kmax);
  c->d_pk_idx = b.take<int>((size_t)c->topk_blocks * B * (K ? K : 1) * c->kmax);
  c->d_rope = b.take<float2>((size_t)c->cap * (f.head_dim / 2));
  size_t e = c->esz;
  c->d_u = b.take<uint8_t>(M * d * e, 1024); c->d_q = b.take<uint8_t>(M * HD * e, 1024);
  c->d_attn = b.take<uint8_t>(M * HD * e, 1024); c->d_act = b.take<uint8_t>(M * F * e, 1024);
  c->d_hq = b.take<uint8_t>(M * d * e, 1024); c->d_hq_last = b.take<uint8_t>(round_up((size_t)B, 16) * d * e, 1024);
  c->d_r = b.take<uint8_t>(round_up((size_t)B * (K ? K : 1), 16) * d * e, 1024);
  c->geom = KVGeom{f.n_layers, f.n_kv_heads, f.head_dim, f.page_size, c->pages_per_seq, B};
  size_t pool_elems = (size_t)B * c->pages_per_seq * c->geom.page_elems();
  c->d_pool = b.take<uint8_t>(pool_elems * e, 1024);
  return round_up(b.off, 1024);
}

#define CUDA_OK(call)                                                                          \
  do {                                                                                         \
    cudaError_t e_ = (call);                                                                   \
    if (e_ != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

#define LAUNCH_CHECK(name)                                                                     \
  do {                                                                                         \
    c->launches++;                                                                             \
    cudaError_t e_ = cudaGetLastError();                                                       \
    if (e_ != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string(name) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// Brackets one launch with events when that kernel kind is being profiled.
struct ProfScope {
  spec_ctx* c;
  bool on;
  ProfScope(spec_ctx* ctx, int kind) : c(ctx), on(ctx->profile_kind == kind && kind != 0) {
    if (!on) return;
    if ((size_t)c->prof_used + 2 > c->prof_ev.size()) {
      cudaEvent_t a, b;
      if (cudaEventCreate(&a) != cudaSuccess || cudaEventCreate(&b) != cudaSuccess) { on = false; return; }
      c->prof_ev.push_back(a); c->prof_ev.push_back(b);
    }
    cudaEventRecord(c->prof_ev[c->prof_used], c->stream);
  }
  ~ProfScope() {
    if (!on) return;
    cudaEventRecord(c->prof_ev[c->prof_used + 1], c->stream);
    c->prof_used += 2;
  }
};

Rows make_rows(spec_ctx* c, int R, bool chain) {
  Rows r;
  r.R = R; r.B = c->B;
  r.tok = c->d_tok; r.pos = c->d_pos; r.slot = c->d_slot; r.n = c->d_n; r.cnt = c->d_cnt;
  r.seq = nullptr;
  r.anc = chain ? c->d_anc_chain : c->d_anc_tree;
  return r;
}

const char* gemm_kind_name(int kind) {
  switch (kind) {
    case SPEC_PROFILE_GATE_UP: return "gemm_gate_up";
    case SPEC_PROFILE_QKV: return "gemm_qkv";
    case SPEC_PROFILE_WO: return "gemm_wo";
    case SPEC_PROFILE_DOWN: return "gemm_down";
    default: return "gemm";
  }
}

// CTA count for a GEMM of n_tiles weight tiles, at most cap: one that lets the CTAs' runs end on tile
// boundaries (p CTAs per q tiles, q as small as possible), so that a tile's partial sums come from as few
// CTAs as possible and the consumers read fewer slots; within 15% of cap, else cap itself.
int aligned_ctas(int n_tiles, int cap) {
  for (int q = 1; q <= 4; ++q) {
    long long p = (long long)cap * q / n_tiles;
    while (p >= 1 && (n_tiles * p) % q) --p;
    if (p < 1) continue;
    const int G = (int)(n_tiles * p / q);
    if (G * 100 >= cap * 85) return G;
  }
  return cap;
}

// CTAs of the weight streamer for a launch of n_tiles weight tiles.
int stream_ctas(const spec_ctx* c, int n_tiles) { return aligned_ctas(n_tiles, n_tiles <= 48 ? std::min(c->gemm_ctas, c->small_gemm_ctas) : c->gemm_ctas); }

// ---- many rows: the two-SM kernel, the step after the projection in its epilogue ----
bool pair_gemm_ok(const spec_ctx* c, int M, int K) { return c->wide_gemm && M > 128 && K % 64 == 0; }

// Clusters that share each tile of a launch (PairGemmParams::parts): as many as there are for it where the tiles employ less than
// half of the clusters, at most four, eight for a long inner dimension (the CTA that finishes a tile adds the parts up, about
// 1 us each). A tile of fewer than GP_SPLIT_KC chunks is short (16 chunks: 6 us) and the exchange takes most of what
// sharing saves; it stays whole and keeps one order of the sums for every number of rows.
int pair_parts(int tiles, int KC, int clusters) {
  if (KC < GP_SPLIT_KC || tiles * 2 > clusters) return 1;
  return std::min(clusters / tiles, KC >= 2 * GP_SPLIT_KC ? 8 : 4);
}

// Pairs of weight tiles of the stacked query, key and value projections.
int qkv_pairs(const spec_config& f) {
  const int HD = f.n_heads * f.head_dim, KD = f.n_kv_heads * f.head_dim;
  return ((HD + 127) / 128 + 2 * ((KD + 127) / 128) + 1) / 2;
}

// What a launch of `tiles` = w_pairs * ceil(M / rows) tiles takes in microseconds, the tiles of its last wave cut in `cut`. Fitted to 45 kernels of 15 tile
// heights each (M 384 to 2304 on d_model 4096, 1024 and 512, event-timed at 1.9 GHz; within 10% of most): a K chunk on all clusters takes
// (0.002 + 0.0013 rows) us, the operands' way out of L2 (0.335 at 256 rows, the same per row from 176 rows on), on few clusters 0.00107 rows, the MMAs,
// and never less than 0.18, the issue; a tile's epilogue 0.0165 us a row where it adds to the residual stream, 0.028 in the other
// modes, under the next tile's MMAs, but for the last.
float pair_cost(int tiles, int rows, int cut, int KC, int clusters, float epilogue) {
  auto chunk = [&](int h, int n) { return std::max(std::max(0.18f, 0.00107f * h), std::max(0.16f + 0.0004f * h, 0.002f + 0.0013f * h) * n / GP_MAX_CLUSTERS); };
  auto waves = [&](int items, int h, bool last) {
    const int full = items / clusters, rest = items % clusters;
    const float wave = std::max(KC * chunk(h, clusters), epilogue * h) + 1.f;
    float us = full * wave;
    if (rest) us += KC * chunk(h, rest) + 1.f;
    return us + (last ? epilogue * h : 0.f);
  };
  if (cut == 1) return waves(tiles, rows, true);
  const int rest = tiles % clusters;
  return waves(tiles - rest, rows, rest == 0) + (rest ? waves(rest * cut, rows / cut, true) : 0.f);
}

// How a launch is cut into items (gemm_pair.cuh), by M, KC, w_pairs and plan_tiles of `p`; with `may_share` the K chunks of few tiles go to several
// clusters. Otherwise the tile height that pair_cost likes best: 256 rows, less where that fills the last wave better or brings more
// clusters to work on a narrow projection, or 256 with the last wave's tiles cut. The choice moves no sum: every element's inner dimension
// runs through as before. 7B shape: q/k/v of 2048 rows 141 -> 127 us (last wave in quarters), output and down projections of 1536 rows 50 -> 40 and
// 124 -> 95 (176 rows). Inside a step, from the end of the kernel before: d_model 1024, 896 rows 16.2 -> 10.4, 12.1 -> 8.5, gate+up 21.5 -> 17.1, down
// 20.2 -> 13.3; from the output to the down projection of a prompt's last row on the 7B shape 149 -> 97 (16 rows, a ring of eleven stages).
void plan_pair(PairGemmParams* p, int mode, bool may_share, int max_clusters = GP_MAX_CLUSTERS) {
  const int clusters = std::min(GP_MAX_CLUSTERS, max_clusters), tall = p->w_pairs * ((p->M + GP_NT - 1) / GP_NT);
  p->tile_rows = GP_NT; p->cut = 1;
  p->parts = may_share && p->runs == 0 ? pair_parts(p->plan_tiles ? p->plan_tiles : tall, p->KC, clusters) : 1;
  const float epilogue = mode == GP_RESIDUAL ? 0.0165f : 0.028f;
  if (p->runs > 0) {
    // a run an accumulator; where tensor memory holds one item's only, its epilogue is not under the next one's MMAs
    float best = 1e30f;
    for (int rows = std::min({GP_NT, (int)round_up(p->M, 16), 512 / p->runs / 16 * 16}); rows >= 16; rows -= 16) {
      const int tiles = p->w_pairs * ((p->M + rows - 1) / rows), bufs = 2 * p->runs * rows <= 512 ? 2 : 1;
      const float us = pair_cost(tiles, rows, 1, p->KC, clusters, epilogue) + (bufs == 1 ? (tiles - 1) / clusters * epilogue * rows : 0.f);
      if (us < 0.99f * best) { best = us; p->tile_rows = rows; p->run_bufs = bufs; }
    }
  } else if (p->parts == 1) {
    // Lower tiles take more bytes out of L2 for the same work, which a launch of several waves pays for in power, and with it in clock: they have to
    // look better by a tenth (1024 rows in tiles of 176 were 4% faster by themselves and slower in a step of 16 sequences).
    const int most = std::min(GP_NT, (int)round_up(p->M, 16));
    auto cost = [&](int rows, int cut) { return pair_cost(p->w_pairs * ((p->M + rows - 1) / rows), rows, cut, p->KC, clusters, epilogue); };
    float best = cost(most, 1);
    const float low = 0.9f * best;
    p->tile_rows = most;
    if (most == GP_NT)
      for (int cut = 2; cut <= 4; cut *= 2) {
        const float us = cost(most, cut);
        if (us < 0.98f * best) { best = us; p->cut = cut; }
      }
    for (int rows = most - 16; rows >= 16; rows -= 16) {
      const float us = cost(rows, 1);
      if (us < low && us < 0.99f * best) { best = us; p->tile_rows = rows; p->cut = 1; }
    }
  }
  p->m_tiles = (p->M + p->tile_rows - 1) / p->tile_rows;
  const int tiles = p->w_pairs * p->m_tiles;
  p->cut_first = p->cut > 1 ? tiles / clusters * clusters : tiles;
  if (p->cut_first == tiles) p->cut = 1;
  p->stages = PairCfg<GP_NT>::stages(p->tile_rows);
}
int pair_items(const PairGemmParams& p) { return p.parts > 1 ? p.w_pairs * p.m_tiles * p.parts : p.cut_first + (p.w_pairs * p.m_tiles - p.cut_first) * p.cut; }

template <int MODE>
cudaError_t launch_gp(cudaStream_t st, bool pdl, const PairTmaps& tm, const PairGemmParams& p, int max_clusters = GP_MAX_CLUSTERS) {
  static bool attr_set_dev[kAttrDevices] = {};
  bool& attr_set = *attr_flag(attr_set_dev);
  if (!attr_set) {
    cudaError_t e = cudaFuncSetAttribute(gemm_pair<MODE, GP_NT, GP_WHOLE>, cudaFuncAttributeMaxDynamicSharedMemorySize, PairCfg<GP_NT>::SMEM_BYTES);
    if constexpr (MODE != GP_PLAIN) {
      if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_pair<MODE, GP_NT, GP_SHARED>, cudaFuncAttributeMaxDynamicSharedMemorySize, PairCfg<GP_NT>::SMEM_BYTES);
      if (e == cudaSuccess) e = cudaFuncSetAttribute(gemm_pair<MODE, GP_NT, GP_RUNS>, cudaFuncAttributeMaxDynamicSharedMemorySize, PairCfg<GP_NT>::SMEM_BYTES);
    }
    if (e != cudaSuccess) return e;
    attr_set = true;
  }
  const int items = pair_items(p), grid = 2 * (p.parts > 1 ? items : std::min(items, std::min(GP_MAX_CLUSTERS, max_clusters)));
  auto kernel = gemm_pair<MODE, GP_NT, GP_WHOLE>;
  if constexpr (MODE != GP_PLAIN) {
    if (p.parts > 1) kernel = gemm_pair<MODE, GP_NT, GP_SHARED>;
    if (p.runs > 0) kernel = gemm_pair<MODE, GP_NT, GP_RUNS>;
  }
  return launch_k(pdl, kernel, dim3(grid), dim3(GP_THREADS), (size_t)PairCfg<GP_NT>::SMEM_BYTES, st, tm, p);
}

// x[M,K] * [mats]^T with the epilogue of `mode`; the caller has filled in the fields its mode uses.
int run_gemm_pair(spec_ctx* c, int mode, const void* x, int M, int K, int n_mats, const void* const* mats, const int* rows,
                  PairGemmParams* w, int kind) {
  PairTmaps tm{};
  w->M = M; w->KC = K / 64; w->n_mats = n_mats; w->packed = c->packed;
  const uint32_t box = mode == GP_SWIGLU ? 64 : 128;      // SwiGLU: 64 gate rows and 64 up rows make a CTA's tile
  int t0 = 0;
  for (int i = 0; i < n_mats; ++i) {
    const int t = (rows[i] + 127) / 128;
    w->mat_tile0[i] = t0;
    t0 += t;
    const CUtensorMap* ta = c->packed ? c->tmap(mats[i], (uint64_t)t * w->KC * 128, 64, box, true) : c->tmap(mats[i], rows[i], K, box);
    if (!ta) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (weights)");
    tm.a[i] = *ta;
  }
  for (int i = n_mats; i <= GS_MAX_MATS; ++i) w->mat_tile0[i] = t0;
  w->n_tiles = mode == GP_SWIGLU ? w->mat_tile0[1] : t0;
  w->w_pairs = mode == GP_SWIGLU ? w->n_tiles : (w->n_tiles + 1) / 2;
  const bool may_share = mode != GP_PLAIN && c->part_floats >= GP_PART_FLOATS;   // (a plain projection's sums go to the scratch)
  plan_pair(w, mode, may_share);
  w->part = c->d_part; w->arrive = c->d_pair_arrive;
  const CUtensorMap* tb = c->tmap(x, round_up(M, 16), K, w->tile_rows / 2);
  if (!tb) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (activations)");
  tm.b = *tb;
  if (w->cut > 1) {
    if (!(tb = c->tmap(x, round_up(M, 16), K, w->tile_rows / w->cut / 2))) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (activations)");
    tm.b_cut = *tb;
  }
  w->status = c->d_status; w->trace = c->next_trace(gemm_kind_name(kind));
  cudaError_t e;
  {
    ProfScope ps(c, kind);
    switch (mode) {
      case GP_RESIDUAL: e = launch_gp<GP_RESIDUAL>(c->stream, c->pdl, tm, *w); break;
      case GP_SWIGLU: e = launch_gp<GP_SWIGLU>(c->stream, c->pdl, tm, *w); break;
      case GP_ROPE: e = launch_gp<GP_ROPE>(c->stream, c->pdl, tm, *w); break;
      default: e = launch_gp<GP_PLAIN>(c->stream, c->pdl, tm, *w); break;
    }
    c->launches++;
  }
  if (e != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string("gemm_pair launch: ") + cudaGetErrorString(e));
  return SPEC_OK;
}

// ---- tensor-core linear (bf16): partial sums of x[M,K] * [mats]^T ----
// kind: SPEC_PROFILE_* of the call site. On success *view describes the partial sums.
int run_gemm(spec_ctx* c, const void* x, int M, int K, int n_mats, const void* const* mats, const int* rows, int kind,
             PartView* view) {
  GemmPlan g;
  int tiles_all = 0;
  for (int i = 0; i < n_mats; ++i) tiles_all += (rows[i] + 127) / 128;
  if (pair_gemm_ok(c, M, K)) {
    // many rows: the compute-bound kernel, whole tiles (one "slot" of finished sums)
    PairGemmParams w{};
    const long long total = (long long)tiles_all * ((M + GP_NT - 1) / GP_NT) * (K / 64);
    if ((size_t)M * tiles_all * 128 > c->part_floats) return c->fail(SPEC_E_NOMEM, "partial-sum scratch too small");
    if (total > 0x3fffffff || (total + 1) * (long long)(tiles_all * ((M + GP_NT - 1) / GP_NT)) >= 0x7fffffffLL) return c->fail(SPEC_E_BADARG, "unsupported linear shape");
    w.out = c->d_part; w.ld = (size_t)tiles_all * 128; w.n_cols = tiles_all * 128;
    int r = run_gemm_pair(c, GP_PLAIN, x, M, K, n_mats, mats, rows, &w, kind);
    if (r) return r;
    // the consumers see one finished slot per tile: a dealing of the units with one CTA per (weight tile, activation tile)
    PartView v{};
    v.part = c->d_part; v.slot_stride = (size_t)M * tiles_all * 128; v.ld = tiles_all * 128;
    v.seg.KC = K / 64; v.seg.m_tiles = (M + GP_NT - 1) / GP_NT; v.seg.G = w.n_tiles * v.seg.m_tiles; v.seg.total = (int)total;
    v.mt_shift = 8;
    v.single = 1;
    *view = v;
    return SPEC_OK;
  }
  if (!plan_gemm(M, K, n_mats, rows, stream_ctas(c, tiles_all), &g))
    return c->fail(SPEC_E_BADARG, "unsupported linear shape");
  if (plan_part_floats(g) > c->part_floats) return c->fail(SPEC_E_NOMEM, "partial-sum scratch too small");
  StreamTmaps tm{};
  for (int i = 0; i < n_mats; ++i) {
    if (c->packed) { g.p.packed[i] = static_cast<const uint8_t*>(mats[i]); continue; }
    const CUtensorMap* t = c->tmap(mats[i], rows[i], K, 128);
    if (!t) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (weights)");
    tm.a[i] = *t;
  }
  const CUtensorMap* tb = c->tmap(x, std::max<size_t>(round_up(M, 16), g.MT), K, g.MT);
  if (!tb) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (activations)");
  tm.b = *tb;
  g.p.part = c->d_part;
  g.p.slot_stride = (size_t)M * g.p.n_tiles * 128;
  g.p.l2_prefetch = c->l2_prefetch;
  g.p.status = c->d_status;
  g.p.trace = c->next_trace(gemm_kind_name(kind));
  {
    ProfScope ps(c, kind);
    cudaError_t e = launch_gs(c->stream, c->pdl, g, tm);
    c->launches++;
    if (e != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string("gemm_stream launch: ") + cudaGetErrorString(e));
  }
  *view = plan_view(g);
  return SPEC_OK;
}

// Can the cluster-reduced GEMM take this shape? One activation tile, and enough K chunks for every CTA
// of the cluster to get a run.
bool cluster_gemm_ok(const spec_ctx* c, int mode, int M, int K) {
  const int bit = mode == GC_RESIDUAL ? 1 : (mode == GC_SWIGLU ? 2 : 4);
  if (!(c->cluster_epilogue & bit) || M < 1 || M > 128 || K % 64) return false;
  const int KC = K / 64;
  if (mode == GC_RESIDUAL) return KC >= GC_RES_CLUSTER;
  // (gate+up of more than 64 rows keeps the weight streamer's split of the inner dimension, in gemm_glu where that is the same for all tiles, and of
  // fewer the clusters of three whatever the number of tiles: the split decides how the operands of the next projection round, and with
  // them which of two candidates that lie close comes first, that is, at which step a token is emitted.)
  if (mode == GC_SWIGLU) return KC >= 3 && M <= 64;
  return KC >= GC_ROPE_CLUSTER && (c->cfg.head_dim == 64 || c->cfg.head_dim == 128);
}

// x[M,N] += in[M,K] * W^T (GC_RESIDUAL, mats[0] = W), act_out[M,N] = bf16(SiLU(in W_g^T) * in W_u^T)
// (GC_SWIGLU, mats = gate, up) or q / cache rows of layer `layer` = RoPE(in [W_q; W_k; W_v]^T) (GC_ROPE, mats =
// q, k, v; rows = the pass's row bookkeeping; kv_alone: without q), finished inside the kernel. Caller checked cluster_gemm_ok.
int run_gemm_cluster(spec_ctx* c, int mode, const void* in, int M, int K, const void* const* mats, int N, float* x,
                     bf16* act_out, int kind, int layer = -1, const Rows* rows = nullptr, bool kv_alone = false) {
  const spec_config& f = c->cfg;
  const int MT = mt_for_rows(M), n_mats = mode == GC_RESIDUAL ? 1 : (mode == GC_SWIGLU ? 2 : 3);
  ClusterGemmParams p{};
  p.M = M; p.K = K; p.KC = K / 64; p.N = N;
  const int HD = f.n_heads * f.head_dim, KD = f.n_kv_heads * f.head_dim;
  StreamTmaps tm{};
  for (int i = 0; i < n_mats; ++i) {
    if (c->packed) { p.packed[i] = static_cast<const uint8_t*>(mats[i]); continue; }
    const int rws = mode == GC_ROPE ? (i == 0 ? HD : KD) : N;
    const CUtensorMap* t = c->tmap(mats[i], rws, K, 128);
    if (!t) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (weights)");
    tm.a[i] = *t;
  }
  const CUtensorMap* tb = c->tmap(in, round_up(M, 16), K, (uint32_t)round_up(M, 16));
  if (!tb) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (activations)");
  tm.b = *tb;
  p.x = x; p.ss_part = mode == GC_RESIDUAL ? c->d_ss_part : nullptr; p.act = act_out; p.status = c->d_status;
  int n_tiles = (N + 127) / 128;
  if (mode == GC_ROPE) {
    const int tq = (HD + 127) / 128, tk = (KD + 127) / 128;
    p.tile0[0] = 0; p.tile0[1] = tq; p.tile0[2] = tq + tk;
    p.tile_first = kv_alone ? tq : 0;
    n_tiles = (kv_alone ? 0 : tq) + 2 * tk;
    p.H = f.n_heads; p.layer = layer; p.rows = *rows; p.cs = c->d_rope; p.q = static_cast<bf16*>(c->d_q);
    p.pool = static_cast<bf16*>(c->d_pool); p.g = c->geom; p.page_table = c->d_page_table;
  }
  p.trace = c->next_trace(gemm_kind_name(kind));
  const int cs = mode == GC_SWIGLU ? GC_GLU_CLUSTER : mode == GC_ROPE ? GC_ROPE_CLUSTER : GC_RES_CLUSTER;
  cudaError_t e = cudaErrorInvalidValue;
  {
    ProfScope ps(c, kind);
    bool* as = c->gc_attr_set;
    if (mode == GC_RESIDUAL) {
      switch (MT) {
        case 16: e = launch_gc_mt<16, GC_RESIDUAL>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 0); break;
        case 32: e = launch_gc_mt<32, GC_RESIDUAL>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 1); break;
        case 64: e = launch_gc_mt<64, GC_RESIDUAL>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 2); break;
        default: e = launch_gc_mt<128, GC_RESIDUAL>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 3); break;
      }
    } else if (mode == GC_SWIGLU) {
      switch (MT) {
        case 16: e = launch_gc_mt<16, GC_SWIGLU>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 4); break;
        case 32: e = launch_gc_mt<32, GC_SWIGLU>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 5); break;
        default: e = launch_gc_mt<64, GC_SWIGLU>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 6); break;
      }
    } else {
      switch (MT) {
        case 16: e = launch_gc_mt<16, GC_ROPE>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 7); break;
        case 32: e = launch_gc_mt<32, GC_ROPE>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 8); break;
        case 64: e = launch_gc_mt<64, GC_ROPE>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 9); break;
        default: e = launch_gc_mt<128, GC_ROPE>(c->stream, c->pdl, n_tiles, cs, tm, p, as + 10); break;
      }
    }
    c->launches++;
  }
  if (e != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string("gemm_cluster launch: ") + cudaGetErrorString(e));
  return SPEC_OK;
}

// CTAs that share a (gate tile, up tile) pair in gemm_glu, 0 where the weight streamer and swiglu_reduce_tc serve: the streamer's plan has to cut the K chunks
// of every tile into the same runs (then it has no run that crosses a tile), at most eight, and all clusters have to fit the chip at one CTA
// an SM: a second wave would wait for the whole chain of the first.
int glu_cluster(const spec_ctx* c, int M, int K) {
  if (!(c->cluster_epilogue & 2) || M <= 64 || M > 128 || K % 64) return 0;
  const int F = c->cfg.d_ffn, tiles = 2 * ((F + 127) / 128), rows[2] = {F, F};
  GemmPlan g;
  if (!plan_gemm(M, K, 2, rows, stream_ctas(c, tiles), &g) || g.grid % tiles) return 0;
  const int cs = g.grid / tiles;
  return cs <= GLU_MAX_CLUSTER && tiles / 2 <= CLUSTERS_ALONE[cs] ? cs : 0;
}

int run_gemm_glu(spec_ctx* c, const void* in, int M, int K, int cs, const void* const* mats, bf16* act) {
  const int F = c->cfg.d_ffn, units = (K / 64 + cs - 1) / cs;
  GluGemmParams p{};
  StreamTmaps tm{};
  p.M = M; p.KC = K / 64; p.N = F; p.stages = std::min(units, GLU_MAX_STAGES); p.act = act; p.status = c->d_status;
  for (int i = 0; i < 2; ++i) {
    if (c->packed) { p.packed[i] = static_cast<const uint8_t*>(mats[i]); continue; }
    const CUtensorMap* t = c->tmap(mats[i], F, K, 128);
    if (!t) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (weights)");
    tm.a[i] = *t;
  }
  const CUtensorMap* tb = c->tmap(in, round_up(M, 16), K, (uint32_t)round_up(M, 16));
  if (!tb) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (activations)");
  tm.b = *tb;
  p.trace = c->next_trace(gemm_kind_name(SPEC_PROFILE_GATE_UP));
  static bool attr_set_dev[kAttrDevices] = {};
  bool& attr_set = *attr_flag(attr_set_dev);
  if (!attr_set) {
    CUDA_OK(cudaFuncSetAttribute(gemm_glu, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024));
    attr_set = true;
  }
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = dim3((F + 127) / 128 * cs); cfg.blockDim = dim3(GLU_THREADS); cfg.dynamicSmemBytes = (size_t)glu_smem_bytes(M, cs, p.stages); cfg.stream = c->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = cs; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = c->pdl ? 2 : 1;
  cudaError_t e;
  {
    ProfScope ps(c, SPEC_PROFILE_GATE_UP);
    e = cudaLaunchKernelEx(&cfg, gemm_glu, tm, p);
    c->launches++;
  }
  if (e != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string("gemm_glu launch: ") + cudaGetErrorString(e));
  return SPEC_OK;
}

#define KLAUNCH(name, kernel, grid, block, smem, ...)                                            \
  do {                                                                                         \
    cudaError_t e_ = launch_k(c->pdl, kernel, grid, block, smem, c->stream, __VA_ARGS__, c->next_trace(name)); \
    c->launches++;                                                                             \
    if (e_ != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string(name) + ": " + cudaGetErrorString(e_)); \
  } while (0)

// y[M, rows of all matrices] = x * [mats]^T on the CUDA cores, act = SiLU(x W_0^T) * (x W_1^T) (LR_SWIGLU, float32 y unused)
// or y += x * W_0^T (LR_RESIDUAL). ldy: row pitch of y.
// best (may be null): set to where each row's largest in every tile (every tiles-th piece of `piece` columns, `tile` of them in all) lies, if the kernel leaves them (in the buffer of the partial sums).
struct RowBest { float* val; int* idx; int tiles, tile, piece; };
template <typename T, int MODE>
int linear_simple(spec_ctx* c, const char* name, const T* x, int n_mats, const void* const* mats, const int* rows, float* y, size_t ldy, T* act,
                  int M, int K, RowBest* best = nullptr, const RopeStore<T>* rope = nullptr) {
  RowLinear<T> w{};
  w.n_mats = n_mats;
  int groups = 0;
  for (int i = 0; i < n_mats; ++i) {
    w.w[i] = static_cast<const T*>(mats[i]); w.rows[i] = rows[i]; w.group0[i] = groups;
    if (MODE != LR_SWIGLU) groups += (rows[i] + LR_N - 1) / LR_N;
  }
  if (MODE == LR_SWIGLU) groups = (rows[0] + LR_N / 2 - 1) / (LR_N / 2);
  const RowLinearShape sh = linear_rows_shape<T>(groups, M, K);
  if constexpr (std::is_same<T, float>::value && MODE == LR_PLAIN)
    if (n_mats == 1 && linear_held(sh, K)) {
      const HeldShape h = linear_held_shape(sh, M, rows[0]);
      RowBest at{};
      if (best && 2 * (size_t)M * h.grid.x <= c->part_floats)
        *best = at = RowBest{c->d_part, reinterpret_cast<int*>(c->d_part + (size_t)M * h.grid.x), (int)h.grid.x, (int)round_up(rows[0], h.piece * h.grid.x) / (int)h.grid.x, h.piece};
      KLAUNCH(name, (h.cols == 8 ? linear_rows_held<8, 4> : linear_rows_held<4, 8>), h.grid, dim3(LR_WARPS * 32), 0, x, w.w[0], y, ldy, M, rows[0], K, h.ms,
              at.val, at.idx);
      return SPEC_OK;
    }
  KLAUNCH(name, (linear_rows<T, MODE>), sh.grid, dim3(LR_WARPS * 32), 0, x, w, y, ldy, act, M, K, groups, sh.ks, sh.ms, rope ? *rope : RopeStore<T>{});
  return SPEC_OK;
}

// Passes with several 16-row blocks whose (sequence, head, row block) CTAs fit the SMs in one wave
// use the kernel that needs no merge across CTAs and no length-dependent launch shape. (A single row block, trees of at most 16 nodes,
// stays with the kernel that splits the keys: a step with 16 nodes, grouped heads of 64 and six layers takes 247 / 269 / 286 us at 500 /
// 1000 / 1900 positions with it and 207 / 225 / 257 without splits, but the other order of the sums rounds to other operands, and tokens
// were emitted at other steps.)
bool attn_rows_mode(const spec_ctx* c, int R, int groups) {
  const int nw = (R + 15) / 16;
  return nw > 1 && c->cfg.n_heads * groups * nw <= SM_SLOTS / 2;
}

// Context length from which a pass of R rows goes to the long-context kernels: the option's value, but at most
// ATTN_WAVES_KEYS for passes of more than 32 rows whose (sequence, head, 16-row block) CTAs do not fit one wave
// (batched verification): there the tcgen05 kernel, one CTA per (sequence, head, 64 rows), already wins.
constexpr int ATTN_WAVES_KEYS = 512;
int attn_long_threshold(const spec_ctx* c, int R, int groups) {
  const bool umma = c->attn_umma && c->tm_kv_ok && c->cfg.head_dim == 128;
  if (c->long_attn_keys > 0 && umma && R > 32 && !attn_rows_mode(c, R, groups)) return std::min(c->long_attn_keys, ATTN_WAVES_KEYS);
  return c->long_attn_keys;
}
// Passes of more than 32 rows (any pass with the tcgen05 kernel) over a context that may exceed that length.
bool attn_long_mode(const spec_ctx* c, int R, int groups, int keys_hi) {
  const bool umma = c->attn_umma && c->tm_kv_ok && c->cfg.head_dim == 128;
  const int thr = attn_long_threshold(c, R, groups);
  return thr > 0 && (R > 32 || umma) && keys_hi > thr;
}

// Key splits of the tcgen05 kernel = its cluster: one CTA per SM, at most a wave of them.
int attn_umma_splits(const spec_ctx* c, int R, int groups) {
  return std::max(1, std::min(std::min(c->nsplit_attn, AU_MAX_CLUSTER), (SM_SLOTS / 2) / (c->cfg.n_heads * groups)));
}
// First positions of a sequence that the attention kernel of such a pass may fetch ahead of its dependency wait, where they
// lie below the host's lower bound of the committed length. A bound beyond them makes no difference to the kernel.
int attn_fetch_ahead(const spec_ctx* c, int R, int groups, int keys_hi) {
  if (!c->tc) return 0;
  if (attn_long_mode(c, R, groups, keys_hi)) {
    if (c->attn_umma && c->tm_kv_ok && c->cfg.head_dim == 128) return 2 * attn_umma_splits(c, R, groups) * AU_KT;   // two tiles a split
    if (R > 32) return 0;
  }
  if (attn_rows_mode(c, R, groups)) return ATTN_ROWS_WARPS * ATTN_ROWS_BUFS * ATTN_ROWS_SUB;
  return keys_hi <= ATTN_SINGLE_TILES * 64 ? ATTN_STAGES * 64 : 0;
}

// Number of positions that a step's launches are planned for where a sequence may reach `keys` of them: the most with which
// launch_attention_tc takes the kernel and the launch shape that it takes for `keys`.
int attn_plan_bound(const spec_ctx* c, int R, int groups, int keys) {
  if (attn_long_mode(c, R, groups, keys)) return c->cap;                       // the long-context kernels: any length
  const bool may_get_long = attn_long_mode(c, R, groups, 1 << 30);
  const int below_long = may_get_long ? attn_long_threshold(c, R, groups) / 64 * 64 : c->cap;
  if (attn_rows_mode(c, R, groups)) return std::min(below_long, c->cap);       // a CTA per 16 rows: any length below the threshold
  const int single = ATTN_SINGLE_TILES * 64;                                   // one split of the keys up to here, several beyond
  if (keys <= single) return std::min(single, c->cap);
  return std::min(may_get_long ? std::max(below_long, single) : c->cap, c->cap);
}

// n_hi_pass / n_lo_pass: host bounds of the cached length the pass's rows sit on, per sequence
// (n_lo_pass may be null: nothing is fetched before the dependency wait).
// part: the groups of R rows that are computed, where they are not all of the pass's (the kernel and its splits are chosen for the whole
// pass, so that a row's sums do not depend on which rows are left out).
// len_now: the computed groups' lengths as well as the host knows them (what the longest-first order goes by).
int launch_attention_tc(spec_ctx* c, const Rows& pass, int l, const int* n_hi_pass, const int* n_lo_pass, const int* len_now, const Rows* part = nullptr) {
  const spec_config& f = c->cfg;
  const int H = f.n_heads, D = f.head_dim, R = pass.R, B = pass.B;
  const Rows& rows = part ? *part : pass;
  const int G = rows.B;                                          // groups computed
  AttnTcArgs a{};
  a.q = static_cast<const bf16*>(c->d_q); a.part_o = c->d_part_o; a.part_ml = c->d_part_ml;
  a.pool = static_cast<const bf16*>(c->d_pool); a.g = c->geom; a.page_table = c->d_page_table; a.rows = rows;
  a.layer = l; a.H = H; a.scale_log2 = 1.4426950408889634f / sqrtf((float)D);
  a.out = static_cast<bf16*>(c->d_attn); a.arrive = c->d_attn_arrive;
  a.status = c->d_status;
  int tiles_hi = 1;
  for (int b = 0; b < B; ++b) {
    tiles_hi = std::max(tiles_hi, (n_hi_pass[b] + R + 63) / 64);
    if (b < ATTN_MAX_SEQS) a.n_lo[b] = n_lo_pass ? n_lo_pass[b] : 0;
  }
  const int nw = (R + 15) / 16;
  if (attn_long_mode(c, R, B, tiles_hi * 64) && c->attn_umma && c->tm_kv_ok && D == 128) {
    // long contexts: scores and P V on tcgen05, a CTA per (head, 64 rows, key split)
    // passes of more than 64 rows (prompt chunks, trees of up to 128 nodes): a CTA takes 128 rows and reads the keys once for
    // them; 64 rows or fewer fill the 128-row MMAs twice, with two halves of the keys
    const bool tall = R > 64;
    if (G <= ATTN_MAX_SEQS) {
      int idx[ATTN_MAX_SEQS];
      for (int b = 0; b < G; ++b) idx[b] = b;
      std::stable_sort(idx, idx + G, [&](int x, int y) { return len_now[x] > len_now[y]; });
      for (int b = 0; b < G; ++b) a.order[b] = (unsigned char)idx[b];
    }
    // the key splits of a (sequence, head) are one cluster; without splits a CTA takes one (sequence, head) after another
    a.nsplit = attn_umma_splits(c, R, B);
    const dim3 grid = a.nsplit > 1 ? dim3(H, a.nsplit, G) : dim3(std::min(H * G, SM_SLOTS / 2), 1, 1);
    ProfScope ps_attn(c, SPEC_PROFILE_ATTENTION);
    static bool set_dev[kAttrDevices] = {};
    bool& set_ = *attr_flag(set_dev);
    if (!set_) {
      CUDA_OK(cudaFuncSetAttribute(attention_umma<128, 64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attention_umma_smem()));
      CUDA_OK(cudaFuncSetAttribute(attention_umma<128, 128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attention_umma_smem()));
      set_ = true;
    }
    cudaLaunchConfig_t cfg{};
    cfg.gridDim = grid; cfg.blockDim = dim3(AU_THREADS); cfg.dynamicSmemBytes = attention_umma_smem(); cfg.stream = c->stream;
    cudaLaunchAttribute at[2];
    int n_at = 0;
    if (a.nsplit > 1) {
      at[n_at].id = cudaLaunchAttributeClusterDimension;
      at[n_at].val.clusterDim.x = 1; at[n_at].val.clusterDim.y = (unsigned)a.nsplit; at[n_at].val.clusterDim.z = 1;
      ++n_at;
    }
    if (c->pdl) {
      at[n_at].id = cudaLaunchAttributeProgrammaticStreamSerialization;
      at[n_at].val.programmaticStreamSerializationAllowed = 1;
      ++n_at;
    }
    cfg.attrs = at; cfg.numAttrs = (unsigned)n_at;
    const CUtensorMap* tq = c->tmap(c->d_q, c->Mcap, (uint64_t)H * D, 64);
    if (!tq) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (query rows)");
    cudaError_t e_ = cudaLaunchKernelEx(&cfg, tall ? attention_umma<128, 128> : attention_umma<128, 64>, c->tm_kv, *tq, a, c->next_trace("attention_tc"));
    c->launches++;
    if (e_ != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string("attention_umma: ") + cudaGetErrorString(e_));
    return SPEC_OK;
  }
  if (attn_long_mode(c, R, B, tiles_hi * 64) && R > 32) {
    // long contexts, more than 32 rows: K/V tiles shared by the row blocks of a CTA, keys split across CTAs
    const int halves = (R + AS_RB * 16 - 1) / (AS_RB * 16);
    a.nsplit = std::max(1, std::min(c->nsplit_attn, (SM_SLOTS / 2) / (H * B * halves)));
    a.stages = AS_NB; a.split_tiles = AS_SPLIT_SUB;
    dim3 grid(H, a.nsplit, G * halves);
    ProfScope ps_attn(c, SPEC_PROFILE_ATTENTION);
    static bool set_dev[2][kAttrDevices] = {};
    bool& set_ = *attr_flag(set_dev[D == 128 ? 0 : 1]);
    if (D == 128) {
      if (!set_) { CUDA_OK(cudaFuncSetAttribute(attention_shared<128>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attention_shared_smem(128))); set_ = true; }
      KLAUNCH("attention_tc", (attention_shared<128>), grid, dim3(AS_RB * AS_KP * 32), attention_shared_smem(128), a);
    } else {
      if (!set_) { CUDA_OK(cudaFuncSetAttribute(attention_shared<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attention_shared_smem(64))); set_ = true; }
      KLAUNCH("attention_tc", (attention_shared<64>), grid, dim3(AS_RB * AS_KP * 32), attention_shared_smem(64), a);
    }
    return SPEC_OK;
  }
  if (attn_rows_mode(c, R, B)) {
    // few sequences: a CTA per (head, 16 query rows) walks the whole context, whatever its length
    a.nsplit = 1; a.stages = 2; a.split_tiles = 1;
    dim3 grid(H, nw, G);
    ProfScope ps_attn(c, SPEC_PROFILE_ATTENTION);
    if (D == 128) {
      static bool set_dev[kAttrDevices] = {};
      bool& set_ = *attr_flag(set_dev);
      if (!set_) { CUDA_OK(cudaFuncSetAttribute(attention_rows<128, ATTN_ROWS_WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attention_rows_smem(128, ATTN_ROWS_WARPS))); set_ = true; }
      KLAUNCH("attention_tc", (attention_rows<128, ATTN_ROWS_WARPS>), grid, dim3(ATTN_ROWS_WARPS * 32), attention_rows_smem(128, ATTN_ROWS_WARPS), a);
    } else {
      static bool set_dev[kAttrDevices] = {};
      bool& set_ = *attr_flag(set_dev);
      if (!set_) { CUDA_OK(cudaFuncSetAttribute(attention_rows<64, ATTN_ROWS_WARPS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attention_rows_smem(64, ATTN_ROWS_WARPS))); set_ = true; }
      KLAUNCH("attention_tc", (attention_rows<64, ATTN_ROWS_WARPS>), grid, dim3(ATTN_ROWS_WARPS * 32), attention_rows_smem(64, ATTN_ROWS_WARPS), a);
    }
    return SPEC_OK;
  }
  // more sequences: one CTA per (sequence, head) and KV split, all query rows. Short contexts (host
  // bound of at most ATTN_SINGLE_TILES tiles) get one split and no merge step; longer ones as many
  // split CTAs as fit beside each other, of which the kernel uses min(that, tiles / split_tiles)
  const int slots1 = attn_splits(c->nsplit_attn, H, B);
  a.nsplit = tiles_hi <= ATTN_SINGLE_TILES ? 1 : slots1;
  a.split_tiles = ATTN_SPLIT_TILES;
  a.stages = ATTN_STAGES;
  // With one split the query rows of a (sequence, head) go to several CTAs where there are SMs for them: a row's sums depend neither on the rows
  // beside it nor on who computes it, only on the key groups, and those go by all the rows of the pass. (32 heads of 128, 128 rows at 256
  // positions: 20.1 us a layer on 32 CTAs, 13.2 on 128.)
  a.row_parts = 1;
  if (a.nsplit == 1)
    while (nw > 2 * a.row_parts && H * G * a.row_parts * 2 <= SM_SLOTS / 2) a.row_parts *= 2;
  const int nwp = (nw + a.row_parts - 1) / a.row_parts;          // 16-row blocks of a CTA
  dim3 grid(H, a.nsplit, G * a.row_parts);
#define ATTN_CASE(HDV, NWV, KGV)                                                                         \
  {                                                                                                    \
    size_t sm = attention_tc_smem(HDV, NWV, a.stages);                                                 \
    static bool set_dev[kAttrDevices] = {};                                                            \
    bool& set_ = *attr_flag(set_dev);                                                                  \
    if (!set_) { CUDA_OK(cudaFuncSetAttribute(attention_tc<HDV, NWV, KGV>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)attention_tc_smem(HDV, NWV, ATTN_MAX_STAGES))); set_ = true; } \
    KLAUNCH("attention_tc", (attention_tc<HDV, NWV, KGV>), grid, dim3(NWV * KGV * 32), sm, a);         \
  }
  {
    // up to 64 rows: two key groups of warps per CTA; more rows: one
    ProfScope ps_attn(c, SPEC_PROFILE_ATTENTION);
    if (D == 128) {
      if (nw <= 1) ATTN_CASE(128, 1, 2) else if (nw <= 4 && nwp <= 2) ATTN_CASE(128, 2, 2) else if (nw <= 4) ATTN_CASE(128, 4, 2)
      else if (nwp <= 2) ATTN_CASE(128, 2, 1) else if (nwp <= 4) ATTN_CASE(128, 4, 1) else ATTN_CASE(128, 8, 1)
    } else {
      if (nw <= 1) ATTN_CASE(64, 1, 2) else if (nw <= 4 && nwp <= 2) ATTN_CASE(64, 2, 2) else if (nw <= 4) ATTN_CASE(64, 4, 2)
      else if (nwp <= 2) ATTN_CASE(64, 2, 1) else if (nwp <= 4) ATTN_CASE(64, 4, 1) else ATTN_CASE(64, 8, 1)
    }
  }
#undef ATTN_CASE
  return SPEC_OK;
}

// Of a prompt-processing pass, the last tokens of prompts that it holds: sequences [seq0, seq0 + count).
struct PromptEnds {
  int count, seq0;
  // device tables by sequence: row of the last token within its pass, its position, the sequence itself, 1; first position of the
  // token's chunk and the chunk's rows
  int *row, *pos, *seq, *one, *start, *cnt;
  const int* start_host;
  bool* pruned;                         // out: the last layer was computed for these rows alone, their results are in d_h_last / d_hq_last
};

// The rest of a prompt's last layer once its keys and values are stored: nobody reads the other rows' results, so only the last
// tokens go on, through the kernels that the whole pass of M rows would take: their attention with its chunk, the projections
// with the pass's sharing of the tiles, so that every sum is the whole pass's, bit for bit. On the 7B shape a whole layer takes 0.7 ms at 2304 rows and this
// 0.25 (the kernels that a pass of so few rows would take by itself, 0.09; but a first token's hidden state that rounds otherwise puts other
// candidates first).
int finish_prompt_ends(spec_ctx* c, const Rows& pass, const int* n_hi_pass, const PromptEnds& e) {
  const spec_config& f = c->cfg;
  const int G = e.count, d = f.d_model, F = f.d_ffn, HD = f.n_heads * f.head_dim, l = f.n_layers - 1, R = pass.R;
  if (G == 0) return SPEC_OK;
  const int m_tiles = (pass.B * R + GP_NT - 1) / GP_NT, d_pairs = ((d + 127) / 128 + 1) / 2;
  float* x = c->d_hid;
  bf16 *u = static_cast<bf16*>(c->d_u), *u_end = static_cast<bf16*>(c->d_hq), *act = static_cast<bf16*>(c->d_act), *attn_end = static_cast<bf16*>(c->d_q);
  KLAUNCH("gather_prompt_ends", gather_prompt_ends, dim3(G), dim3(256), 0, (const int*)(e.row + e.seq0), (const int*)(e.pos + e.seq0), (const float*)c->d_x,
          (const bf16*)u, x, u_end, c->d_n + e.seq0, d);
  int r;
  {
    Rows ends = make_rows(c, 1, true);
    ends.B = G; ends.seq = e.seq + e.seq0; ends.cnt = e.one;
    ends.tok = nullptr; ends.pos = ends.slot = ends.n = e.pos + e.seq0;
    const void* mats[1] = {c->wq[l]};
    const int rws[1] = {HD};
    PairGemmParams w{};
    w.plan_tiles = qkv_pairs(f) * m_tiles;
    w.H = f.n_heads; w.layer = l; w.rows = ends; w.cs = c->d_rope; w.q = static_cast<bf16*>(c->d_q); w.q_chunk = R;
    w.pool = static_cast<bf16*>(c->d_pool); w.g = c->geom; w.page_table = c->d_page_table;
    if ((r = run_gemm_pair(c, GP_ROPE, u_end, G, d, 1, mats, rws, &w, SPEC_PROFILE_QKV))) return r;
  }
  {
    // (of a chunk's other rows the queries are whatever is there: a row's scores and output depend on no other row)
    Rows chunks = pass;
    chunks.B = G; chunks.seq = e.seq + e.seq0; chunks.n = e.start + e.seq0; chunks.cnt = e.cnt + e.seq0;
    if ((r = launch_attention_tc(c, pass, l, n_hi_pass, nullptr, e.start_host + e.seq0, &chunks))) return r;
    KLAUNCH("gather_attention_ends", gather_attention_ends, dim3(G), dim3(256), 0, (const int*)(e.pos + e.seq0), static_cast<const bf16*>(c->d_attn), attn_end, R, HD);
  }
  {
    const void* mats[1] = {c->wo[l]};
    const int rws[1] = {d};
    PairGemmParams w{};
    w.plan_tiles = d_pairs * m_tiles; w.out = x; w.n_cols = d;
    if ((r = run_gemm_pair(c, GP_RESIDUAL, attn_end, G, HD, 1, mats, rws, &w, SPEC_PROFILE_WO))) return r;
  }
  KLAUNCH("norm_reduce_tc", norm_rows_wide<false>, dim3(G), dim3(NORMW_THREADS), 0, x, PartView{}, c->fn[l], f.rms_eps, u, (float*)nullptr, d);
  {
    const void* mats[2] = {c->wg[l], c->wu[l]};
    const int rws[2] = {F, F};
    PairGemmParams w{};
    w.plan_tiles = (F + 127) / 128 * m_tiles; w.act = act; w.n_cols = F;
    if ((r = run_gemm_pair(c, GP_SWIGLU, u, G, d, 2, mats, rws, &w, SPEC_PROFILE_GATE_UP))) return r;
  }
  {
    const void* mats[1] = {c->wd[l]};
    const int rws[1] = {d};
    PairGemmParams w{};
    w.plan_tiles = d_pairs * m_tiles; w.out = x; w.n_cols = d;
    if ((r = run_gemm_pair(c, GP_RESIDUAL, act, G, F, 1, mats, rws, &w, SPEC_PROFILE_DOWN))) return r;
  }
  KLAUNCH("norm_reduce_tc", norm_rows_wide<false>, dim3(G), dim3(NORMW_THREADS), 0, x, PartView{}, c->final_norm, f.rms_eps,
          static_cast<bf16*>(c->d_hq_last) + (size_t)e.seq0 * d, c->d_h_last + (size_t)e.seq0 * d, d);
  return SPEC_OK;
}

// Does the last layer of a prompt-processing pass go on with the prompts' last rows alone? Where the pass ends no prompt, always
// (its last layer then ends with the keys and values). Otherwise from 129 rows on: up to 128 the projections are bound by
// the weights, which cross memory either way, and the separate pass has one launch more.
bool prompt_ends_alone(const spec_ctx* c, int M, int G) {
  const spec_config& f = c->cfg;
  const int d = f.d_model, HD = f.n_heads * f.head_dim;
  if (G == 0) return pair_gemm_ok(c, M, d) || cluster_gemm_ok(c, GC_ROPE, M, d);
  return pair_gemm_ok(c, M, d) && pair_gemm_ok(c, M, HD) && pair_gemm_ok(c, M, f.d_ffn);
}

// act = SiLU(u W_g^T) * (u W_u^T) of layer l without the many-row kernel.
int gate_up_act(spec_ctx* c, const bf16* u, int M, int l, bf16* act) {
  const spec_config& f = c->cfg;
  const int d = f.d_model, F = f.d_ffn, up0 = (F + 127) / 128 * 128;             // padded column of the up projection in the partial sums
  const void* mats[2] = {c->wg[l], c->wu[l]};
  const int rws[2] = {F, F};
  if (cluster_gemm_ok(c, GC_SWIGLU, M, d)) return run_gemm_cluster(c, GC_SWIGLU, u, M, d, mats, F, nullptr, act, SPEC_PROFILE_GATE_UP);
  if (const int cs = glu_cluster(c, M, d)) return run_gemm_glu(c, u, M, d, cs, mats, act);
  PartView vg{};
  int r = run_gemm(c, u, M, d, 2, mats, rws, SPEC_PROFILE_GATE_UP, &vg);
  if (r) return r;
  int slots = 0;
  for (int t = 0; t < 2 * (up0 / 128) * vg.seg.m_tiles; ++t) slots = std::max(slots, vg.seg.nseg(t));
  if (slots <= 2) {
    KLAUNCH("swiglu_reduce_tc", swiglu_reduce_tc<SWIGLU_ROWS>, dim3((F / 4 + 255) / 256, (M + SWIGLU_ROWS - 1) / SWIGLU_ROWS), dim3(256), 0, vg, 0, up0, act, M, F);
  } else {
    KLAUNCH("swiglu_reduce_tc", swiglu_reduce_tc<1>, dim3((F / 4 + 255) / 256, M), dim3(256), 0, vg, 0, up0, act, M, F);
  }
  return SPEC_OK;
}

// ---- a lone prompt of two chunks ----
// Its sums are those of its chunks one after the other, through the projections that stream the weights (see prefill_t). Where those cut every inner dimension
// into a few runs, the same for a gate tile as for its up tile, both chunks go through the layers together: GP_RUNS adds the runs up in the
// same order, the norm makes the pieces' sums that the residual clusters leave, and the attention takes the kernel that a chunk by itself
// takes. The last layer goes on with the second chunk alone, from its attention output on with that chunk's own kernels.
// On the 7B shape a layer of 256 rows takes 165 us (q/k/v 36, attention 14, output 19, gate+up 49, down 40, norms 7), of two chunks by themselves 224: a prompt through
// four layers 1.03 -> 0.78 ms with the set-up, what bounds it being the chain of these kernels (weights 62 us, MMAs 65).
// Fills in how gate and up are dealt out; false: chunk by chunk.
bool two_chunks_at_once(const spec_ctx* c, SegMap* gate_up, int* gate_up_runs) {
  const spec_config& f = c->cfg;
  const int d = f.d_model, F = f.d_ffn, HD = f.n_heads * f.head_dim, R = PREFILL_ROWS, ft = (F + 127) / 128, rows[2] = {F, F};
  if (!c->tc || c->chunk_cap < 2 || !pair_gemm_ok(c, 2 * R, d) || !pair_gemm_ok(c, 2 * R, HD) || !pair_gemm_ok(c, 2 * R, F) || d > 16 * NORM_PIECES) return false;
  if (!cluster_gemm_ok(c, GC_ROPE, R, d) || !cluster_gemm_ok(c, GC_RESIDUAL, R, HD) || !cluster_gemm_ok(c, GC_RESIDUAL, R, F)) return false;
  if (attn_long_mode(c, R, 1, 2 * R)) return false;
  GemmPlan g;
  if (!plan_gemm(R, d, 2, rows, stream_ctas(c, 2 * ft), &g)) return false;
  const SegMap& s = g.p.seg;
  int most = 0;
  for (int t = 0; t < ft; ++t) {
    const int n = s.nseg(t), at = s.owner(t * s.KC), up = s.owner((t + ft) * s.KC);
    if (s.nseg(t + ft) != n) return false;
    for (int r = 1; r < n; ++r)
      if (s.lo(at + r) - t * s.KC != s.lo(up + r) - (t + ft) * s.KC) return false;
    most = std::max(most, n);
  }
  *gate_up = s; *gate_up_runs = most;
  return most <= 8;
}

int forward_two_chunks(spec_ctx* c, const Rows& both, int M, const SegMap& gate_up, int gate_up_runs) {
  const spec_config& f = c->cfg;
  const int d = f.d_model, F = f.d_ffn, H = f.n_heads, HD = H * f.head_dim, KD = f.n_kv_heads * f.head_dim, R = PREFILL_ROWS;
  bf16 *u = static_cast<bf16*>(c->d_u), *act = static_cast<bf16*>(c->d_act), *attn = static_cast<bf16*>(c->d_attn);
  Rows one = both;                           // a chunk by itself, which the attention's kernel is chosen for
  one.B = 1;
  const int cached[2] = {0, R};
  int r;
  for (int l = 0; l < f.n_layers; ++l) {
    if (l == 0) {
      KLAUNCH("norm_reduce_tc", norm_reduce_tc, dim3(M, NORM_CLUSTER), dim3(NORM_THREADS), 0, c->d_x, PartView{}, c->an[l], f.rms_eps, u, (float*)nullptr, d);
    } else {
      KLAUNCH("norm_reduce_tc", norm_pieces_tc, dim3(M), dim3(NORM_THREADS), 0, (const float*)c->d_x, c->an[l], f.rms_eps, u, d);
    }
    {
      const void* mats[3] = {c->wq[l], c->wk[l], c->wv[l]};
      const int rws[3] = {HD, KD, KD};
      PairGemmParams w{};
      w.runs = GC_ROPE_CLUSTER;
      w.H = H; w.layer = l; w.rows = both; w.cs = c->d_rope; w.q = static_cast<bf16*>(c->d_q);
      w.pool = static_cast<bf16*>(c->d_pool); w.g = c->geom; w.page_table = c->d_page_table;
      if ((r = run_gemm_pair(c, GP_ROPE, u, M, d, 3, mats, rws, &w, SPEC_PROFILE_QKV))) return r;
    }
    if ((r = launch_attention_tc(c, one, l, cached + 1, nullptr, cached, &both))) return r;
    if (l == f.n_layers - 1) break;
    {
      const void* mats[1] = {c->wo[l]};
      const int rws[1] = {d};
      PairGemmParams w{};
      w.runs = GC_RES_CLUSTER; w.out = c->d_x; w.n_cols = d;
      if ((r = run_gemm_pair(c, GP_RESIDUAL, attn, M, HD, 1, mats, rws, &w, SPEC_PROFILE_WO))) return r;
    }
    KLAUNCH("norm_reduce_tc", norm_pieces_tc, dim3(M), dim3(NORM_THREADS), 0, (const float*)c->d_x, c->fn[l], f.rms_eps, u, d);
    {
      const void* mats[2] = {c->wg[l], c->wu[l]};
      const int rws[2] = {F, F};
      PairGemmParams w{};
      w.runs = gate_up_runs; w.seg = gate_up; w.act = act; w.n_cols = F;
      if ((r = run_gemm_pair(c, GP_SWIGLU, u, M, d, 2, mats, rws, &w, SPEC_PROFILE_GATE_UP))) return r;
    }
    {
      const void* mats[1] = {c->wd[l]};
      const int rws[1] = {d};
      PairGemmParams w{};
      w.runs = GC_RES_CLUSTER; w.out = c->d_x; w.n_cols = d;
      if ((r = run_gemm_pair(c, GP_RESIDUAL, act, M, F, 1, mats, rws, &w, SPEC_PROFILE_DOWN))) return r;
    }
  }
  // the second chunk's rows, whole
  const int l = f.n_layers - 1, n_ss = ((d + 127) / 128) * GC_RES_CLUSTER;
  float* x = c->d_x + (size_t)R * d;
  {
    const void* mats[1] = {c->wo[l]};
    if ((r = run_gemm_cluster(c, GC_RESIDUAL, attn + (size_t)R * HD, R, HD, mats, d, x, nullptr, SPEC_PROFILE_WO))) return r;
  }
  KLAUNCH("norm_reduce_tc", norm_scaled_tc, dim3(R, NORM_CLUSTER), dim3(NORM_THREADS), 0, (const float*)x, (const float*)c->d_ss_part, n_ss, c->fn[l], f.rms_eps, u, (float*)nullptr, d);
  if ((r = gate_up_act(c, u, R, l, act))) return r;
  {
    const void* mats[1] = {c->wd[l]};
    if ((r = run_gemm_cluster(c, GC_RESIDUAL, act, R, F, mats, d, x, nullptr, SPEC_PROFILE_DOWN))) return r;
  }
  KLAUNCH("norm_reduce_tc", norm_scaled_tc, dim3(R, NORM_CLUSTER), dim3(NORM_THREADS), 0, (const float*)x, (const float*)c->d_ss_part, n_ss, c->final_norm, f.rms_eps,
          static_cast<bf16*>(c->d_hq), c->d_hid, d);
  return SPEC_OK;
}

// One pass of the base model over M = groups * R rows whose tokens/positions/slots are prepared and
// whose embeddings are in d_x: bf16 tensor-core path. Leaves the final hidden state in d_hid
// (float32) and d_hq (bf16). ends: of a prompt-processing pass, else null.
int forward_layers_tc(spec_ctx* c, const Rows& rows, const int* n_hi_pass, const int* n_lo_pass, const int* len_now, const PromptEnds* ends) {
  const spec_config& f = c->cfg;
  const int M = rows.B * rows.R, d = f.d_model, F = f.d_ffn, H = f.n_heads, D = f.head_dim, HD = H * D, KD = f.n_kv_heads * D;
  bf16* u = static_cast<bf16*>(c->d_u);
  bf16* act = static_cast<bf16*>(c->d_act);
  const int kp0 = (HD + 127) / 128 * 128, vp0 = kp0 + (KD + 127) / 128 * 128;   // padded columns of k and v in the QKV partials
  // (passes of more than 128 rows are bound by bandwidth, not by a row's latency: one plain CTA per row)
  // (after a residual cluster epilogue the pieces' sums of squares exist already: ss_ready)
  bool ss_ready = false;
  const int n_ss = ((d + 127) / 128) * GC_RES_CLUSTER;
#define NORM_LAUNCH(pv, gain, uq, hid)                                                                   \
  if (ss_ready && M <= 128) {                                                                            \
    KLAUNCH("norm_reduce_tc", norm_scaled_tc, dim3(M, NORM_CLUSTER), dim3(NORM_THREADS), 0, (const float*)c->d_x, (const float*)c->d_ss_part, n_ss, gain, f.rms_eps, uq, hid, d); \
  } else if (M > 128) {                                                                                         \
    if (pv.part) {                                                                                       \
      KLAUNCH("norm_reduce_tc", norm_rows_wide<true>, dim3(M), dim3(NORMW_THREADS), 0, c->d_x, pv, gain, f.rms_eps, uq, hid, d); \
    } else {                                                                                             \
      KLAUNCH("norm_reduce_tc", norm_rows_wide<false>, dim3(M), dim3(NORMW_THREADS), 0, c->d_x, pv, gain, f.rms_eps, uq, hid, d); \
    }                                                                                                    \
  } else {                                                                                               \
    KLAUNCH("norm_reduce_tc", norm_reduce_tc, dim3(M, NORM_CLUSTER), dim3(NORM_THREADS), 0, c->d_x, pv, gain, f.rms_eps, uq, hid, d); \
  }
  PartView pend{};              // partial sums of the previous down-projection still to be added to x
  for (int l = 0; l < f.n_layers; ++l) {
    NORM_LAUNCH(pend, c->an[l], u, (float*)nullptr);
    int r;
    {
      const void* mats[3] = {c->wq[l], c->wk[l], c->wv[l]};
      int rws[3] = {HD, KD, KD};
      const bool kv_alone = ends && l == f.n_layers - 1 && prompt_ends_alone(c, M, ends->count);
      if (pair_gemm_ok(c, M, d)) {
        PairGemmParams w{};
        w.kind0 = kv_alone; w.plan_tiles = qkv_pairs(f) * ((M + GP_NT - 1) / GP_NT);
        w.H = H; w.layer = l; w.rows = rows; w.cs = c->d_rope; w.q = static_cast<bf16*>(c->d_q);
        w.pool = static_cast<bf16*>(c->d_pool); w.g = c->geom; w.page_table = c->d_page_table;
        if ((r = run_gemm_pair(c, GP_ROPE, u, M, d, 3 - w.kind0, mats + w.kind0, rws + w.kind0, &w, SPEC_PROFILE_QKV))) return r;
      } else if (cluster_gemm_ok(c, GC_ROPE, M, d)) {
        // the clusters rotate q and k and store q and the cache rows themselves
        if ((r = run_gemm_cluster(c, GC_ROPE, u, M, d, mats, 0, nullptr, nullptr, SPEC_PROFILE_QKV, l, &rows, kv_alone))) return r;
      } else {
        PartView vq{};
        if ((r = run_gemm(c, u, M, d, 3, mats, rws, SPEC_PROFILE_QKV, &vq))) return r;
        KLAUNCH("rope_store_tc", rope_store_tc, dim3(M, M <= 128 ? 8 : 2), dim3(256), 0, vq, 0, kp0, vp0, rows, c->d_rope,
                static_cast<bf16*>(c->d_q), static_cast<bf16*>(c->d_pool), c->geom, c->d_page_table, l, H);
      }
    }
    if (ends && l == f.n_layers - 1 && prompt_ends_alone(c, M, ends->count)) {
      *ends->pruned = true;
      return finish_prompt_ends(c, rows, n_hi_pass, *ends);
    }
    if ((r = launch_attention_tc(c, rows, l, n_hi_pass, n_lo_pass, len_now))) return r;
    PartView vo{};
    {
      const void* mats[1] = {c->wo[l]};
      int rws[1] = {d};
      if (pair_gemm_ok(c, M, HD)) {
        PairGemmParams w{};
        w.out = c->d_x; w.n_cols = d;
        if ((r = run_gemm_pair(c, GP_RESIDUAL, c->d_attn, M, HD, 1, mats, rws, &w, SPEC_PROFILE_WO))) return r;
      } else if (cluster_gemm_ok(c, GC_RESIDUAL, M, HD)) {
        // the cluster adds its split-K sums and the residual stream itself: nothing left for the norm kernel to add
        if ((r = run_gemm_cluster(c, GC_RESIDUAL, c->d_attn, M, HD, mats, d, c->d_x, nullptr, SPEC_PROFILE_WO))) return r;
        ss_ready = true;
      } else {
        ss_ready = false;
        if ((r = run_gemm(c, c->d_attn, M, HD, 1, mats, rws, SPEC_PROFILE_WO, &vo))) return r;
      }
    }
    NORM_LAUNCH(vo, c->fn[l], u, (float*)nullptr);
    {
      const void* mats[2] = {c->wg[l], c->wu[l]};
      int rws[2] = {F, F};
      if (pair_gemm_ok(c, M, d)) {
        PairGemmParams w{};
        w.act = act; w.n_cols = F;
        if ((r = run_gemm_pair(c, GP_SWIGLU, u, M, d, 2, mats, rws, &w, SPEC_PROFILE_GATE_UP))) return r;
      } else if ((r = gate_up_act(c, u, M, l, act))) {
        return r;
      }
    }
    {
      const void* mats[1] = {c->wd[l]};
      int rws[1] = {d};
      pend = PartView{};
      if (pair_gemm_ok(c, M, F)) {
        PairGemmParams w{};
        w.out = c->d_x; w.n_cols = d;
        if ((r = run_gemm_pair(c, GP_RESIDUAL, act, M, F, 1, mats, rws, &w, SPEC_PROFILE_DOWN))) return r;
      } else if (cluster_gemm_ok(c, GC_RESIDUAL, M, F)) {
        if ((r = run_gemm_cluster(c, GC_RESIDUAL, act, M, F, mats, d, c->d_x, nullptr, SPEC_PROFILE_DOWN))) return r;
        ss_ready = true;
      } else {
        ss_ready = false;
        if ((r = run_gemm(c, act, M, F, 1, mats, rws, SPEC_PROFILE_DOWN, &pend))) return r;
      }
    }
  }
  NORM_LAUNCH(pend, c->final_norm, static_cast<bf16*>(c->d_hq), c->d_hid);
#undef NORM_LAUNCH
  return SPEC_OK;
}

template <typename T, int EPL, int ROWS>
int launch_attention_plain_rows(spec_ctx* c, const Rows& rows, int l) {
  static bool set_dev[kAttrDevices] = {};
  bool& set_ = *attr_flag(set_dev);
  const size_t sm = attention_plain_smem(EPL * 32);
  if (!set_) { CUDA_OK(cudaFuncSetAttribute(attention_plain<T, EPL, ROWS>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm)); set_ = true; }
  KLAUNCH("attention_plain", (attention_plain<T, EPL, ROWS>), dim3(c->cfg.n_heads, rows.B, (rows.R + ROWS - 1) / ROWS), dim3(AP_WARPS * 32), sm,
          static_cast<const T*>(c->d_q), static_cast<T*>(c->d_attn), static_cast<const T*>(c->d_pool), c->geom, (const int*)c->d_page_table, rows, l,
          c->cfg.n_heads, 1.0f / sqrtf((float)c->cfg.head_dim));
  return SPEC_OK;
}
template <typename T, int EPL>
int launch_attention_plain(spec_ctx* c, const Rows& rows, int l) {
  // several warps a row while the SMs take all of the CTAs that makes at once, a warp a row beyond (each CTA stages its head's keys and values for itself)
  const bool few = (long long)c->cfg.n_heads * rows.B * ((rows.R + AP_FEW - 1) / AP_FEW) <= 2 * 148;
  return few ? launch_attention_plain_rows<T, EPL, AP_FEW>(c, rows, l) : launch_attention_plain_rows<T, EPL, AP_WARPS>(c, rows, l);
}

// The same pass with the plain CUDA-core kernels (float32 configurations and the bf16 debug mode).
template <typename T>
int forward_layers(spec_ctx* c, const Rows& rows, const int* n_hi_pass, const int* n_lo_pass, const int* len_now, const PromptEnds* ends = nullptr) {
  if (c->tc) return forward_layers_tc(c, rows, n_hi_pass, n_lo_pass, len_now, ends);
  const spec_config& f = c->cfg;
  const int R = rows.R, M = rows.B * R, d = f.d_model, F = f.d_ffn, H = f.n_heads, D = f.head_dim, HD = H * D, KD = f.n_kv_heads * D;
  T* u = static_cast<T*>(c->d_u);
  T* q = static_cast<T*>(c->d_q);
  T* attn = static_cast<T*>(c->d_attn);
  T* act = static_cast<T*>(c->d_act);
  T* pool = static_cast<T*>(c->d_pool);
  for (int l = 0; l < f.n_layers; ++l) {
    int r;
    KLAUNCH("rmsnorm_rows", rmsnorm_rows<T>, dim3(M), dim3(256), 0, (const float*)c->d_x, c->an[l], f.rms_eps, u, (float*)nullptr, d);
    {
      const void* mats[3] = {c->wq[l], c->wk[l], c->wv[l]};
      const int rws[3] = {HD, KD, KD};
      const RopeStore<T> rs{rows, c->d_rope, q, pool, c->geom, c->d_page_table, l, H};
      if ((r = linear_simple<T, LR_ROPE>(c, "linear_qkv", u, 3, mats, rws, nullptr, 0, nullptr, M, d, nullptr, &rs))) return r;
    }
    switch (D / 32) {
      case 1: r = launch_attention_plain<T, 1>(c, rows, l); break;
      case 2: r = launch_attention_plain<T, 2>(c, rows, l); break;
      case 3: r = launch_attention_plain<T, 3>(c, rows, l); break;
      case 4: r = launch_attention_plain<T, 4>(c, rows, l); break;
      case 5: r = launch_attention_plain<T, 5>(c, rows, l); break;
      case 6: r = launch_attention_plain<T, 6>(c, rows, l); break;
      case 7: r = launch_attention_plain<T, 7>(c, rows, l); break;
      default: r = launch_attention_plain<T, 8>(c, rows, l); break;
    }
    if (r) return r;
    {
      const void* mats[1] = {c->wo[l]};
      if ((r = linear_simple<T, LR_RESIDUAL>(c, "linear_wo", attn, 1, mats, &d, c->d_x, d, nullptr, M, HD))) return r;
    }
    KLAUNCH("rmsnorm_rows", rmsnorm_rows<T>, dim3(M), dim3(256), 0, (const float*)c->d_x, c->fn[l], f.rms_eps, u, (float*)nullptr, d);
    {
      const void* mats[2] = {c->wg[l], c->wu[l]};
      const int rws[2] = {F, F};
      if ((r = linear_simple<T, LR_SWIGLU>(c, "linear_gate_up", u, 2, mats, rws, nullptr, 0, act, M, d))) return r;
    }
    {
      const void* mats[1] = {c->wd[l]};
      if ((r = linear_simple<T, LR_RESIDUAL>(c, "linear_down", act, 1, mats, &d, c->d_x, d, nullptr, M, F))) return r;
    }
  }
  // final norm: hidden (float32) and its operand-typed copy
  KLAUNCH("rmsnorm_rows", rmsnorm_rows<T>, dim3(M), dim3(256), 0, (const float*)c->d_x, c->final_norm, f.rms_eps, static_cast<T*>(c->d_hq), c->d_hid, d);
  return SPEC_OK;
}

// A [rows][ld] matrix of finished float32 values seen as one slot of partial sums.
PartView plain_view(const float* p, int rows, int ld) {
  PartView v{};
  v.part = p; v.slot_stride = (size_t)rows * ld; v.ld = ld;
  v.seg.KC = 1; v.seg.m_tiles = 1; v.seg.G = v.seg.total = (ld + 127) / 128;
  v.mt_shift = 30;                     // all rows are one activation tile
  v.single = 1;
  return v;
}

// Per-head top-k over the logits of `rows` (sequence, head) rows from `row0` on into the candidate table.
int heads_top_k(spec_ctx* c, const PartView& pl, int row0, int rows, const int* ov) {
  const int kmax = c->kmax, V = c->cfg.vocab;
  // the row's last-arriving CTA merges the slices' lists: no merge kernel
  // about 296 CTAs whatever the number of rows, and up to 1024 while that is at most 16 a row (64 rows with four slices each left the SMs at
  // two CTAs: 27 us, now 21): more slices would only lengthen the lists to merge (and at least as many as let a slice fit 40 KB)
  const int want = std::min(c->topk_blocks, std::max(std::max(std::max(4, std::min(16, 1024 / rows)), (V + 10239) / 10240), SM_SLOTS / rows));
  const int slice = (int)round_up((V + want - 1) / want, 4), blocks = (V + slice - 1) / slice;
  const size_t sm_topk = std::max((size_t)slice * sizeof(float), (size_t)blocks * kmax * 8);
  if (sm_topk > 44 * 1024) return c->fail(SPEC_E_BADARG, "top-k lists do not fit the merge's shared memory");
  KLAUNCH("topk_slices_tc", topk_slices_tc, dim3(blocks, rows), dim3(256), sm_topk,
          pl, V, row0, slice, kmax, c->d_pk_val, c->d_pk_idx, c->d_row_arrive, c->K, (const int*)c->d_root, ov, c->d_cand);
  return SPEC_OK;
}

// lm_head over up to 128 rows with its sums finished in the kernel (0: this shape goes to the weight streamer).
int lm_head_cluster(const spec_ctx* c, int M) {
  return c->tc && M <= 128 ? plain_cluster((c->cfg.vocab + 127) / 128, c->cfg.d_model / 64, SM_SLOTS) : 0;
}
// y (may be null): [M][ldy] logits; best_val / best_idx (may be null): [M][tiles] each row's largest in each tile of 128 tokens.
int run_lm_head(spec_ctx* c, const void* x, int M, int cluster, float* y, size_t ldy, float* best_val, int* best_idx) {
  const int V = c->cfg.vocab, d = c->cfg.d_model, MT = mt_for_rows(M);
  ClusterGemmParams p{};
  StreamTmaps tm{};
  p.M = M; p.K = d; p.KC = d / 64; p.N = V; p.y = y; p.ldy = ldy; p.best_val = best_val; p.best_idx = best_idx; p.status = c->d_status;
  if (c->packed) {
    p.packed[0] = static_cast<const uint8_t*>(c->lm_head);
  } else {
    const CUtensorMap* t = c->tmap(c->lm_head, V, d, 128);
    if (!t) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (weights)");
    tm.a[0] = *t;
  }
  const CUtensorMap* tb = c->tmap(x, round_up(M, 16), d, (uint32_t)round_up(M, 16));
  if (!tb) return c->fail(SPEC_E_CUDA, "cuTensorMapEncodeTiled failed (activations)");
  tm.b = *tb;
  p.trace = c->next_trace(gemm_kind_name(SPEC_PROFILE_OFF));
  cudaError_t e = launch_gc_plain(c->stream, c->pdl, (V + 127) / 128, cluster, tm, p);
  c->launches++;
  if (e != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string("gemm_cluster launch: ") + cudaGetErrorString(e));
  return SPEC_OK;
}

// Extra decoding heads on the tensor cores: residual blocks (head matrices stacked along the
// output dimension, up to four per launch), shared lm_head, per-head top-k.
int heads_tc(spec_ctx* c, const int* ov) {
  const spec_config& f = c->cfg;
  const int B = c->B, K = c->K, d = f.d_model, rows_total = B * K;
  const int dpad = (d + 127) / 128 * 128;
  for (int k0 = 0; k0 < K; k0 += GS_MAX_MATS) {
    const int nk = std::min(GS_MAX_MATS, K - k0);
    const void* mats[GS_MAX_MATS];
    int rws[GS_MAX_MATS];
    for (int i = 0; i < nk; ++i) { mats[i] = c->mw[k0 + i]; rws[i] = d; }
    PartView pv{};
    int r = run_gemm(c, c->d_hq_last, B, d, nk, mats, rws, SPEC_PROFILE_OFF, &pv);
    if (r) return r;
    KLAUNCH("medusa_act_tc", medusa_act_tc, dim3(B * nk, 4), dim3(256), 0, pv, dpad, (const bf16*)c->d_hq_last,
            reinterpret_cast<const bf16* const*>(c->d_mb), static_cast<bf16*>(c->d_r), K, k0, nk, d);
  }
  PartView pl{};
  if (const int cs = lm_head_cluster(c, rows_total)) {
    const int ldz = (int)round_up(f.vocab, 4);                  // (fits: partial sums of this shape would be rows of whole tiles)
    const int tiles = (f.vocab + 127) / 128;
    // (the logits and behind them the tiles' maxima: partial sums of this shape would be rows of whole tiles, in two slots at least)
    float* val = c->d_part + (size_t)rows_total * ldz;
    int* idx = reinterpret_cast<int*>(val + (size_t)rows_total * tiles);
    const bool maxima = tiles >= c->kmax && tiles <= TOPK_MAX_TILES && (size_t)rows_total * (ldz + 2 * (size_t)tiles) <= c->part_floats;
    int r = run_lm_head(c, c->d_r, rows_total, cs, c->d_part, ldz, maxima ? val : nullptr, maxima ? idx : nullptr);
    if (r) return r;
    if (maxima) {
      KLAUNCH("topk_tiles", topk_tiles, dim3(rows_total), dim3(256), 0, (const float*)c->d_part, ldz, (const float*)val, (const int*)idx, tiles, 128, 128, f.vocab, c->kmax, K,
              (const int*)c->d_root, ov, c->d_cand);
      return SPEC_OK;
    }
    pl = plain_view(c->d_part, rows_total, ldz);
  } else {
    const void* mats[1] = {c->lm_head};
    int rws[1] = {f.vocab};
    int r = run_gemm(c, c->d_r, rows_total, d, 1, mats, rws, SPEC_PROFILE_OFF, &pl);
    if (r) return r;
  }
  return heads_top_k(c, pl, 0, rows_total, ov);
}

// lm_head over `M` operand rows at `src`, leaving per-row argmax partials (and logits).
template <typename T>
int lm_head_argmax(spec_ctx* c, const T* src, int M) {
  const spec_config& f = c->cfg;
  PartView pl{};
  const void* mats[1] = {c->lm_head};
  int rws[1] = {f.vocab};
  if (const int cs = lm_head_cluster(c, M)) {
    // a tile's largest of every row comes out of the projection; the tiles' are compared here (behind partial sums, whose consumer has to read
    // 16 MB, the two steps took 12.6 us after the projection on the 7B shape with 64 rows)
    const int tiles = (f.vocab + 127) / 128;
    float* val = c->d_part;
    int* idx = reinterpret_cast<int*>(val + (size_t)M * tiles);
    int r = run_lm_head(c, src, M, cs, c->keep_logits ? c->d_logits : nullptr, f.vocab, val, idx);
    if (r) return r;
    KLAUNCH("argmax_tiles", argmax_tiles, dim3((M + 7) / 8), dim3(256), 0, (const float*)val, (const int*)idx, M, tiles, c->d_pval2, c->d_pidx2);
    return SPEC_OK;
  }
  if (c->tc && pair_gemm_ok(c, M, f.d_model)) {
    // (the same with the projection of many rows, whose logits nobody else needs: written and read back they were 131 MB and a
    // kernel of 53 us behind 195 for 16 sequences of 64 rows; now 14 behind 202)
    const int slots = 4 * ((f.vocab + 127) / 128);
    PairGemmParams w{};
    w.out = c->keep_logits ? c->d_logits : nullptr; w.ld = (size_t)f.vocab; w.n_cols = f.vocab;
    w.best_val = c->d_part; w.best_idx = reinterpret_cast<int*>(c->d_part + (size_t)slots * M);
    int r = run_gemm_pair(c, GP_PLAIN, src, M, f.d_model, 1, mats, rws, &w, SPEC_PROFILE_OFF);
    if (r) return r;
    KLAUNCH("argmax_slots", argmax_slots, dim3((M + 31) / 32), dim3(1024), 0, (const float*)w.best_val, (const int*)w.best_idx, M, slots, c->d_pval2, c->d_pidx2);
    return SPEC_OK;
  }
  if (c->tc) {
    int r = run_gemm(c, src, M, f.d_model, 1, mats, rws, SPEC_PROFILE_OFF, &pl);
    if (r) return r;
  } else {
    RowBest best{};
    int r = linear_simple<T, LR_PLAIN>(c, "linear_lm_head", src, 1, mats, rws, c->d_logits, f.vocab, nullptr, M, f.d_model, &best);
    if (r) return r;
    if (best.val) {
      KLAUNCH("argmax_tiles", argmax_tiles, dim3((M + 7) / 8), dim3(256), 0, (const float*)best.val, (const int*)best.idx, M, best.tiles, c->d_pval2, c->d_pidx2);
      return SPEC_OK;
    }
    pl = plain_view(c->d_logits, M, f.vocab);
  }
  KLAUNCH("argmax_partials_tc", argmax_partials_tc, dim3(M, c->n_argmax), dim3(256), 0, pl, f.vocab,
          c->tc && c->keep_logits ? c->d_logits : (float*)nullptr, c->d_pval, c->d_pidx, c->d_row_arrive, c->d_pval2, c->d_pidx2);
  return SPEC_OK;
}

AcceptArgs make_accept(spec_ctx* c, int R, int mode) {
  AcceptArgs a{};
  a.rows = make_rows(c, R, false);
  a.pidx = c->d_pidx2;
  a.hq_last = c->tc ? static_cast<bf16*>(c->d_hq_last) : nullptr;
  a.parent = c->d_parent; a.depth = c->d_depth; a.edge_ok = nullptr;
  a.K = c->K; a.frag_token = c->cfg.frag_token; a.d = c->cfg.d_model; a.mode = mode;
  a.hid = c->d_hid; a.am = c->d_am; a.path = c->d_path; a.count = c->d_count; a.out_tok = c->d_out_tok;
  a.n_old = c->d_n_old; a.root_tok = c->d_root; a.h_last = c->d_h_last;
  a.gen_log = c->d_gen_log; a.gen_cnt = c->d_gen_cnt; a.gen_cap = c->gen_cap;
  a.status = c->d_status; a.host_status = c->h_result_dev;
  return a;
}

int report_status(spec_ctx* c, const int* st) {
  if (st[0] == ST_OK) return SPEC_OK;
  char buf[128];
  snprintf(buf, sizeof(buf), "device status %d at %d (detail %d)", st[0], st[1], st[2]);
  return c->fail(st[0] == ST_TIMEOUT ? SPEC_E_TIMEOUT : (st[0] == ST_SEQLEN ? SPEC_E_SEQLEN : SPEC_E_BADARG), buf);
}

int check_status(spec_ctx* c) {
  cudaError_t e = cudaMemcpyAsync(c->h_result, c->d_status, 4 * sizeof(int), cudaMemcpyDeviceToHost, c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) return c->fail(SPEC_E_CUDA, std::string("status read: ") + cudaGetErrorString(e));
  return report_status(c, c->h_result);
}

// Waits for a stream at the end of its scope, unless that has been done.
struct StreamWait {
  cudaStream_t st;
  bool through = false;
  ~StreamWait() { if (!through) cudaStreamSynchronize(st); }
};

template <typename T>
int prefill_t(spec_ctx* c, int batch, const int32_t* tokens, const int32_t* offsets) {
  const spec_config& f = c->cfg;
  int maxlen = 0;
  for (int b = 0; b < batch; ++b) {
    int len = offsets[b + 1] - offsets[b];
    if (len < 1) return c->fail(SPEC_E_BADARG, "empty prompt");
    if (len + c->K + 1 > f.max_seq) return c->fail(SPEC_E_SEQLEN, "prompt leaves no room to generate within max_seq");
    if (offsets[b + 1] - offsets[0] > batch * f.max_seq) return c->fail(SPEC_E_SEQLEN, "prompts exceed the prompt buffer");
    maxlen = std::max(maxlen, len);
  }
  c->B = batch;
  c->prefilled = false;
  c->prefills++;      // a recorded step stays valid while its plan covers the new sequences (step_t looks)
  std::vector<int> off(batch + 1);
  for (int b = 0; b <= batch; ++b) off[b] = offsets[b] - offsets[0];
  // (an error on the way leaves it open what has been written)
  const std::vector<int> before = c->written;
  c->written.assign(f.max_batch, c->cap);
  // The prompts are cut into chunks of R tokens and the chunks of all prompts, one prompt after another, are dealt to as
  // few passes as the row buffers allow, evenly. A chunk sees the chunks before it in the cache whether they belong to an
  // earlier pass or to this one: a layer stores the keys and values of all its rows before its attention starts.
  // (without the many-row projection kernel a pass takes as many chunks as there are sequences)
  const int cap = c->tc && !c->wide_gemm ? f.max_batch : c->chunk_cap;
  // The 16-bit path keeps whole chunks also for shorter prompts: the projections' kernels go by the number of rows, here a multiple
  // of 128 whatever the lengths. (In float32 a row's sums do not depend on the others.)
  const int R = c->tc ? PREFILL_ROWS : std::min(PREFILL_ROWS, (int)round_up(maxlen, 16));
  std::vector<int> cseq, cpos;
  for (int b = 0; b < batch; ++b)
    for (int p = 0; p < off[b + 1] - off[b]; p += R) { cseq.push_back(b); cpos.push_back(p); }
  const int chunks = (int)cseq.size();
  // A lone prompt of two chunks has the sums of its chunks one after the other, through the projections that stream the weights: the order of sums that the
  // prompt of one chunk and a lone sequence's verification steps have. (Both chunks at once where that can be had, see two_chunks_at_once.) Nothing more is promised: prompts of more chunks, and any prompt processed together with
  // others, take the many-row projections, whose order of sums is another one (and, up to 512 rows, depends on the rows).
  const int passes = batch == 1 && chunks == 2 ? 2 : (chunks + cap - 1) / cap;
  // the prompts' last rows, by sequence (the edge flags of the acceptance step are not in use while prompts are processed)
  static_assert(PREFILL_ROWS >= 6, "a place of the edge flags a table entry");
  std::vector<int> ends(6 * (size_t)batch);
  PromptEnds pe{};
  bool pruned = false;
  pe.row = c->d_edge; pe.pos = pe.row + batch; pe.seq = pe.pos + batch; pe.one = pe.seq + batch; pe.start = pe.one + batch; pe.cnt = pe.start + batch;
  pe.start_host = ends.data() + 4 * (size_t)batch; pe.pruned = &pruned;
  for (int pass = 0, ch = 0; pass < passes; ++pass) {
    const int g = (chunks - ch + passes - pass - 1) / (passes - pass);
    for (int v = ch; v < ch + g; ++v) {
      const int b = cseq[v], last = off[b + 1] - off[b] - 1;
      if (last >= cpos[v] + R) continue;
      const int entry[6] = {(v - ch) * R + last - cpos[v], last, b, 1, cpos[v], last - cpos[v] + 1};
      for (int k = 0; k < 6; ++k) ends[(size_t)k * batch + b] = entry[k];
    }
    ch += g;
  }
  StreamWait wait{c->stream};     // (page-locked tokens are read until their copy is through, which a return with an error must not leave behind)
  CUDA_OK(cudaMemcpyAsync(c->d_prompt, tokens + offsets[0], (size_t)off[batch] * sizeof(int), cudaMemcpyHostToDevice, c->stream));
  const int pair_vecs = (int)(c->geom.block_elems() * 2 * c->esz / 16);   // 16-byte vectors of a page's K and V of one layer and head
  const int lh = f.n_layers * f.n_kv_heads, most_share = (int)std::max<long long>(1, std::min<long long>(c->pages_per_seq, 8 * SM_SLOTS / ((long long)lh * f.max_batch)));
  uint4* pool = static_cast<uint4*>(c->d_pool);
  const size_t lh_vecs = c->geom.pool_pages() * pair_vecs;
  if (f.max_batch <= PS_SEQS && chunks <= PS_CHUNKS) {
    PrefillSetup ps{};
    ps.batch = batch; ps.max_batch = f.max_batch; ps.chunks = chunks;
    int pages = 1;                                             // most that a sequence has to clear
    for (int b = 0; b < f.max_batch; ++b) {
      ps.page_end[b] = std::min(c->pages_per_seq, (before[b] + f.page_size - 1) / f.page_size);
      pages = std::max(pages, ps.page_end[b] - (b < batch ? (off[b + 1] - off[b]) / f.page_size : 0));
    }
    std::copy(off.begin(), off.end(), ps.offsets);
    std::copy(cseq.begin(), cseq.end(), ps.chunk_seq);
    std::copy(cpos.begin(), cpos.end(), ps.chunk_pos);
    std::copy(ends.begin(), ends.end(), ps.ends);
    PrefillTargets to{c->d_offsets, c->d_chunk_seq, c->d_chunk_pos, c->d_edge, c->d_status, c->d_gen_cnt, c->d_draws, c->d_pair_arrive, c->d_attn_arrive, GP_ARRIVE};
    const int share = std::min(most_share, pages);
    for (int lh0 = 0; lh0 < lh; lh0 += 65535) {
      prefill_setup<<<dim3((unsigned)share * (unsigned)f.max_batch, (unsigned)std::min(65535, lh - lh0)), 256, 0, c->stream>>>(
          ps, to, pool + (size_t)lh0 * lh_vecs, c->pages_per_seq, f.page_size, pair_vecs, share);
      to.status = nullptr;                                     // (the tables are written)
      LAUNCH_CHECK("prefill_setup");
    }
  } else {
    CUDA_OK(cudaMemsetAsync(c->d_status, 0, 4 * sizeof(int), c->stream));
    CUDA_OK(cudaMemcpyAsync(c->d_offsets, off.data(), (batch + 1) * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    for (int lh0 = 0; lh0 < lh; lh0 += 65535)
      clear_free_pages<<<dim3((unsigned)most_share * (unsigned)f.max_batch, (unsigned)std::min(65535, lh - lh0)), 256, 0, c->stream>>>(
          pool + (size_t)lh0 * lh_vecs, c->d_offsets, batch, c->pages_per_seq, f.max_batch, f.page_size, pair_vecs, most_share, c->d_attn_arrive);
    LAUNCH_CHECK("clear_free_pages");
    CUDA_OK(cudaMemsetAsync(c->d_pair_arrive, 0, GP_ARRIVE * sizeof(unsigned int), c->stream));
    CUDA_OK(cudaMemsetAsync(c->d_gen_cnt, 0, batch * sizeof(int), c->stream));
    CUDA_OK(cudaMemsetAsync(c->d_draws, 0, batch * sizeof(int), c->stream));
    CUDA_OK(cudaMemcpyAsync(c->d_chunk_seq, cseq.data(), chunks * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    CUDA_OK(cudaMemcpyAsync(c->d_chunk_pos, cpos.data(), chunks * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    CUDA_OK(cudaMemcpyAsync(c->d_edge, ends.data(), ends.size() * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    CUDA_OK(cudaStreamSynchronize(c->stream));   // the host staging vectors go out of scope
  }
  SegMap gate_up{};
  int gate_up_runs = 0;
  const bool at_once = c->tc && batch == 1 && chunks == 2 && two_chunks_at_once(c, &gate_up, &gate_up_runs);
  if (at_once) {
    Rows rows = make_rows(c, R, true);
    rows.B = 2; rows.seq = c->d_chunk_seq; rows.n = c->d_chunk_n; rows.cnt = c->d_chunk_cnt;
    prepare_prefill_rows<T><<<2 * R, 128, 0, c->stream>>>(rows, c->d_prompt, c->d_offsets, c->d_chunk_pos, static_cast<const T*>(c->embed), c->d_x, f.d_model,
                                                        f.vocab, c->d_status);
    LAUNCH_CHECK("prepare_prefill_rows");
    int r = forward_two_chunks(c, rows, (int)round_up(off[1], 16), gate_up, gate_up_runs);
    if (r) return r;
    rows.B = 1; rows.seq += 1; rows.n += 1; rows.cnt += 1;
    prefill_keep_last<T><<<1, 256, 0, c->stream>>>(rows, c->d_offsets, c->d_chunk_pos + 1, c->d_hid, c->d_h_last, static_cast<T*>(c->d_hq_last), c->d_n, f.d_model);
    LAUNCH_CHECK("prefill_keep_last");
  }
  for (int pass = 0, ch = 0; !at_once && pass < passes; ++pass) {
    const int g = (chunks - ch + passes - pass - 1) / (passes - pass);    // chunks of this pass
    pe.seq0 += pe.count;
    pe.count = 0;
    for (int v = ch; v < ch + g; ++v) pe.count += cpos[v] + R >= off[cseq[v] + 1] - off[cseq[v]];
    pruned = false;
    Rows rows = make_rows(c, R, true);
    rows.B = g; rows.seq = c->d_chunk_seq + ch; rows.n = c->d_chunk_n; rows.cnt = c->d_chunk_cnt;
    prepare_prefill_rows<T><<<g * R, 128, 0, c->stream>>>(rows, c->d_prompt, c->d_offsets, c->d_chunk_pos + ch, static_cast<const T*>(c->embed),
                                                        c->d_x, f.d_model, f.vocab, c->d_status);
    LAUNCH_CHECK("prepare_prefill_rows");
    int r = forward_layers<T>(c, rows, cpos.data() + ch, nullptr, cpos.data() + ch, &pe);
    if (r) return r;
    if (!pruned) {
      prefill_keep_last<T><<<g, 256, 0, c->stream>>>(rows, c->d_offsets, c->d_chunk_pos + ch, c->d_hid, c->d_h_last, static_cast<T*>(c->d_hq_last),
                                                     c->d_n, f.d_model);
      LAUNCH_CHECK("prefill_keep_last");
    }
    ch += g;
  }
  int r = lm_head_argmax<T>(c, static_cast<const T*>(c->d_hq_last), batch);
  if (r) return r;
  AcceptArgs a = make_accept(c, 1, 1);
  KLAUNCH("accept_kernel", accept_kernel, dim3(batch), dim3(256), 0, a);
  if (f.sampling) {
    KLAUNCH("sample_root", sample_root, dim3(SAMPLE_CLUSTER, batch), dim3(SAMPLE_THREADS), 0, (const float*)c->d_logits, (const float*)c->d_pval2, f.vocab, 1, c->K,
            (const int*)c->d_path, (const int*)c->d_count, f.temperature, f.seed_lo, f.seed_hi, c->d_draws, c->d_root, 1);
  }
  // (accept_kernel has put the status word into host memory)
  wait.through = true;
  CUDA_OK(cudaStreamSynchronize(c->stream));
  if ((r = report_status(c, c->h_result))) return r;
  for (int b = 0; b < f.max_batch; ++b) c->written[b] = b < batch ? off[b + 1] - off[b] : 0;
  c->n_hi.assign(batch, 0);
  for (int b = 0; b < batch; ++b) c->n_hi[b] = offsets[b + 1] - offsets[b];
  c->n_lo = c->n_hi;
  c->n_copy_pending = false;
  c->prefilled = true;
  return SPEC_OK;
}

// Phase boundary i of the step (only with SPEC_OPT_PHASE_TIMING: an event between two kernels costs the
// programmatic overlap of that pair): an event record, an external-event node while the step is captured.
void step_event(spec_ctx* c, int i) {
  if (!c->phase_timing) return;
  if (c->capturing) cudaEventRecordWithFlags(c->phase_ev[i], c->stream, cudaEventRecordExternal);
  else cudaEventRecord(c->phase_ev[i], c->stream);
}

// Enqueues the kernels of one step (or records them, when the stream is capturing). ov: device
// candidate overrides or null; n_hi_plan / n_lo_plan: the length bounds the attention launches are planned for.
template <typename T>
int step_body(spec_ctx* c, const int* ov, const int* n_hi_plan, const int* n_lo_plan) {
  const spec_config& f = c->cfg;
  int B = c->B, K = c->K, T_ = c->T, d = f.d_model, kmax = c->kmax;
  step_event(c, 0);
  // (1) extra heads -> shared lm_head -> per-head top-k -> candidate table
  if (K > 0 && c->tc) {
    int r = heads_tc(c, ov);
    if (r) return r;
  } else if (K > 0) {
    constexpr int MC = 4;
    dim3 g1((K * d + 7) / 8, (B + MC - 1) / MC);
    KLAUNCH("medusa_resblock", (medusa_resblock<T, MC>), g1, dim3(256), 0, (const float*)c->d_h_last,
            reinterpret_cast<const T* const*>(c->d_mw), reinterpret_cast<const T* const*>(c->d_mb), static_cast<T*>(c->d_r), B, K, d);
    const void* mats[1] = {c->lm_head};
    const int ldz = (int)round_up(f.vocab, 4);
    for (int r0 = 0; r0 < B * K; r0 += c->head_rows) {
      const int rows_now = std::min(c->head_rows, B * K - r0);
      RowBest best{};
      int r = linear_simple<T, LR_PLAIN>(c, "linear_heads", static_cast<const T*>(c->d_r) + (size_t)r0 * d, 1, mats, &f.vocab, c->d_logits, ldz, nullptr,
                                         rows_now, d, &best);
      if (r) return r;
      if (best.val && rows_now == B * K && best.tiles >= kmax && best.tiles <= TOPK_MAX_TILES && best.tile <= 512) {   // (beyond, a tile is much to read again)
        KLAUNCH("topk_tiles", topk_tiles, dim3(rows_now), dim3(256), 0, (const float*)c->d_logits, ldz, (const float*)best.val, (const int*)best.idx, best.tiles, best.tile, best.piece,
                f.vocab, kmax, K, (const int*)c->d_root, ov, c->d_cand);
        break;
      }
      if ((r = heads_top_k(c, plain_view(c->d_logits, rows_now, ldz), r0, rows_now, ov))) return r;
    }
  } else {
    CUDA_OK(cudaMemcpyAsync(c->d_cand, c->d_root, B * sizeof(int), cudaMemcpyDeviceToDevice, c->stream));
  }
  step_event(c, 1);
  // (2) candidate tree -> rows
  int M = B * T_;
  Rows rows = make_rows(c, T_, false);
  KLAUNCH("prepare_verify_rows", prepare_verify_rows<T>, dim3(M), dim3(256), 0, rows, (const int*)c->d_cand, (K + 1) * kmax, kmax,
          (const int*)c->d_depth, (const int*)c->d_rank, c->cap, static_cast<const T*>(c->embed), c->d_x, d, f.vocab, c->d_status);
  step_event(c, 2);
  // (3) verification forward
  // (the order the attention CTAs are handed out in goes by the host's current bounds, not by the bounds the launch is
  // planned for: those are the same for all sequences)
  int r = forward_layers<T>(c, rows, n_hi_plan, n_lo_plan, c->n_hi.data());
  if (r) return r;
  r = lm_head_argmax<T>(c, static_cast<const T*>(c->d_hq), M);
  if (r) return r;
  step_event(c, 3);
  // (4) acceptance
  AcceptArgs a = make_accept(c, T_, 0);
  if (f.accept_mode == 1) {
    KLAUNCH("typical_edges", typical_edges, dim3(M), dim3(TYP_THREADS), 0, (const float*)c->d_logits, f.vocab, rows, (const int*)c->d_parent,
            f.typ_eps, f.typ_delta, 1.0f / (f.temperature > 0.f ? f.temperature : 1.0f), c->d_edge);
    a.edge_ok = c->d_edge;
  }
  KLAUNCH("accept_kernel", accept_kernel, dim3(B), dim3(256), 0, a);
  if (f.sampling) {
    KLAUNCH("sample_root", sample_root, dim3(SAMPLE_CLUSTER, B), dim3(SAMPLE_THREADS), 0, (const float*)c->d_logits, (const float*)c->d_pval2, f.vocab, T_, K,
            (const int*)c->d_path, (const int*)c->d_count, f.temperature, f.seed_lo, f.seed_hi, c->d_draws, c->d_root, 0);
  }
  step_event(c, 4);
  // (5) KV compaction
  dim3 gc(f.n_layers * 2 * ((f.n_kv_heads + COMPACT_HEADS - 1) / COMPACT_HEADS), B);
  KLAUNCH("compact_kv", compact_kv<T>, gc, dim3(128), 0, static_cast<T*>(c->d_pool), c->geom, (const int*)c->d_page_table,
          (const int*)c->d_path, (const int*)c->d_count, (const int*)c->d_n_old, K, (const int*)c->d_result, c->h_result_dev, 4 + f.max_batch * (K + 3));
  step_event(c, 5);
  return SPEC_OK;
}

template <typename T>
int step_t(spec_ctx* c, int32_t* out_tokens, int32_t* out_counts, const int32_t* cand_override) {
  const spec_config& f = c->cfg;
  int B = c->B, K = c->K, T_ = c->T, kmax = c->kmax;
  for (int b = 0; b < B; ++b)
    if (c->n_hi[b] + K + 1 > f.max_seq) return c->fail(SPEC_E_SEQLEN, "sequence would exceed max_seq");
  for (int i = 0; i < 6; ++i)
    if (!c->phase_ev[i]) CUDA_OK(cudaEventCreate(&c->phase_ev[i]));
  c->prof_used = 0;
  if (c->trace_on) {
    c->trace_n = 0;
    c->trace_names.clear();
    CUDA_OK(cudaMemcpyAsync(c->d_trace, c->trace_init.data(), c->trace_init.size() * 8, cudaMemcpyHostToDevice, c->stream));
  }
  const int* ov = nullptr;
  if (cand_override && K > 0) {
    CUDA_OK(cudaMemcpyAsync(c->d_cand_ov, cand_override, (size_t)B * K * kmax * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    ov = c->d_cand_ov;
  }
  for (int b = 0; b < B; ++b) c->written[b] = std::max(c->written[b], std::min(c->cap, c->n_hi[b] + T_));
  // (the kernels take the lengths themselves from the device, so a recorded step serves every length below its bounds)
  std::vector<int> n_hi_plan(B), n_lo_plan(B);
  for (int b = 0; b < B; ++b) n_hi_plan[b] = attn_plan_bound(c, T_, B, c->n_hi[b] + T_) - T_;
  // a recorded step serves every sequence that is at least as long as the part it fetches ahead
  const int ahead = attn_fetch_ahead(c, T_, B, (*std::max_element(n_hi_plan.begin(), n_hi_plan.end()) + T_ + 63) / 64 * 64);
  for (int b = 0; b < B; ++b) n_lo_plan[b] = std::min(c->n_lo[b], ahead);
  const bool use_graph = c->graph_on && !c->trace_on && c->profile_kind == 0;
  if (!use_graph) {
    int r = step_body<T>(c, ov, n_hi_plan.data(), n_lo_plan.data());
    if (r) return r;
  } else {
    spec_ctx::StepGraph& g = c->step_graph[ov ? 1 : 0];
    bool valid = g.exec && g.epoch == c->graph_epoch && g.B == B;
    for (int b = 0; valid && b < B; ++b) valid = c->n_hi[b] <= g.n_hi_plan[b] && c->n_lo[b] >= g.n_lo_plan[b];
    // after a prefill: the same launch shape as a new recording would get (a shorter bound may choose another kernel) and the
    // same order of the sequences
    std::vector<int> order;
    if (!valid || g.prefills != c->prefills) {
      order.resize(B);
      for (int b = 0; b < B; ++b) order[b] = b;
      std::stable_sort(order.begin(), order.end(), [&](int x, int y) { return c->n_hi[x] > c->n_hi[y]; });
      if (valid) valid = g.n_hi_plan == n_hi_plan && g.order == order;
      if (valid) g.prefills = c->prefills;
    }
    if (!valid) {
      // record the step once, then replay it until a sequence outgrows the planned bound
      cudaGraph_t graph = nullptr;
      const long long l0 = c->launches;
      // recorded on a stream of the library's own (the caller's may be the legacy default stream,
      // which cannot be captured); the graph is then launched on the caller's stream
      if (!c->cap_stream) CUDA_OK(cudaStreamCreateWithFlags(&c->cap_stream, cudaStreamNonBlocking));
      CUDA_OK(cudaStreamBeginCapture(c->cap_stream, cudaStreamCaptureModeThreadLocal));
      cudaStream_t user_stream = c->stream;
      c->stream = c->cap_stream;
      c->capturing = true;
      int r = step_body<T>(c, ov, n_hi_plan.data(), n_lo_plan.data());
      c->capturing = false;
      c->stream = user_stream;
      cudaError_t e = cudaStreamEndCapture(c->cap_stream, &graph);
      if (r) { if (graph) cudaGraphDestroy(graph); c->launches = l0; return r; }
      if (e != cudaSuccess || !graph) { c->launches = l0; return c->fail(SPEC_E_CUDA, std::string("step capture: ") + cudaGetErrorString(e)); }
      if (g.exec) { cudaGraphExecDestroy(g.exec); g.exec = nullptr; }
      e = cudaGraphInstantiate(&g.exec, graph, 0);
      cudaGraphDestroy(graph);
      if (e != cudaSuccess) { g.exec = nullptr; c->launches = l0; return c->fail(SPEC_E_CUDA, std::string("step graph instantiate: ") + cudaGetErrorString(e)); }
      g.epoch = c->graph_epoch; g.B = B; g.n_launches = c->launches - l0;
      g.n_hi_plan = n_hi_plan; g.n_lo_plan = n_lo_plan;
      g.prefills = c->prefills; g.order = order;
      c->launches = l0;
      c->graph_captures++;
    }
    CUDA_OK(cudaGraphLaunch(g.exec, c->stream));
    c->launches += g.n_launches;
  }
  c->phase_valid = c->phase_timing;
  if (c->profile_kind) {
    CUDA_OK(cudaStreamSynchronize(c->stream));
    for (int i = 0; i + 1 < c->prof_used; i += 2) {
      float ms = 0.f;
      if (cudaEventElapsedTime(&ms, c->prof_ev[i], c->prof_ev[i + 1]) == cudaSuccess) { c->prof_ms += ms; c->prof_launches++; }
    }
  }
  if (out_tokens || out_counts) {
    // (the step's last kernel has put the result block into host memory)
    const int cap = f.max_batch;
    CUDA_OK(cudaStreamSynchronize(c->stream));
    const int *nn = c->h_result + 4, *counts = nn + cap, *toks = counts + cap;
    if (out_tokens) memcpy(out_tokens, toks, (size_t)B * (K + 1) * sizeof(int));
    if (out_counts) memcpy(out_counts, counts, (size_t)B * sizeof(int));
    int r = report_status(c, c->h_result);
    if (r) return r;
    for (int b = 0; b < B; ++b) c->n_hi[b] = c->n_lo[b] = nn[b];
    c->n_copy_pending = false;
  } else {
    for (int b = 0; b < B; ++b) { c->n_hi[b] += K + 1; c->n_lo[b] += 1; }
    if (c->h_n_pinned && c->n_ev) {
      if (c->n_copy_pending) {
        c->n_copy_steps_after++;
        // the host stays at most MAX_STEPS_AHEAD steps ahead of the device, so that its bounds stay close
        if (c->n_copy_steps_after >= MAX_STEPS_AHEAD) cudaEventSynchronize(c->n_ev);
        if (cudaEventQuery(c->n_ev) == cudaSuccess) {
          // the copy shows the lengths after an earlier step; every step since added 1..K+1 tokens
          for (int b = 0; b < B; ++b) {
            c->n_lo[b] = std::max(c->n_lo[b], c->h_n_pinned[b] + c->n_copy_steps_after);
            c->n_hi[b] = std::min(c->n_hi[b], c->h_n_pinned[b] + c->n_copy_steps_after * (K + 1));
          }
          c->n_copy_pending = false;
        }
      }
      // a copy between two steps costs the overlap of the step's last kernel with the next step's first:
      // one every N_COPY_EVERY steps keeps the bounds tight enough
      if (!c->n_copy_pending && ++c->steps_since_n_copy >= N_COPY_EVERY && (c->steps_since_n_copy = 0, true) &&
          cudaMemcpyAsync(c->h_n_pinned, c->d_n, (size_t)B * sizeof(int), cudaMemcpyDeviceToHost, c->stream) == cudaSuccess &&
          cudaEventRecord(c->n_ev, c->stream) == cudaSuccess) {
        c->n_copy_pending = true;
        c->n_copy_steps_after = 0;
      }
    }
  }
  return SPEC_OK;
}

}  // namespace

extern "C" {

size_t spec_workspace_bytes(const spec_config* cfg, const spec_tree* tree) {
  std::string why;
  if (!cfg || !tree || !validate_config(cfg, &why)) return 0;
  spec_ctx tmp{};
  tmp.cfg = *cfg;
  if (!validate_tree(cfg, tree, &tmp.kmax, &why)) return 0;
  tmp.T = tree->n_nodes; tmp.K = cfg->n_medusa;
  tmp.tc = cfg->dtype == 1 && !(cfg->flags & SPEC_FLAG_SIMPLE_KERNELS);
  tmp.esz = cfg->dtype == 1 ? 2 : 4;
  return carve(&tmp, nullptr, full_chunk_cap(&tmp), true);
}

int spec_create(const spec_config* cfg, const spec_weights* w, const spec_tree* tree, void* workspace,
                size_t workspace_bytes, void* cuda_stream, spec_ctx** out) {
  std::string why;
  if (!cfg || !w || !tree || !workspace || !out) { g_create_error = "null argument"; return SPEC_E_BADARG; }
  if (!validate_config(cfg, &why)) { g_create_error = why; return SPEC_E_BADARG; }
  int kmax = 1;
  if (!validate_tree(cfg, tree, &kmax, &why)) { g_create_error = why; return SPEC_E_BADTREE; }
  if (!w->embed || !w->lm_head || !w->final_norm || !w->attn_norm || !w->wq || !w->wk || !w->wv || !w->wo ||
      !w->ffn_norm || !w->w_gate || !w->w_up || !w->w_down || (cfg->n_medusa > 0 && (!w->medusa_w || !w->medusa_b))) {
    g_create_error = "null weight pointer"; return SPEC_E_BADARG;
  }
  if (reinterpret_cast<uintptr_t>(workspace) % 1024) { g_create_error = "workspace must be 1024-byte aligned"; return SPEC_E_BADARG; }
  spec_ctx* c = new spec_ctx();
  c->cfg = *cfg;
  c->stream = static_cast<cudaStream_t>(cuda_stream);
  c->T = tree->n_nodes; c->K = cfg->n_medusa; c->kmax = kmax; c->B = cfg->max_batch;
  c->tc = cfg->dtype == 1 && !(cfg->flags & SPEC_FLAG_SIMPLE_KERNELS);
  c->packed = (cfg->flags & SPEC_FLAG_PACKED_WEIGHTS) != 0;
  c->esz = cfg->dtype == 1 ? 2 : 4;
  // a smaller workspace than spec_workspace_bytes: prompts in passes of fewer chunks, at least one a sequence
  int chunks = full_chunk_cap(c);
  size_t need = carve(c, workspace, chunks, true);
  while (need > workspace_bytes && chunks > cfg->max_batch) need = carve(c, workspace, --chunks, true);
  if (need > workspace_bytes) need = carve(c, workspace, chunks, false);
  if (need > workspace_bytes) { g_create_error = "workspace too small"; delete c; return SPEC_E_NOMEM; }
  c->written.assign(cfg->max_batch, c->cap);
  c->h_parent.assign(tree->parent, tree->parent + c->T);
  c->h_depth.assign(tree->depth, tree->depth + c->T);
  c->h_rank.assign(tree->rank, tree->rank + c->T);
  int L = cfg->n_layers;
  c->embed = w->embed; c->lm_head = w->lm_head; c->final_norm = w->final_norm;
  c->qkv_fused = true;
  size_t qn = (size_t)cfg->n_heads * cfg->head_dim * cfg->d_model * c->esz, kn = (size_t)cfg->n_kv_heads * cfg->head_dim * cfg->d_model * c->esz;
  for (int l = 0; l < L; ++l) {
    if (!w->attn_norm[l] || !w->wq[l] || !w->wk[l] || !w->wv[l] || !w->wo[l] || !w->ffn_norm[l] || !w->w_gate[l] || !w->w_up[l] || !w->w_down[l]) {
      g_create_error = "null layer weight pointer"; delete c; return SPEC_E_BADARG;
    }
    c->an.push_back(w->attn_norm[l]); c->fn.push_back(w->ffn_norm[l]);
    c->wq.push_back(w->wq[l]); c->wk.push_back(w->wk[l]); c->wv.push_back(w->wv[l]); c->wo.push_back(w->wo[l]);
    c->wg.push_back(w->w_gate[l]); c->wu.push_back(w->w_up[l]); c->wd.push_back(w->w_down[l]);
    const uint8_t* q0 = static_cast<const uint8_t*>(w->wq[l]);
    if (static_cast<const uint8_t*>(w->wk[l]) != q0 + qn || static_cast<const uint8_t*>(w->wv[l]) != q0 + qn + kn) c->qkv_fused = false;
  }
  for (int k = 0; k < c->K; ++k) { c->mw.push_back(w->medusa_w[k]); c->mb.push_back(w->medusa_b[k]); }
  if (c->tc && !get_encode_fn()) { g_create_error = "cuTensorMapEncodeTiled entry point unavailable"; delete c; return SPEC_E_CUDA; }

  // host-made tables: tree arrays, ancestor bitsets (tree and chain), page table, RoPE table
  std::vector<uint32_t> anc_tree(SPEC_MAX_NODES * 4, 0), anc_chain(PREFILL_ROWS * 4, 0);
  for (int v = 0; v < c->T; ++v) {
    if (v > 0) for (int wd = 0; wd < 4; ++wd) anc_tree[v * 4 + wd] = anc_tree[c->h_parent[v] * 4 + wd];
    anc_tree[v * 4 + (v >> 5)] |= 1u << (v & 31);
  }
  for (int v = 0; v < PREFILL_ROWS; ++v)
    for (int u = 0; u <= v; ++u) anc_chain[v * 4 + (u >> 5)] |= 1u << (u & 31);
  std::vector<int> pt((size_t)cfg->max_batch * c->pages_per_seq);
  for (int b = 0; b < cfg->max_batch; ++b)
    for (int p = 0; p < c->pages_per_seq; ++p) pt[(size_t)b * c->pages_per_seq + p] = p * cfg->max_batch + b;
  int half = cfg->head_dim / 2;
  std::vector<float2> rope((size_t)c->cap * half);
  for (int i = 0; i < half; ++i) {
    double inv = pow((double)cfg->rope_base, -2.0 * i / cfg->head_dim);
    for (int p = 0; p < c->cap; ++p) {
      double ang = (double)p * inv;
      rope[(size_t)p * half + i] = make_float2((float)cos(ang), (float)sin(ang));
    }
  }
  cudaError_t e = cudaSuccess;
  auto up = [&](void* dst, const void* src, size_t bytes) {
    if (e == cudaSuccess && bytes) e = cudaMemcpyAsync(dst, src, bytes, cudaMemcpyHostToDevice, c->stream);
  };
  up(c->d_parent, c->h_parent.data(), c->T * sizeof(int));
  up(c->d_depth, c->h_depth.data(), c->T * sizeof(int));
  up(c->d_rank, c->h_rank.data(), c->T * sizeof(int));
  up(c->d_anc_tree, anc_tree.data(), anc_tree.size() * 4);
  up(c->d_anc_chain, anc_chain.data(), anc_chain.size() * 4);
  up(c->d_page_table, pt.data(), pt.size() * sizeof(int));
  up(c->d_rope, rope.data(), rope.size() * sizeof(float2));
  up(c->d_mw, c->mw.data(), c->mw.size() * sizeof(void*));
  up(c->d_mb, c->mb.data(), c->mb.size() * sizeof(void*));
  if (e == cudaSuccess) e = cudaMemsetAsync(c->d_status, 0, 4 * sizeof(int), c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->d_attn_arrive, 0, (size_t)c->chunk_cap * cfg->n_heads * 2 * sizeof(unsigned int), c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->d_row_arrive, 0, (size_t)c->Mcap * sizeof(unsigned int), c->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(c->d_cand, 0, (size_t)cfg->max_batch * (c->K + 1) * c->kmax * sizeof(int), c->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(c->stream);
  if (e != cudaSuccess) { g_create_error = std::string("set-up copies: ") + cudaGetErrorString(e); delete c; return SPEC_E_CUDA; }
  // one pinned block: a step's result, then the copy of the committed lengths
  if (cudaHostAlloc(reinterpret_cast<void**>(&c->h_result), (4 + (size_t)cfg->max_batch * (c->K + 4)) * sizeof(int), cudaHostAllocMapped) != cudaSuccess ||
      cudaHostGetDevicePointer(reinterpret_cast<void**>(&c->h_result_dev), c->h_result, 0) != cudaSuccess) {
    if (c->h_result) cudaFreeHost(c->h_result);
    g_create_error = "pinned host memory for a step's result"; delete c; return SPEC_E_CUDA;
  }
  c->h_n_pinned = c->h_result + 4 + (size_t)cfg->max_batch * (c->K + 3);
  if (cudaEventCreateWithFlags(&c->n_ev, cudaEventDisableTiming) != cudaSuccess) c->n_ev = nullptr;
  cudaGetLastError();
  if (c->tc && cfg->head_dim == 128 && cfg->page_size == 16) {
    // 5-D view of the page pool for the tcgen05 attention: (64 dims of a slab row, the 64 slab rows of a page's
    // K|V pair = 4 slabs x 16 rows, sequence, page, layer * kv_heads + head); page p of sequence b is pool
    // page p * max_batch + b (the table written above), so both are strided dimensions
    EncodeTiledFn fn = get_encode_fn();
    const cuuint64_t pair_bytes = (cuuint64_t)c->geom.block_elems() * 2 * 2;
    cuuint64_t dims[5] = {64, 64, (cuuint64_t)cfg->max_batch, (cuuint64_t)c->pages_per_seq, (cuuint64_t)cfg->n_layers * cfg->n_kv_heads};
    cuuint64_t strides[4] = {128, pair_bytes, pair_bytes * (cuuint64_t)cfg->max_batch, pair_bytes * (cuuint64_t)c->geom.pool_pages()};
    cuuint32_t box[5] = {64, 16, 1, AU_KT / 16, 1};
    cuuint32_t estr[5] = {1, 1, 1, 1, 1};
    c->tm_kv_ok = fn && fn(&c->tm_kv, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, c->d_pool, dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                           CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
  }
  *out = c;
  return SPEC_OK;
}

int spec_prefill(spec_ctx* c, int32_t batch, const int32_t* tokens, const int32_t* offsets) {
  if (!c) return SPEC_E_BADARG;
  if (!tokens || !offsets) return c->fail(SPEC_E_BADARG, "null argument");
  if (batch < 1 || batch > c->cfg.max_batch) return c->fail(SPEC_E_BADARG, "batch out of range");
  return c->cfg.dtype == 1 ? prefill_t<bf16>(c, batch, tokens, offsets) : prefill_t<float>(c, batch, tokens, offsets);
}

int spec_step(spec_ctx* c, int32_t* out_tokens, int32_t* out_counts, const int32_t* cand_override) {
  if (!c) return SPEC_E_BADARG;
  if (!c->prefilled) return c->fail(SPEC_E_STATE, "spec_step before spec_prefill");
  const int r = c->cfg.dtype == 1 ? step_t<bf16>(c, out_tokens, out_counts, cand_override)
                                  : step_t<float>(c, out_tokens, out_counts, cand_override);
  // (a failed step may have moved the device's lengths on while the host's bounds stay: what later ones write is not known here)
  if (r != SPEC_OK) c->written.assign(c->cfg.max_batch, c->cap);
  return r;
}

int spec_read_generated(spec_ctx* c, int32_t seq, int32_t* out, int32_t max_tokens, int32_t* n_generated) {
  if (!c) return SPEC_E_BADARG;
  if (!c->prefilled) return c->fail(SPEC_E_STATE, "nothing generated yet");
  if (seq < 0 || seq >= c->B || !n_generated || max_tokens < 0) return c->fail(SPEC_E_BADARG, "bad argument");
  int r = check_status(c);
  if (r) return r;
  int cnt = 0;
  CUDA_OK(cudaMemcpyAsync(&cnt, c->d_gen_cnt + seq, sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  CUDA_OK(cudaStreamSynchronize(c->stream));
  int stored = cnt < c->gen_cap ? cnt : c->gen_cap;
  int ncopy = stored < max_tokens ? stored : max_tokens;
  if (out && ncopy > 0) {
    CUDA_OK(cudaMemcpyAsync(out, c->d_gen_log + (size_t)seq * c->gen_cap, ncopy * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
    CUDA_OK(cudaStreamSynchronize(c->stream));
  }
  *n_generated = cnt;
  std::vector<int> nn(c->B);
  CUDA_OK(cudaMemcpyAsync(nn.data(), c->d_n, c->B * sizeof(int), cudaMemcpyDeviceToHost, c->stream));
  CUDA_OK(cudaStreamSynchronize(c->stream));
  for (int b = 0; b < c->B; ++b) c->n_hi[b] = c->n_lo[b] = nn[b];
  return SPEC_OK;
}

int spec_destroy(spec_ctx* c) {
  if (!c) return SPEC_E_BADARG;
  cudaStreamSynchronize(c->stream);
  for (int i = 0; i < 6; ++i) if (c->phase_ev[i]) cudaEventDestroy(c->phase_ev[i]);
  for (cudaEvent_t e : c->prof_ev) cudaEventDestroy(e);
  for (auto& g : c->step_graph) if (g.exec) cudaGraphExecDestroy(g.exec);
  if (c->cap_stream) cudaStreamDestroy(c->cap_stream);
  if (c->n_ev) cudaEventDestroy(c->n_ev);
  if (c->h_result) cudaFreeHost(c->h_result);
  delete c;
  return SPEC_OK;
}

const char* spec_last_error(const spec_ctx* c) { return c ? c->err.c_str() : g_create_error.c_str(); }

int64_t spec_query(const spec_ctx* c, int32_t what) {
  if (!c) return -1;
  const spec_config& f = c->cfg;
  switch (what) {
    case SPEC_Q_KMAX: return c->kmax;
    case SPEC_Q_KERNEL_LAUNCHES: return c->launches;
    case SPEC_Q_N_NODES: return c->T;
    case SPEC_Q_BATCH: return c->B;
    case SPEC_Q_GRAPH_CAPTURES: return c->graph_captures;
    case SPEC_Q_WIDE_GEMM: return c->tc && c->wide_gemm ? 1 : 0;
    case SPEC_Q_CLUSTER_GATE_UP: return c->tc && (cluster_gemm_ok(c, GC_SWIGLU, c->B * c->T, f.d_model) || glu_cluster(c, c->B * c->T, f.d_model)) ? 1 : 0;
    case SPEC_Q_ALGO_BYTES_PER_STEP: {
      double d = f.d_model, F = f.d_ffn, V = f.vocab, HD = (double)f.n_heads * f.head_dim, KD = (double)f.n_kv_heads * f.head_dim;
      double layer = d * HD + 2 * d * KD + HD * d + 3 * d * F;
      double bytes = (f.n_layers * layer + 2 * V * d + c->K * (d * d + d)) * (double)c->esz;
      return (int64_t)(bytes / 1024.0);
    }
    default: return -1;
  }
}

int spec_set_option(spec_ctx* c, int32_t what, int32_t value) {
  if (!c) return SPEC_E_BADARG;
  switch (what) {
    case SPEC_OPT_GEMM_CTAS: case SPEC_OPT_SMALL_GEMM_CTAS:
      if (value < 1 || value > SM_SLOTS) return c->fail(SPEC_E_BADARG, "gemm CTA count out of range");
      break;
    case SPEC_OPT_L2_PREFETCH:
      if (value < 0 || value > 64) return c->fail(SPEC_E_BADARG, "L2 prefetch depth out of range");
      break;
    case SPEC_OPT_GRAPH: case SPEC_OPT_PHASE_TIMING: case SPEC_OPT_PDL: case SPEC_OPT_TRACE: case SPEC_OPT_CLUSTER_EPILOGUE: case SPEC_OPT_WIDE_GEMM: case SPEC_OPT_ATTN_UMMA: break;
    case SPEC_OPT_LONG_ATTN_KEYS:
      if (value < 0) return c->fail(SPEC_E_BADARG, "context threshold must not be negative");
      break;
    default: return c->fail(SPEC_E_BADARG, "unknown option");
  }
  c->graph_epoch++;   // the option is valid: a recorded step no longer matches the options
  switch (what) {
    case SPEC_OPT_GRAPH:
      c->graph_on = value != 0; return SPEC_OK;
    case SPEC_OPT_PHASE_TIMING:
      c->phase_timing = value != 0; c->phase_valid = false; return SPEC_OK;
    case SPEC_OPT_PDL: c->pdl = value != 0; return SPEC_OK;
    case SPEC_OPT_GEMM_CTAS:
      if (value < 1 || value > SM_SLOTS) return c->fail(SPEC_E_BADARG, "gemm CTA count out of range");
      c->gemm_ctas = value; return SPEC_OK;
    case SPEC_OPT_L2_PREFETCH:
      if (value < 0 || value > 64) return c->fail(SPEC_E_BADARG, "L2 prefetch depth out of range");
      c->l2_prefetch = value; return SPEC_OK;
    case SPEC_OPT_SMALL_GEMM_CTAS:
      if (value < 1 || value > SM_SLOTS) return c->fail(SPEC_E_BADARG, "out of range");
      c->small_gemm_ctas = value; return SPEC_OK;
    case SPEC_OPT_CLUSTER_EPILOGUE: c->cluster_epilogue = value & 7; return SPEC_OK;
    case SPEC_OPT_WIDE_GEMM: c->wide_gemm = value != 0; return SPEC_OK;
    case SPEC_OPT_LONG_ATTN_KEYS: c->long_attn_keys = value; return SPEC_OK;
    case SPEC_OPT_ATTN_UMMA: c->attn_umma = value != 0; return SPEC_OK;
    case SPEC_OPT_TRACE:
      c->trace_on = value != 0;
      if (c->trace_on && c->trace_init.empty()) {
        c->trace_init.resize((size_t)TRACE_CAP * 4);
        for (int i = 0; i < TRACE_CAP; ++i) { c->trace_init[4 * i] = ~0ull; c->trace_init[4 * i + 1] = 0; c->trace_init[4 * i + 2] = ~0ull; c->trace_init[4 * i + 3] = 0; }
      }
      return SPEC_OK;
    default: return c->fail(SPEC_E_BADARG, "unknown option");
  }
}

int spec_trace_read(spec_ctx* c, int32_t max_records, char* names, uint64_t* stamps, int32_t* n_records) {
  if (!c || !n_records || max_records < 0 || (max_records > 0 && (!names || !stamps))) return SPEC_E_BADARG;
  if (!c->trace_on) return c->fail(SPEC_E_STATE, "tracing is off (SPEC_OPT_TRACE)");
  int n = c->trace_n < max_records ? c->trace_n : max_records;
  if (n > 0) {
    CUDA_OK(cudaMemcpyAsync(stamps, c->d_trace, (size_t)n * 32, cudaMemcpyDeviceToHost, c->stream));
    CUDA_OK(cudaStreamSynchronize(c->stream));
    for (int i = 0; i < n; ++i) {
      strncpy(names + (size_t)i * SPEC_TRACE_NAME_LEN, c->trace_names[i].c_str(), SPEC_TRACE_NAME_LEN - 1);
      names[(size_t)i * SPEC_TRACE_NAME_LEN + SPEC_TRACE_NAME_LEN - 1] = 0;
    }
  }
  *n_records = c->trace_n;
  return SPEC_OK;
}

int spec_last_step_phase_ms(spec_ctx* c, float* ms) {
  if (!c || !ms) return SPEC_E_BADARG;
  if (!c->phase_valid) return c->fail(SPEC_E_STATE, "no step has run with SPEC_OPT_PHASE_TIMING on");
  CUDA_OK(cudaStreamSynchronize(c->stream));
  for (int i = 0; i < 5; ++i) CUDA_OK(cudaEventElapsedTime(&ms[i], c->phase_ev[i], c->phase_ev[i + 1]));
  return SPEC_OK;
}

int spec_profile_kernel(spec_ctx* c, int32_t kind) {
  if (!c || kind < 0 || kind > SPEC_PROFILE_ATTENTION) return SPEC_E_BADARG;
  c->profile_kind = kind;
  c->prof_ms = 0.0;
  c->prof_launches = 0;
  return SPEC_OK;
}

int spec_profile_read(spec_ctx* c, double* total_ms, int64_t* launches) {
  if (!c || !total_ms || !launches) return SPEC_E_BADARG;
  *total_ms = c->prof_ms;
  *launches = c->prof_launches;
  return SPEC_OK;
}

int spec_debug_read(spec_ctx* c, int32_t what, void* host_buf, size_t bytes) {
  if (!c || !host_buf) return SPEC_E_BADARG;
  const spec_config& f = c->cfg;
  size_t rows = (size_t)c->B * c->T;
  const void* src = nullptr;
  size_t need = 0;
  switch (what) {
    case SPEC_DBG_TOK: src = c->d_tok; need = rows * 4; break;
    case SPEC_DBG_POS: src = c->d_pos; need = rows * 4; break;
    case SPEC_DBG_LOGITS: src = c->d_logits; need = rows * f.vocab * 4; break;
    case SPEC_DBG_HIDDEN: src = c->d_hid; need = rows * f.d_model * 4; break;
    case SPEC_DBG_ARGMAX: src = c->d_am; need = rows * 4; break;
    case SPEC_DBG_PATH: src = c->d_path; need = (size_t)c->B * (c->K + 1) * 4; break;
    case SPEC_DBG_CAND: src = c->d_cand; need = (size_t)c->B * (c->K + 1) * c->kmax * 4; break;
    case SPEC_DBG_SEQLEN: src = c->d_n; need = (size_t)c->B * 4; break;
    case SPEC_DBG_NEXT_ROOT: src = c->d_root; need = (size_t)c->B * 4; break;
    case SPEC_DBG_H_LAST: src = c->d_h_last; need = (size_t)c->B * f.d_model * 4; break;
    case SPEC_DBG_STATUS: src = c->d_status; need = 16; break;
    default: return c->fail(SPEC_E_BADARG, "unknown debug tap");
  }
  if (!src) return c->fail(SPEC_E_STATE, "tap not available (logits need SPEC_FLAG_KEEP_LOGITS)");
  if (bytes < need) return c->fail(SPEC_E_BADARG, "host buffer too small");
  CUDA_OK(cudaMemcpyAsync(host_buf, src, need, cudaMemcpyDeviceToHost, c->stream));
  CUDA_OK(cudaStreamSynchronize(c->stream));
  return SPEC_OK;
}

int spec_debug_wait_timeout(spec_ctx* c, int32_t limit_us) {
  if (!c) return SPEC_E_BADARG;
  if (limit_us < 1 || limit_us > 100000) return c->fail(SPEC_E_BADARG, "limit must be 1..100000 microseconds");
  CUDA_OK(cudaStreamSynchronize(c->stream));
  wait_probe<<<1, 32, 0, c->stream>>>(c->d_status, (unsigned long long)limit_us * 1000ull);
  LAUNCH_CHECK("wait_probe");
  int r = check_status(c);           // reads the status word: SPEC_E_TIMEOUT with the probe's place code
  // the probe is the only writer here: clear the word so that the context stays usable
  CUDA_OK(cudaMemsetAsync(c->d_status, 0, 4 * sizeof(int), c->stream));
  CUDA_OK(cudaStreamSynchronize(c->stream));
  return r;
}

int spec_debug_read_kv(spec_ctx* c, int32_t seq, int32_t layer, int32_t slot0, int32_t n_slots, float* host_k, float* host_v) {
  if (!c || !host_k || !host_v) return SPEC_E_BADARG;
  const spec_config& f = c->cfg;
  if (seq < 0 || seq >= f.max_batch || layer < 0 || layer >= f.n_layers || slot0 < 0 || n_slots < 0 || slot0 + n_slots > c->cap)
    return c->fail(SPEC_E_BADARG, "bad KV range");
  int D = f.head_dim, Hkv = f.n_kv_heads, ps = f.page_size;
  std::vector<uint8_t> blk(c->geom.block_elems() * c->esz);
  CUDA_OK(cudaStreamSynchronize(c->stream));
  for (int kv = 0; kv < 2; ++kv) {
    float* dst = kv ? host_v : host_k;
    for (int h = 0; h < Hkv; ++h) {
      int cur_page = -1;
      for (int sl = slot0; sl < slot0 + n_slots; ++sl) {
        int page = (sl / ps) * f.max_batch + seq;   // same mapping as the device page table
        if (page != cur_page) {
          const uint8_t* src = static_cast<const uint8_t*>(c->d_pool) + c->geom.block_offset(page, layer, kv, h) * c->esz;
          CUDA_OK(cudaMemcpy(blk.data(), src, blk.size(), cudaMemcpyDeviceToHost));
          cur_page = page;
        }
        int row = sl % ps;
        for (int e = 0; e < D; ++e) {
          float v;
          if (c->esz == 2) {
            uint16_t raw = reinterpret_cast<uint16_t*>(blk.data())[(size_t)row * D + kv_elem<bf16>(row, e, D, ps)];
            uint32_t u32 = (uint32_t)raw << 16;
            memcpy(&v, &u32, 4);
          } else {
            v = reinterpret_cast<float*>(blk.data())[(size_t)row * D + e];
          }
          dst[((size_t)(sl - slot0) * Hkv + h) * D + e] = v;
        }
      }
    }
  }
  return SPEC_OK;
}

namespace {
// Status words of stand-alone calls in pinned host memory, where the kernels report a wait that ran out: nothing has to be cleared before
// them and nothing copied after them (a memset and a 16-byte copy to pageable memory took 12 of the call's 53 us at 64 rows of 4096 x
// 11008). One block a process, made by the first call that asks and kept; a word is taken for a call and given back when the call's kernels
// are through. Where there is none, the caller's words on the device serve.
class StatusWords {
 public:
  int* take(int** dev) {
    std::lock_guard<std::mutex> lock(m_);
    if (!block_) {
      allocations_++;
      if (cudaHostAlloc(reinterpret_cast<void**>(&block_), (size_t)WORDS * 64, cudaHostAllocPortable | cudaHostAllocMapped) != cudaSuccess) block_ = nullptr;
      busy_ = 0;
    }
    void* d = nullptr;
    if (block_ && cudaHostGetDevicePointer(&d, block_, 0) != cudaSuccess) block_ = nullptr;   // (the device has been reset: the block went with it)
    if (!block_ || busy_ == ~0ull) { cudaGetLastError(); return nullptr; }
    int i = 0;
    while ((busy_ >> i) & 1) ++i;
    busy_ |= 1ull << i;
    *dev = static_cast<int*>(d) + i * 16;
    memset(block_ + i * 16, 0, 4 * sizeof(int));
    return block_ + i * 16;
  }
  void give(const int* word) {
    std::lock_guard<std::mutex> lock(m_);
    if (block_ && word >= block_ && word < block_ + WORDS * 16) busy_ &= ~(1ull << ((word - block_) / 16));
  }
  int allocations() { std::lock_guard<std::mutex> lock(m_); return allocations_; }
 private:
  static constexpr int WORDS = 64;                               // bits of busy_; a word has 64 bytes of the block
  std::mutex m_;
  int* block_ = nullptr;
  unsigned long long busy_ = 0;
  int allocations_ = 0;
};
StatusWords& status_words() { static StatusWords* w = new StatusWords; return *w; }   // (never destroyed: a call may come late in the process's exit)

// The status of one call: four ints `words` of the caller's on the device, which get it, and where `pinned` a host word that the kernels report into.
class OpStatus {
 public:
  OpStatus(int* words, bool pinned, cudaStream_t st) : words_(words), st_(st) {
    if (pinned) host_ = status_words().take(&dev_);
    if (!host_) { dev_ = words; ok_ = cudaMemsetAsync(words, 0, 4 * sizeof(int), st) == cudaSuccess; }
  }
  ~OpStatus() {
    if (!host_) return;
    if (!through_) cudaStreamSynchronize(st_);                   // a call that failed behind its first launch: its kernel may still report
    status_words().give(host_);
  }
  OpStatus(const OpStatus&) = delete;
  OpStatus& operator=(const OpStatus&) = delete;
  bool ok() const { return ok_; }
  int* report() const { return dev_; }                           // what the kernels report into
  int* clear() const { return host_ ? words_ : nullptr; }        // what they set to zero
  int finish() {                                                 // waits for the call's kernels
    int st[4] = {};
    if (!host_ && cudaMemcpyAsync(st, words_, sizeof(st), cudaMemcpyDeviceToHost, st_) != cudaSuccess) return SPEC_E_CUDA;
    if (cudaStreamSynchronize(st_) != cudaSuccess) return SPEC_E_CUDA;
    through_ = true;
    if (!host_) return st[0] == 0 ? SPEC_OK : SPEC_E_TIMEOUT;
    if (*static_cast<const volatile int*>(host_) == 0) return SPEC_OK;
    if (cudaMemcpyAsync(words_, host_, sizeof(st), cudaMemcpyHostToDevice, st_) != cudaSuccess || cudaStreamSynchronize(st_) != cudaSuccess) return SPEC_E_CUDA;
    return SPEC_E_TIMEOUT;
  }
 private:
  int *words_, *dev_ = nullptr, *host_ = nullptr;
  cudaStream_t st_;
  bool ok_ = true, through_ = false;
};
// Shared body of the two stand-alone linear entry points (bf16): scratch holds the partial
// sums followed by the four-int status word. pinned: the status may come through pinned host memory.
int op_linear_bf16(const void* x, const void* w, float* y, int M, int N, int K, int ctas, float* scratch,
                   size_t scratch_floats, bool pinned, cudaStream_t st) {
  GemmPlan g;
  int rws[1] = {N};
  if (!plan_gemm(M, K, 1, rws, ctas, &g)) return SPEC_E_BADARG;
  StreamTmaps tm{};
  OpStatus status(reinterpret_cast<int*>(scratch + scratch_floats), pinned, st);
  if (!status.ok()) return SPEC_E_CUDA;
  if (M > 128 && (long long)g.p.n_tiles * g.p.seg.m_tiles >= 2LL * g.grid) {
    // many rows: whole tiles on pairs of SMs, finished sums straight into y (M = 1008, N = 11008, K = 4096: 94 us a call; weight streaming fetches the
    // weights once per 128 rows and adds up partial sums: 204). With few tiles a CTA the streaming kernel is closer to the exact result, since it cuts
    // the inner dimension into more separately rounded sums than the two that this kernel adds: 256 x 4096 x 4096 (0.2 tiles a CTA) 8.1e-7 off
    // 64-bit products against 2.1e-6, 52 us against 47. The line was drawn at two tiles a CTA when the kernel had one tile height; with the heights it
    // has, it is the more exact one from about 0.7 on (512 x 11008 x 4096, 1.2 a CTA: 3.3e-6 and 117 us here, 2.1e-6 and 66 there).
    PairGemmParams p{};
    PairTmaps pm{};
    p.M = M; p.KC = K / 64; p.n_mats = 1;
    p.n_tiles = g.p.n_tiles; p.w_pairs = (g.p.n_tiles + 1) / 2;
    plan_pair(&p, GP_PLAIN, false, std::max(1, ctas / 2));
    if (!make_tmap(&pm.a[0], w, N, K, 128) || !make_tmap(&pm.b, x, M, K, p.tile_rows / 2) || (p.cut > 1 && !make_tmap(&pm.b_cut, x, M, K, p.tile_rows / p.cut / 2))) return SPEC_E_CUDA;
    for (int i = 1; i <= GS_MAX_MATS; ++i) p.mat_tile0[i] = p.n_tiles;
    p.out = y; p.ld = (size_t)N; p.n_cols = N;
    p.status = status.report(); p.clear = status.clear();
    if (launch_gp<GP_PLAIN>(st, false, pm, p, std::max(1, ctas / 2)) != cudaSuccess) return SPEC_E_CUDA;
    return status.finish();
  }
  const int cs = M <= 128 ? plain_cluster(g.p.n_tiles, K / 64, ctas) : 0;
  const bool cluster = 2LL * g.p.n_tiles * cs >= g.grid;
  if (!make_tmap(&tm.a[0], w, N, K, 128) || !make_tmap(&tm.b, x, M, K, cluster ? M : g.MT)) return SPEC_E_CUDA;   // (M % 16 == 0)
  if (cluster) {
    // few rows: the CTAs of a tile finish its sums on the chip. Not where their half runs would be longer than the streaming kernel's
    // runs (few tiles and a long inner dimension): the error of a running sum grows with its length.
    ClusterGemmParams p{};
    p.M = M; p.K = K; p.KC = K / 64; p.N = N; p.y = y; p.ldy = (size_t)N;
    p.status = status.report(); p.clear = status.clear();
    if (launch_gc_plain(st, false, g.p.n_tiles, cs, tm, p) != cudaSuccess) return SPEC_E_CUDA;
    return status.finish();
  }
  g.p.part = scratch;
  g.p.slot_stride = (size_t)M * g.p.n_tiles * 128;
  g.p.l2_prefetch = 0;
  g.p.status = status.report();
  // (the partial sums are fully overwritten before they are read)
  if (launch_gs(st, false, g, tm) != cudaSuccess) return SPEC_E_CUDA;
  size_t total = (size_t)M * ((N + 3) / 4);
  if (launch_k(true, part_sum_rows, dim3((unsigned)std::min<size_t>((total + 255) / 256, 4096)), dim3(256), 0, st, plan_view(g), y, M, N, status.clear()) != cudaSuccess)
    return SPEC_E_CUDA;
  return status.finish();
}
int op_linear_f32(const void* x, const void* w, float* y, int M, int N, int K, cudaStream_t st) {
  RowLinear<float> rl{};
  rl.w[0] = static_cast<const float*>(w); rl.rows[0] = N; rl.n_mats = 1;
  const int groups = (N + LR_N - 1) / LR_N;
  const RowLinearShape sh = linear_rows_shape<float>(groups, M, K);
  const float* xf = static_cast<const float*>(x);
  if (linear_held(sh, K)) {
    const HeldShape h = linear_held_shape(sh, M, N);
    (h.cols == 8 ? linear_rows_held<8, 4> : linear_rows_held<4, 8>)<<<h.grid, LR_WARPS * 32, 0, st>>>(xf, rl.w[0], y, (size_t)N, M, N, K, h.ms, nullptr, nullptr, nullptr);
  } else {
    linear_rows<float, LR_PLAIN><<<sh.grid, LR_WARPS * 32, 0, st>>>(xf, rl, y, (size_t)N, nullptr, M, K, groups, sh.ks, sh.ms, RopeStore<float>{}, nullptr);
  }
  return cudaGetLastError() == cudaSuccess ? SPEC_OK : SPEC_E_CUDA;
}
bool op_linear_args_ok(int32_t dtype, const void* x, const void* w, const float* y, int M, int N, int K, int ctas) {
  if (!x || !w || !y || M < 1 || N < 1 || K < 8 || K % 8 || M > 2048) return false;
  if (dtype == 0) return true;
  return dtype == 1 && K % 64 == 0 && M % 16 == 0 && N >= 128 && ctas >= 1 && ctas <= 1024;
}
}  // namespace

int spec_debug_op_wait_timeout(int32_t limit_us, int32_t pinned, int32_t* words, void* cuda_stream) {
  if (!words || limit_us < 1 || limit_us > 100000) return SPEC_E_BADARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  OpStatus status(words, pinned != 0, st);
  if (!status.ok()) return SPEC_E_CUDA;
  wait_probe<<<1, 32, 0, st>>>(status.report(), (unsigned long long)limit_us * 1000ull);
  if (cudaGetLastError() != cudaSuccess) return SPEC_E_CUDA;
  return status.finish();
}

int spec_debug_cluster_residency(int32_t mode, int32_t rows, int32_t tiles, int32_t cluster, int32_t chunks, int32_t* out) {
  constexpr int size[4] = {GC_RES_CLUSTER, GC_GLU_CLUSTER, GC_ROPE_CLUSTER, 0};
  if (!out || mode < 0 || mode > 3 || rows < 1 || rows > (mode == GC_SWIGLU ? 64 : 128) || tiles < 1 || tiles > 1024 || chunks < 1 || chunks > 4096) return SPEC_E_BADARG;
  if (cluster < 1 || cluster > 8 || (size[mode] && cluster != size[mode])) return SPEC_E_BADARG;
  cudaError_t e = cudaErrorInvalidValue;
#define MODES(MT)                                                                       \
  switch (mode) {                                                                       \
    case GC_RESIDUAL: e = cluster_residency<MT, GC_RESIDUAL>(tiles, cluster, chunks, out); break; \
    case GC_ROPE: e = cluster_residency<MT, GC_ROPE>(tiles, cluster, chunks, out); break;         \
    case GC_PLAIN: e = cluster_residency<MT, GC_PLAIN>(tiles, cluster, chunks, out); break;       \
    default:                                                                            \
      if constexpr (MT < 128) e = cluster_residency<MT, GC_SWIGLU>(tiles, cluster, chunks, out);  \
  }
  switch (mt_for_rows(rows)) {
    case 16: MODES(16) break;
    case 32: MODES(32) break;
    case 64: MODES(64) break;
    default: MODES(128) break;
  }
#undef MODES
  return e == cudaSuccess ? SPEC_OK : SPEC_E_CUDA;
}

int spec_debug_pinned_allocations(void) { return status_words().allocations(); }

int spec_build_labels(const int32_t* tokens, int32_t n_seq, int32_t seq_len, int32_t num_heads, int32_t frag_token,
                      int32_t pad_token, int32_t ignore_token, int32_t* labels, void* cuda_stream) {
  if (n_seq == 0 || seq_len == 0) return SPEC_OK;
  if (!tokens || !labels || n_seq < 0 || seq_len < 0 || num_heads < 0 || num_heads > LABEL_MAX_HEADS || n_seq > 65535)
    return SPEC_E_BADARG;
  const bool vec = seq_len % 4 == 0 && (reinterpret_cast<uintptr_t>(labels) & 15) == 0;
  const int threads = vec ? LABEL_VEC_THREADS : LABEL_THREADS, cols = vec ? LABEL_VEC_COLS : LABEL_THREADS;
  auto kernel = vec ? build_labels_vec : build_labels_kernel;
  kernel<<<dim3((seq_len + cols - 1) / cols, n_seq), threads, 0, static_cast<cudaStream_t>(cuda_stream)>>>(tokens, seq_len, num_heads, frag_token, pad_token,
                                                                                                        ignore_token, labels);
  return cudaGetLastError() == cudaSuccess ? SPEC_OK : SPEC_E_CUDA;
}

size_t spec_packed_weight_bytes(int32_t rows, int32_t cols) {
  if (rows < 1 || cols < 64 || cols % 64) return 0;
  return (size_t)((rows + 127) / 128) * (size_t)(cols / 64) * 16384;
}

int spec_pack_weight(const void* w, int32_t rows, int32_t cols, void* packed, void* cuda_stream) {
  const size_t bytes = spec_packed_weight_bytes(rows, cols);
  if (!w || !packed || bytes == 0 || (reinterpret_cast<uintptr_t>(packed) & 15) || (reinterpret_cast<uintptr_t>(w) & 15)) {
    g_create_error = "spec_pack_weight: null or unaligned pointer, or cols not a multiple of 64";
    return SPEC_E_BADARG;
  }
  const size_t units = bytes / 16384;
  if (units > 0x7fffffffu) { g_create_error = "spec_pack_weight: matrix too large"; return SPEC_E_BADARG; }
  pack_weight_tiles<<<(unsigned)units, 256, 0, static_cast<cudaStream_t>(cuda_stream)>>>(static_cast<const bf16*>(w), rows, cols,
                                                                                        static_cast<uint8_t*>(packed));
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) { g_create_error = std::string("pack_weight_tiles: ") + cudaGetErrorString(e); return SPEC_E_CUDA; }
  return SPEC_OK;
}

size_t spec_op_linear_scratch_floats(int32_t M, int32_t N, int32_t K, int32_t ctas) {
  GemmPlan g;
  int rws[1] = {N};
  if (M < 1 || N < 1 || ctas < 1 || !plan_gemm(M, K, 1, rws, ctas, &g)) return 0;
  return plan_part_floats(g);
}

int spec_op_linear(int32_t dtype, const void* x, const void* w, float* y, int32_t M, int32_t N, int32_t K,
                   int32_t ctas, float* scratch, void* cuda_stream) {
  if (!op_linear_args_ok(dtype, x, w, y, M, N, K, ctas)) return SPEC_E_BADARG;
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (dtype == 0) {
    return op_linear_f32(x, w, y, M, N, K, st);
  }
  if (!scratch) return SPEC_E_BADARG;
  return op_linear_bf16(x, w, y, M, N, K, ctas, scratch, spec_op_linear_scratch_floats(M, N, K, ctas), true, st);
}

}  // extern "C"

// ---- the linear operation for callers that cannot allocate device memory ----
// The partial sums and the status word of spec_op_linear_static live here instead of in a
// caller-provided buffer. Every context that loads the library holds these bytes until exit.
static __device__ __align__(256) float g_static_linear_scratch[SPEC_STATIC_SCRATCH_FLOATS + 4];

namespace {
constexpr int kMaxDevices = 64;
float* g_static_scratch_addr[kMaxDevices] = {};   // device address of the array, per device ordinal
}  // namespace

extern "C" int spec_op_linear_static(int32_t dtype, const void* x, const void* w, float* y, int32_t M, int32_t N, int32_t K,
                                     int32_t ctas, void* cuda_stream) {
  if (!op_linear_args_ok(dtype, x, w, y, M, N, K, ctas)) { g_create_error = "spec_op_linear_static: bad argument"; return SPEC_E_BADARG; }
  cudaStream_t st = static_cast<cudaStream_t>(cuda_stream);
  if (dtype == 0) {
    return op_linear_f32(x, w, y, M, N, K, st);
  }
  const size_t need = spec_op_linear_scratch_floats(M, N, K, ctas);
  if (need == 0) { g_create_error = "spec_op_linear_static: bad argument"; return SPEC_E_BADARG; }
  if (need > (size_t)SPEC_STATIC_SCRATCH_FLOATS) {
    char buf[200];
    snprintf(buf, sizeof(buf), "spec_op_linear_static: %zu floats of partial sums exceeds the built-in scratch of %u floats",
             need, (unsigned)SPEC_STATIC_SCRATCH_FLOATS);
    g_create_error = buf;
    return SPEC_E_NOMEM;
  }
  // Set-up, once per device: the array's name is only a host-side handle here, so ask the
  // runtime for its address on the current device and keep it.
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) { g_create_error = "spec_op_linear_static: cudaGetDevice failed"; return SPEC_E_CUDA; }
  float* scratch = g_static_scratch_addr[dev];
  if (!scratch) {
    void* ptr = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&ptr, g_static_linear_scratch);
    if (e != cudaSuccess || !ptr) { g_create_error = std::string("spec_op_linear_static: cudaGetSymbolAddress: ") + cudaGetErrorString(e); return SPEC_E_CUDA; }
    scratch = static_cast<float*>(ptr);
    g_static_scratch_addr[dev] = scratch;
  }
  // the status word sits at the fixed end of the array (not in pinned memory: this entry allocates nothing, on any thread)
  int r = op_linear_bf16(x, w, y, M, N, K, ctas, scratch, (size_t)SPEC_STATIC_SCRATCH_FLOATS, false, st);
  if (r) g_create_error = "spec_op_linear_static: launch or device status failed";
  return r;
}
