// libtarflow: host side of the selective-Jacobi TarFlow engine and its C ABI (see include/tarflow.h).
//
// One tf_model owns: the weights of K flow blocks (fp32, or bf16 matrices + fp32 vectors), two
// token-sequence buffers that ping-pong between blocks, the activation workspace of one causal pass
// over up to max_batch * L rows, the per-layer key/value cache of the sequential path, and the
// sweep-control words.  All sequences stay in raster token order; the block permutation (reversal
// on odd blocks) is folded into the index arithmetic of the embedding and update kernels.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <climits>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <map>
#include <mutex>
#include <string>
#include <tuple>
#include <type_traits>
#include <vector>

#include "../../include/tarflow.h"
#include "attention_mma.cuh"
#include "attention_tc.cuh"
#include "common.cuh"
#include "epilogue.cuh"
#include "f32_engine.cuh"
#include "gemm_tc.cuh"
#include "gemm_tc2.cuh"
#include "gemm_few.cuh"
#include "kernels_simt.cuh"
#include "seq_decode.cuh"
#include "seq_persist.cuh"

// ------------------------------------------------------------------------------------------------
// errors
// ------------------------------------------------------------------------------------------------
static thread_local char g_err[512] = "";
static int fail(int code, const char* fmt, ...) {
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(g_err, sizeof(g_err), fmt, ap);
  va_end(ap);
  return code;
}
#define CU_OK(expr)                                                                       \
  do {                                                                                    \
    cudaError_t e__ = (expr);                                                             \
    if (e__ != cudaSuccess) return fail(TF_ECUDA, "%s: %s", #expr, cudaGetErrorString(e__)); \
  } while (0)
#define TF_TRY(expr)            \
  do {                          \
    int r__ = (expr);           \
    if (r__ < 0) return r__;    \
  } while (0)

// ------------------------------------------------------------------------------------------------
// TMA tensor maps (driver entry point fetched at run time; libcuda is not linked)
// ------------------------------------------------------------------------------------------------
typedef CUresult (*encode_tiled_fn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                    const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                    CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static encode_tiled_fn get_encode_fn() {
  static encode_tiled_fn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<encode_tiled_fn>(p);
  }
  return fn;
}
// bf16 matrix [rows, K] row-major; box = 64 (K) x box_rows, 128-byte swizzle, zero fill outside.
static int make_map_bf16(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t K, uint32_t box_rows) {
  encode_tiled_fn fn = get_encode_fn();
  if (!fn) return fail(TF_ECUDA, "cuTensorMapEncodeTiled entry point not available");
  if ((reinterpret_cast<uintptr_t>(ptr) & 15) || (K * 2) % 16) return fail(TF_EINVAL, "TMA operand not 16-byte aligned");
  cuuint64_t dims[2] = {K, rows};
  cuuint64_t strides[1] = {K * 2};
  cuuint32_t box[2] = {64, box_rows};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(TF_ECUDA, "cuTensorMapEncodeTiled failed (%d)", (int)r);
  return TF_OK;
}

// Store map for the bulk-store epilogues: matrix [rows, cols] row-major of 2-byte (bf16) or 4-byte (fp32) elements,
// box = 128 bytes of a row x 32 rows, 128-byte swizzle.
static int make_map_store(CUtensorMap* map, const void* ptr, uint64_t rows, uint64_t cols, int elem_bytes) {
  encode_tiled_fn fn = get_encode_fn();
  if (!fn) return fail(TF_ECUDA, "cuTensorMapEncodeTiled entry point not available");
  if ((reinterpret_cast<uintptr_t>(ptr) & 15) || (cols * elem_bytes) % 16) return fail(TF_EINVAL, "TMA operand not 16-byte aligned");
  cuuint64_t dims[2] = {cols, rows};
  cuuint64_t strides[1] = {cols * (uint64_t)elem_bytes};
  cuuint32_t box[2] = {(cuuint32_t)(128 / elem_bytes), 32};
  cuuint32_t estr[2] = {1, 1};
  CUresult r = fn(map, elem_bytes == 2 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2,
                  const_cast<void*>(ptr), dims, strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                  CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(TF_ECUDA, "cuTensorMapEncodeTiled (store map) failed (%d)", (int)r);
  return TF_OK;
}

// bf16 tensor [slots][L][cols] seen as 3-D, box = 64 columns x box_rows positions of one slot, 128-byte swizzle:
// positions >= L read as zeros and are not written, whatever L is.
static int make_map_3d(CUtensorMap* map, const void* ptr, uint64_t slots, uint64_t L, uint64_t cols, uint32_t box_rows) {
  encode_tiled_fn fn = get_encode_fn();
  if (!fn) return fail(TF_ECUDA, "cuTensorMapEncodeTiled entry point not available");
  if ((reinterpret_cast<uintptr_t>(ptr) & 15) || (cols * 2) % 16) return fail(TF_EINVAL, "TMA operand not 16-byte aligned");
  cuuint64_t dims[3] = {cols, L, slots};
  cuuint64_t strides[2] = {cols * 2, L * cols * 2};
  cuuint32_t box[3] = {64, box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(TF_ECUDA, "cuTensorMapEncodeTiled (3-D map) failed (%d)", (int)r);
  return TF_OK;
}

// ------------------------------------------------------------------------------------------------
// model
// ------------------------------------------------------------------------------------------------
enum KernelClass {
  KC_LAYOUT, KC_EMBED, KC_LN, KC_GEMM_QKV, KC_ATTN, KC_GEMM_O, KC_GEMM_MLP1, KC_GEMM_MLP2, KC_GEMM_HEAD_UPDATE,
  KC_GEMM_HEAD, KC_AFFINE, KC_CTRL, KC_SEQ_EMBED, KC_SEQ_LN, KC_SEQ_GEMM, KC_SEQ_ATTN, KC_SEQ_UPDATE, KC_SEQ_BLOCK, KC_COUNT
};
static const char* kKernelClassNames[KC_COUNT] = {
    "layout", "embed", "layernorm", "gemm_qkv", "attention", "gemm_out", "gemm_mlp_up", "gemm_mlp_down",
    "gemm_head_update", "gemm_head", "forward_affine", "sweep_control", "seq_embed", "seq_layernorm", "seq_gemm",
    "seq_attention", "seq_update", "seq_block"};

struct Matrix {       // a linear layer's weight [N, K]
  void* w = nullptr;  // float* or bf16*
  int N = 0, K = 0;
  CUtensorMap map;    // bf16 engine: box 64 x bn
  int bn = 0;
  CUtensorMap map_seq;  // bf16 engine: box 64 x 128 for the sequential-step GEMM
  CUtensorMap map_few;  // bf16 engine: box 64 x few_bn for sweeps over few rows
  int few_bn = 0;
  const int2* bounds = nullptr;  // masked layers: per 128 columns the k slabs that hold weights (null: all)
};
struct LayerW {
  float *ln1_g, *ln1_b, *b_qkv, *b_o, *ln2_g, *ln2_b, *b_1, *b_2;
  Matrix w_qkv, w_o, w_1, w_2;
};
struct BlockW {
  float *w_in_t, *b_in, *pos, *cls, *lnf_g, *lnf_b, *b_out;  // b_out interleaved (mu_c, alpha_c)
  Matrix w_out;                                                // rows interleaved the same way
  std::vector<LayerW> layers;
};

struct tf_model {
  tf_config cfg;
  int L, D, d, hid, hd;
  int num_sms = 148;
  std::vector<BlockW> blocks;
  std::vector<void*> allocs;
  std::vector<unsigned char*> guards;   // start of every guard region (two per allocation)
  unsigned char** guards_dev = nullptr; // the same list on the device, built by the first check
  int* guard_count = nullptr;
  int64_t device_bytes = 0;
  // workspace
  float *seq_a = nullptr, *seq_b = nullptr, *h = nullptr, *o = nullptr, *maxdiff = nullptr;
  void *xn = nullptr, *qkv = nullptr, *att = nullptr, *mlp = nullptr, *kcache = nullptr, *vcache = nullptr;
  void *xn_lo = nullptr, *qkv_lo = nullptr, *att_lo = nullptr, *mlp_lo = nullptr;  // second terms (bf16 engine)
  CUtensorMap map_xn, map_att, map_mlp, map_xn_lo, map_att_lo, map_mlp_lo;
  enum { SM_QKV, SM_QKV_LO, SM_MLP, SM_MLP_LO, SM_H, SM_ATT3, SM_ATT3_LO, SM_PART, SM_COUNT };
  CUtensorMap map_qkv3, map_kv3, map_qkv3_lo, map_kv3_lo;  // qkv as [slot][position][3d] for the tensor-core attention (query / key boxes)
  bool use_tc_attention = true;   // single-operand attention on tcgen05 (TARFLOW_ATTN_TC=0: the mma.sync kernel)
  bool use_tc_attention_split = true;  // two-term attention on tcgen05 too (TARFLOW_ATTN_TC_SPLIT=0: mma.sync)
  CUtensorMap* store_maps = nullptr;  // device copy of the bulk-store maps of qkv, qkv_lo, mlp, mlp_lo, h
  CUtensorMap map_seq_a[3][3];  // sequential-step GEMM operands {xn, att, mlp} x row tile {16, 32, 64}
  bool use_pair_gemm = true;    // sweep GEMMs on 2-CTA tile pairs (false: one CTA per tile)
  bool seq_use_tc = true;       // sequential-step GEMMs on tcgen05 (false: the mma.sync kernel)
  int seq_fuse_tail = -1;       // step tail (final LN, head, update, embed, next LN) in one kernel: -1 = when the head
                                // matrix is at most 64 KB, 0 = never, 1 = always
  bool seq_fuse_gelu = false;   // MLP-up step GEMM with K <= 512 applies bias + GELU itself (no K split): one kernel
                                // less per layer, but 16 CTAs instead of 64 stream the weights; measured slower
  int *idx = nullptr, *idx_tmp = nullptr, *phase = nullptr, *ctrl = nullptr, *iters_sample = nullptr, *err = nullptr;
  // sweep control of large batches (more than FIN_CHUNK samples): per-slot decisions and per-CTA counts
  unsigned char* fin_code = nullptr;
  int *fin_cnt = nullptr, *fin_flag = nullptr;
  float* fin_top = nullptr;
  // precision policy of Jacobi blocks on the bf16 engine: 0 = escalate per sample, 1 = single bf16
  // operands only, 2 = two-term operands for every sweep
  int precision_mode = 0;
  float switch_threshold = 0.03125f;   // a sample's sweeps use two-term operands once its max|du| <= this
  float single_ok_tau = 0.015625f;     // tau at or above this never escalates
  int* ctrl_host = nullptr;  // pinned, written by the sweep-control kernels themselves (HOST_* words of kernels_simt.cuh)
  int sweep_seq = 0;         // sweep-control launches so far: the value their sequence word has to reach
  // sequential decoding on the bf16 engine: step counter on the device, model-owned copy of the labels
  // (fixed address for captured graphs), one instantiated graph of `unroll` steps per (block, batch)
  int* step_ctr = nullptr;
  int* labels_own = nullptr;
  cudaStream_t cap_stream = nullptr;
  struct SeqGraph { cudaGraphExec_t exec = nullptr; int unroll = 0; int nodes = 0; };
  std::map<std::tuple<int, int, int, int>, SeqGraph> seq_graphs;  // (block g, first sample, samples, buffer set) of a chain
  enum { MAX_CHAINS = 4 };
  cudaStream_t seq_streams[MAX_CHAINS] = {nullptr};  // one stream per chain of a sequential block
  cudaEvent_t seq_fork = nullptr, seq_join[MAX_CHAINS] = {nullptr};
  int seq_chains_force = 0;  // TARFLOW_SEQ_CHAINS=1|2|4: chains per sequential block (0 = by the size of the weights)
  enum { SEQ_TICKETS = 1024 };
  int* seq_tickets = nullptr;      // [MAX_CHAINS][SEQ_TICKETS]
  float2* seq_stats = nullptr;     // [MAX_CHAINS][16 column tiles][max_batch]
  bool seq_kbn8 = true;            // TARFLOW_SEQ_KBN8=0: finishing launches never take eight k slabs per CTA
  // TARFLOW_SEQ_FIN=1: five kernels per layer instead of eight (the last K slice of a projection finishes its tile, the
  // next projection normalises its own operand slice).  Off by default: measured 55.8 / 144.7 / 416 ms per block against
  // 28.3 / 84.1 / 283 ms for the eight-kernel chain (256 tokens width 512, 256 tokens width 1024, 1024 tokens): the
  // fence + ticket + fence of the last arriver and its one-CTA reduction cost more than the kernel boundary and the
  // many-CTA consumer kernel they replace.
  bool seq_fin = false;
  // bf16 engine: blocks decoded by one cooperative launch (seq_persist.cuh)
  std::vector<seqp::Layer*> seqp_layers;       // per block, device memory
  std::vector<float*> seqp_vecs;
  int seqp_groups[2] = {0, 0};                 // groups of 16 / 32 samples that fit the GPU side by side (0: not eligible)
  uint32_t seqp_seq = 1;                       // sequence number of the next exchange
  unsigned long long *seqp_part = nullptr, *seqp_row = nullptr;
  size_t seqp_part_words = 0, seqp_row_words = 0;
  CUtensorMap seqp_cache[2];                   // keys, values
  bool seq_use_persist = true;                 // TARFLOW_SEQ_PERSIST=0: the chain of kernels
  int seqp_turn = -1;                          // device whose SeqpTurn this model shares (-1: none)
  bool seqp_debug_refuse = false;              // tf_debug_set: the launch asks for what no CTA can have
  int seq_attn_threads = 0;  // TARFLOW_SEQ_ATTN_THREADS=128|256: CTA size of the step attention (0 = by the number of CTAs)
  int seq_kbn_force = 0;     // TARFLOW_SEQ_KBN
  bool seq_nc_forced = false;  // TARFLOW_SEQ_NC is set
  // Jacobi sweeps over few rows are replayed from graphs: one per (block, single-term slots, two-term slots, buffers).  The
  // current slot list is one of the buffers: idx and idx_tmp change places after every sweep of more than FIN_CHUNK samples.
  std::map<std::tuple<int, int, int, const void*, const void*, const void*, const void*, const void*>, SeqGraph> sweep_graphs;
  int small_m_rows = 1024;      // TARFLOW_SMALL_M_ROWS: sweeps of at most this many rows use 128 x 128 single-CTA tiles
  int split_m_rows = 4096;      // TARFLOW_SPLIT_M_ROWS: up to this many rows the residual projections on pair tiles are cut in K too
  bool small_m_split = true;    // TARFLOW_SMALL_M_SPLIT=0: the residual projections of such sweeps keep whole-K tiles
  float* sweep_part = nullptr;  // K-slice partial products of the residual projections of such sweeps [part_cap_rows, d]
  int part_cap_rows = 0;
  int64_t sweep_graph_rows = 4096;  // TARFLOW_SWEEP_GRAPH_ROWS: largest slots x tokens replayed from a graph (0 = never)
  // fp32 engine: blocks that fit a cluster's shared memory are decoded by one launch (f32_engine.cuh)
  f32::SeqPlan seq_plan;
  std::vector<float*> seq_image;              // per block, the images of a cluster's CTAs
  int seq_clusters = 0;                       // clusters that fit the GPU side by side (0: not eligible)
  int seq_cluster_smem[3] = {0, 0, 0};        // dynamic shared memory with 1, 2, 4 samples per cluster (0: does not fit)
  int seq_cluster_tail[3] = {0, 0, 0};        // how much of the head and embedding matrices is in shared memory too
  int seq_variant = 0;       // 0: the block's own token buffers, 1: the compact buffers of the sequential fall-back
  size_t seq_part_row_floats = 0;  // floats of partial tiles available per sample
  bool use_graphs = true;
  int seq_check_steps = 0;    // 1 when a replayed graph can run past the last step (kernels then test the counter)
  float* seq_part = nullptr;  // fp32 partial tiles [K slices][B][N] of the projection in flight
  size_t seq_part_floats = 0;
  float *cmp_v = nullptr, *cmp_u = nullptr, *ref_seq = nullptr;  // compact token buffers (fall-back), reference state
  int* cmp_labels = nullptr;
  float* trace_l2 = nullptr;            // [n_blocks][trace_l2_sweeps][max_batch] when the trace is on
  int trace_l2_sweeps = 0;
  std::vector<int> trace_l2_count;      // sweeps recorded per block in the last call
  // second workload: MLP-based autoregressive flow (MADE networks, App. E.3).  Such a model reuses the token buffers
  // (L = D values of token dimension 1), the sweep control and the GEMM machinery; the TarFlow calls refuse it.
  bool is_maf = false;
  struct MafBlock { Matrix w1, w2, w3; float *b1 = nullptr, *b2 = nullptr, *b3 = nullptr; };
  std::vector<MafBlock> maf_blocks;
  int maf_H = 0;
  void *maf_a0 = nullptr, *maf_a0_lo = nullptr, *maf_h1 = nullptr, *maf_h1_lo = nullptr, *maf_h2 = nullptr, *maf_h2_lo = nullptr;
  CUtensorMap maf_map[3][2];               // A-operand maps of {a0, h1, h2} x {hi, lo}
  CUtensorMap* maf_store_maps = nullptr;   // device copy: bulk-store maps of h1, h1_lo, h2, h2_lo, o (fp32)
  float *io_z = nullptr, *io_x = nullptr;  // staging for the host-buffer entry point
  int* io_labels = nullptr;
  cudaStream_t stream = nullptr;
  int64_t launches = 0;
  // profiling
  bool prof_on = false;
  int prof_mode = 0;       // 1: every launch; 2: sweep kernels per launch, a sequential block as one timed unit (from its graph)
  bool prof_suspend = false;
  std::vector<cudaEvent_t> ev_pool;
  std::vector<std::pair<cudaEvent_t, cudaEvent_t>> ev_pending[KC_COUNT];
  double prof_ms[KC_COUNT] = {0};
  int64_t prof_n[KC_COUNT] = {0};
  double prof_rows[KC_COUNT] = {0};  // activation rows the timed launches of a class processed
  int64_t cur_rows = 0;              // rows of the launches being issued (set by the pass drivers)
  cudaEvent_t cur_start = nullptr;
  // convergence trace (one record per sweep of the last inverse call)
  struct TraceRec { int block, sweep, active; float maxdiff; };
  bool trace_on = false;
  std::vector<TraceRec> trace;
  std::vector<cudaEvent_t> block_ev;  // n_blocks + 1 events bracketing the blocks of the last inverse call
  bool block_ev_valid = false;

  cudaEvent_t get_event() {
    if (!ev_pool.empty()) {
      cudaEvent_t e = ev_pool.back();
      ev_pool.pop_back();
      return e;
    }
    cudaEvent_t e;
    cudaEventCreate(&e);
    return e;
  }
  void pre(int) {
    if (prof_on && !prof_suspend) {
      cur_start = get_event();
      cudaEventRecord(cur_start, stream);
    }
  }
  void drop() {  // the launch announced by pre() did not take place
    if (prof_on && !prof_suspend) ev_pool.push_back(cur_start);
  }
  void post(int cls) {
    ++launches;
    if (prof_on && !prof_suspend) {
      cudaEvent_t e = get_event();
      cudaEventRecord(e, stream);
      ev_pending[cls].push_back({cur_start, e});
      prof_rows[cls] += (double)cur_rows;
    }
  }
  void prof_collect() {
    for (int c = 0; c < KC_COUNT; ++c) {
      for (auto& pr : ev_pending[c]) {
        float ms = 0.f;
        cudaEventSynchronize(pr.second);
        cudaEventElapsedTime(&ms, pr.first, pr.second);
        prof_ms[c] += ms;
        prof_n[c] += 1;
        ev_pool.push_back(pr.first);
        ev_pool.push_back(pr.second);
      }
      ev_pending[c].clear();
    }
  }
};

#define LAUNCH(m, cls, kern, grid, block, smem, ...)           \
  do {                                                         \
    (m)->pre(cls);                                             \
    kern<<<(grid), (block), (smem), (m)->stream>>>(__VA_ARGS__); \
    (m)->post(cls);                                            \
  } while (0)

// Launch with programmatic stream serialization: only for kernels that call pdl_wait() before they touch global
// memory, so their CTAs may be scheduled while the previous kernel of the stream drains.
template <class... KArgs, class... Args>
static void launch_pdl_raw(cudaStream_t stream, void (*kern)(KArgs...), dim3 grid, dim3 block, size_t smem, Args... args) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = block;
  lc.dynamicSmemBytes = smem;
  lc.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  cudaLaunchKernelEx(&lc, kern, static_cast<KArgs>(args)...);  // errors surface in check_launch()
}
#define LAUNCH_PDL(m, cls, kern, grid, block, smem, ...)                                        \
  do {                                                                                          \
    (m)->pre(cls);                                                                              \
    launch_pdl_raw((m)->stream, kern, dim3(grid), dim3(block), (size_t)(smem), __VA_ARGS__);    \
    (m)->post(cls);                                                                             \
  } while (0)

static int check_launch(const char* what) {
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return fail(TF_ECUDA, "%s: %s", what, cudaGetErrorString(e));
  return TF_OK;
}

// Per-device host state (kernel attributes set, error words, symbol addresses) is indexed by device ordinal.
constexpr int kMaxDevices = 64;
static int current_device() {
  int dev = -1;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return -1;
  return dev;
}

// Every device buffer of a model sits between two guard regions of GUARD_BYTES filled with a fixed pattern.  A kernel
// that writes outside its buffer (the kind of fault a memory checker would report) damages a guard instead of a
// neighbouring buffer, and tf_debug_check_guards counts the damaged words after any call.
constexpr size_t GUARD_BYTES = 256;
constexpr unsigned char GUARD_BYTE = 0xA5;

template <class T>
static int dev_alloc(tf_model* m, T** p, size_t count) {
  size_t bytes = ((count * sizeof(T)) + 255) & ~(size_t)255;
  if (bytes == 0) bytes = 256;
  void* q = nullptr;
  cudaError_t e = cudaMalloc(&q, bytes + 2 * GUARD_BYTES);
  if (e != cudaSuccess) {
    cudaGetLastError();
    return fail(TF_ENOMEM, "cudaMalloc(%zu bytes) failed: %s", bytes, cudaGetErrorString(e));
  }
  m->allocs.push_back(q);
  unsigned char* base = reinterpret_cast<unsigned char*>(q);
  CU_OK(cudaMemset(base, GUARD_BYTE, GUARD_BYTES));
  CU_OK(cudaMemset(base + GUARD_BYTES + bytes, GUARD_BYTE, GUARD_BYTES));
  m->guards.push_back(base);
  m->guards.push_back(base + GUARD_BYTES + bytes);
  m->device_bytes += (int64_t)(bytes + 2 * GUARD_BYTES);
  *p = reinterpret_cast<T*>(base + GUARD_BYTES);
  return TF_OK;
}

// ------------------------------------------------------------------------------------------------
// GEMM dispatch
// ------------------------------------------------------------------------------------------------
template <int BN, int STAGES, class Epi>
static int launch_gemm_tc(tf_model* m, int cls, cudaStream_t stream, const CUtensorMap& ma, const CUtensorMap* ma_lo,
                          const CUtensorMap& mw, int M, int N, int K, const Epi& epi, int* err, int num_sms,
                          int64_t* launches, int ksplit = 1, int part_rows = 0, const int2* bounds = nullptr) {
  using SL = tc::SmemLayout<BN, STAGES>;
  if (ksplit < 1 || ksplit > (K + tc::BK - 1) / tc::BK || (ksplit > 1 && Epi::kTmaCols == 0))
    return fail(TF_EINVAL, "gemm_tc_kernel: bad K split %d", ksplit);
  auto kern = tc::gemm_tc_kernel<BN, STAGES, Epi>;
  static bool configured[kMaxDevices] = {false};  // per instantiation and device
  const int dev = current_device();
  if (dev < 0) return fail(TF_ECUDA, "no usable current device");
  if (!configured[dev]) {
    CU_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, SL::TOTAL));
    configured[dev] = true;
  }
  int tiles = ((M + tc::BM - 1) / tc::BM) * ((N + BN - 1) / BN) * ksplit;
  int grid = tiles < num_sms ? tiles : num_sms;
  if (m) m->pre(cls);
  launch_pdl_raw(stream, kern, dim3(grid), dim3(tc::NUM_THREADS), (size_t)SL::TOTAL, ma, ma_lo ? *ma_lo : ma, mw, M, N, K,
                 ma_lo ? 1 : 0, epi, err, ksplit, part_rows, bounds);
  if (m) m->post(cls); else if (launches) ++*launches;
  return check_launch("gemm_tc_kernel");
}

// pair kernel: 256 x 256 tiles on clusters of two CTAs (N % 256 == 0, bulk-store epilogues)
template <class Epi>
static int launch_gemm_tc2(tf_model* m, int cls, const CUtensorMap& ma, const CUtensorMap* ma_lo, const CUtensorMap& mw, int M,
                           int N, int K, const Epi& epi, int ksplit = 1, int part_rows = 0, const int2* bounds = nullptr) {
  if (ksplit < 1 || ksplit > (K + tc::BK - 1) / tc::BK) return fail(TF_EINVAL, "gemm_tc2_kernel: bad K split %d", ksplit);
  auto kern = tc2::gemm_tc2_kernel<Epi>;
  static bool configured[kMaxDevices] = {false};  // per instantiation and device
  const int dev = current_device();
  if (dev < 0) return fail(TF_ECUDA, "no usable current device");
  if (!configured[dev]) {
    CU_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, tc2::Smem2::TOTAL));
    configured[dev] = true;
  }
  const int tiles = ((M + 2 * tc::BM - 1) / (2 * tc::BM)) * (N / tc2::BN2) * ksplit;
  int pairs = m->num_sms / 2;
  if (tiles < pairs) pairs = tiles;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(2 * pairs);
  lc.blockDim = dim3(tc::NUM_THREADS);
  lc.dynamicSmemBytes = tc2::Smem2::TOTAL;
  lc.stream = m->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = 2;
  at[0].val.clusterDim.y = 1;
  at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 2;
  m->pre(cls);
  cudaError_t e = cudaLaunchKernelEx(&lc, kern, ma, ma_lo ? *ma_lo : ma, mw, M, N, K, ma_lo ? 1 : 0, epi, m->err, ksplit, part_rows, bounds);
  m->post(cls);
  if (e != cudaSuccess) return fail(TF_ECUDA, "gemm_tc2_kernel launch failed: %s", cudaGetErrorString(e));
  return TF_OK;
}

// few rows: one 128 x BN tile, or a K slice of one, per CTA (gemm_few.cuh); W.map_few has a box of BN rows
template <int BN, class Epi>
static int launch_few(tf_model* m, int cls, const CUtensorMap& ma, const CUtensorMap* ma_lo, const Matrix& W, int M, const Epi& epi,
                      const float* bias, int ksplit = 1, int part_rows = 0) {
  using C = few::Cfg<BN>;
  if (ksplit < 1 || ksplit > (W.K + tc::BK - 1) / tc::BK || W.few_bn != BN) return fail(TF_EINVAL, "gemm_few_kernel: bad K split %d or tile %d", ksplit, BN);
  auto kern = few::gemm_few_kernel<BN, Epi>;
  static bool configured[kMaxDevices] = {false};  // per instantiation and device
  const int dev = current_device();
  if (dev < 0) return fail(TF_ECUDA, "no usable current device");
  if (!configured[dev]) {
    CU_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::MAX_RING + C::EXTRA));
    configured[dev] = true;
  }
  const int per = ((W.K + tc::BK - 1) / tc::BK + ksplit - 1) / ksplit, want = ma_lo ? few::STAGES_SPLIT : few::STAGES;
  int ring = (per < want ? per : want) * ((ma_lo ? 2 : 1) * C::A_BYTES + C::W_BYTES);
  if (ring < 8 * few::BOX) ring = 8 * few::BOX;  // the epilogue's boxes
  const int tiles = (M + tc::BM - 1) / tc::BM * ((W.N + BN - 1) / BN);
  LAUNCH_PDL(m, cls, kern, tiles * ksplit, few::THREADS, ring + C::EXTRA, ma, ma_lo ? *ma_lo : ma, W.map_few, M, W.N, W.K, ma_lo ? 1 : 0, epi, bias,
             m->err, ksplit, part_rows, ring);
  return check_launch("gemm_few_kernel");
}

// Whether the narrow tiles of a product fit the GPU at once: beyond one wave the wider tiles of the other kernels win (256-token
// sweeps of width 1024, narrow / wide tiles everywhere: 1 sample 335 / 385 us and, with two-term operands, 414 / 522; 4 samples
// 809 / 567).
static bool few_fits(const tf_model* m, int M, const Matrix& W) {
  return m->small_m_rows > 0 && W.few_bn > 0 && (M + tc::BM - 1) / tc::BM * ((W.N + W.few_bn - 1) / W.few_bn) <= m->num_sms;
}

template <int BM, int BN, int TM, class Epi>
static int launch_gemm_f32(tf_model* m, int cls, const float* A, const Matrix& W, int M, const Epi& epi) {
  using C = f32::GemmCfg<BM, BN, TM>;
  auto kern = f32::gemm_kernel<BM, BN, TM, Epi>;
  static bool configured[kMaxDevices] = {false};  // per instantiation and device
  const int dev = current_device();
  if (dev < 0) return fail(TF_ECUDA, "no usable current device");
  if (!configured[dev]) {
    CU_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, C::SMEM));
    configured[dev] = true;
  }
  LAUNCH_PDL(m, cls, kern, dim3((W.N + BN - 1) / BN, (M + BM - 1) / BM), C::THREADS, C::SMEM, A, reinterpret_cast<const float*>(W.w), M,
             W.N, W.K, epi);
  return check_launch("f32::gemm_kernel");
}

// fp32 product.  The tile shrinks until about every SM has one: the kernels are short and few, so spreading a product over
// more SMs matters more than operand reuse.  Rows per thread were chosen by the reads from shared memory that an output costs
// (sweeps of 64 tokens, width 128: 16 x 32 tiles with 1 / 2 / 4 rows per thread 89.4 / 76.8 / 78.3 us at 4 samples, 32 x 32 tiles with
// 2 / 4 116 / 104 us at 16; 16 x 16 tiles where 16 x 32 ones would reach half of the SMs at most: 71.6 -> 67.3 us at 4, 62 -> 54 at 1).
// The head with the update in its epilogue keeps two rows per thread in 32 x 32 tiles (width 32, 256 samples 199.2 us with four, 195.7 with
// two; width 64 325.2 and 321.6).
// K % 4 != 0 (an MLP flow of odd dimension) takes the scalar-load kernel.
template <class T, class Epi>
static int launch_gemm_simt(tf_model* m, int cls, const T* A, const Matrix& W, int M, const Epi& epi) {
  if constexpr (sizeof(T) == 4) {
    if (W.K % 4 == 0) {
      auto tiles = [&](int bm, int bn) { return ((M + bm - 1) / bm) * ((W.N + bn - 1) / bn); };
      if (tiles(64, 64) >= 2 * m->num_sms) return launch_gemm_f32<64, 64, 8>(m, cls, A, W, M, epi);
      constexpr int TM32 = std::is_same<Epi, EpiHeadUpdate>::value ? 2 : 4;
      if (tiles(32, 32) >= m->num_sms) return launch_gemm_f32<32, 32, TM32>(m, cls, A, W, M, epi);
      if (tiles(16, 32) * 2 <= m->num_sms) return launch_gemm_f32<16, 16, 1>(m, cls, A, W, M, epi);
      return launch_gemm_f32<16, 32, 2>(m, cls, A, W, M, epi);
    }
  }
  dim3 grid((W.N + 63) / 64, (M + 63) / 64);
  LAUNCH(m, cls, (gemm_simt_kernel<T, Epi>), grid, 256, 0, A, reinterpret_cast<const T*>(W.w), M, W.N, W.K, epi);
  return check_launch("gemm_simt_kernel");
}

// A [M, K] activations (type T) times W^T.  bf16 engine: tensor-core kernel (map_a_lo != null: A is a
// two-term pair); fp32 engine: SIMT kernel.
template <class T, class Epi>
static int gemm(tf_model* m, int cls, const T* A, const CUtensorMap* map_a, const CUtensorMap* map_a_lo,
                const Matrix& W, int M, const Epi& epi, int ksplit = 1, int part_rows = 0) {
  if constexpr (sizeof(T) == 2) {
    if constexpr (Epi::kTmaCols > 0) {
      // few rows: 128 x 128 tiles on single CTAs put four times as many SMs on the weights as 256 x 256 pair tiles,
      // and K slices (ksplit > 1: partial products, added by the consumer) fill the rest of the GPU
      if (M <= m->small_m_rows && W.N % 128 == 0)
        return launch_gemm_tc<128, 6, Epi>(m, cls, m->stream, *map_a, map_a_lo, W.map_seq, M, W.N, W.K, epi, m->err,
                                           m->num_sms, nullptr, ksplit, part_rows, W.bounds);
      if (m->use_pair_gemm && W.N % 256 == 0 && M >= 256)
        return launch_gemm_tc2<Epi>(m, cls, *map_a, map_a_lo, W.map_seq, M, W.N, W.K, epi, ksplit, part_rows, W.bounds);
    }
    if (ksplit > 1) return fail(TF_EINVAL, "no K-split kernel for this shape");
    if (W.bn == 256)
      return launch_gemm_tc<256, 4, Epi>(m, cls, m->stream, *map_a, map_a_lo, W.map, M, W.N, W.K, epi, m->err,
                                         m->num_sms, nullptr, 1, 0, W.bounds);
    return launch_gemm_tc<128, 6, Epi>(m, cls, m->stream, *map_a, map_a_lo, W.map, M, W.N, W.K, epi, m->err,
                                       m->num_sms, nullptr, 1, 0, W.bounds);
  } else {
    return launch_gemm_simt<T, Epi>(m, cls, A, W, M, epi);
  }
}

// ------------------------------------------------------------------------------------------------
// one causal pass over n_slots * L rows (a Jacobi sweep, or the forward direction)
// ------------------------------------------------------------------------------------------------
// A projection into the residual stream that was left as K-slice partial products: the LayerNorm after it adds them.
struct SplitSum {
  const float* part;
  int ksplit, part_rows;
  const float* bias;
};

template <class T>
static int layernorm(tf_model* m, int cls, const float* x, const float* g, const float* b, T* y, T* y_lo, int rows,
                     const SplitSum* ss = nullptr) {
  int d = m->d;
  if (ss != nullptr) {  // d % 128 == 0 and d <= 4096 on this path
    LAUNCH_PDL(m, cls, resid_sum_ln_kernel<T>, rows, d / 4, 0, const_cast<float*>(x), ss->part, ss->ksplit, ss->part_rows, ss->bias,
               g, b, y, y_lo, d);
    return check_launch("resid_sum_ln_kernel");
  }
  if (sizeof(T) == 2 && rows <= m->small_m_rows && d % 128 == 0 && d <= 4096) {  // few rows: a CTA per row
    LAUNCH_PDL(m, cls, resid_sum_ln_kernel<T>, rows, d / 4, 0, const_cast<float*>(x), (const float*)nullptr, 0, 0, (const float*)nullptr,
               g, b, y, y_lo, d);
    return check_launch("resid_sum_ln_kernel");
  }
  // a warp per row; CTAs of two warps while there are few (256 rows of width 128: sweep 71.6 -> 68 us), else of eight
  const int threads = rows <= 16 * m->num_sms ? 64 : 256, blocks = (int)(((int64_t)rows * 32 + threads - 1) / threads);
  if (d <= 128 * 1) LAUNCH_PDL(m, cls, (layernorm_kernel<T, 1>), blocks, threads, 0, x, g, b, y, y_lo, rows, d);
  else if (d <= 128 * 4) LAUNCH_PDL(m, cls, (layernorm_kernel<T, 4>), blocks, threads, 0, x, g, b, y, y_lo, rows, d);
  else if (d <= 128 * 8) LAUNCH_PDL(m, cls, (layernorm_kernel<T, 8>), blocks, threads, 0, x, g, b, y, y_lo, rows, d);
  else LAUNCH_PDL(m, cls, (layernorm_kernel<T, 16>), blocks, threads, 0, x, g, b, y, y_lo, rows, d);
  return check_launch("layernorm_kernel");
}

enum PassMode { PASS_JACOBI, PASS_FORWARD };

// hp: every bf16 operand travels as a two-term pair (bf16 engine only).
template <class T>
static int run_pass(tf_model* m, int g, int n_slots, const float* u_src, const int* idx, const int* labels,
                    PassMode mode, const float* v, float* u_upd, bool hp) {
  const BlockW& bw = m->blocks[g];
  const int L = m->L, D = m->D, d = m->d, M = n_slots * L, rev = g & 1;
  T* xn = reinterpret_cast<T*>(m->xn);
  T* qkv = reinterpret_cast<T*>(m->qkv);
  T* att = reinterpret_cast<T*>(m->att);
  T* mlp = reinterpret_cast<T*>(m->mlp);
  T* xn_lo = hp ? reinterpret_cast<T*>(m->xn_lo) : nullptr;
  T* qkv_lo = hp ? reinterpret_cast<T*>(m->qkv_lo) : nullptr;
  T* att_lo = hp ? reinterpret_cast<T*>(m->att_lo) : nullptr;
  T* mlp_lo = hp ? reinterpret_cast<T*>(m->mlp_lo) : nullptr;
  const CUtensorMap* mxl = hp ? &m->map_xn_lo : nullptr;
  const CUtensorMap* mal = hp ? &m->map_att_lo : nullptr;
  const CUtensorMap* mml = hp ? &m->map_mlp_lo : nullptr;
  int ethreads = d < 256 ? d : 256;
  m->cur_rows = M;
  // embedding fused with the first LayerNorm when a thread can own four columns of a row
  const bool fused_embed = d % 4 == 0 && d <= 1024 && (size_t)16 * D * sizeof(float) <= EMBED_TOKEN_BYTES;
  if (fused_embed) {
    const LayerW& l0 = bw.layers[0];
    // Fewer CTAs of sixteen rows than SMs: four rows each instead, as long as fetching the weights four times as often costs less than
    // it saves.  Sweep of four layers, four / sixteen rows: width 256 154 / 164 us (1280 rows), 180 / 178 (2304), width 128 144 / 153 (2304),
    // width 512 213 / 216 (1280) and 251 / 245 (2304); width 1024 with 48 values per token 323 / 324 (1280) and 411 / 400 (2304), with
    // 192 values 361 / 349 (1280) and 486 / 443 (2304), with 12 values 321 / 326 (1536) and 359 / 361 (1792); width 384 183 / 187 (1536).
    const int64_t weights = (int64_t)D * d;
    const int few_rows = d <= 256 ? 16 * m->num_sms : weights <= 24 * 1024 ? 12 * m->num_sms : weights <= 48 * 1024 ? 10 * m->num_sms : 1024;
    const bool few = M <= few_rows;
    const int R = few ? 4 : 16, threads = ((d / 4 + 31) / 32) * 32;
    int cc = EMBED_WEIGHT_BYTES / (2 * d * (int)sizeof(float));  // token values per weight buffer
    cc = cc > D ? D : cc;
    const size_t smem = (size_t)(2 * cc * d + R * D) * sizeof(float);
    if (few)
      LAUNCH_PDL(m, KC_EMBED, (embed_ln_rows_kernel<T, 4>), (M + 3) / 4, threads, smem, u_src, idx, labels, bw.w_in_t, bw.b_in, bw.pos,
                 bw.cls, m->h, l0.ln1_g, l0.ln1_b, xn, xn_lo, L, D, d, rev, M, cc);
    else
      LAUNCH_PDL(m, KC_EMBED, (embed_ln_rows_kernel<T, 16>), (M + 15) / 16, threads, smem, u_src, idx, labels, bw.w_in_t, bw.b_in, bw.pos,
                 bw.cls, m->h, l0.ln1_g, l0.ln1_b, xn, xn_lo, L, D, d, rev, M, cc);
  } else {
    LAUNCH_PDL(m, KC_EMBED, embed_rows_kernel<16>, (M + 15) / 16, ethreads, 16 * D * sizeof(float), u_src, idx, labels,
               bw.w_in_t, bw.b_in, bw.pos, bw.cls, m->h, L, D, d, rev, M);
  }
  TF_TRY(check_launch("embed_kernel"));
  // Few rows (bf16 engine): the two projections into the residual stream have d / 64 or d / 128 column tiles per 128 rows, too few
  // CTAs to stream their weights, so they are cut into K slices that leave partial products; the LayerNorm that follows
  // (this layer's second, the next layer's first, or the block's last) adds them to the stream in slice order.
  const int m_pad = (M + 127) / 128 * 128;
  struct Slices { int n; bool narrow; };  // {1, false}: no partial products, the projection adds to the stream itself
  auto slices_for = [&](const Matrix& W) -> Slices {
    if (sizeof(T) != 2 || m->sweep_part == nullptr || !m->small_m_split || d > 4096) return {1, false};
    auto slices = [&](int tiles, int ctas) {
      int ks = ctas / tiles;
      if (ks > W.K / (2 * tc::BK)) ks = W.K / (2 * tc::BK);  // at least two k slabs per slice
      if (ks > 8) ks = 8;
      if (ks > m->part_cap_rows / m_pad) ks = m->part_cap_rows / m_pad;
      return ks < 1 ? 1 : ks;
    };
    Slices wide = {1, false};
    const bool single = M <= m->small_m_rows, pairs = !single && m->use_pair_gemm && d % 256 == 0 && M >= 256;
    if (single) wide.n = slices((m_pad / 128) * (d / 128), m->num_sms);                                       // 128 x 128 tiles
    else if (pairs && M <= m->split_m_rows) wide.n = slices((M + 255) / 256 * (d / 256), m->num_sms / 2);     // pair tiles
    // A narrow product leaves its sums in the partial buffer however few its slices are: its rows must fit there, and the LayerNorm
    // reads them beside the stream.  Against 128 x 128 tiles that reduce into the stream this pays up to 4096 rows (width 128, narrow /
    // wide: sweep 180 / 178 us, two-term 212 / 223 at 4096 rows, 205 / 199 and 242 / 236 at 5120, 241 / 208 and 290 / 256 at 8192).
    if (m_pad > m->part_cap_rows || !few_fits(m, M, W) || (!single && !pairs && M > 4096)) return wide;
    // Microseconds of a tile's k slabs, plus what the other form costs on top: a further slice for the LayerNorm, a longer epilogue.
    // Per layer at four layers, narrow / wide: down projection, 512 rows of width 1024 8.0 / 6.6 (measured: wide 2.2 faster), 256 rows
    // 4.0 / 4.9 (narrow 0.9 faster), 1280 rows of width 768 12 / 8.1 (wide 5.2 faster), of width 256 1.3 / 4.6 (narrow 4.6 faster);
    // out-projection, 1024 rows of width 1024 4.0 / 3.5 (wide 0.5 faster), 1280 rows of width 512 2.0 / 4.3 (narrow 2.2 faster).
    const int n = slices((m_pad / 128) * (d / 64), m->num_sms);
    const float slabs = (float)(W.K / tc::BK), more = 0.45f * (wide.n - n);
    if (slabs * 0.25f / n > slabs * (pairs ? 0.38f : 0.33f) / wide.n + (pairs ? 2.2f : 0.45f) + more) return wide;
    return {n, true};
  };
  SplitSum pend{nullptr, 0, 0, nullptr};
  bool has_pend = false;
  bool first_layer = true;
  // a projection into the residual stream, W over the activations a (maps ma, ma_lo)
  auto into_stream = [&](int cls, const T* a, const CUtensorMap* ma, const CUtensorMap* ma_lo, const Matrix& W, const float* bias) -> int {
    if constexpr (sizeof(T) == 2) {
      const Slices ks = slices_for(W);
      if (ks.n == 1 && !ks.narrow) return gemm<T>(m, cls, a, ma, ma_lo, W, M, EpiResidTma{bias, m->store_maps + tf_model::SM_H});
      // rows behind the buffer's end would be lost on the way in and read from other memory on the way out
      if ((int64_t)ks.n * m_pad > m->part_cap_rows) return fail(TF_EINVAL, "%d slices of %d rows exceed the partial buffer", ks.n, m_pad);
      const CUtensorMap* part = m->store_maps + tf_model::SM_PART;
      if (ks.narrow) TF_TRY(launch_few<64>(m, cls, *ma, ma_lo, W, M, few::StoreF32{part}, nullptr, ks.n, m_pad));
      else TF_TRY(gemm<T>(m, cls, a, ma, ma_lo, W, M, EpiStoreF32Tma{nullptr, part}, ks.n, m_pad));
      pend = SplitSum{m->sweep_part, ks.n, m_pad, bias};
      has_pend = true;
      return TF_OK;
    } else {
      return gemm<T>(m, cls, a, ma, ma_lo, W, M, EpiResid{m->h, bias, d});
    }
  };
  for (const LayerW& lw : bw.layers) {
    if (!(first_layer && fused_embed)) TF_TRY(layernorm<T>(m, KC_LN, m->h, lw.ln1_g, lw.ln1_b, xn, xn_lo, M, has_pend ? &pend : nullptr));
    has_pend = false;
    first_layer = false;
    if constexpr (sizeof(T) == 2) {
      const CUtensorMap* sm = m->store_maps;
      if (few_fits(m, M, lw.w_qkv)) TF_TRY(launch_few<64>(m, KC_GEMM_QKV, m->map_xn, mxl, lw.w_qkv, M, few::Store<ACT_NONE>{sm + tf_model::SM_QKV, hp ? sm + tf_model::SM_QKV_LO : nullptr}, lw.b_qkv));
      else TF_TRY(gemm<T>(m, KC_GEMM_QKV, xn, &m->map_xn, mxl, lw.w_qkv, M,
                     EpiStoreTma<false>{lw.b_qkv, sm + tf_model::SM_QKV, hp ? sm + tf_model::SM_QKV_LO : nullptr}));
    } else {
      TF_TRY(gemm<T>(m, KC_GEMM_QKV, xn, &m->map_xn, mxl, lw.w_qkv, M, EpiStore<T, false>{qkv, lw.b_qkv, 3 * d, qkv_lo}));
    }
    if constexpr (sizeof(T) == 2) {
      dim3 grid((L + attn::BQ - 1) / attn::BQ, m->cfg.n_heads, n_slots);
      const float sl2 = 1.4426950408889634f / sqrtf((float)m->hd);
      const dim3 grid_tc((L + attn_tc::BQ - 1) / attn_tc::BQ, m->cfg.n_heads, n_slots);
      if (hp && m->use_tc_attention && m->use_tc_attention_split)
        LAUNCH_PDL(m, KC_ATTN, attn_tc::attention_tc_kernel<true>, grid_tc, attn_tc::NUM_THREADS_ATTN, attn_tc::Cfg<true>::SMEM_BYTES,
                   m->map_qkv3, m->map_kv3, m->map_qkv3_lo, m->map_kv3_lo, m->store_maps + tf_model::SM_ATT3,
                   m->store_maps + tf_model::SM_ATT3_LO, L, d, sl2, m->err);
      else if (hp)
        LAUNCH(m, KC_ATTN, attn::attention_mma_kernel<true>, grid, 128, attn::smem_bytes<true>(), qkv, qkv_lo, att,
               att_lo, L, d, sl2);
      else if (m->use_tc_attention)
        LAUNCH_PDL(m, KC_ATTN, attn_tc::attention_tc_kernel<false>, grid_tc, attn_tc::NUM_THREADS_ATTN, attn_tc::Cfg<false>::SMEM_BYTES,
                   m->map_qkv3, m->map_kv3, m->map_qkv3, m->map_kv3, m->store_maps + tf_model::SM_ATT3,
                   m->store_maps + tf_model::SM_ATT3, L, d, sl2, m->err);
      else
        LAUNCH(m, KC_ATTN, attn::attention_mma_kernel<false>, grid, 128, attn::smem_bytes<false>(), qkv, qkv_lo, att,
               att_lo, L, d, sl2);
    } else if (m->hd % 4 == 0 && m->hd <= 128) {
      const dim3 grid((L + f32::AT_Q - 1) / f32::AT_Q, m->cfg.n_heads, n_slots);
      const size_t smem = f32::attention_smem_floats(m->hd) * sizeof(float);
      const float scale = 1.0f / sqrtf((float)m->hd);
      if ((int64_t)grid.x * grid.y * grid.z <= 4 * m->num_sms)
        LAUNCH_PDL(m, KC_ATTN, f32::attention_kernel<1>, grid, 32 * f32::AT_Q, smem, qkv, att, L, d, m->hd, scale);
      else
        LAUNCH_PDL(m, KC_ATTN, f32::attention_kernel<2>, grid, 16 * f32::AT_Q, smem, qkv, att, L, d, m->hd, scale);
    } else {
      const int warps = 4;
      dim3 grid((L + warps - 1) / warps, m->cfg.n_heads, n_slots);
      size_t smem = (size_t)warps * (L + m->hd) * sizeof(float);
      LAUNCH(m, KC_ATTN, (attention_simt_kernel<T>), grid, warps * 32, smem, qkv, att, L, d, m->hd,
             1.0f / sqrtf((float)m->hd));
    }
    TF_TRY(check_launch("attention kernel"));
    TF_TRY(into_stream(KC_GEMM_O, att, &m->map_att, mal, lw.w_o, lw.b_o));
    TF_TRY(layernorm<T>(m, KC_LN, m->h, lw.ln2_g, lw.ln2_b, xn, xn_lo, M, has_pend ? &pend : nullptr));
    has_pend = false;
    if constexpr (sizeof(T) == 2) {
      const CUtensorMap* sm = m->store_maps;
      if (few_fits(m, M, lw.w_1)) TF_TRY(launch_few<64>(m, KC_GEMM_MLP1, m->map_xn, mxl, lw.w_1, M, few::Store<ACT_GELU>{sm + tf_model::SM_MLP, hp ? sm + tf_model::SM_MLP_LO : nullptr}, lw.b_1));
      else TF_TRY(gemm<T>(m, KC_GEMM_MLP1, xn, &m->map_xn, mxl, lw.w_1, M,
                     EpiStoreTma<true>{lw.b_1, sm + tf_model::SM_MLP, hp ? sm + tf_model::SM_MLP_LO : nullptr}));
    } else {
      TF_TRY(gemm<T>(m, KC_GEMM_MLP1, xn, &m->map_xn, mxl, lw.w_1, M, EpiStore<T, true>{mlp, lw.b_1, m->hid, mlp_lo}));
    }
    TF_TRY(into_stream(KC_GEMM_MLP2, mlp, &m->map_mlp, mml, lw.w_2, lw.b_2));
  }
  TF_TRY(layernorm<T>(m, KC_LN, m->h, bw.lnf_g, bw.lnf_b, xn, xn_lo, M, has_pend ? &pend : nullptr));
  if (mode == PASS_JACOBI) {
    if (sizeof(T) == 2 && few_fits(m, M, bw.w_out) && D % 2 == 0) {
      if constexpr (sizeof(T) == 2) {
        if (D % 4 == 0) TF_TRY(launch_few<32>(m, KC_GEMM_HEAD_UPDATE, m->map_xn, mxl, bw.w_out, M, few::HeadUpdate<4>{v, u_upd, m->maxdiff, idx, L, D, rev}, bw.b_out));
        else TF_TRY(launch_few<32>(m, KC_GEMM_HEAD_UPDATE, m->map_xn, mxl, bw.w_out, M, few::HeadUpdate<2>{v, u_upd, m->maxdiff, idx, L, D, rev}, bw.b_out));
      }
    } else {
      EpiHeadUpdate epi{v, u_upd, m->maxdiff, idx, bw.b_out, L, D, rev};
      TF_TRY(gemm<T>(m, KC_GEMM_HEAD_UPDATE, xn, &m->map_xn, mxl, bw.w_out, M, epi));
    }
  } else {
    TF_TRY(gemm<T>(m, KC_GEMM_HEAD, xn, &m->map_xn, mxl, bw.w_out, M, EpiStore<float, false>{m->o, bw.b_out, 2 * D}));
  }
  return TF_OK;
}

// ------------------------------------------------------------------------------------------------
// sequential block with KV cache (Eq. 5): L-1 single-token passes
// ------------------------------------------------------------------------------------------------
// fp32 models whose block fits a cluster's shared memory: the whole block in one launch
static int run_sequential_cluster(tf_model* m, int g, int B, const int* labels, const float* v, float* u) {
  const BlockW& bw = m->blocks[g];
  // one sample per cluster while the clusters fit the GPU side by side, then as many as shared memory allows
  int S = 1;
  while (S < 4 && B > S * m->seq_clusters && m->seq_cluster_smem[S == 1 ? 1 : 2] > 0) S *= 2;
  const int si = S == 1 ? 0 : S == 2 ? 1 : 2;
  static decltype(&f32::seq_cluster_kernel<1, 0>) const kernels[3][3] = {
      {f32::seq_cluster_kernel<1, 0>, f32::seq_cluster_kernel<1, 1>, f32::seq_cluster_kernel<1, 2>},
      {f32::seq_cluster_kernel<2, 0>, f32::seq_cluster_kernel<2, 1>, f32::seq_cluster_kernel<2, 2>},
      {f32::seq_cluster_kernel<4, 0>, f32::seq_cluster_kernel<4, 1>, f32::seq_cluster_kernel<4, 2>}};
  auto kern = kernels[si][m->seq_cluster_tail[si]];
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(f32::SC * ((B + S - 1) / S));
  lc.blockDim = dim3(f32::ST);
  lc.dynamicSmemBytes = m->seq_cluster_smem[si];
  lc.stream = m->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = f32::SC;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  m->cur_rows = (int64_t)B * (m->L - 1);
  m->pre(KC_SEQ_GEMM);
  cudaError_t e = cudaLaunchKernelEx(&lc, kern, m->seq_plan, (const float*)m->seq_image[g], v, u, labels,
                                     (const float*)bw.pos, (const float*)bw.cls, reinterpret_cast<float*>(m->kcache),
                                     reinterpret_cast<float*>(m->vcache), m->cfg.max_batch, B, g & 1, m->err);
  m->post(KC_SEQ_GEMM);
  if (e != cudaSuccess) return fail(TF_ECUDA, "seq_cluster_kernel launch failed: %s", cudaGetErrorString(e));
  return TF_OK;
}

template <class T>
static int run_sequential_block(tf_model* m, int g, int B, const int* labels, const float* v, float* u) {
  const BlockW& bw = m->blocks[g];
  const int L = m->L, D = m->D, d = m->d, rev = g & 1, nl = m->cfg.n_layers;
  T* xn = reinterpret_cast<T*>(m->xn);
  T* q = reinterpret_cast<T*>(m->qkv);
  T* att = reinterpret_cast<T*>(m->att);
  T* mlp = reinterpret_cast<T*>(m->mlp);
  const size_t layer_stride = (size_t)m->cfg.max_batch * L * d;
  const float scale = 1.0f / sqrtf((float)m->hd);
  int ethreads = d < 256 ? d : 256;
  if (m->seq_clusters > 0) return run_sequential_cluster(m, g, B, labels, v, u);
  m->cur_rows = B;
  LAUNCH(m, KC_SEQ_UPDATE, copy_first_token_kernel, (B * D + 127) / 128, 128, 0, v, u, B, L, D, rev);
  for (int t = 0; t + 1 < L; ++t) {
    LAUNCH(m, KC_SEQ_EMBED, embed_kernel, B, ethreads, D * sizeof(float), u, (const int*)nullptr, labels, bw.w_in_t,
           bw.b_in, bw.pos, bw.cls, m->h, L, D, d, rev, t);
    for (int i = 0; i < nl; ++i) {
      const LayerW& lw = bw.layers[i];
      T* kc = reinterpret_cast<T*>(m->kcache) + i * layer_stride;
      T* vc = reinterpret_cast<T*>(m->vcache) + i * layer_stride;
      TF_TRY(layernorm<T>(m, KC_SEQ_LN, m->h, lw.ln1_g, lw.ln1_b, xn, (T*)nullptr, B));
      TF_TRY(launch_gemm_simt<T>(m, KC_SEQ_GEMM, xn, lw.w_qkv, B, EpiQKVCache<T>{q, kc, vc, lw.b_qkv, d, L, t}));
      size_t smem = (size_t)(L + m->hd + 8 + 4 * m->hd) * sizeof(float);
      LAUNCH(m, KC_SEQ_ATTN, (attention_step_kernel<T>), dim3(m->cfg.n_heads, B), 128, smem, q, kc, vc, att, L, d,
             m->hd, t, scale);
      TF_TRY(launch_gemm_simt<T>(m, KC_SEQ_GEMM, att, lw.w_o, B, EpiResid{m->h, lw.b_o, d}));
      TF_TRY(layernorm<T>(m, KC_SEQ_LN, m->h, lw.ln2_g, lw.ln2_b, xn, (T*)nullptr, B));
      TF_TRY(launch_gemm_simt<T>(m, KC_SEQ_GEMM, xn, lw.w_1, B, EpiStore<T, true>{mlp, lw.b_1, m->hid}));
      TF_TRY(launch_gemm_simt<T>(m, KC_SEQ_GEMM, mlp, lw.w_2, B, EpiResid{m->h, lw.b_2, d}));
    }
    TF_TRY(layernorm<T>(m, KC_SEQ_LN, m->h, bw.lnf_g, bw.lnf_b, xn, (T*)nullptr, B));
    TF_TRY(launch_gemm_simt<T>(m, KC_SEQ_GEMM, xn, bw.w_out, B, EpiStore<float, false>{m->o, bw.b_out, 2 * D}));
    LAUNCH(m, KC_SEQ_UPDATE, seq_update_kernel, (B * D + 127) / 128, 128, 0, m->o, v, u, B, L, D, rev, t);
  }
  return check_launch("sequential block");
}

// ---- bf16 engine: fused-LayerNorm skinny GEMMs on tensor cores, replayed from a CUDA graph -------
// Launch of a sequential-step kernel with programmatic dependent launch, so that consecutive kernels of
// the chain overlap their launch latency and weight prefetch (see seq_decode.cuh).
template <class... KArgs, class... Args>
static int launch_seq(tf_model* m, int cls, void (*kern)(KArgs...), dim3 grid, int threads, int smem, Args... args) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = grid;
  lc.blockDim = dim3(threads);
  lc.dynamicSmemBytes = smem;
  lc.stream = m->stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  m->pre(cls);
  cudaError_t e = cudaLaunchKernelEx(&lc, kern, static_cast<KArgs>(args)...);
  m->post(cls);
  if (e != cudaSuccess) return fail(TF_ECUDA, "sequential-step kernel launch failed: %s", cudaGetErrorString(e));
  return TF_OK;
}

// A chain decodes the samples b0 .. b0 + B - 1 of a sequential block on its own stream, with its own step counter
// and its own region of the partial-tile buffer.  Samples are independent, so a block's batch may be split over a few
// chains that run side by side: every kernel of a decoding step is bound by the latency of its dependent chain, not
// by throughput, and the chains fill each other's idle time.  A sample's arithmetic does not depend on the split.
struct SeqCtx {
  int b0 = 0, B = 0;
  int* step_ctr = nullptr;
  float* part = nullptr;
  int* tickets = nullptr;    // last-arriver tickets of the step GEMMs' column tiles (zero between launches)
  float2* stats = nullptr;   // per column tile and sample: (sum, sum of squares) of the residual row, for the next LayerNorm
};

// One skinny GEMM of a decoding step: part[ks][B, N] = A[B, K slice ks] W[N, K slice ks]^T.  Returns the number of
// K slices in *nsplit; the kernel that consumes the tiles adds them up.  CTAs of 64 columns x 256 of K read as many
// activation bytes as weight bytes and give a grid of (N / 64) * (K / 256) CTAs.
// gelu_bias / gelu_out non-null: the caller wants bf16(GELU(product + bias)) in gelu_out.  When the whole reduction
// fits one CTA (K <= 512) the GEMM writes that itself and *nsplit = 0; otherwise it writes partial tiles as usual
// and the caller runs the bias + GELU kernel.
static int seq_gemm(tf_model* m, const SeqCtx& cx, int cls, int abuf, const Matrix& W, int step_off, int* nsplit,
                    const float* gelu_bias = nullptr, bf16* gelu_out = nullptr, const seq::SeqFin* fin = nullptr,
                    const seq::SeqLnA* lna = nullptr) {
  const int N = W.N, K = W.K, n_steps = m->L - 1, B = cx.B;
  const bf16* A = reinterpret_cast<const bf16*>(abuf == 0 ? m->xn : abuf == 1 ? m->att : m->mlp) + (size_t)cx.b0 * K;
  const bf16* w = reinterpret_cast<const bf16*>(W.w);
  const size_t part_cap = (size_t)B * m->seq_part_row_floats;
  if (m->seq_use_tc && gelu_out != nullptr && m->seq_fuse_gelu && K % 64 == 0 && K / 64 <= 8 && N % 4 == 0) {
    *nsplit = 0;
    dim3 grid((N + 127) / 128, 1, (B + 63) / 64);
    return launch_seq(m, cls, seq::seq_gemm_tc_kernel<64, 8>, grid, 128, seq::gemm_tc_smem_bytes<64, 8>(), W.map_seq,
                      m->map_seq_a[abuf][2], cx.b0, B, N, K / 64, cx.part, cx.step_ctr, step_off, n_steps, m->seq_check_steps,
                      m->err, gelu_bias, gelu_out + (size_t)cx.b0 * N, seq::SeqFin{}, seq::SeqLnA{});
  }
  if (m->seq_use_tc) {  // tcgen05 kernel: CTAs of 128 columns x kbn slabs of 64 k
    const int slabs = K / 64;
    int kbn = slabs % 4 == 0 ? 4 : slabs % 2 == 0 ? 2 : 1;
    // two slabs per CTA (more CTAs) while the grid is below one wave and the partial tiles stay <= 16
    if (kbn == 4 && ((N + 127) / 128) * (slabs / 4) < m->num_sms && slabs / 2 <= 16) kbn = 2;
    // a launch whose last K slice finishes the tile reads all partials of it: keep them to eight where that is possible
    if (fin != nullptr && slabs / kbn > 8 && slabs % 4 == 0) kbn = 4;
    if (fin != nullptr && slabs / kbn > 8 && slabs % 8 == 0 && m->seq_kbn8) kbn = 8;  // eight slab buffers per CTA
    if (m->seq_kbn_force > 0 && slabs % m->seq_kbn_force == 0 && slabs / m->seq_kbn_force <= 16) kbn = m->seq_kbn_force;
    const int ksplit = slabs / kbn;
    if (ksplit > 16) return fail(TF_EINVAL, "sequential decoding: reduction length %d not supported", K);
    *nsplit = fin != nullptr ? 0 : ksplit;  // with a finishing launch nothing is left for the consumer to add up
    if ((size_t)ksplit * B * N > part_cap) return fail(TF_EINVAL, "sequential decoding: partial-tile buffer too small");
    const int ri = B <= 16 ? 0 : B <= 32 ? 1 : 2, rt = 16 << ri;
    dim3 grid((N + 127) / 128, ksplit, (B + rt - 1) / rt);
    if (fin != nullptr && (int)(grid.x * grid.z) > tf_model::SEQ_TICKETS) return fail(TF_EINVAL, "sequential decoding: too many column tiles");
    const seq::SeqFin fin_v = fin ? *fin : seq::SeqFin{};
    const seq::SeqLnA lna_v = lna ? *lna : seq::SeqLnA{};
#define TF_SEQ_TC_CASE(RTV)                                                                                              \
  if (rt == RTV)                                                                                                         \
    return launch_seq(m, cls, seq::seq_gemm_tc_kernel<RTV>, grid, 128, seq::gemm_tc_smem_bytes<RTV>(), W.map_seq,         \
                      m->map_seq_a[abuf][ri], cx.b0, B, N, kbn, cx.part, cx.step_ctr, step_off, n_steps,                 \
                      m->seq_check_steps, m->err, (const float*)nullptr, (bf16*)nullptr, fin_v, lna_v);
#define TF_SEQ_TC_CASE8(RTV)                                                                                             \
  if (rt == RTV && kbn == 8)                                                                                             \
    return launch_seq(m, cls, seq::seq_gemm_tc_kernel<RTV, 8>, grid, 128, seq::gemm_tc_smem_bytes<RTV, 8>(), W.map_seq,   \
                      m->map_seq_a[abuf][ri], cx.b0, B, N, kbn, cx.part, cx.step_ctr, step_off, n_steps,                 \
                      m->seq_check_steps, m->err, (const float*)nullptr, (bf16*)nullptr, fin_v, lna_v);
    TF_SEQ_TC_CASE8(16)
    TF_SEQ_TC_CASE8(32)
    TF_SEQ_TC_CASE8(64)
#undef TF_SEQ_TC_CASE8
    TF_SEQ_TC_CASE(16)
    TF_SEQ_TC_CASE(32)
    TF_SEQ_TC_CASE(64)
#undef TF_SEQ_TC_CASE
  }
  if (fin != nullptr || lna != nullptr) return fail(TF_EINVAL, "fused step kernels need the tcgen05 step GEMM");
  const int row_tiles = (B + seq::ROWS - 1) / seq::ROWS;
  int klen = (K % 256 == 0) ? 256 : K;
  while (K / klen > 16 && K % (klen * 2) == 0) klen *= 2;  // at most 16 partial tiles
  if (klen > seq::KC || K / klen > 16) return fail(TF_EINVAL, "sequential decoding: reduction length %d not supported", K);
  const int ksplit = K / klen;
  *nsplit = ksplit;
  if ((size_t)ksplit * B * N > part_cap) return fail(TF_EINVAL, "sequential decoding: partial-tile buffer too small");
  // column slices: the narrowest (most CTAs, shortest per-warp MMA chain) that keeps the grid within two waves; the
  // warps of a CTA split its K slice, which needs klen % (32 * 64 / NC) == 0
  int nc = 64;
  if (klen % 256 == 0 && ((N + 7) / 8) * ksplit <= 2 * m->num_sms) nc = 8;
  else if (klen % 128 == 0 && ((N + 15) / 16) * ksplit <= 2 * m->num_sms) nc = 16;
  else if (klen % 64 == 0 && ((N + 31) / 32) * ksplit <= 2 * m->num_sms) nc = 32;
  if (const char* e = getenv("TARFLOW_SEQ_NC")) {  // tuning aid: force the slice width where it is valid
    const int f = atoi(e);
    if ((f == 8 && klen % 256 == 0) || (f == 16 && klen % 128 == 0) || (f == 32 && klen % 64 == 0) || f == 64) nc = f;
  }
  dim3 grid((N + nc - 1) / nc, ksplit, row_tiles);
  const int smem = seq::gemm_smem_bytes(klen);
#define TF_SEQ_GEMM_CASE(NCV)                                                                                            \
  if (nc == NCV)                                                                                                         \
    return launch_seq(m, cls, seq::seq_gemm_kernel<NCV>, grid, seq::THREADS, smem, A, w, B, N, K, klen, cx.part,         \
                      cx.step_ctr, step_off, n_steps, m->seq_check_steps);
  TF_SEQ_GEMM_CASE(8)
  TF_SEQ_GEMM_CASE(16)
  TF_SEQ_GEMM_CASE(32)
  TF_SEQ_GEMM_CASE(64)
#undef TF_SEQ_GEMM_CASE
  return fail(TF_EINVAL, "no sequential GEMM variant for this shape");
}

static int seq_resid_ln(tf_model* m, const SeqCtx& cx, const float* bias, int nsplit, const float* gamma, const float* beta,
                        int step_off) {
  return launch_seq(m, KC_SEQ_LN, seq::seq_resid_ln_kernel, dim3(cx.B), m->d / 4, 0, m->h + (size_t)cx.b0 * m->d, cx.part, bias,
                    nsplit, gamma, beta, reinterpret_cast<bf16*>(m->xn) + (size_t)cx.b0 * m->d, cx.B, m->d, cx.step_ctr, step_off,
                    m->L - 1, m->seq_check_steps);
}

static bool seq_tail_fused(const tf_model* m) {
  if (m->d % 8 != 0 || m->d > 1024) return false;
  if (m->seq_fuse_tail >= 0) return m->seq_fuse_tail != 0;
  return (size_t)2 * m->D * m->d * sizeof(bf16) <= 64 * 1024;
}

// the fused tail of step step_off (first = 0) or the block's start (first = 1)
static int seq_tail(tf_model* m, const SeqCtx& cx, int g, const int* labels, const float* v, float* u,
                    const float* pending_bias, int pending, int first, int step_off) {
  const BlockW& bw = m->blocks[g];
  const LayerW& l0 = bw.layers[0];
  const int smem = (m->d + 3 * m->D) * (int)sizeof(float);
  const size_t tok0 = (size_t)cx.b0 * m->L * m->D;
  return launch_seq(m, KC_SEQ_UPDATE, seq::seq_tail_kernel, dim3(cx.B), 256, smem, m->h + (size_t)cx.b0 * m->d, cx.part,
                    pending_bias, pending, bw.lnf_g, bw.lnf_b, reinterpret_cast<const bf16*>(bw.w_out.w), bw.b_out, cx.B,
                    v + tok0, u + tok0, labels ? labels + cx.b0 : nullptr, bw.w_in_t, bw.b_in, bw.pos, bw.cls, l0.ln1_g, l0.ln1_b,
                    reinterpret_cast<bf16*>(m->xn) + (size_t)cx.b0 * m->d, m->L, m->D, m->d, g & 1, first, cx.step_ctr, step_off,
                    m->L - 1);
}

static bool seq_chain_fused(const tf_model* m) {
  return m->seq_fin && m->seq_use_tc && !m->seq_fuse_gelu && m->d % 128 == 0 && m->hid % 4 == 0 && m->d / 128 <= 16;
}

static int seq_update_embed(tf_model* m, const SeqCtx& cx, int g, const int* labels, const float* v, float* u, int ns,
                            int first, int step_off) {
  const BlockW& bw = m->blocks[g];
  const int d = m->d, D = m->D, ethreads = d < 128 ? d : 128;
  const size_t tok0 = (size_t)cx.b0 * m->L * D;
  return launch_seq(m, KC_SEQ_UPDATE, seq::seq_update_embed_kernel, dim3(cx.B, (d + ethreads - 1) / ethreads), ethreads,
                    (int)(D * sizeof(float)), cx.part, ns, bw.b_out, cx.B, v + tok0, u + tok0, labels ? labels + cx.b0 : nullptr,
                    bw.w_in_t, bw.b_in, bw.pos, bw.cls, m->h + (size_t)cx.b0 * d, m->L, D, d, g & 1, first, cx.step_ctr, step_off,
                    m->L - 1, (seq_chain_fused(m) && ethreads == 128) ? cx.stats : (float2*)nullptr);
}

// attention of the new token of every (sample, head) of the chain over its cache rows
static int seq_attention(tf_model* m, const SeqCtx& cx, int ns, const float* b_qkv, bf16* kc, bf16* vc, bf16* att, int step_off) {
  const int heads = m->cfg.n_heads, L = m->L;
  const float sl2 = 1.4426950408889634f / sqrtf((float)m->hd);
  // more (sample, head) pairs than three 256-thread CTAs per SM hold at once: the 128-thread form runs as one wave
  const bool small = m->seq_attn_threads == 128 || (m->seq_attn_threads == 0 && heads * cx.B > 3 * m->num_sms);
  if (small)
    return launch_seq(m, KC_SEQ_ATTN, seq::seq_attention_kernel<128>, dim3(heads, cx.B), 128, 0, cx.part, ns, b_qkv, kc, vc, att,
                      cx.B, L, m->d, heads, sl2, cx.step_ctr, step_off, L - 1);
  return launch_seq(m, KC_SEQ_ATTN, seq::seq_attention_kernel<256>, dim3(heads, cx.B), 256, 0, cx.part, ns, b_qkv, kc, vc, att,
                    cx.B, L, m->d, heads, sl2, cx.step_ctr, step_off, L - 1);
}

// kernels of decoding steps step_off .. step_off+count-1 relative to the chain's device step counter
static int seq_enqueue_steps(tf_model* m, const SeqCtx& cx, int g, const int* labels, const float* v, float* u, int count) {
  const BlockW& bw = m->blocks[g];
  const int L = m->L, d = m->d, nl = m->cfg.n_layers, B = cx.B;
  bf16* att = reinterpret_cast<bf16*>(m->att) + (size_t)cx.b0 * d;
  bf16* mlp = reinterpret_cast<bf16*>(m->mlp) + (size_t)cx.b0 * m->hid;
  const size_t layer_stride = (size_t)m->cfg.max_batch * L * d, kv0 = (size_t)cx.b0 * L * d;
  m->cur_rows = B;
  const bool tail = seq_tail_fused(m);
  // Fused form (opt-in, measured slower): the last K slice of a residual projection adds the finished sums to h and
  // leaves the row statistics, the next projection normalises its own K slice of h while staging it, the MLP-up
  // projection applies bias + GELU itself: five kernels per layer instead of eight.
  const bool fused = seq_chain_fused(m);
  float* hrow = m->h + (size_t)cx.b0 * d;
  for (int s = 0; s < count; ++s) {
    const float* pending_bias = nullptr;  // bias of the projection whose partial tiles are not yet in h
    int pending = 0, ns = 0;
    for (int i = 0; i < nl; ++i) {
      const LayerW& lw = bw.layers[i];
      bf16* kc = reinterpret_cast<bf16*>(m->kcache) + i * layer_stride + kv0;
      bf16* vc = reinterpret_cast<bf16*>(m->vcache) + i * layer_stride + kv0;
      if (fused) {
        const seq::SeqLnA ln1{hrow, cx.stats, lw.ln1_g, lw.ln1_b}, ln2{hrow, cx.stats, lw.ln2_g, lw.ln2_b};
        const seq::SeqFin fin_o{2, cx.tickets, lw.b_o, nullptr, hrow, cx.stats};
        const seq::SeqFin fin_1{1, cx.tickets, lw.b_1, mlp, nullptr, nullptr};
        const seq::SeqFin fin_2{2, cx.tickets, lw.b_2, nullptr, hrow, cx.stats};
        if (i == 0 && tail) {  // layer 0's input was normalised by the fused tail of the previous step
          TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 0, lw.w_qkv, s, &ns));
        } else {  // (for layer 0 the statistics come from the embedding kernel)
          TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 0, lw.w_qkv, s, &ns, nullptr, nullptr, nullptr, &ln1));
        }
        TF_TRY(seq_attention(m, cx, ns, lw.b_qkv, kc, vc, att, s));
        int none = 0;
        TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 1, lw.w_o, s, &none, nullptr, nullptr, &fin_o));
        TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 0, lw.w_1, s, &none, nullptr, nullptr, &fin_1, &ln2));
        TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 2, lw.w_2, s, &none, nullptr, nullptr, &fin_2));
        pending_bias = nullptr;
        pending = 0;
        continue;
      }
      // layer 0's input comes from the fused tail of the previous step (or of the block's start) when that is on
      if (!(tail && i == 0)) TF_TRY(seq_resid_ln(m, cx, pending_bias, pending, lw.ln1_g, lw.ln1_b, s));
      TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 0, lw.w_qkv, s, &ns));
      TF_TRY(seq_attention(m, cx, ns, lw.b_qkv, kc, vc, att, s));
      TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 1, lw.w_o, s, &pending));
      TF_TRY(seq_resid_ln(m, cx, lw.b_o, pending, lw.ln2_g, lw.ln2_b, s));
      TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 0, lw.w_1, s, &ns, lw.b_1, reinterpret_cast<bf16*>(m->mlp)));
      if (ns > 0)  // the GEMM left partial tiles: sum them, add the bias, apply GELU
        TF_TRY(launch_seq(m, KC_SEQ_LN, seq::seq_bias_gelu_kernel, dim3((B * (m->hid / 4) + 255) / 256), 256, 0, cx.part, ns,
                          lw.b_1, mlp, B, m->hid, cx.step_ctr, s, L - 1, m->seq_check_steps));
      TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 2, lw.w_2, s, &pending));
      pending_bias = lw.b_2;
    }
    if (tail) {
      TF_TRY(seq_tail(m, cx, g, labels, v, u, pending_bias, pending, 0, s));
      continue;
    }
    if (fused) {  // the head normalises h itself (statistics from the last MLP-down projection)
      const seq::SeqLnA lnf{hrow, cx.stats, bw.lnf_g, bw.lnf_b};
      TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 0, bw.w_out, s, &ns, nullptr, nullptr, nullptr, &lnf));
    } else {
      TF_TRY(seq_resid_ln(m, cx, pending_bias, pending, bw.lnf_g, bw.lnf_b, s));
      TF_TRY(seq_gemm(m, cx, KC_SEQ_GEMM, 0, bw.w_out, s, &ns));
    }
    TF_TRY(seq_update_embed(m, cx, g, labels, v, u, ns, 0, s));
  }
  return check_launch("sequential step kernels");
}

static int seq_unroll(int n_steps) {  // steps per graph: a divisor of n_steps close to 16, so no step is a no-op
  int best = 1;
  for (int c = 1; c <= 32 && c <= n_steps; ++c)
    if (n_steps % c == 0) best = c;
  return best >= 4 ? best : (n_steps < 16 ? n_steps : 16);
}

// How many chains decode a batch of B samples side by side.  Measured (one block, ms): width 512, 4 layers, batch 64:
// 34.8 / 28.3 / 28.4 with 1 / 2 / 4 chains; width 1024, 8 layers, batch 64: 82.0 / 76.0 / 86.1; 1024 tokens, batch 16:
// 287 / 303 / 359.  A chain of 16 samples takes as long as one of 64: the block's time is the length of the dependent
// kernel chain, and a split only hides the small throughput-bound part (attention over the cache, partial sums), while
// every chain streams the weights again.  So: two chains from 32 samples up, otherwise one.
static int seq_chain_count(const tf_model* m, int B) {
  int n = m->seq_chains_force > 0 ? m->seq_chains_force : (B >= 32 ? 2 : 1);
  if (n > tf_model::MAX_CHAINS) n = tf_model::MAX_CHAINS;
  while (n > 1 && B / n < 4) n /= 2;  // at least four samples per chain
  return n < 1 ? 1 : n;
}

// all decoding steps of one chain, enqueued on m->stream (the chain's stream)
static int run_sequential_chain(tf_model* m, const SeqCtx& cx, int g, const int* labels, const float* v, float* u) {
  const int n_steps = m->L - 1;
  CU_OK(cudaMemsetAsync(cx.step_ctr, 0, sizeof(int), m->stream));
  CU_OK(cudaMemsetAsync(cx.tickets, 0, tf_model::SEQ_TICKETS * sizeof(int), m->stream));  // after an aborted launch
  m->cur_rows = cx.B;
  if (seq_tail_fused(m)) TF_TRY(seq_tail(m, cx, g, labels, v, u, nullptr, 0, 1, 0));
  else TF_TRY(seq_update_embed(m, cx, g, labels, v, u, 0, 1, 0));
  if ((m->prof_on && m->prof_mode == 1) || !m->use_graphs) {  // direct launches (per-kernel events need them)
    for (int t = 0; t < n_steps; ++t) {
      TF_TRY(seq_enqueue_steps(m, cx, g, labels, v, u, 1));
      TF_TRY(launch_seq(m, KC_CTRL, seq::seq_advance_kernel, dim3(1), 32, 0, cx.step_ctr, 1));
    }
    return check_launch("sequential block");
  }
  cudaStream_t run_stream = m->stream;
  auto key = std::make_tuple(g, cx.b0, cx.B, m->seq_variant);
  auto it = m->seq_graphs.find(key);
  if (it == m->seq_graphs.end()) {
    tf_model::SeqGraph sg;
    sg.unroll = seq_unroll(n_steps);
    const int64_t before = m->launches;
    cudaGraph_t graph = nullptr;
    m->stream = m->cap_stream;
    cudaError_t e = cudaStreamBeginCapture(m->cap_stream, cudaStreamCaptureModeThreadLocal);
    int r = TF_OK;
    if (e == cudaSuccess) {
      r = seq_enqueue_steps(m, cx, g, labels, v, u, sg.unroll);
      if (r == TF_OK) r = launch_seq(m, KC_CTRL, seq::seq_advance_kernel, dim3(1), 32, 0, cx.step_ctr, sg.unroll);
      e = cudaStreamEndCapture(m->cap_stream, &graph);
    }
    m->stream = run_stream;
    sg.nodes = (int)(m->launches - before);
    m->launches = before;
    if (e != cudaSuccess || r != TF_OK || !graph) {
      if (graph) cudaGraphDestroy(graph);
      cudaGetLastError();
      return r != TF_OK ? r : fail(TF_ECUDA, "capturing the sequential-step graph failed: %s", cudaGetErrorString(e));
    }
    e = cudaGraphInstantiate(&sg.exec, graph, 0);
    cudaGraphDestroy(graph);
    if (e != cudaSuccess) return fail(TF_ECUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(e));
    it = m->seq_graphs.emplace(key, sg).first;
  }
  const tf_model::SeqGraph& sg = it->second;
  const int replays = (n_steps + sg.unroll - 1) / sg.unroll;  // steps past n_steps return at once
  for (int i = 0; i < replays; ++i) CU_OK(cudaGraphLaunch(sg.exec, run_stream));
  m->launches += (int64_t)replays * sg.nodes;
  return TF_OK;
}

// ---- blocks decoded by one cooperative launch
using SeqpKernel = void (*)(seqp::Job);
struct SeqpShape { SeqpKernel kern; int smem, cs, heads; size_t part, row; };  // exchange words per group
template <int D, int RT>
static SeqpShape seqp_shape() {
  using C = seqp::Cfg<D, RT>;
  return {seqp::seq_block_kernel<D, RT>, C::TOTAL, C::CS, C::HEADS, (size_t)RT * C::HEADS * D, (size_t)RT * D / 2};
}
static SeqpShape seqp_shape_of(int d, int rt) {
  if (rt == 16) return d == 1024 ? seqp_shape<1024, 16>() : d == 512 ? seqp_shape<512, 16>() : d == 256 ? seqp_shape<256, 16>() : seqp_shape<128, 16>();
  return d == 1024 ? seqp_shape<1024, 32>() : d == 512 ? seqp_shape<512, 32>() : d == 256 ? seqp_shape<256, 32>() : seqp_shape<128, 32>();
}

constexpr int kLaunchRefused = 1;
// Launches (max_clusters == nullptr), or asks how many clusters fit the GPU side by side.  Returns kLaunchRefused when the
// launch was turned down and the context is none the worse for it (fewer SMs than at load, a tool that allows no such launch).
static int seqp_launch(tf_model* m, const SeqpShape& sh, int groups, const seqp::Job* job, int* max_clusters) {
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(groups * sh.heads * sh.cs);
  lc.blockDim = dim3(seqp::NTHREADS + 32);
  lc.dynamicSmemBytes = sh.smem;
  lc.stream = m->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = sh.cs;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeCooperative;  // the clusters wait on one another
  at[1].val.cooperative = 1;
  lc.attrs = at;
  lc.numAttrs = max_clusters ? 1 : 2;
  if (max_clusters) {
    if (cudaOccupancyMaxActiveClusters(max_clusters, sh.kern, &lc) != cudaSuccess) {
      cudaGetLastError();
      *max_clusters = 0;
    }
    return TF_OK;
  }
  if (m->seqp_debug_refuse) lc.dynamicSmemBytes = 1u << 20;
  const cudaError_t e = cudaLaunchKernelEx(&lc, sh.kern, *job);
  if (e == cudaSuccess) return TF_OK;
  cudaGetLastError();
  if (cudaPeekAtLastError() == cudaSuccess && e != cudaErrorLaunchFailure) return kLaunchRefused;  // an error of the context stays
  return fail(TF_ECUDA, "seq_block_kernel launch failed: %s", cudaGetErrorString(e));
}

// The one-launch blocks of a device take turns.  The CTAs of such a launch wait on one another, so two of them that start side
// by side (two models, two streams) could each hold SMs that the other one's missing CTAs need, until the waits run out.  Every
// launch therefore waits for the one before it; the event lives as long as a model that may launch.  A chain of launches on
// one stream is ordered anyway and pays for an event record and a wait per block.
struct SeqpTurn {
  std::mutex mu;
  int models = 0;
  cudaEvent_t done = nullptr;
};
static SeqpTurn g_seqp_turn[kMaxDevices];
static int seqp_turn_join(tf_model* m) {
  const int dev = current_device();
  if (dev < 0) return fail(TF_ECUDA, "no usable current device");
  SeqpTurn& t = g_seqp_turn[dev];
  std::lock_guard<std::mutex> lock(t.mu);
  if (t.models == 0) CU_OK(cudaEventCreateWithFlags(&t.done, cudaEventDisableTiming));
  ++t.models;
  m->seqp_turn = dev;
  return TF_OK;
}
static void seqp_turn_leave(tf_model* m) {
  if (m->seqp_turn < 0) return;
  SeqpTurn& t = g_seqp_turn[m->seqp_turn];
  std::lock_guard<std::mutex> lock(t.mu);
  if (--t.models == 0) {
    cudaEventDestroy(t.done);
    t.done = nullptr;
  }
  m->seqp_turn = -1;
}

// at load: whether the shape fits, the layers' tables, the exchange buffers
static int seqp_setup(tf_model* m) {
  const int d = m->d;
  if ((d != 128 && d != 256 && d != 512 && d != 1024) || m->hid != 4 * d || m->hd != 64 || m->D > (d == 1024 ? 256 : 128)) return TF_OK;
  size_t part = 0, row = 0;
  for (int i = 0; i < 2; ++i) {
    const SeqpShape sh = seqp_shape_of(d, 16 << i);
    CU_OK(cudaFuncSetAttribute(sh.kern, cudaFuncAttributeMaxDynamicSharedMemorySize, sh.smem));
    int n = 0;
    TF_TRY(seqp_launch(m, sh, 1, nullptr, &n));
    int groups = n / sh.heads;
    if (groups > m->cfg.max_batch) groups = m->cfg.max_batch;
    m->seqp_groups[i] = groups;
    if (groups * sh.part > part) part = groups * sh.part;
    if (groups * sh.row > row) row = groups * sh.row;
  }
  if (m->seqp_groups[0] == 0 || m->seqp_groups[1] == 0) return TF_OK;
  const int64_t cache_rows = (int64_t)m->cfg.n_layers * m->cfg.max_batch * m->cfg.n_heads * m->L;
  if (cache_rows > INT_MAX - 32) return TF_OK;
  TF_TRY(seqp_turn_join(m));
  TF_TRY(make_map_bf16(&m->seqp_cache[0], m->kcache, cache_rows, seqp::HD, 32));
  TF_TRY(make_map_bf16(&m->seqp_cache[1], m->vcache, cache_rows, seqp::HD, 32));
  TF_TRY(dev_alloc(m, &m->seqp_part, part));
  TF_TRY(dev_alloc(m, &m->seqp_row, row));
  m->seqp_part_words = part;
  m->seqp_row_words = row;
  CU_OK(cudaMemset(m->seqp_part, 0, part * sizeof(*m->seqp_part)));
  CU_OK(cudaMemset(m->seqp_row, 0, row * sizeof(*m->seqp_row)));
  for (BlockW& bw : m->blocks) {
    std::vector<seqp::Layer> table;
    float* vecs = nullptr;
    TF_TRY(dev_alloc(m, &vecs, (size_t)seqp::V_COUNT * d * bw.layers.size()));
    m->seqp_vecs.push_back(vecs);
    for (LayerW& lw : bw.layers) {
      seqp::Layer ly;
      TF_TRY(make_map_bf16(&ly.qkv, lw.w_qkv.w, lw.w_qkv.N, lw.w_qkv.K, 64));
      TF_TRY(make_map_bf16(&ly.wo, lw.w_o.w, lw.w_o.N, lw.w_o.K, 64));
      TF_TRY(make_map_bf16(&ly.w1, lw.w_1.w, lw.w_1.N, lw.w_1.K, 64));
      TF_TRY(make_map_bf16(&ly.w2, lw.w_2.w, lw.w_2.N, lw.w_2.K, 64));
      const float* parts[] = {lw.ln1_g, lw.ln1_b, lw.b_qkv, lw.b_o, lw.ln2_g, lw.ln2_b, lw.b_1, lw.b_2};
      const int starts[] = {seqp::V_LN1G, seqp::V_LN1B, seqp::V_BQKV, seqp::V_BO, seqp::V_LN2G, seqp::V_LN2B, seqp::V_B1, seqp::V_B2, seqp::V_COUNT};
      for (int i = 0; i < 8; ++i)
        CU_OK(cudaMemcpy(vecs + (size_t)starts[i] * d, parts[i], (size_t)(starts[i + 1] - starts[i]) * d * sizeof(float), cudaMemcpyDeviceToDevice));
      vecs += (size_t)seqp::V_COUNT * d;
      table.push_back(ly);
    }
    seqp::Layer* dev = nullptr;
    TF_TRY(dev_alloc(m, &dev, table.size()));
    CU_OK(cudaMemcpy(dev, table.data(), table.size() * sizeof(seqp::Layer), cudaMemcpyHostToDevice));
    m->seqp_layers.push_back(dev);
  }
  return TF_OK;
}

// Batches that need more than one launch go to the chain of kernels, whose cost hardly grows with the batch.  Width 1024, 256
// tokens: 64 samples take 61.8 ms in one launch, 74.6 in the chain; 96 samples would take 61.8 + 38.9 ms in two launches, 92.9 in
// the chain, 128 samples 123.6 and 107.  Width 512: 128 samples 26.6 ms and 37.9, 160 samples 39 either way.
static bool seqp_on(const tf_model* m, int B) {
  // a switch of the step kernels asks for the chain they belong to
  const bool chain_wanted = !m->seq_use_tc || m->seq_fin || m->seq_fuse_gelu || m->seq_fuse_tail >= 0 || m->seq_chains_force > 0 ||
                            m->seq_kbn_force > 0 || m->seq_attn_threads > 0 || m->seq_nc_forced || !m->seq_kbn8;
  return !m->seqp_layers.empty() && m->seq_use_persist && !chain_wanted && B <= 32 * m->seqp_groups[1];
}

// TF_OK, kLaunchRefused (nothing has run) or an error
static int run_sequential_persistent(tf_model* m, int g, int B, const int* labels, const float* v, float* u) {
  const BlockW& bw = m->blocks[g];
  const int L = m->L, D = m->D, nl = m->cfg.n_layers, n_steps = L - 1;
  constexpr size_t kL2Half = 64u << 20;  // what may be expected to stay in L2 from one step to the next
  const size_t weights = (size_t)nl * 12 * m->d * m->d * sizeof(bf16);
  // All groups that fit, however few samples each (the groups run side by side and a step's length grows with a group's
  // samples); the 16-sample kernel (shorter exchanges) where that is enough.
  const int i = B <= 16 * m->seqp_groups[0] ? 0 : 1;
  const SeqpShape sh = seqp_shape_of(m->d, 16 << i);
  const int want = B < m->seqp_groups[i] ? B : m->seqp_groups[i];
  seqp::Job job = {};
  job.rows = (B + want - 1) / want;
  job.layers = m->seqp_layers[g];
  job.vecs = m->seqp_vecs[g];
  job.lnf_g = bw.lnf_g; job.lnf_b = bw.lnf_b; job.w_in_t = bw.w_in_t; job.b_in = bw.b_in; job.pos = bw.pos; job.cls = bw.cls;
  job.b_out = bw.b_out; job.w_out = reinterpret_cast<const bf16*>(bw.w_out.w);
  job.v = v; job.u = u; job.labels = labels;
  job.kc = reinterpret_cast<bf16*>(m->kcache); job.vc = reinterpret_cast<bf16*>(m->vcache);
  job.kmap = m->seqp_cache[0]; job.vmap = m->seqp_cache[1];
  job.layer_rows = m->cfg.max_batch * m->cfg.n_heads * L;
  job.xpart = m->seqp_part; job.xrow = m->seqp_row;
  job.n_layers = nl; job.B = B; job.L = L; job.Dt = D; job.reversed = g & 1;
  // Words are recognised by their sequence number alone.  Before the numbers would start over (34 680 a call at 256 tokens and
  // eight blocks of eight layers) what is left of them in the buffers is cleared, rows that few batches reach included.
  const uint32_t numbers = (uint32_t)((2 * nl + 1) * n_steps + 1);
  if (UINT32_MAX - m->seqp_seq < numbers) {
    CU_OK(cudaMemsetAsync(m->seqp_part, 0, m->seqp_part_words * sizeof(*m->seqp_part), m->stream));
    CU_OK(cudaMemsetAsync(m->seqp_row, 0, m->seqp_row_words * sizeof(*m->seqp_row), m->stream));
    m->seqp_seq = 1;
  }
  job.seq0 = m->seqp_seq;
  m->seqp_seq += numbers;
  // One block of width 1024, without / with: 28.5 / 28.5 ms (1 sample), 29.5 / 29.1 (8), 32.5 / 32.4 (16), 38.8 / 39.0 (32),
  // 61.8 / 62.0 (64); 1024 tokens, 16 samples: 177.2 / 178.4.
  job.prefetch_w = weights > kL2Half;
  job.scale_log2e = 1.4426950408889634f / sqrtf((float)m->hd);
  job.err = m->err;
  m->cur_rows = (int64_t)B * n_steps;
  int r;
  {
    SeqpTurn& turn = g_seqp_turn[m->seqp_turn];
    std::lock_guard<std::mutex> lock(turn.mu);
    CU_OK(cudaStreamWaitEvent(m->stream, turn.done, 0));
    m->pre(KC_SEQ_BLOCK);
    r = seqp_launch(m, sh, (B + job.rows - 1) / job.rows, &job, nullptr);
    if (r == TF_OK) m->post(KC_SEQ_BLOCK);
    else m->drop();
    if (r == TF_OK) CU_OK(cudaEventRecord(turn.done, m->stream));
  }
  return r;
}

static int run_sequential_block_bf16(tf_model* m, int g, int B, const int* labels, const float* v, float* u) {
  if (seqp_on(m, B)) {
    const int r = run_sequential_persistent(m, g, B, labels, v, u);
    if (r != kLaunchRefused) return r;  // refused: the chain of kernels needs no cooperation
  }
  const int n_steps = m->L - 1;
  cudaStream_t user = m->stream;
  const bool direct = (m->prof_on && m->prof_mode == 1) || !m->use_graphs;
  m->seq_check_steps = direct ? 0 : (n_steps % seq_unroll(n_steps) != 0);
  const int nch = direct ? 1 : seq_chain_count(m, B);
  if (nch == 1) {
    SeqCtx cx;
    cx.b0 = 0; cx.B = B; cx.step_ctr = m->step_ctr; cx.part = m->seq_part;
    cx.tickets = m->seq_tickets; cx.stats = m->seq_stats;
    return run_sequential_chain(m, cx, g, labels, v, u);
  }
  // fork: the chains start once everything enqueued on the caller's stream so far has completed; join: the caller's
  // stream continues once every chain has finished
  CU_OK(cudaEventRecord(m->seq_fork, user));
  int r = TF_OK;
  for (int c = 0; c < nch && r == TF_OK; ++c) {
    SeqCtx cx;
    cx.b0 = (int)((int64_t)B * c / nch);
    cx.B = (int)((int64_t)B * (c + 1) / nch) - cx.b0;
    cx.step_ctr = m->step_ctr + 16 * c;
    cx.part = m->seq_part + (size_t)cx.b0 * m->seq_part_row_floats;
    cx.tickets = m->seq_tickets + (size_t)c * tf_model::SEQ_TICKETS;
    cx.stats = m->seq_stats + (size_t)c * 16 * m->cfg.max_batch;
    m->stream = m->seq_streams[c];
    cudaError_t e = cudaStreamWaitEvent(m->stream, m->seq_fork, 0);
    if (e != cudaSuccess) r = fail(TF_ECUDA, "cudaStreamWaitEvent: %s", cudaGetErrorString(e));
    if (r == TF_OK) r = run_sequential_chain(m, cx, g, labels, v, u);
    if (r == TF_OK && (e = cudaEventRecord(m->seq_join[c], m->stream)) != cudaSuccess)
      r = fail(TF_ECUDA, "cudaEventRecord: %s", cudaGetErrorString(e));
    if (r == TF_OK && (e = cudaStreamWaitEvent(user, m->seq_join[c], 0)) != cudaSuccess)
      r = fail(TF_ECUDA, "cudaStreamWaitEvent: %s", cudaGetErrorString(e));
  }
  m->stream = user;
  return r;
}

// ------------------------------------------------------------------------------------------------
// Jacobi block (Algorithm 1) with per-sample stopping and active-set compaction
// ------------------------------------------------------------------------------------------------
// A recorded device-side timeout is reported once and the word is cleared, so the model stays usable: kernels
// launched after the word was set returned without work, the ones launched after this call run normally.
static int report_timeout(tf_model* m) {
  const int code = m->ctrl_host[HOST_ERR];
  cudaMemsetAsync(m->err, 0, sizeof(int), m->stream);
  cudaStreamSynchronize(m->stream);
  return fail(TF_ETIMEOUT, "device-side wait expired (code %d)", code);
}

// Waits until the sweep-control kernel of the last sweep enqueued has written its words into pinned host memory.  The
// host polls the sequence word instead of copying the words and synchronising the stream: the next sweep can be
// enqueued about 10 us earlier (three small copies and a stream synchronisation: 12-15 us between sweeps).  Every few
// thousand polls the stream is queried, so a failed launch or fault ends the wait with an error.
static int read_ctrl(tf_model* m) {
  volatile int* seq = m->ctrl_host + HOST_SEQ;
  for (unsigned spin = 1; *seq != m->sweep_seq; ++spin) {
    if ((spin & 8191u) == 0) {
      const cudaError_t e = cudaStreamQuery(m->stream);
      if (e == cudaSuccess && *seq != m->sweep_seq) return fail(TF_ECUDA, "sweep control did not report");
      if (e != cudaSuccess && e != cudaErrorNotReady) return fail(TF_ECUDA, "sweep: %s", cudaGetErrorString(e));
    }
  }
  __atomic_thread_fence(__ATOMIC_ACQUIRE);
  if (m->ctrl_host[HOST_ERR] != 0 || m->ctrl_host[HOST_BAD] != 0) CU_OK(cudaStreamSynchronize(m->stream));
  if (m->ctrl_host[HOST_ERR] != 0) return report_timeout(m);
  if (m->ctrl_host[HOST_BAD] != 0) return fail(TF_ENONFINITE, "non-finite value in the convergence reduction");
  return TF_OK;
}

// synchronise the stream and turn a recorded device-side timeout into an error
static int sync_check(tf_model* m) {
  CU_OK(cudaMemcpyAsync(m->ctrl_host + HOST_ERR, m->err, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
  CU_OK(cudaStreamSynchronize(m->stream));
  if (m->ctrl_host[HOST_ERR] != 0) return report_timeout(m);
  return TF_OK;
}

// Class labels come from the caller's device memory and index the class-embedding table: copy them into the
// model-owned array (a fixed address for captured graphs) clamped to [0, n_classes), and fail with TF_EINVAL when one
// was out of range -- no kernel ever indexes the table with an unchecked id.
static int take_labels(tf_model* m, const int** labels, int B) {
  if (!*labels) return TF_OK;
  if (m->cfg.n_classes <= 0) {  // an unconditional model has no table: the labels are not read at all
    *labels = nullptr;
    return TF_OK;
  }
  LAUNCH(m, KC_CTRL, labels_check_kernel, (B + 127) / 128, 128, 0, *labels, m->labels_own, B, m->cfg.n_classes, m->ctrl + CTRL_LABEL_FLAG);
  TF_TRY(check_launch("labels_check_kernel"));
  CU_OK(cudaMemcpyAsync(m->ctrl_host + HOST_LABEL, m->ctrl + CTRL_LABEL_FLAG, sizeof(int), cudaMemcpyDeviceToHost, m->stream));
  CU_OK(cudaStreamSynchronize(m->stream));
  if (m->ctrl_host[HOST_LABEL] != 0) {
    CU_OK(cudaMemsetAsync(m->ctrl + CTRL_LABEL_FLAG, 0, sizeof(int), m->stream));
    return fail(TF_EINVAL, "a class label lies outside [0, %d)", m->cfg.n_classes);
  }
  *labels = m->labels_own;
  return TF_OK;
}

// Options of one inverse call beyond the policy (all optional; see tf_jacobi_opts in tarflow.h).
struct InvOpts {
  int init_mode = 0;
  const float* u0_img = nullptr;        // [n_blocks][B][C][H][W]
  const float* tau_block = nullptr;     // host [n_blocks]
  int fallback_sweeps = 0;
  float* states_img = nullptr;          // out [n_blocks][B][C][H][W]
  const float* ref_img = nullptr;       // in  [n_blocks][B][C][H][W]
};

static int layout(tf_model* m, float* img, float* seq, int B, int to_seq);
template <class T>
static int run_sequential_any(tf_model* m, int g, int B, const int* labels, const float* v, float* u);
template <class T>
static int maf_pass(tf_model* m, int g, int n_slots, const float* u_src, const int* idx, int mode, const float* v, float* u_upd,
                    bool hp, int only_col);

// one causal pass of a Jacobi sweep over the listed slots, whichever flow the model is
template <class T>
static int sweep_pass(tf_model* m, int g, int n_slots, const float* u_src, const int* idx, const int* labels, const float* v,
                      float* u_upd, bool hp) {
  if (m->is_maf) return maf_pass<T>(m, g, n_slots, u_src, idx, 0, v, u_upd, hp, -1);
  return run_pass<T>(m, g, n_slots, u_src, idx, labels, PASS_JACOBI, v, u_upd, hp);
}

// the pass over sample 0 alone, its head output (biases included) left in m->o
template <class T>
static int first_pass(tf_model* m, int g, const float* u_src, bool hp) {
  if (m->is_maf) return maf_pass<T>(m, g, 1, u_src, nullptr, 1, nullptr, nullptr, hp, -1);
  return run_pass<T>(m, g, 1, u_src, nullptr, nullptr, PASS_FORWARD, nullptr, nullptr, hp);
}

template <class T>
static int run_jacobi_block(tf_model* m, int g, int B, const int* labels, const float* v, float* u, float tau,
                            int max_iters, const InvOpts& op, int* sweeps_out, int* iters_row) {
  const size_t n = (size_t)B * m->L * m->D, img = (size_t)B * m->cfg.C * m->cfg.H * m->cfg.W;
  // u^0 = 0 without class labels: the first sweep's pass is the same for every sample and runs for one of them only
  const bool shared_first = op.init_mode == 0 && labels == nullptr && B > 1;
  if (op.init_mode == 0) CU_OK(cudaMemsetAsync(u, 0, (shared_first ? n / B : n) * sizeof(float), m->stream));
  else if (op.init_mode == 1) CU_OK(cudaMemcpyAsync(u, v, n * sizeof(float), cudaMemcpyDeviceToDevice, m->stream));
  else TF_TRY(layout(m, const_cast<float*>(op.u0_img) + (size_t)g * img, u, B, 1));
  const bool l2 = m->trace_on && op.ref_img != nullptr && m->trace_l2 != nullptr;
  if (l2) TF_TRY(layout(m, const_cast<float*>(op.ref_img) + (size_t)g * img, m->ref_seq, B, 1));
  // precision policy (bf16 engine): which sweeps of a sample use two-term operands
  int start_phase = 0;
  float sw = -1.f;  // never escalate
  if (sizeof(T) == 2) {
    if (m->precision_mode == 2) start_phase = 1;
    else if (m->precision_mode == 0 && tau >= 0.f && tau < m->single_ok_tau) sw = m->switch_threshold;
  }
  LAUNCH(m, KC_CTRL, jacobi_begin_kernel, (B + 1023) / 1024 < 64 ? (B + 1023) / 1024 : 64, 256, 0, m->maxdiff, m->idx, m->phase,
         m->ctrl, B, start_phase, tau, sw, m->sweep_seq);
  int n_active = B, n_hp = start_phase ? B : 0, t = 0;
  const int cap = (op.fallback_sweeps > 0 && op.fallback_sweeps < max_iters) ? op.fallback_sweeps : max_iters;
  // everything one sweep launches: the pass over the single-term samples, the pass over the two-term samples, the
  // sweep control (which takes the sweep number and the thresholds from device memory)
  auto enqueue_sweep = [&](int n_lp, int n_hpp, bool first) -> int {
    if (first) {
      TF_TRY(first_pass<T>(m, g, u, n_hpp > 0));
      const long long units = (long long)B * ((m->L * m->D + FIRST_CHUNK - 1) / FIRST_CHUNK);
      LAUNCH_PDL(m, KC_AFFINE, jacobi_first_update_kernel, (unsigned)((units + 7) / 8), 256, 0, m->o, v, u, m->maxdiff, B, m->L, m->D,
                 m->is_maf ? 0 : g & 1, m->is_maf ? 0 : 1);
      TF_TRY(check_launch("jacobi_first_update_kernel"));
    } else if (n_lp > 0) TF_TRY(sweep_pass<T>(m, g, n_lp, u, m->idx, labels, v, u, false));
    if (!first && n_hpp > 0) TF_TRY(sweep_pass<T>(m, g, n_hpp, u, m->idx + n_lp, labels, v, u, true));
    const int na = n_lp + n_hpp;
    if (na <= FIN_CHUNK || m->fin_code == nullptr) {
      LAUNCH_PDL(m, KC_CTRL, jacobi_finalize_kernel, 1, 256, 0, m->maxdiff, m->idx, m->idx_tmp, m->phase, m->ctrl, iters_row,
                 m->err, m->ctrl_host);
    } else {  // large batches: count / scan / scatter over all SMs; the new slot list is written to the other buffer
      const int nblk = (na + FIN_CHUNK - 1) / FIN_CHUNK;
      LAUNCH(m, KC_CTRL, jacobi_finalize_count_kernel, nblk, FIN_CHUNK, 0, m->maxdiff, m->idx, m->phase, m->ctrl, iters_row,
             m->fin_code, m->fin_cnt, m->fin_top, m->fin_flag, nblk);
      LAUNCH(m, KC_CTRL, jacobi_finalize_scan_kernel, 1, 256, 0, m->fin_cnt, m->fin_top, m->fin_flag, m->ctrl, nblk,
             m->err, m->ctrl_host);
      LAUNCH(m, KC_CTRL, jacobi_finalize_scatter_kernel, nblk, FIN_CHUNK, 0, m->idx, m->idx_tmp, m->fin_code, m->fin_cnt, m->ctrl,
             nblk);
      int* sw_idx = m->idx; m->idx = m->idx_tmp; m->idx_tmp = sw_idx;
    }
    return check_launch("sweep control kernels");
  };
  while (t < cap && n_active > 0) {
    ++t;
    ++m->sweep_seq;
    const int n_lp = n_active - n_hp;
    const bool first = shared_first && t == 1;
    // Few rows: a sweep is a chain of short kernels whose launch cost exceeds their run time, so the whole sweep is
    // captured once per (block, single-term slots, two-term slots) and replayed as a graph afterwards.
    const bool as_graph = m->use_graphs && m->cap_stream != nullptr && !m->prof_on && n_active <= FIN_CHUNK && (int64_t)(first ? 1 : n_active) * m->L <= m->sweep_graph_rows;
    if (as_graph) {
      const auto key = std::make_tuple(g, first ? -1 - n_lp : n_lp, n_hp, (const void*)v, (const void*)u, (const void*)labels, (const void*)iters_row,
                                       (const void*)m->idx);
      auto it = m->sweep_graphs.find(key);
      if (it == m->sweep_graphs.end() && m->sweep_graphs.size() < 2048) {
        tf_model::SeqGraph sg;
        const int64_t before = m->launches;
        cudaStream_t user = m->stream;
        cudaGraph_t graph = nullptr;
        m->stream = m->cap_stream;
        cudaError_t e = cudaStreamBeginCapture(m->cap_stream, cudaStreamCaptureModeRelaxed);
        int r = TF_OK;
        if (e == cudaSuccess) {
          r = enqueue_sweep(n_lp, n_hp, first);
          e = cudaStreamEndCapture(m->cap_stream, &graph);
        }
        m->stream = user;
        sg.nodes = (int)(m->launches - before);
        m->launches = before;
        if (e != cudaSuccess || r != TF_OK || !graph) {
          if (graph) cudaGraphDestroy(graph);
          cudaGetLastError();
          return r != TF_OK ? r : fail(TF_ECUDA, "capturing a sweep graph failed: %s", cudaGetErrorString(e));
        }
        e = cudaGraphInstantiate(&sg.exec, graph, 0);
        cudaGraphDestroy(graph);
        if (e != cudaSuccess) return fail(TF_ECUDA, "cudaGraphInstantiate: %s", cudaGetErrorString(e));
        it = m->sweep_graphs.emplace(key, sg).first;
      }
      if (it != m->sweep_graphs.end()) {
        CU_OK(cudaGraphLaunch(it->second.exec, m->stream));
        m->launches += it->second.nodes;
      } else {
        TF_TRY(enqueue_sweep(n_lp, n_hp, first));
      }
    } else {
      TF_TRY(enqueue_sweep(n_lp, n_hp, first));
    }
    if (l2 && t <= m->trace_l2_sweeps) {
      LAUNCH(m, KC_CTRL, l2_distance_kernel, B, 256, 0, u, m->ref_seq,
             m->trace_l2 + ((size_t)g * m->trace_l2_sweeps + (t - 1)) * m->cfg.max_batch, m->L * m->D);
      m->trace_l2_count[g] = t;
    }
    if (tau >= 0.f || t == cap || m->trace_on) {
      const int before = n_active;
      TF_TRY(read_ctrl(m));
      n_active = m->ctrl_host[HOST_ACTIVE];
      n_hp = m->ctrl_host[HOST_TWO_TERM];
      if (m->trace_on) {
        float top;
        memcpy(&top, &m->ctrl_host[HOST_TOP], sizeof(float));
        m->trace.push_back({g, t, before, top});
      }
    }
  }
  *sweeps_out = t;
  if (tau >= 0.f && n_active > 0 && cap < max_iters) {
    // Fall-back: the samples still in the active list are decoded sequentially from the block's input (Eq. 5), as a
    // dense batch of their own; their count becomes sweeps + L - 1.
    const int nf = m->L * m->D, nb = n_active;
    int gb = (int)(((size_t)nb * nf + 255) / 256);
    if (gb > 148 * 16) gb = 148 * 16;
    LAUNCH(m, KC_LAYOUT, gather_rows_kernel, gb, 256, 0, v, m->cmp_v, m->idx, nb, nf, 1);
    const int* lab_c = nullptr;
    if (labels) {
      LAUNCH(m, KC_LAYOUT, gather_int_kernel, (nb + 127) / 128, 128, 0, labels, m->cmp_labels, m->idx, nb);
      lab_c = m->cmp_labels;
    }
    TF_TRY(check_launch("gather kernels"));
    m->seq_variant = 1;
    int r = run_sequential_any<T>(m, g, nb, lab_c, m->cmp_v, m->cmp_u);
    m->seq_variant = 0;
    TF_TRY(r);
    LAUNCH(m, KC_LAYOUT, gather_rows_kernel, gb, 256, 0, m->cmp_u, u, m->idx, nb, nf, 0);
    LAUNCH(m, KC_CTRL, add_int_rows_kernel, (nb + 127) / 128, 128, 0, iters_row, m->idx, nb, m->L - 1);
    TF_TRY(check_launch("scatter kernels"));
    *sweeps_out = t + m->L - 1;
    return TF_OK;
  }
  return (tau >= 0.f && n_active > 0) ? TF_MAXITER : TF_OK;
}

// ------------------------------------------------------------------------------------------------
// whole-model drivers
// ------------------------------------------------------------------------------------------------
static int layout(tf_model* m, float* img, float* seq, int B, int to_seq) {
  size_t n = (size_t)B * m->cfg.C * m->cfg.H * m->cfg.W;
  int blocks = (int)((n + 255) / 256);
  if (blocks > 148 * 16) blocks = 148 * 16;
  LAUNCH(m, KC_LAYOUT, patchify_kernel, blocks, 256, 0, img, seq, B, m->cfg.C, m->cfg.H, m->cfg.W, m->cfg.patch, to_seq);
  return check_launch("patchify_kernel");
}

template <class T>
static int run_sequential_any(tf_model* m, int g, int B, const int* labels, const float* v, float* u) {
  const bool unit = m->prof_on && m->prof_mode == 2;  // time the whole block as one unit of class seq_block
  if (unit) {
    m->cur_rows = (int64_t)B * (m->L - 1);
    m->pre(KC_SEQ_BLOCK);
    m->prof_suspend = true;
  }
  int r;
  if constexpr (sizeof(T) == 2) r = run_sequential_block_bf16(m, g, B, labels, v, u);
  else r = run_sequential_block<T>(m, g, B, labels, v, u);
  if (unit) {
    m->prof_suspend = false;
    m->cur_rows = (int64_t)B * (m->L - 1);
    const int64_t keep = m->launches;
    m->post(KC_SEQ_BLOCK);
    m->launches = keep;
  }
  return r;
}

template <class T>
static int inverse_impl(tf_model* m, const float* z, const int* labels, int B, const uint8_t* policy, float tau,
                        int max_iters, const InvOpts& op, float* x, int* iters_block_host, int* iters_sample_dev) {
  const int K = m->cfg.n_blocks;
  const size_t img = (size_t)B * m->cfg.C * m->cfg.H * m->cfg.W;
  float *v = m->seq_a, *u = m->seq_b;
  m->trace.clear();
  m->trace_l2_count.assign(K, 0);
  TF_TRY(take_labels(m, &labels, B));
  TF_TRY(layout(m, const_cast<float*>(z), v, B, 1));
  int status = TF_OK;
  for (int g = 0; g < K; ++g) {
    int* iters_row = m->iters_sample + (size_t)g * m->cfg.max_batch;
    int sweeps = m->L - 1;
    if (m->block_ev[g]) cudaEventRecord(m->block_ev[g], m->stream);
    if (policy[g] == 0) {
      TF_TRY(run_sequential_any<T>(m, g, B, labels, v, u));
      LAUNCH(m, KC_CTRL, fill_int_kernel, (B + 127) / 128, 128, 0, iters_row, B, m->L - 1);
    } else {
      const float tau_g = op.tau_block ? op.tau_block[g] : tau;
      int r = run_jacobi_block<T>(m, g, B, labels, v, u, tau_g, max_iters, op, &sweeps, iters_row);
      if (r < 0) return r;
      if (r == TF_MAXITER) status = TF_MAXITER;
    }
    if (iters_block_host) iters_block_host[g] = sweeps;
    if (op.states_img) TF_TRY(layout(m, op.states_img + (size_t)g * img, u, B, 0));
    float* tmp = v; v = u; u = tmp;
  }
  if (m->block_ev[K]) cudaEventRecord(m->block_ev[K], m->stream);
  m->block_ev_valid = true;
  TF_TRY(layout(m, x, v, B, 0));
  if (iters_sample_dev) {
    for (int g = 0; g < K; ++g)
      CU_OK(cudaMemcpyAsync(iters_sample_dev + (size_t)g * B, m->iters_sample + (size_t)g * m->cfg.max_batch,
                            B * sizeof(int), cudaMemcpyDeviceToDevice, m->stream));
  }
  TF_TRY(sync_check(m));
  return status;
}

static int forward_affine(tf_model* m, int B, const float* u, float* v, float* logdet, int reversed) {
  // By the values of a sample alone: the order of a sample's sum does not depend on its batch.  Eight CTAs / one per sample: 12 288 values
  // 8.6 / 12.7 us (1 sample), 25.7 / 16.3 (64), 81 / 32 (256); 196 608 values 19 / 105 (2 samples).
  if (m->L * m->D < 65536) {
    LAUNCH_PDL(m, KC_AFFINE, forward_affine_kernel<1>, B, affine_threads(m->L * m->D), 0, m->o, u, v, logdet, m->L, m->D, reversed);
    return check_launch("forward_affine_kernel");
  }
  constexpr int CS = 8;
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(B * CS);
  lc.blockDim = dim3(AFFINE_THREADS);
  lc.stream = m->stream;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = CS;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[1].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at;
  lc.numAttrs = 2;
  m->pre(KC_AFFINE);
  const cudaError_t e = cudaLaunchKernelEx(&lc, forward_affine_kernel<CS>, (const float*)m->o, u, v, logdet, m->L, m->D, reversed);
  m->post(KC_AFFINE);
  if (e != cudaSuccess) return fail(TF_ECUDA, "forward_affine_kernel launch failed: %s", cudaGetErrorString(e));
  return TF_OK;
}

template <class T>
static int forward_impl(tf_model* m, const float* x, const int* labels, int B, float* z, float* logdet) {
  float *u = m->seq_a, *v = m->seq_b;
  TF_TRY(take_labels(m, &labels, B));
  TF_TRY(layout(m, const_cast<float*>(x), u, B, 1));
  if (logdet) CU_OK(cudaMemsetAsync(logdet, 0, B * sizeof(float), m->stream));
  for (int g = m->cfg.n_blocks - 1; g >= 0; --g) {
    TF_TRY(run_pass<T>(m, g, B, u, nullptr, labels, PASS_FORWARD, nullptr, nullptr, false));
    TF_TRY(forward_affine(m, B, u, v, logdet, g & 1));
    float* tmp = v; v = u; u = tmp;
  }
  TF_TRY(layout(m, z, u, B, 0));
  return sync_check(m);
}

// ------------------------------------------------------------------------------------------------
// second workload: MLP-based autoregressive flow (App. E.3).  One pass = cast -> three masked linear layers.
//   mode 0: Jacobi update in the last layer's epilogue (only_col >= 0: one step of sequential decoding)
//   mode 1: forward direction, the raw (mu, alpha) go to m->o
// The layer permutation (reversal on odd layers) and the MADE masks are folded into the weights when they are
// loaded, so every buffer here is in the sample's own dimension order.
// ------------------------------------------------------------------------------------------------
template <class T>
static int maf_pass(tf_model* m, int g, int n_slots, const float* u_src, const int* idx, int mode, const float* v, float* u_upd,
                    bool hp, int only_col) {
  const tf_model::MafBlock& bw = m->maf_blocks[g];
  const int D = m->L, H = m->maf_H, M = n_slots;
  T* a0 = reinterpret_cast<T*>(m->maf_a0);
  T* h1 = reinterpret_cast<T*>(m->maf_h1);
  T* h2 = reinterpret_cast<T*>(m->maf_h2);
  T* a0_lo = hp ? reinterpret_cast<T*>(m->maf_a0_lo) : nullptr;
  T* h1_lo = hp ? reinterpret_cast<T*>(m->maf_h1_lo) : nullptr;
  T* h2_lo = hp ? reinterpret_cast<T*>(m->maf_h2_lo) : nullptr;
  m->cur_rows = M;
  int cb = (int)(((size_t)M * ((D & 3) == 0 ? D / 4 : D) + 255) / 256);
  if (cb > 148 * 16) cb = 148 * 16;
  LAUNCH_PDL(m, KC_EMBED, (maf_cast_rows_kernel<T>), cb, 256, 0, u_src, idx, a0, a0_lo, M, D);
  TF_TRY(check_launch("maf_cast_rows_kernel"));
  if constexpr (sizeof(T) == 2) {
    const CUtensorMap* sm = m->maf_store_maps;
    TF_TRY(gemm<T>(m, KC_GEMM_MLP1, a0, &m->maf_map[0][0], hp ? &m->maf_map[0][1] : nullptr, bw.w1, M,
                   EpiStoreTma<ACT_RELU>{bw.b1, sm + 0, hp ? sm + 1 : nullptr}));
    TF_TRY(gemm<T>(m, KC_GEMM_MLP2, h1, &m->maf_map[1][0], hp ? &m->maf_map[1][1] : nullptr, bw.w2, M,
                   EpiStoreTma<ACT_RELU>{bw.b2, sm + 2, hp ? sm + 3 : nullptr}));
  } else {
    TF_TRY(gemm<T>(m, KC_GEMM_MLP1, a0, nullptr, nullptr, bw.w1, M, EpiStore<T, ACT_RELU>{h1, bw.b1, H, h1_lo}));
    TF_TRY(gemm<T>(m, KC_GEMM_MLP2, h1, nullptr, nullptr, bw.w2, M, EpiStore<T, ACT_RELU>{h2, bw.b2, H, h2_lo}));
  }
  const CUtensorMap* map2 = sizeof(T) == 2 ? &m->maf_map[2][0] : nullptr;
  const CUtensorMap* map2_lo = (sizeof(T) == 2 && hp) ? &m->maf_map[2][1] : nullptr;
  if (mode == 0) {
    if constexpr (sizeof(T) == 2) {
      // tensor-core engine: the raw (mu, alpha) leave through bulk stores, a row-per-warp kernel applies the update
      // (measured: 381 us for the fused lane-per-column epilogue against 85 + 60 us for the pair on 69 k rows)
      TF_TRY(gemm<T>(m, KC_GEMM_HEAD_UPDATE, h2, map2, map2_lo, bw.w3, M, EpiStoreF32Tma{bw.b3, m->maf_store_maps + 4}));
      // Launched early, the update's CTAs crowd onto the SMs that the output layer leaves idle and stay there, which costs more than the
      // kernel boundary once there is something to move (early / not: 1000 rows of 784 values 53.5 / 47.1 us per sweep, 3000 of 2048
      // 125 / 97.5, 100 000 of 256 378 / 362; but 500 rows of 784 43.2 / 43.6, 300 of 2048 51.0 / 51.3, 100 of 256 34.3 / 34.8).  Short rows
      // are done before it matters (20 000 rows of 64: 45.0 / 47.2, 100 000: 107 / 107).
      if (only_col < 0 && (int64_t)M * D >= (D >= 256 ? 512 * 1024 : 4 * 1024 * 1024))
        LAUNCH(m, KC_AFFINE, maf_update_kernel, (M + 7) / 8, 256, 0, m->o, v, u_upd, m->maxdiff, idx, M, D, only_col);
      else
        LAUNCH_PDL(m, KC_AFFINE, maf_update_kernel, (M + 7) / 8, 256, 0, m->o, v, u_upd, m->maxdiff, idx, M, D, only_col);
      return check_launch("maf_update_kernel");
    } else {
      EpiMafUpdate epi{v, u_upd, m->maxdiff, idx, bw.b3, D, only_col};
      return gemm<T>(m, KC_GEMM_HEAD_UPDATE, h2, map2, map2_lo, bw.w3, M, epi);
    }
  }
  return gemm<T>(m, KC_GEMM_HEAD, h2, map2, map2_lo, bw.w3, M, EpiStore<float, ACT_NONE>{m->o, bw.b3, 2 * D});
}

template <class T>
static int maf_inverse_impl(tf_model* m, const float* z, int B, bool jacobi, float tau, int max_iters, int init_mode, float* x,
                            int* iters_block_host, int* iters_sample_dev) {
  const int K = m->cfg.n_blocks, D = m->L;
  const size_t n = (size_t)B * D;
  float *v = m->seq_a, *u = m->seq_b;
  m->trace.clear();
  m->trace_l2_count.assign(K, 0);
  CU_OK(cudaMemcpyAsync(v, z, n * sizeof(float), cudaMemcpyDeviceToDevice, m->stream));
  int status = TF_OK;
  InvOpts op;
  op.init_mode = init_mode;
  for (int g = 0; g < K; ++g) {
    int* iters_row = m->iters_sample + (size_t)g * m->cfg.max_batch;
    int sweeps = D;
    if (m->block_ev[g]) cudaEventRecord(m->block_ev[g], m->stream);
    if (!jacobi) {
      // Eq. 5: dimension i (in the layer's own order) is final after pass i; there is no cache, every pass is a whole one
      CU_OK(cudaMemsetAsync(u, 0, n * sizeof(float), m->stream));
      for (int i = 0; i < D; ++i)
        TF_TRY(maf_pass<T>(m, g, B, u, nullptr, 0, v, u, m->precision_mode == 2, (g & 1) ? D - 1 - i : i));
      LAUNCH(m, KC_CTRL, fill_int_kernel, (B + 127) / 128, 128, 0, iters_row, B, D);
      CU_OK(cudaMemsetAsync(m->maxdiff, 0, B * sizeof(float), m->stream));
    } else {
      int r = run_jacobi_block<T>(m, g, B, nullptr, v, u, tau, max_iters, op, &sweeps, iters_row);
      if (r < 0) return r;
      if (r == TF_MAXITER) status = TF_MAXITER;
    }
    if (iters_block_host) iters_block_host[g] = sweeps;
    float* tmp = v; v = u; u = tmp;
  }
  if (m->block_ev[K]) cudaEventRecord(m->block_ev[K], m->stream);
  m->block_ev_valid = true;
  CU_OK(cudaMemcpyAsync(x, v, n * sizeof(float), cudaMemcpyDeviceToDevice, m->stream));
  if (iters_sample_dev)
    for (int g = 0; g < K; ++g)
      CU_OK(cudaMemcpyAsync(iters_sample_dev + (size_t)g * B, m->iters_sample + (size_t)g * m->cfg.max_batch, B * sizeof(int),
                            cudaMemcpyDeviceToDevice, m->stream));
  TF_TRY(sync_check(m));
  return status;
}

template <class T>
static int maf_forward_impl(tf_model* m, const float* x, int B, float* z, float* logdet) {
  const int D = m->L;
  const size_t n = (size_t)B * D;
  float *u = m->seq_a, *v = m->seq_b;
  CU_OK(cudaMemcpyAsync(u, x, n * sizeof(float), cudaMemcpyDeviceToDevice, m->stream));
  if (logdet) CU_OK(cudaMemsetAsync(logdet, 0, B * sizeof(float), m->stream));
  for (int g = m->cfg.n_blocks - 1; g >= 0; --g) {
    TF_TRY(maf_pass<T>(m, g, B, u, nullptr, 1, nullptr, nullptr, false, -1));
    LAUNCH(m, KC_AFFINE, maf_forward_affine_kernel, B, 256, 0, m->o, u, v, logdet, D);
    TF_TRY(check_launch("maf_forward_affine_kernel"));
    float* tmp = v; v = u; u = tmp;
  }
  CU_OK(cudaMemcpyAsync(z, u, n * sizeof(float), cudaMemcpyDeviceToDevice, m->stream));
  return sync_check(m);
}

// ------------------------------------------------------------------------------------------------
// loading
// ------------------------------------------------------------------------------------------------
struct BlobReader {
  const float* p;
  const float* end;
  const float* take(size_t n) {
    const float* r = p;
    p += n;
    return r;
  }
};

static int upload_f32(tf_model* m, float** dst, const float* src, size_t n) {
  TF_TRY(dev_alloc(m, dst, n));
  CU_OK(cudaMemcpy(*dst, src, n * sizeof(float), cudaMemcpyHostToDevice));
  return TF_OK;
}

// matrix [N, K]: fp32 engine keeps fp32; bf16 engine converts on the device (round to nearest even)
// few_bn: columns of the narrow tiles (0: the matrix has none)
static int upload_matrix(tf_model* m, Matrix* W, const float* src, int N, int K, float* staging, int few_bn = 64) {
  W->N = N;
  W->K = K;
  size_t n = (size_t)N * K;
  if (m->cfg.dtype == 0) {
    float* w;
    TF_TRY(upload_f32(m, &w, src, n));
    W->w = w;
    return TF_OK;
  }
  bf16* w;
  TF_TRY(dev_alloc(m, &w, n));
  CU_OK(cudaMemcpy(staging, src, n * sizeof(float), cudaMemcpyHostToDevice));
  f32_to_bf16_kernel<<<148 * 4, 256>>>(staging, w, n);
  CU_OK(cudaDeviceSynchronize());
  W->w = w;
  W->bn = (N % 256 == 0) ? 256 : 128;
  TF_TRY(make_map_bf16(&W->map_seq, w, (uint64_t)N, (uint64_t)K, 128u));
  W->few_bn = few_bn;
  if (few_bn > 0) TF_TRY(make_map_bf16(&W->map_few, w, (uint64_t)N, (uint64_t)K, (uint32_t)few_bn));
  return make_map_bf16(&W->map, w, (uint64_t)N, (uint64_t)K, (uint32_t)W->bn);
}

// Decides whether an fp32 model's blocks are decoded by f32::seq_cluster_kernel and cuts them into the CTAs' shares: whole
// heads round robin, hidden units (multiples of four) so that the bytes come out even.
static int plan_seq_cluster(tf_model* m) {
  const int d = m->d, hid = m->hid, heads = m->cfg.n_heads, hd = m->hd, lpk = hd / 4;
  if (d % 4 || hid % 4 || hd % 4 || hd > 128 || (lpk & (lpk - 1)) || d > 1024) return TF_OK;
  f32::SeqPlan& P = m->seq_plan;
  P.n_layers = m->cfg.n_layers; P.heads = heads; P.hd = hd; P.d = d; P.D = m->D; P.L = m->L;
  P.owners = heads < f32::SC ? heads : f32::SC;
  const int64_t share = ((int64_t)4 * d * d + (int64_t)2 * d * hid) / f32::SC;
  int left = hid;
  for (int r = f32::SC - 1; r >= 0; --r) {  // CTAs without heads come last and take the most hidden units
    P.nown[r] = (heads - r + f32::SC - 1) / f32::SC;
    if (P.nown[r] < 0) P.nown[r] = 0;
    const int64_t room = share - (int64_t)4 * hd * d * P.nown[r];
    int n = room <= 0 ? 0 : (int)(room / (2 * d)) / 4 * 4;
    if (n > left || r == 0) n = left;
    P.nu[r] = n;
    left -= n;
  }
  int64_t most = 0, off = 0;
  for (int r = 0; r < f32::SC; ++r) {
    P.off[r] = (int)off;
    if (P.fixed_floats(r) > most) most = P.fixed_floats(r);
    off += P.fixed_floats(r) + P.tail_floats(2);
    if (off > (1 << 28)) return TF_OK;
  }
  P.off[f32::SC] = (int)off;
  const int limit = 226 * 1024;  // a block may have 227 KB, static shared memory and its padding included
  for (int i = 0; i < 3; ++i) {
    for (int level = 2; level >= 0 && m->seq_cluster_smem[i] == 0; --level) {
      const int64_t need = (most + P.work_floats(1 << i) + P.tail_floats(level)) * (int64_t)sizeof(float);
      if (need > limit) continue;
      m->seq_cluster_tail[i] = level;
      m->seq_cluster_smem[i] = (int)need;
    }
  }
  if (m->seq_cluster_smem[0] == 0) return TF_OK;
  for (auto kern : {f32::seq_cluster_kernel<1, 0>, f32::seq_cluster_kernel<1, 1>, f32::seq_cluster_kernel<1, 2>, f32::seq_cluster_kernel<2, 0>,
                    f32::seq_cluster_kernel<2, 1>, f32::seq_cluster_kernel<2, 2>, f32::seq_cluster_kernel<4, 0>,
                    f32::seq_cluster_kernel<4, 1>, f32::seq_cluster_kernel<4, 2>})
    CU_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, limit));
  cudaLaunchConfig_t lc = {};
  lc.gridDim = dim3(f32::SC);
  lc.blockDim = dim3(f32::ST);
  lc.dynamicSmemBytes = m->seq_cluster_smem[0];
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.x = f32::SC;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  lc.attrs = at;
  lc.numAttrs = 1;
  int n = 0;
  if (cudaOccupancyMaxActiveClusters(&n, f32::seq_cluster_kernel<1, 0>, &lc) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  m->seq_clusters = n;
  return TF_OK;
}

// the images of one block; `layers` is the first layer's tensors in the weight blob, w_out / b_out interleaved
static int upload_seq_images(tf_model* m, const float* layers, const float* lnf, const float* b_in, const float* w_in_t,
                             const float* w_out, const float* b_out) {
  const f32::SeqPlan& P = m->seq_plan;
  const int d = P.d, hid = m->hid, hd = P.hd, D = P.D, No = P.pad4(2 * D), Dp = P.pad4(D);
  std::vector<float> img(P.off[f32::SC], 0.f);
  int unit0 = 0;
  for (int r = 0; r < f32::SC; ++r) {
    const int nown = P.nown[r], nu = P.nu[r], nq = 3 * hd * nown;
    float* o = img.data() + P.off[r];
    const float* q = layers;
    for (int i = 0; i < P.n_layers; ++i) {
      const float *ln1 = q, *w_qkv = ln1 + 2 * d, *b_qkv = w_qkv + (size_t)3 * d * d, *w_o = b_qkv + 3 * d, *b_o = w_o + (size_t)d * d,
                  *ln2 = b_o + d, *w_1 = ln2 + 2 * d, *b_1 = w_1 + (size_t)hid * d, *w_2 = b_1 + hid, *b_2 = w_2 + (size_t)d * hid;
      q = b_2 + d;
      auto row_of = [&](int n) { return (n / hd % 3) * d + (r + f32::SC * (n / (3 * hd))) * hd + n % hd; };  // row of w_qkv
      auto put = [&](const float* p, int n) { memcpy(o, p, n * sizeof(float)); o += n; };
      for (int n = 0; n < nq; ++n) put(w_qkv + (size_t)row_of(n) * d, d);
      for (int n = 0; n < nq; ++n) *o++ = b_qkv[row_of(n)];
      for (int n = 0; n < d; ++n)
        for (int k = 0; k < nown; ++k) put(w_o + (size_t)n * d + (r + f32::SC * k) * hd, hd);
      put(w_1 + (size_t)unit0 * d, nu * d);
      put(b_1 + unit0, nu);
      for (int n = 0; n < d; ++n) put(w_2 + (size_t)n * hid + unit0, nu);
      put(ln1, 2 * d); put(b_o, d); put(ln2, 2 * d); put(b_2, d);
    }
    memcpy(o, lnf, 2 * d * sizeof(float)); o += 2 * d;
    memcpy(o, b_in, d * sizeof(float)); o += d;
    memcpy(o, w_out, (size_t)2 * D * d * sizeof(float)); o += (size_t)No * d;  // the image starts out as zeros
    memcpy(o, b_out, 2 * D * sizeof(float)); o += No;
    for (int j = 0; j < d; ++j)
      for (int c = 0; c < Dp; ++c) *o++ = c < D ? w_in_t[(size_t)c * d + j] : 0.f;
    unit0 += nu;
  }
  float* dev = nullptr;
  TF_TRY(upload_f32(m, &dev, img.data(), img.size()));
  m->seq_image.push_back(dev);
  return TF_OK;
}

static size_t block_floats(const tf_config& c, int L, int D) {
  size_t d = c.width, hid = (size_t)c.mlp_ratio * d;
  size_t n = d * D + d + (size_t)L * d + (size_t)c.n_classes * d;
  n += (size_t)c.n_layers * (2 * d + 3 * d * d + 3 * d + d * d + d + 2 * d + hid * d + hid + d * hid + d);
  n += 2 * d + 2 * (size_t)D * d + 2 * D;
  return n;
}

static int load_impl(tf_model* m, const void* blob, size_t nbytes) {
  const tf_config& c = m->cfg;
  const int L = m->L, D = m->D, d = m->d, hid = m->hid;
  const size_t want = 64 + 4 * block_floats(c, L, D) * c.n_blocks;
  if (nbytes != want) return fail(TF_ESIZE, "weight blob is %zu bytes, configuration needs %zu", nbytes, want);
  const int32_t* hdr = reinterpret_cast<const int32_t*>(blob);
  const int32_t expect[13] = {0x31574654, 1, c.C, c.H, c.W, c.patch, c.n_blocks, c.n_layers, c.width, c.n_heads,
                              c.mlp_ratio, c.n_classes, c.dtype};
  for (int i = 0; i < 13; ++i)
    if (hdr[i] != expect[i]) return fail(TF_ESIZE, "weight blob header field %d is %d, expected %d", i, hdr[i], expect[i]);

  int dev = 0;
  CU_OK(cudaGetDevice(&dev));
  CU_OK(cudaDeviceGetAttribute(&m->num_sms, cudaDevAttrMultiProcessorCount, dev));

  float* staging = nullptr;
  size_t max_mat = (size_t)hid * d;
  if ((size_t)3 * d * d > max_mat) max_mat = (size_t)3 * d * d;
  if (c.dtype == 1) CU_OK(cudaMalloc(&staging, max_mat * sizeof(float)));
  struct Guard { float* p; ~Guard() { if (p) cudaFree(p); } } guard{staging};

  BlobReader rd{reinterpret_cast<const float*>(reinterpret_cast<const char*>(blob) + 64), nullptr};
  m->blocks.resize(c.n_blocks);
  if (c.dtype == 0) TF_TRY(plan_seq_cluster(m));
  std::vector<float> tmp, w_in_t;
  for (int g = 0; g < c.n_blocks; ++g) {
    BlockW& bw = m->blocks[g];
    const float* w_in = rd.take((size_t)d * D);
    w_in_t.resize((size_t)d * D);
    for (int j = 0; j < d; ++j)
      for (int cc = 0; cc < D; ++cc) w_in_t[(size_t)cc * d + j] = w_in[(size_t)j * D + cc];
    TF_TRY(upload_f32(m, &bw.w_in_t, w_in_t.data(), w_in_t.size()));
    const float* b_in = rd.take(d);
    TF_TRY(upload_f32(m, &bw.b_in, b_in, d));
    TF_TRY(upload_f32(m, &bw.pos, rd.take((size_t)L * d), (size_t)L * d));
    bw.cls = nullptr;
    if (c.n_classes > 0) TF_TRY(upload_f32(m, &bw.cls, rd.take((size_t)c.n_classes * d), (size_t)c.n_classes * d));
    bw.layers.resize(c.n_layers);
    const float* layers = rd.p;
    for (LayerW& lw : bw.layers) {
      TF_TRY(upload_f32(m, &lw.ln1_g, rd.take(d), d));
      TF_TRY(upload_f32(m, &lw.ln1_b, rd.take(d), d));
      TF_TRY(upload_matrix(m, &lw.w_qkv, rd.take((size_t)3 * d * d), 3 * d, d, staging));
      TF_TRY(upload_f32(m, &lw.b_qkv, rd.take(3 * d), 3 * d));
      TF_TRY(upload_matrix(m, &lw.w_o, rd.take((size_t)d * d), d, d, staging));
      TF_TRY(upload_f32(m, &lw.b_o, rd.take(d), d));
      TF_TRY(upload_f32(m, &lw.ln2_g, rd.take(d), d));
      TF_TRY(upload_f32(m, &lw.ln2_b, rd.take(d), d));
      TF_TRY(upload_matrix(m, &lw.w_1, rd.take((size_t)hid * d), hid, d, staging));
      TF_TRY(upload_f32(m, &lw.b_1, rd.take(hid), hid));
      TF_TRY(upload_matrix(m, &lw.w_2, rd.take((size_t)d * hid), d, hid, staging));
      TF_TRY(upload_f32(m, &lw.b_2, rd.take(d), d));
    }
    const float* lnf = rd.p;
    TF_TRY(upload_f32(m, &bw.lnf_g, rd.take(d), d));
    TF_TRY(upload_f32(m, &bw.lnf_b, rd.take(d), d));
    // head: interleave rows so that outputs (2c, 2c+1) = (mu~_c, alpha~_c)
    const float* w_out = rd.take((size_t)2 * D * d);
    const float* b_out = rd.take((size_t)2 * D);
    tmp.resize((size_t)2 * D * d);
    std::vector<float> btmp(2 * D);
    for (int cc = 0; cc < D; ++cc) {
      memcpy(&tmp[(size_t)(2 * cc) * d], &w_out[(size_t)cc * d], d * sizeof(float));
      memcpy(&tmp[(size_t)(2 * cc + 1) * d], &w_out[(size_t)(D + cc) * d], d * sizeof(float));
      btmp[2 * cc] = b_out[cc];
      btmp[2 * cc + 1] = b_out[D + cc];
    }
    TF_TRY(upload_matrix(m, &bw.w_out, tmp.data(), 2 * D, d, staging, 32));
    TF_TRY(upload_f32(m, &bw.b_out, btmp.data(), btmp.size()));
    if (m->seq_clusters > 0) TF_TRY(upload_seq_images(m, layers, lnf, b_in, w_in_t.data(), tmp.data(), btmp.data()));
  }

  // workspace
  const size_t B = c.max_batch, M = B * L, esz = c.dtype == 1 ? 2 : 4;
  TF_TRY(dev_alloc(m, &m->seq_a, M * D));
  TF_TRY(dev_alloc(m, &m->seq_b, M * D));
  TF_TRY(dev_alloc(m, &m->cmp_v, M * D));
  TF_TRY(dev_alloc(m, &m->cmp_u, M * D));
  TF_TRY(dev_alloc(m, &m->ref_seq, M * D));
  TF_TRY(dev_alloc(m, &m->cmp_labels, B));
  TF_TRY(dev_alloc(m, &m->h, M * d));
  TF_TRY(dev_alloc(m, &m->o, M * 2 * D));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->xn), M * d * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->qkv), M * 3 * d * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->att), M * d * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->mlp), M * hid * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->kcache), (size_t)c.n_layers * M * d * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->vcache), (size_t)c.n_layers * M * d * esz));
  if (c.dtype == 1) {
    TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->xn_lo), M * d * esz));
    TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->qkv_lo), M * 3 * d * esz));
    TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->att_lo), M * d * esz));
    TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->mlp_lo), M * hid * esz));
  }
  TF_TRY(dev_alloc(m, &m->maxdiff, B));
  TF_TRY(dev_alloc(m, &m->idx, B));
  TF_TRY(dev_alloc(m, &m->idx_tmp, B));
  TF_TRY(dev_alloc(m, &m->phase, B));
  if (B > (size_t)FIN_CHUNK) {
    const size_t nblk = (B + FIN_CHUNK - 1) / FIN_CHUNK;
    TF_TRY(dev_alloc(m, &m->fin_code, B));
    TF_TRY(dev_alloc(m, &m->fin_cnt, 2 * nblk));
    TF_TRY(dev_alloc(m, &m->fin_top, nblk));
    TF_TRY(dev_alloc(m, &m->fin_flag, nblk));
  }
  TF_TRY(dev_alloc(m, &m->ctrl, CTRL_WORDS));
  TF_TRY(dev_alloc(m, &m->err, 1));
  TF_TRY(dev_alloc(m, &m->iters_sample, (size_t)c.n_blocks * B));
  TF_TRY(dev_alloc(m, &m->io_z, B * c.C * c.H * c.W));
  TF_TRY(dev_alloc(m, &m->io_x, B * c.C * c.H * c.W));
  TF_TRY(dev_alloc(m, &m->io_labels, B));
  TF_TRY(dev_alloc(m, &m->labels_own, B));
  TF_TRY(dev_alloc(m, &m->step_ctr, 16 * tf_model::MAX_CHAINS));  // one counter per chain, 64 bytes apart
  if (c.dtype == 1) {  // partial tiles: up to 16 K slices of a [B, d] output, or d/256 slices of the widest one
    const size_t wide = (size_t)(hid > 3 * d ? hid : 3 * d);
    m->seq_part_row_floats = (size_t)16 * d;
    const size_t per_wide = (size_t)(d / 64 < 16 ? d / 64 : 16) * wide;
    if (per_wide > m->seq_part_row_floats) m->seq_part_row_floats = per_wide;
    m->seq_part_floats = m->seq_part_row_floats * B;
    TF_TRY(dev_alloc(m, &m->seq_part, m->seq_part_floats));
  }
  CU_OK(cudaMemset(m->step_ctr, 0, 16 * tf_model::MAX_CHAINS * sizeof(int)));
  CU_OK(cudaMemset(m->ctrl, 0, CTRL_WORDS * sizeof(int)));
  CU_OK(cudaMemset(m->err, 0, sizeof(int)));
  CU_OK(cudaMemset(m->iters_sample, 0, (size_t)c.n_blocks * B * sizeof(int)));
  for (const auto kern : {embed_ln_rows_kernel<bf16, 4>, embed_ln_rows_kernel<bf16, 16>})
    CU_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, EMBED_WEIGHT_BYTES + EMBED_TOKEN_BYTES));
  for (const auto kern : {embed_ln_rows_kernel<float, 4>, embed_ln_rows_kernel<float, 16>})
    CU_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, EMBED_WEIGHT_BYTES + EMBED_TOKEN_BYTES));
  CU_OK(cudaMallocHost(&m->ctrl_host, HOST_WORDS * sizeof(int)));
  memset(m->ctrl_host, 0, HOST_WORDS * sizeof(int));
  m->block_ev.assign(c.n_blocks + 1, nullptr);
  for (auto& e : m->block_ev) CU_OK(cudaEventCreate(&e));
  if (c.dtype == 1) {
    TF_TRY(make_map_bf16(&m->map_xn, m->xn, M, d, tc::BM));
    TF_TRY(make_map_bf16(&m->map_att, m->att, M, d, tc::BM));
    TF_TRY(make_map_bf16(&m->map_mlp, m->mlp, M, hid, tc::BM));
    TF_TRY(make_map_bf16(&m->map_xn_lo, m->xn_lo, M, d, tc::BM));
    TF_TRY(make_map_bf16(&m->map_att_lo, m->att_lo, M, d, tc::BM));
    TF_TRY(make_map_bf16(&m->map_mlp_lo, m->mlp_lo, M, hid, tc::BM));
    {
      CUtensorMap sm[tf_model::SM_COUNT];
      TF_TRY(make_map_store(&sm[tf_model::SM_QKV], m->qkv, M, 3 * d, 2));
      TF_TRY(make_map_store(&sm[tf_model::SM_QKV_LO], m->qkv_lo, M, 3 * d, 2));
      TF_TRY(make_map_store(&sm[tf_model::SM_MLP], m->mlp, M, hid, 2));
      TF_TRY(make_map_store(&sm[tf_model::SM_MLP_LO], m->mlp_lo, M, hid, 2));
      TF_TRY(make_map_store(&sm[tf_model::SM_H], m->h, M, d, 4));
      if (const char* e = getenv("TARFLOW_SMALL_M_ROWS")) m->small_m_rows = atoi(e);
      if (const char* e = getenv("TARFLOW_SPLIT_M_ROWS")) m->split_m_rows = atoi(e);
      if (const char* e = getenv("TARFLOW_SMALL_M_SPLIT")) m->small_m_split = atoi(e) != 0;
      if ((m->small_m_rows > 0 || m->split_m_rows > 0) && d % 128 == 0) {
        m->part_cap_rows = 8192;
        TF_TRY(dev_alloc(m, &m->sweep_part, (size_t)m->part_cap_rows * d));
        TF_TRY(make_map_store(&sm[tf_model::SM_PART], m->sweep_part, (uint64_t)m->part_cap_rows, d, 4));
      } else {
        sm[tf_model::SM_PART] = sm[tf_model::SM_H];
      }
      TF_TRY(make_map_3d(&sm[tf_model::SM_ATT3], m->att, B, L, d, 32));
      TF_TRY(make_map_3d(&m->map_qkv3, m->qkv, B, L, 3 * (uint64_t)d, attn_tc::BQ));
      TF_TRY(make_map_3d(&m->map_kv3, m->qkv, B, L, 3 * (uint64_t)d, attn_tc::BKV));
      TF_TRY(make_map_3d(&sm[tf_model::SM_ATT3_LO], m->att_lo, B, L, d, 32));
      TF_TRY(make_map_3d(&m->map_qkv3_lo, m->qkv_lo, B, L, 3 * (uint64_t)d, attn_tc::BQ));
      TF_TRY(make_map_3d(&m->map_kv3_lo, m->qkv_lo, B, L, 3 * (uint64_t)d, attn_tc::BKV));
      CU_OK(cudaFuncSetAttribute(attn_tc::attention_tc_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 attn_tc::Cfg<false>::SMEM_BYTES));
      CU_OK(cudaFuncSetAttribute(attn_tc::attention_tc_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                 attn_tc::Cfg<true>::SMEM_BYTES));
      if (const char* e = getenv("TARFLOW_ATTN_TC_SPLIT")) m->use_tc_attention_split = atoi(e) != 0;
      if (const char* e = getenv("TARFLOW_ATTN_TC")) m->use_tc_attention = atoi(e) != 0;
      TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->store_maps), sizeof(sm)));
      CU_OK(cudaMemcpy(m->store_maps, sm, sizeof(sm), cudaMemcpyHostToDevice));
    }
    for (int r = 0; r < 3; ++r) {
      const uint32_t rt = 16u << r;
      TF_TRY(make_map_bf16(&m->map_seq_a[0][r], m->xn, M, d, rt));
      TF_TRY(make_map_bf16(&m->map_seq_a[1][r], m->att, M, d, rt));
      TF_TRY(make_map_bf16(&m->map_seq_a[2][r], m->mlp, M, hid, rt));
    }
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_tc_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, seq::gemm_tc_smem_bytes<16>()));
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_tc_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, seq::gemm_tc_smem_bytes<32>()));
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_tc_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, seq::gemm_tc_smem_bytes<64>()));
    if (const char* e = getenv("TARFLOW_SEQ_MMA")) m->seq_use_tc = atoi(e) == 0;
    if (const char* e = getenv("TARFLOW_SEQ_FUSE_GELU")) m->seq_fuse_gelu = atoi(e) != 0;
    if (const char* e = getenv("TARFLOW_SEQ_FUSE_TAIL")) m->seq_fuse_tail = atoi(e) != 0;
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_tc_kernel<64, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, seq::gemm_tc_smem_bytes<64, 8>()));
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_tc_kernel<32, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, seq::gemm_tc_smem_bytes<32, 8>()));
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_tc_kernel<16, 8>, cudaFuncAttributeMaxDynamicSharedMemorySize, seq::gemm_tc_smem_bytes<16, 8>()));
    if (const char* e = getenv("TARFLOW_SEQ_KBN8")) m->seq_kbn8 = atoi(e) != 0;
    if (const char* e = getenv("TARFLOW_PAIR_GEMM")) m->use_pair_gemm = atoi(e) != 0;
    CU_OK(cudaFuncSetAttribute(attn::attention_mma_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               attn::smem_bytes<true>()));
    CU_OK(cudaFuncSetAttribute(attn::attention_mma_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               attn::smem_bytes<false>()));
    const int gsm = seq::gemm_smem_bytes(seq::KC);
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_kernel<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, gsm));
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_kernel<16>, cudaFuncAttributeMaxDynamicSharedMemorySize, gsm));
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_kernel<32>, cudaFuncAttributeMaxDynamicSharedMemorySize, gsm));
    CU_OK(cudaFuncSetAttribute(seq::seq_gemm_kernel<64>, cudaFuncAttributeMaxDynamicSharedMemorySize, gsm));
    CU_OK(cudaStreamCreateWithFlags(&m->cap_stream, cudaStreamNonBlocking));
    for (int c = 0; c < tf_model::MAX_CHAINS; ++c) {
      CU_OK(cudaStreamCreateWithFlags(&m->seq_streams[c], cudaStreamNonBlocking));
      CU_OK(cudaEventCreateWithFlags(&m->seq_join[c], cudaEventDisableTiming));
    }
    CU_OK(cudaEventCreateWithFlags(&m->seq_fork, cudaEventDisableTiming));
    if (const char* e = getenv("TARFLOW_SEQ_CHAINS")) m->seq_chains_force = atoi(e);
    if (const char* e = getenv("TARFLOW_SEQ_KBN")) m->seq_kbn_force = atoi(e);
    if (const char* e = getenv("TARFLOW_SEQ_FIN")) m->seq_fin = atoi(e) != 0;
    if (const char* e = getenv("TARFLOW_SEQ_ATTN_THREADS")) m->seq_attn_threads = atoi(e);
    m->seq_nc_forced = getenv("TARFLOW_SEQ_NC") != nullptr;
    TF_TRY(dev_alloc(m, &m->seq_tickets, (size_t)tf_model::MAX_CHAINS * tf_model::SEQ_TICKETS));
    CU_OK(cudaMemset(m->seq_tickets, 0, (size_t)tf_model::MAX_CHAINS * tf_model::SEQ_TICKETS * sizeof(int)));
    TF_TRY(dev_alloc(m, &m->seq_stats, (size_t)tf_model::MAX_CHAINS * 16 * B));
    if (const char* e = getenv("TARFLOW_SWEEP_GRAPH_ROWS")) m->sweep_graph_rows = atoll(e);
    if (const char* e = getenv("TARFLOW_GRAPHS")) m->use_graphs = atoi(e) != 0;
    TF_TRY(seqp_setup(m));
    if (const char* e = getenv("TARFLOW_SEQ_PERSIST")) m->seq_use_persist = atoi(e) != 0;
  }
  if (c.dtype == 0) {
    for (const auto kern : {f32::attention_kernel<1>, f32::attention_kernel<2>})
      CU_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, f32::attention_smem_floats(128) * (int)sizeof(float)));
    if (const char* e = getenv("TARFLOW_SWEEP_GRAPH_ROWS")) m->sweep_graph_rows = atoll(e);
    if (const char* e = getenv("TARFLOW_GRAPHS")) m->use_graphs = atoi(e) != 0;
    CU_OK(cudaStreamCreateWithFlags(&m->cap_stream, cudaStreamNonBlocking));
  }
  CU_OK(cudaDeviceSynchronize());
  return TF_OK;
}

// Per 128 rows of the weight matrix (= columns of the product) the range of 64-wide k slabs outside which they are all zero.
static int upload_slab_bounds(tf_model* m, Matrix* W, const float* w) {
  if (m->cfg.dtype == 0) return TF_OK;
  const int groups = (W->N + 127) / 128, slabs = (W->K + tc::BK - 1) / tc::BK;
  std::vector<int2> bounds(groups);
  for (int j = 0; j < groups; ++j) {
    int first = W->K, last = -1;
    for (int n = 128 * j; n < W->N && n < 128 * (j + 1); ++n) {
      const float* row = w + (size_t)n * W->K;
      int a = 0, b = W->K - 1;
      while (a < first && row[a] == 0.f) ++a;
      while (b > last && row[b] == 0.f) --b;
      if (a < first) first = a;
      if (b > last) last = b;
    }
    if (last < 0) first = last = 0;  // no weight at all: one slab of zeros
    bounds[j] = make_int2(first / tc::BK, last / tc::BK + 1);
    if (bounds[j].y > slabs) bounds[j].y = slabs;
  }
  int2* dev = nullptr;
  TF_TRY(dev_alloc(m, &dev, groups));
  CU_OK(cudaMemcpy(dev, bounds.data(), groups * sizeof(int2), cudaMemcpyHostToDevice));
  W->bounds = dev;
  return TF_OK;
}

// ---- loading an MLP-based flow: masks and the layer permutation are applied to the weights here ----------------
// Degrees (MADE): input i has degree i + 1, hidden unit j of either hidden layer 1 + (j mod (D - 1)), output i degree
// i + 1.  A hidden unit keeps the weights from inputs / hidden units of degree <= its own, an output those from
// hidden units of degree < its own.  Odd layers act on the reversed dimension order: their first matrix gets its
// columns reversed and their output matrix / bias their rows, so the kernels work in the sample's own order.
static int maf_load_impl(tf_model* m, const void* blob, size_t nbytes, int D, int H) {
  const tf_config& c = m->cfg;
  const size_t per_block = (size_t)H * D + H + (size_t)H * H + H + (size_t)2 * D * H + 2 * D;
  const size_t want = 64 + 4 * per_block * c.n_blocks;
  if (nbytes != want) return fail(TF_ESIZE, "weight blob is %zu bytes, configuration needs %zu", nbytes, want);
  const int32_t* hdr = reinterpret_cast<const int32_t*>(blob);
  const int32_t expect[6] = {0x3146414D, 1, D, H, c.n_blocks, c.dtype};
  for (int i = 0; i < 6; ++i)
    if (hdr[i] != expect[i]) return fail(TF_ESIZE, "weight blob header field %d is %d, expected %d", i, hdr[i], expect[i]);
  int dev = 0;
  CU_OK(cudaGetDevice(&dev));
  CU_OK(cudaDeviceGetAttribute(&m->num_sms, cudaDevAttrMultiProcessorCount, dev));
  float* staging = nullptr;
  size_t max_mat = (size_t)H * H;
  if ((size_t)2 * D * H > max_mat) max_mat = (size_t)2 * D * H;
  if (c.dtype == 1) CU_OK(cudaMalloc(&staging, max_mat * sizeof(float)));
  struct Guard { float* p; ~Guard() { if (p) cudaFree(p); } } guard{staging};

  // Hidden units are kept sorted by degree (rows of a matrix and columns of the next): the masked matrices become block
  // triangular and the GEMMs leave out the k slabs in which a column group has no weight.  unit[j]: unit in place j.
  auto degree = [&](int j) { return 1 + j % (D > 1 ? D - 1 : 1); };
  std::vector<int> unit(H);
  for (int j = 0; j < H; ++j) unit[j] = j;
  std::stable_sort(unit.begin(), unit.end(), [&](int a, int b) { return degree(a) < degree(b); });
  auto deg_hidden = [&](int j) { return degree(unit[j]); };
  std::vector<float> vec(H);
  auto upload_sorted = [&](float** dst, const float* src) -> int {
    for (int j = 0; j < H; ++j) vec[j] = src[unit[j]];
    return upload_f32(m, dst, vec.data(), H);
  };
  BlobReader rd{reinterpret_cast<const float*>(reinterpret_cast<const char*>(blob) + 64), nullptr};
  m->maf_blocks.resize(c.n_blocks);
  std::vector<float> tmp, btmp(2 * D);
  for (int g = 0; g < c.n_blocks; ++g) {
    tf_model::MafBlock& bw = m->maf_blocks[g];
    const bool rev = (g & 1) != 0;
    const float* w1 = rd.take((size_t)H * D);
    tmp.assign((size_t)H * D, 0.f);
    for (int j = 0; j < H; ++j)
      for (int i = 0; i < D; ++i)
        if (deg_hidden(j) >= i + 1) tmp[(size_t)j * D + (rev ? D - 1 - i : i)] = w1[(size_t)unit[j] * D + i];
    TF_TRY(upload_matrix(m, &bw.w1, tmp.data(), H, D, staging, 0));
    TF_TRY(upload_slab_bounds(m, &bw.w1, tmp.data()));
    TF_TRY(upload_sorted(&bw.b1, rd.take(H)));
    const float* w2 = rd.take((size_t)H * H);
    tmp.assign((size_t)H * H, 0.f);
    for (int j = 0; j < H; ++j)
      for (int i = 0; i < H; ++i)
        if (deg_hidden(j) >= deg_hidden(i)) tmp[(size_t)j * H + i] = w2[(size_t)unit[j] * H + unit[i]];
    TF_TRY(upload_matrix(m, &bw.w2, tmp.data(), H, H, staging, 0));
    TF_TRY(upload_slab_bounds(m, &bw.w2, tmp.data()));
    TF_TRY(upload_sorted(&bw.b2, rd.take(H)));
    // output layer [mu | alpha] -> interleaved rows (2 i, 2 i + 1) = (mu_i, alpha_i) in the sample's own order
    const float* w3 = rd.take((size_t)2 * D * H);
    const float* b3 = rd.take((size_t)2 * D);
    tmp.assign((size_t)2 * D * H, 0.f);
    for (int i = 0; i < D; ++i) {
      const int r = rev ? D - 1 - i : i;  // position of the layer's dimension i in the sample's order
      for (int j = 0; j < H; ++j)
        if (i + 1 > deg_hidden(j)) {
          tmp[(size_t)(2 * r) * H + j] = w3[(size_t)i * H + unit[j]];
          tmp[(size_t)(2 * r + 1) * H + j] = w3[(size_t)(D + i) * H + unit[j]];
        }
      btmp[2 * r] = b3[i];
      btmp[2 * r + 1] = b3[D + i];
    }
    TF_TRY(upload_matrix(m, &bw.w3, tmp.data(), 2 * D, H, staging, 0));
    TF_TRY(upload_slab_bounds(m, &bw.w3, tmp.data()));
    TF_TRY(upload_f32(m, &bw.b3, btmp.data(), btmp.size()));
  }

  const size_t B = c.max_batch, esz = c.dtype == 1 ? 2 : 4;
  TF_TRY(dev_alloc(m, &m->seq_a, B * D));
  TF_TRY(dev_alloc(m, &m->seq_b, B * D));
  TF_TRY(dev_alloc(m, &m->o, B * 2 * D));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->maf_a0), B * D * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->maf_a0_lo), B * D * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->maf_h1), B * H * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->maf_h1_lo), B * H * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->maf_h2), B * H * esz));
  TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->maf_h2_lo), B * H * esz));
  TF_TRY(dev_alloc(m, &m->maxdiff, B));
  TF_TRY(dev_alloc(m, &m->idx, B));
  TF_TRY(dev_alloc(m, &m->idx_tmp, B));
  TF_TRY(dev_alloc(m, &m->phase, B));
  if (B > (size_t)FIN_CHUNK) {
    const size_t nblk = (B + FIN_CHUNK - 1) / FIN_CHUNK;
    TF_TRY(dev_alloc(m, &m->fin_code, B));
    TF_TRY(dev_alloc(m, &m->fin_cnt, 2 * nblk));
    TF_TRY(dev_alloc(m, &m->fin_top, nblk));
    TF_TRY(dev_alloc(m, &m->fin_flag, nblk));
  }
  TF_TRY(dev_alloc(m, &m->ctrl, CTRL_WORDS));
  TF_TRY(dev_alloc(m, &m->err, 1));
  TF_TRY(dev_alloc(m, &m->iters_sample, (size_t)c.n_blocks * B));
  CU_OK(cudaMemset(m->ctrl, 0, CTRL_WORDS * sizeof(int)));
  CU_OK(cudaMemset(m->err, 0, sizeof(int)));
  CU_OK(cudaMemset(m->maxdiff, 0, B * sizeof(float)));
  CU_OK(cudaMemset(m->iters_sample, 0, (size_t)c.n_blocks * B * sizeof(int)));
  CU_OK(cudaMallocHost(&m->ctrl_host, HOST_WORDS * sizeof(int)));
  memset(m->ctrl_host, 0, HOST_WORDS * sizeof(int));
  m->block_ev.assign(c.n_blocks + 1, nullptr);
  for (auto& e : m->block_ev) CU_OK(cudaEventCreate(&e));
  if (c.dtype == 1) {
    void* bufs[3][2] = {{m->maf_a0, m->maf_a0_lo}, {m->maf_h1, m->maf_h1_lo}, {m->maf_h2, m->maf_h2_lo}};
    const int cols[3] = {D, H, H};
    for (int i = 0; i < 3; ++i)
      for (int t = 0; t < 2; ++t) TF_TRY(make_map_bf16(&m->maf_map[i][t], bufs[i][t], B, cols[i], tc::BM));
    CUtensorMap sm[5];
    TF_TRY(make_map_store(&sm[4], m->o, B, 2 * (uint64_t)D, 4));
    TF_TRY(make_map_store(&sm[0], m->maf_h1, B, H, 2));
    TF_TRY(make_map_store(&sm[1], m->maf_h1_lo, B, H, 2));
    TF_TRY(make_map_store(&sm[2], m->maf_h2, B, H, 2));
    TF_TRY(make_map_store(&sm[3], m->maf_h2_lo, B, H, 2));
    TF_TRY(dev_alloc(m, reinterpret_cast<char**>(&m->maf_store_maps), sizeof(sm)));
    CU_OK(cudaMemcpy(m->maf_store_maps, sm, sizeof(sm), cudaMemcpyHostToDevice));
    if (const char* e = getenv("TARFLOW_PAIR_GEMM")) m->use_pair_gemm = atoi(e) != 0;
    if (const char* e = getenv("TARFLOW_SWEEP_GRAPH_ROWS")) m->sweep_graph_rows = atoll(e);
    CU_OK(cudaStreamCreateWithFlags(&m->cap_stream, cudaStreamNonBlocking));
  }
  CU_OK(cudaDeviceSynchronize());
  return TF_OK;
}

static int check_call(tf_model* m, int B, bool want_maf = false) {
  if (!m) return fail(TF_EINVAL, "model is NULL");
  if (m->is_maf != want_maf)
    return fail(TF_EINVAL, want_maf ? "this call needs a model loaded with tf_maf_load" : "this call needs a model loaded with tf_load");
  if (B < 1 || B > m->cfg.max_batch) return fail(TF_EINVAL, "B=%d outside [1, max_batch=%d]", B, m->cfg.max_batch);
  return TF_OK;
}

// ------------------------------------------------------------------------------------------------
// C ABI
// ------------------------------------------------------------------------------------------------
extern "C" {

const char* tf_last_error(void) { return g_err; }

int tf_load(const tf_config* cfg, const void* weights_host, size_t nbytes, tf_model** out) {
  g_err[0] = 0;
  if (!cfg || !weights_host || !out) return fail(TF_EINVAL, "NULL argument");
  *out = nullptr;
  const tf_config& c = *cfg;
  if (c.C < 1 || c.H < 1 || c.W < 1 || c.patch < 1 || c.H % c.patch || c.W % c.patch)
    return fail(TF_EINVAL, "image %dx%dx%d not divisible by patch %d", c.C, c.H, c.W, c.patch);
  if (c.n_blocks < 1 || c.n_layers < 1 || c.width < 4 || c.n_heads < 1 || c.width % c.n_heads || c.width % 4 ||
      c.mlp_ratio < 1 || c.n_classes < 0 || c.max_batch < 1)
    return fail(TF_EINVAL, "bad model dimensions");
  if (c.dtype != 0 && c.dtype != 1) return fail(TF_EINVAL, "dtype must be 0 (fp32) or 1 (bf16)");
  if (c.dtype == 1 && (c.width % 64 || c.width / c.n_heads != 64))
    return fail(TF_EINVAL, "bf16 engine needs width %% 64 == 0 and head_dim == 64");
  if (c.width > 2048) return fail(TF_EINVAL, "width > 2048 not supported");
  if (c.dtype == 1 && c.width > 1024) return fail(TF_EINVAL, "bf16 engine: width > 1024 not supported");
  tf_model* m = new (std::nothrow) tf_model();
  if (!m) return fail(TF_ENOMEM, "host allocation failed");
  m->cfg = c;
  m->L = (c.H / c.patch) * (c.W / c.patch);
  m->D = c.C * c.patch * c.patch;
  m->d = c.width;
  m->hid = c.mlp_ratio * c.width;
  m->hd = c.width / c.n_heads;
  if (m->L < 2) { delete m; return fail(TF_EINVAL, "need at least 2 tokens"); }
  int r = load_impl(m, weights_host, nbytes);
  if (r != TF_OK) {
    tf_free(m);
    return r;
  }
  *out = m;
  return TF_OK;
}

void tf_free(tf_model* m) {
  if (!m) return;
  cudaDeviceSynchronize();
  m->prof_collect();
  seqp_turn_leave(m);
  for (cudaEvent_t e : m->ev_pool) cudaEventDestroy(e);
  for (cudaEvent_t e : m->block_ev) if (e) cudaEventDestroy(e);
  for (auto& kv : m->seq_graphs) if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
  for (auto& kv : m->sweep_graphs) if (kv.second.exec) cudaGraphExecDestroy(kv.second.exec);
  if (m->cap_stream) cudaStreamDestroy(m->cap_stream);
  for (int c = 0; c < tf_model::MAX_CHAINS; ++c) {
    if (m->seq_streams[c]) cudaStreamDestroy(m->seq_streams[c]);
    if (m->seq_join[c]) cudaEventDestroy(m->seq_join[c]);
  }
  if (m->seq_fork) cudaEventDestroy(m->seq_fork);
  for (void* p : m->allocs) cudaFree(p);
  if (m->guards_dev) cudaFree(m->guards_dev);
  if (m->guard_count) cudaFree(m->guard_count);
  if (m->ctrl_host) cudaFreeHost(m->ctrl_host);
  delete m;
}

int tf_forward(tf_model* m, const float* x_dev, const int32_t* labels_dev, int32_t B, float* z_dev, float* logdet_dev,
               void* cuda_stream) {
  g_err[0] = 0;
  TF_TRY(check_call(m, B));
  if (!x_dev || !z_dev) return fail(TF_EINVAL, "NULL buffer");
  if (m->cfg.n_classes > 0 && !labels_dev) return fail(TF_EINVAL, "class-conditional model needs labels");
  m->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
  return m->cfg.dtype == 1 ? forward_impl<bf16>(m, x_dev, labels_dev, B, z_dev, logdet_dev)
                           : forward_impl<float>(m, x_dev, labels_dev, B, z_dev, logdet_dev);
}

static int inverse_checked(tf_model* m, const float* z_dev, const int32_t* labels_dev, int32_t B, const uint8_t* policy_host,
                           float tau, int32_t max_iters, const InvOpts& op, float* x_dev, int32_t* iters_block_host,
                           int32_t* iters_sample_dev, void* cuda_stream) {
  TF_TRY(check_call(m, B));
  if (!z_dev || !x_dev || !policy_host) return fail(TF_EINVAL, "NULL buffer");
  if (m->cfg.n_classes > 0 && !labels_dev) return fail(TF_EINVAL, "class-conditional model needs labels");
  if (max_iters < 1) return fail(TF_EINVAL, "max_iters must be >= 1");
  if (op.init_mode < 0 || op.init_mode > 2) return fail(TF_EINVAL, "init_mode must be 0, 1 or 2");
  if (op.init_mode == 2 && !op.u0_img) return fail(TF_EINVAL, "init_mode 2 needs u0_dev");
  if (op.fallback_sweeps < 0) return fail(TF_EINVAL, "fallback_sweeps must be >= 0");
  if (tau != tau) return fail(TF_EINVAL, "tau is NaN");
  for (int g = 0; g < m->cfg.n_blocks; ++g) {
    if (policy_host[g] > 1) return fail(TF_EINVAL, "policy[%d]=%d is neither 0 nor 1", g, (int)policy_host[g]);
    if (op.tau_block && op.tau_block[g] != op.tau_block[g]) return fail(TF_EINVAL, "tau_block[%d] is NaN", g);
  }
  m->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
  return m->cfg.dtype == 1 ? inverse_impl<bf16>(m, z_dev, labels_dev, B, policy_host, tau, max_iters, op, x_dev,
                                                iters_block_host, iters_sample_dev)
                           : inverse_impl<float>(m, z_dev, labels_dev, B, policy_host, tau, max_iters, op, x_dev,
                                                 iters_block_host, iters_sample_dev);
}

int tf_inverse_jacobi(tf_model* m, const float* z_dev, const int32_t* labels_dev, int32_t B, const uint8_t* policy_host,
                      float tau, int32_t max_iters, int32_t init_mode, float* x_dev, int32_t* iters_block_host,
                      int32_t* iters_sample_dev, void* cuda_stream) {
  g_err[0] = 0;
  if (init_mode != 0 && init_mode != 1) return fail(TF_EINVAL, "init_mode must be 0 or 1");
  InvOpts op;
  op.init_mode = init_mode;
  return inverse_checked(m, z_dev, labels_dev, B, policy_host, tau, max_iters, op, x_dev, iters_block_host, iters_sample_dev,
                         cuda_stream);
}

int tf_inverse_jacobi_ex(tf_model* m, const float* z_dev, const int32_t* labels_dev, int32_t B, const uint8_t* policy_host,
                         float tau, int32_t max_iters, const tf_jacobi_opts* opts, float* x_dev, int32_t* iters_block_host,
                         int32_t* iters_sample_dev, void* cuda_stream) {
  g_err[0] = 0;
  InvOpts op;
  if (opts) {
    if (opts->struct_bytes != (int32_t)sizeof(tf_jacobi_opts)) return fail(TF_EINVAL, "tf_jacobi_opts.struct_bytes is %d, expected %d", opts->struct_bytes, (int)sizeof(tf_jacobi_opts));
    op.init_mode = opts->init_mode;
    op.u0_img = opts->u0_dev;
    op.tau_block = opts->tau_block_host;
    op.fallback_sweeps = opts->fallback_sweeps;
    op.states_img = opts->states_dev;
    op.ref_img = opts->ref_states_dev;
  }
  return inverse_checked(m, z_dev, labels_dev, B, policy_host, tau, max_iters, op, x_dev, iters_block_host, iters_sample_dev,
                         cuda_stream);
}

int tf_block_times(tf_model* m, float* ms_host, int32_t cap) {
  if (!m) return fail(TF_EINVAL, "model is NULL");
  const int K = m->cfg.n_blocks;
  if (!m->block_ev_valid) return 0;
  for (int g = 0; g < K && g < cap; ++g) {
    float ms = 0.f;
    if (cudaEventElapsedTime(&ms, m->block_ev[g], m->block_ev[g + 1]) != cudaSuccess) { cudaGetLastError(); return 0; }
    if (ms_host) ms_host[g] = ms;
  }
  return K;
}

int tf_inverse_sequential(tf_model* m, const float* z_dev, const int32_t* labels_dev, int32_t B, float* x_dev,
                          void* cuda_stream) {
  if (!m) return fail(TF_EINVAL, "model is NULL");
  std::vector<uint8_t> policy(m->cfg.n_blocks, 0);
  return tf_inverse_jacobi(m, z_dev, labels_dev, B, policy.data(), 0.f, 1, 0, x_dev, nullptr, nullptr, cuda_stream);
}

int tf_inverse_jacobi_host(tf_model* m, const float* z_host, const int32_t* labels_host, int32_t B,
                           const uint8_t* policy_host, float tau, int32_t max_iters, int32_t init_mode, float* x_host,
                           int32_t* iters_block_host, int32_t* iters_sample_host, void* cuda_stream) {
  g_err[0] = 0;
  TF_TRY(check_call(m, B));
  if (!z_host || !x_host) return fail(TF_EINVAL, "NULL buffer");
  if (m->cfg.n_classes > 0 && !labels_host) return fail(TF_EINVAL, "class-conditional model needs labels");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  size_t n = (size_t)B * m->cfg.C * m->cfg.H * m->cfg.W;
  CU_OK(cudaMemcpyAsync(m->io_z, z_host, n * sizeof(float), cudaMemcpyHostToDevice, st));
  if (labels_host) CU_OK(cudaMemcpyAsync(m->io_labels, labels_host, B * sizeof(int), cudaMemcpyHostToDevice, st));
  int r = tf_inverse_jacobi(m, m->io_z, labels_host ? m->io_labels : nullptr, B, policy_host, tau, max_iters, init_mode,
                            m->io_x, iters_block_host, nullptr, cuda_stream);
  if (r < 0) return r;
  CU_OK(cudaMemcpyAsync(x_host, m->io_x, n * sizeof(float), cudaMemcpyDeviceToHost, st));
  if (iters_sample_host)
    for (int g = 0; g < m->cfg.n_blocks; ++g)
      CU_OK(cudaMemcpyAsync(iters_sample_host + (size_t)g * B, m->iters_sample + (size_t)g * m->cfg.max_batch,
                            B * sizeof(int), cudaMemcpyDeviceToHost, st));
  CU_OK(cudaStreamSynchronize(st));
  return r;
}

int tf_maf_load(const tf_maf_config* cfg, const void* weights_host, size_t nbytes, tf_model** out) {
  g_err[0] = 0;
  if (!cfg || !weights_host || !out) return fail(TF_EINVAL, "NULL argument");
  *out = nullptr;
  if (cfg->D < 2 || cfg->hidden < 1 || cfg->n_blocks < 1 || cfg->max_batch < 1) return fail(TF_EINVAL, "bad model dimensions");
  if (cfg->dtype != 0 && cfg->dtype != 1) return fail(TF_EINVAL, "dtype must be 0 (fp32) or 1 (bf16)");
  if (cfg->dtype == 1 && (cfg->D % 8 || cfg->hidden % 64))
    return fail(TF_EINVAL, "bf16 engine needs D %% 8 == 0 and hidden %% 64 == 0");
  tf_model* m = new (std::nothrow) tf_model();
  if (!m) return fail(TF_ENOMEM, "host allocation failed");
  m->is_maf = true;
  m->small_m_rows = m->split_m_rows = 0;  // the MLP flow keeps one tile shape from 256 rows up: results do not depend on the batch
  m->cfg = tf_config{1, cfg->D, 1, 1, cfg->n_blocks, 2, cfg->hidden, 1, 1, 0, cfg->dtype, cfg->max_batch};
  m->L = cfg->D;  // D values per sample, token dimension 1
  m->D = 1;
  m->d = m->hid = m->maf_H = cfg->hidden;
  m->hd = cfg->hidden;
  int r = maf_load_impl(m, weights_host, nbytes, cfg->D, cfg->hidden);
  if (r != TF_OK) {
    tf_free(m);
    return r;
  }
  *out = m;
  return TF_OK;
}

int tf_maf_forward(tf_model* m, const float* x_dev, int32_t B, float* z_dev, float* logdet_dev, void* cuda_stream) {
  g_err[0] = 0;
  TF_TRY(check_call(m, B, true));
  if (!x_dev || !z_dev) return fail(TF_EINVAL, "NULL buffer");
  m->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
  return m->cfg.dtype == 1 ? maf_forward_impl<bf16>(m, x_dev, B, z_dev, logdet_dev) : maf_forward_impl<float>(m, x_dev, B, z_dev, logdet_dev);
}

int tf_maf_inverse_sequential(tf_model* m, const float* z_dev, int32_t B, float* x_dev, void* cuda_stream) {
  g_err[0] = 0;
  TF_TRY(check_call(m, B, true));
  if (!z_dev || !x_dev) return fail(TF_EINVAL, "NULL buffer");
  m->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
  return m->cfg.dtype == 1 ? maf_inverse_impl<bf16>(m, z_dev, B, false, 0.f, 1, 0, x_dev, nullptr, nullptr)
                           : maf_inverse_impl<float>(m, z_dev, B, false, 0.f, 1, 0, x_dev, nullptr, nullptr);
}

int tf_maf_inverse_jacobi(tf_model* m, const float* z_dev, int32_t B, float tau, int32_t max_iters, int32_t init_mode,
                          float* x_dev, int32_t* iters_block_host, int32_t* iters_sample_dev, void* cuda_stream) {
  g_err[0] = 0;
  TF_TRY(check_call(m, B, true));
  if (!z_dev || !x_dev) return fail(TF_EINVAL, "NULL buffer");
  if (max_iters < 1) return fail(TF_EINVAL, "max_iters must be >= 1");
  if (init_mode != 0 && init_mode != 1) return fail(TF_EINVAL, "init_mode must be 0 or 1");
  if (tau != tau) return fail(TF_EINVAL, "tau is NaN");
  m->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
  return m->cfg.dtype == 1
             ? maf_inverse_impl<bf16>(m, z_dev, B, true, tau, max_iters, init_mode, x_dev, iters_block_host, iters_sample_dev)
             : maf_inverse_impl<float>(m, z_dev, B, true, tau, max_iters, init_mode, x_dev, iters_block_host, iters_sample_dev);
}

int tf_jacobi_update(const float* o_dev, const float* v_dev, float* u_dev, float* maxdiff_dev, int32_t B, int32_t L,
                     int32_t D, int32_t reversed, void* cuda_stream) {
  g_err[0] = 0;
  if (!o_dev || !v_dev || !u_dev || !maxdiff_dev) return fail(TF_EINVAL, "NULL buffer");
  if (B < 1 || L < 2 || D < 1) return fail(TF_EINVAL, "bad sizes");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  CU_OK(cudaMemsetAsync(maxdiff_dev, 0, B * sizeof(float), st));
  size_t n = (size_t)B * L * D;
  int blocks = (int)((n + 255) / 256);
  if (blocks > 148 * 8) blocks = 148 * 8;
  jacobi_update_kernel<<<blocks, 256, 0, st>>>(o_dev, v_dev, u_dev, maxdiff_dev, nullptr, B * L, L, D, reversed, 0);
  return check_launch("jacobi_update_kernel");
}

static int* g_gemm_err[kMaxDevices] = {nullptr};  // error word of the model-less GEMM entry point (one per device)

int tf_gemm_bf16(const void* a_dev, const void* w_dev, const float* bias_dev, float* c_dev, int32_t M, int32_t N,
                 int32_t K, void* cuda_stream) {
  g_err[0] = 0;
  if (!a_dev || !w_dev || !c_dev) return fail(TF_EINVAL, "NULL buffer");
  if (M < 1 || N < 8 || K < 64 || K % 64 || N % 8) return fail(TF_EINVAL, "need M>=1, N%%8==0, K%%64==0");
  const int dev = current_device();
  if (dev < 0) return fail(TF_EINVAL, "no current device with an ordinal below %d", kMaxDevices);
  if (!g_gemm_err[dev]) {
    CU_OK(cudaMalloc(&g_gemm_err[dev], sizeof(int)));
    CU_OK(cudaMemset(g_gemm_err[dev], 0, sizeof(int)));
  }
  int sms = 148;
  CU_OK(cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev));
  const int bn = (N % 256 == 0) ? 256 : 128;
  CUtensorMap ma, mw;
  TF_TRY(make_map_bf16(&ma, a_dev, M, K, tc::BM));
  TF_TRY(make_map_bf16(&mw, w_dev, N, K, bn));
  EpiStore<float, false> epi{c_dev, bias_dev, N};
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  if (bn == 256) return launch_gemm_tc<256, 4>(nullptr, 0, st, ma, nullptr, mw, M, N, K, epi, g_gemm_err[dev], sms, nullptr);
  return launch_gemm_tc<128, 6>(nullptr, 0, st, ma, nullptr, mw, M, N, K, epi, g_gemm_err[dev], sms, nullptr);
}

int tf_gemm_status(void* cuda_stream) {
  g_err[0] = 0;
  CU_OK(cudaStreamSynchronize(reinterpret_cast<cudaStream_t>(cuda_stream)));
  const int dev = current_device();
  if (dev < 0 || !g_gemm_err[dev]) return TF_OK;
  int e = 0;
  CU_OK(cudaMemcpy(&e, g_gemm_err[dev], sizeof(int), cudaMemcpyDeviceToHost));
  if (e != 0) {  // reported once, then cleared: later launches run normally
    CU_OK(cudaMemset(g_gemm_err[dev], 0, sizeof(int)));
    return fail(TF_ETIMEOUT, "device-side wait expired in tf_gemm_bf16 (code %d)", e);
  }
  return TF_OK;
}

// ------------------------------------------------------------------------------------------------
// Allocation-free skinny GEMM (see tf_skinny_gemm_noalloc in tarflow.h).  The split-K partial tiles and
// the step-counter word the kernel reads live in a static device array instead of cudaMalloc'd memory.
// ------------------------------------------------------------------------------------------------
#define TF_NOALLOC_HEADER_BYTES 256u
static __device__ __align__(256) unsigned char g_noalloc_scratch[TF_NOALLOC_SCRATCH_BYTES];
static unsigned char* g_noalloc_ptr[kMaxDevices] = {nullptr};  // device address of the array, per device ordinal

// c[m, n] = bias[n] + sum over K slices of part[s][m][n], slices added in index order
__global__ void noalloc_reduce_kernel(const float* __restrict__ part, const float* __restrict__ bias,
                                      float* __restrict__ c, int nsplit, int M, int N) {
  const size_t total = (size_t)M * N;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < total; i += (size_t)gridDim.x * blockDim.x) {
    float acc = bias ? bias[i % N] : 0.f;
    for (int sl = 0; sl < nsplit; ++sl) acc += part[(size_t)sl * total + i];
    c[i] = acc;
  }
}

int tf_skinny_gemm_noalloc(const void* a_dev, const void* w_dev, const float* bias_dev, float* c_dev, int32_t M, int32_t N,
                           int32_t K, void* cuda_stream) {
  g_err[0] = 0;
  if (!a_dev || !w_dev || !c_dev) return fail(TF_EINVAL, "NULL buffer");
  if (M < 1 || N < 8 || N % 8 || K < 256 || K % 256) return fail(TF_EINVAL, "need M >= 1, N %% 8 == 0, K %% 256 == 0");
  // the kernel reads A and W with 16-byte accesses and the reduction reads/writes 4-byte floats: a misaligned pointer
  // would fault on the device, so it is refused here
  if ((reinterpret_cast<uintptr_t>(a_dev) | reinterpret_cast<uintptr_t>(w_dev)) & 15)
    return fail(TF_EINVAL, "tf_skinny_gemm_noalloc: a_dev and w_dev must be 16-byte aligned");
  if ((reinterpret_cast<uintptr_t>(c_dev) | reinterpret_cast<uintptr_t>(bias_dev)) & 3)
    return fail(TF_EINVAL, "tf_skinny_gemm_noalloc: c_dev and bias_dev must be 4-byte aligned");
  const int klen = 256, ksplit = K / klen;
  const size_t need = (size_t)ksplit * M * N * sizeof(float);
  if (need > (size_t)TF_NOALLOC_SCRATCH_BYTES - TF_NOALLOC_HEADER_BYTES)
    return fail(TF_EINVAL, "tf_skinny_gemm_noalloc: (K/256)*M*N*4 = %zu bytes of partial tiles exceed the %zu-byte static scratch",
                need, (size_t)TF_NOALLOC_SCRATCH_BYTES - TF_NOALLOC_HEADER_BYTES);
  const int dev = current_device();
  if (dev < 0) return fail(TF_EINVAL, "no current device with an ordinal below %d", kMaxDevices);
  using Kern = void (*)(const bf16*, const bf16*, int, int, int, int, float*, const int*, int, int, int);
  Kern kern = seq::seq_gemm_kernel<8>;
  const int smem = seq::gemm_smem_bytes(klen);
  if (!g_noalloc_ptr[dev]) {  // once per device, with that device current: resolve the symbol to a device address
    unsigned char* p = nullptr;
    CU_OK(cudaGetSymbolAddress(reinterpret_cast<void**>(&p), g_noalloc_scratch));
    // the same limit tf_load sets for this kernel, so a model loaded earlier keeps its larger K slices
    CU_OK(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, seq::gemm_smem_bytes(seq::KC)));
    g_noalloc_ptr[dev] = p;
  }
  unsigned char* base = g_noalloc_ptr[dev];
  int* step_word = reinterpret_cast<int*>(base);
  float* part = reinterpret_cast<float*>(base + TF_NOALLOC_HEADER_BYTES);
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  // the array keeps whatever the last call left: the step word must read 0; the tiles are fully overwritten
  CU_OK(cudaMemsetAsync(step_word, 0, sizeof(int), st));
  dim3 grid((N + 7) / 8, ksplit, (M + seq::ROWS - 1) / seq::ROWS);
  kern<<<grid, seq::THREADS, smem, st>>>(reinterpret_cast<const bf16*>(a_dev), reinterpret_cast<const bf16*>(w_dev), M, N, K,
                                         klen, part, step_word, 0, 1, 0);
  TF_TRY(check_launch("seq_gemm_kernel (no-alloc)"));
  const size_t total = (size_t)M * N;
  int blocks = (int)((total + 255) / 256);
  if (blocks > 148 * 8) blocks = 148 * 8;
  noalloc_reduce_kernel<<<blocks, 256, 0, st>>>(part, bias_dev, c_dev, ksplit, M, N);
  return check_launch("noalloc_reduce_kernel");
}

int tf_selftest_wait_timeout(tf_model* m, int32_t limit_us, void* cuda_stream) {
  g_err[0] = 0;
  if (!m) return fail(TF_EINVAL, "model is NULL");
  if (limit_us < 1 || limit_us > 1000000) return fail(TF_EINVAL, "limit_us must lie in [1, 1000000]");
  m->stream = reinterpret_cast<cudaStream_t>(cuda_stream);
  LAUNCH(m, KC_CTRL, tc::wait_selftest_kernel, 1, 32, 0, m->err, (unsigned long long)limit_us * 1000ull);
  TF_TRY(check_launch("wait_selftest_kernel"));
  int r = sync_check(m);
  // the polled pair of words is a part of the control words that nothing writes: zero, where the number waited for is 1
  for (int which = 0; which < 2 && r == TF_ETIMEOUT; ++which) {
    CU_OK(cudaMemsetAsync(m->ctrl + CTRL_SELFTEST, 0, 4 * sizeof(int), m->stream));
    LAUNCH(m, KC_CTRL, seqp::wait_selftest_kernel, 1, 32, 0, m->err, which,
           reinterpret_cast<const unsigned long long*>(m->ctrl + CTRL_SELFTEST));
    TF_TRY(check_launch("seqp::wait_selftest_kernel"));
    r = sync_check(m);
  }
  return r == TF_OK ? fail(TF_ECUDA, "a wait that nothing satisfies did not run out") : r;
}

int64_t tf_debug_check_guards(tf_model* m, void* cuda_stream) {
  g_err[0] = 0;
  if (!m) return fail(TF_EINVAL, "model is NULL");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(cuda_stream);
  const int n = (int)m->guards.size();
  if (!m->guards_dev) {  // plain cudaMalloc: these two are not themselves guarded
    CU_OK(cudaMalloc(&m->guards_dev, (size_t)n * sizeof(unsigned char*)));
    CU_OK(cudaMalloc(&m->guard_count, sizeof(int)));
    CU_OK(cudaMemcpy(m->guards_dev, m->guards.data(), (size_t)n * sizeof(unsigned char*), cudaMemcpyHostToDevice));
  }
  CU_OK(cudaMemsetAsync(m->guard_count, 0, sizeof(int), st));
  guard_check_kernel<<<n, (int)(GUARD_BYTES / 4), 0, st>>>(m->guards_dev, m->guard_count, 0x01010101u * GUARD_BYTE);
  TF_TRY(check_launch("guard_check_kernel"));
  int bad = 0;
  CU_OK(cudaMemcpyAsync(&bad, m->guard_count, sizeof(int), cudaMemcpyDeviceToHost, st));
  CU_OK(cudaStreamSynchronize(st));
  if (bad != 0) fail(TF_OK, "%d guard words next to the model's device buffers were overwritten", bad);
  return bad;
}

int tf_debug_set(tf_model* m, int32_t what, int64_t value) {
  g_err[0] = 0;
  if (!m) return fail(TF_EINVAL, "model is NULL");
  switch (what) {
    case TF_DEBUG_REFUSE_BLOCK_LAUNCH: m->seqp_debug_refuse = value != 0; return TF_OK;
    case TF_DEBUG_EXCHANGE_NUMBER:
      if (value < (int64_t)m->seqp_seq || value > (int64_t)UINT32_MAX) return fail(TF_EINVAL, "sequence numbers only grow, up to 2^32 - 1");
      m->seqp_seq = (uint32_t)value;
      return TF_OK;
  }
  return fail(TF_EINVAL, "unknown debug setting %d", what);
}

int tf_profile_enable(tf_model* m, int32_t on) {
  if (!m) return fail(TF_EINVAL, "model is NULL");
  cudaDeviceSynchronize();
  m->prof_collect();
  for (int c = 0; c < KC_COUNT; ++c) { m->prof_ms[c] = 0; m->prof_n[c] = 0; m->prof_rows[c] = 0; }
  m->prof_on = on != 0;
  m->prof_mode = on == 2 ? 2 : (on != 0 ? 1 : 0);
  return TF_OK;
}

int tf_profile_read(tf_model* m, const char** names, double* ms, int64_t* launches, double* rows, int32_t cap) {
  if (!m) return fail(TF_EINVAL, "model is NULL");
  m->prof_collect();
  for (int c = 0; c < KC_COUNT && c < cap; ++c) {
    if (names) names[c] = kKernelClassNames[c];
    if (ms) ms[c] = m->prof_ms[c];
    if (launches) launches[c] = m->prof_n[c];
    if (rows) rows[c] = m->prof_rows[c];
  }
  return KC_COUNT;
}

int tf_set_precision(tf_model* m, int32_t mode, float switch_threshold, float single_ok_tau) {
  if (!m) return fail(TF_EINVAL, "model is NULL");
  if (mode < 0 || mode > 2) return fail(TF_EINVAL, "precision mode must be 0, 1 or 2");
  m->precision_mode = mode;
  m->switch_threshold = switch_threshold > 0.f ? switch_threshold : 0.03125f;
  m->single_ok_tau = single_ok_tau > 0.f ? single_ok_tau : 0.015625f;
  return TF_OK;
}

int tf_trace_enable(tf_model* m, int32_t on) {
  if (!m) return fail(TF_EINVAL, "model is NULL");
  m->trace_on = on != 0;
  m->trace.clear();
  m->trace_l2_count.assign(m->cfg.n_blocks, 0);
  if (m->trace_on && !m->trace_l2) {  // distance records: up to L + 2 sweeps per block
    m->trace_l2_sweeps = m->L + 2;
    TF_TRY(dev_alloc(m, &m->trace_l2, (size_t)m->cfg.n_blocks * m->trace_l2_sweeps * m->cfg.max_batch));
  }
  return TF_OK;
}

int tf_trace_read_l2(tf_model* m, int32_t block, int32_t B, float* l2_host, int32_t cap_sweeps) {
  if (!m) return fail(TF_EINVAL, "model is NULL");
  if (block < 0 || block >= m->cfg.n_blocks || B < 1 || B > m->cfg.max_batch) return fail(TF_EINVAL, "bad block or batch");
  if (!m->trace_l2 || m->trace_l2_count.empty()) return 0;
  const int n = m->trace_l2_count[block];
  for (int t = 0; t < n && t < cap_sweeps && l2_host; ++t)
    CU_OK(cudaMemcpy(l2_host + (size_t)t * B, m->trace_l2 + ((size_t)block * m->trace_l2_sweeps + t) * m->cfg.max_batch,
                     B * sizeof(float), cudaMemcpyDeviceToHost));
  return n;
}

int tf_trace_read(tf_model* m, int32_t* block, int32_t* sweep, int32_t* active, float* maxdiff, int32_t cap) {
  if (!m) return fail(TF_EINVAL, "model is NULL");
  int n = (int)m->trace.size();
  for (int i = 0; i < n && i < cap; ++i) {
    if (block) block[i] = m->trace[i].block;
    if (sweep) sweep[i] = m->trace[i].sweep;
    if (active) active[i] = m->trace[i].active;
    if (maxdiff) maxdiff[i] = m->trace[i].maxdiff;
  }
  return n;
}

int64_t tf_launch_count(tf_model* m) { return m ? m->launches : 0; }
int64_t tf_device_bytes(tf_model* m) { return m ? m->device_bytes : 0; }

}  // extern "C"
