// pdADMM-G / pdADMM-G-Q on one B200: context, host orchestration of one iteration, C ABI.
//
// Data layout (device): every N x width matrix is node-major with its leading dimension padded to a
// multiple of 16 or 32 floats (row_ld) and zero padding columns.  Per layer l the context keeps p_l, z_l, q_l, u_l,
// W_l, b_l and the linear residual r_l = W_l p_l + b_l - z_l, which every step of the iteration
// updates in place instead of recomputing the product:
//     p+ = p - g/tau        =>  r <- r - (W g)/tau            (pdADMM-G-Q: r <- r + W (p+ - p))
//     W+ = W - G/theta      =>  r <- r - (G p+)/theta
//     b+ = b - mean_j r     =>  r <- r - mean_j r      (mean_j r from column sums of r and p+)
//     z+                    =>  r <- (r + z) - z+
// so one iteration of a layer costs four dense products: W^T r (the p-gradient), W g (tau),
// r^T p+ (the W-gradient, contraction over the nodes) and G p+ (theta).
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <map>
#include <memory>
#include <tuple>
#include <vector>

#include "common.cuh"
#include "elementwise.cuh"
#include "gemm_simt.cuh"
#include "gemm_tc.cuh"
#include "graph.cuh"
#include "host_io.cuh"
#include "pools.cuh"

namespace pd {

// ---- kernel classes for the per-kernel timing -----------------------------------------------------
enum KClass {
  KC_GEMM_RESID = 0,  // r = P W^T + b - z                    (after init / set_tensor only)
  KC_GEMM_GRADP,      // g = nu r W + u + rho (p - q), ||g||^2
  KC_GEMM_WG,         // W g (or W d), squared norm
  KC_GEMM_GRADW,      // partial tiles of r^T p+ over node slices
  KC_GRADW_REDUCE,    // sum of the partial tiles, nu, ||G||^2
  KC_GEMM_GP,         // G p+, squared norm
  KC_AXPY,            // p -= g/tau, r -= (Wg)/tau
  KC_QUANT,           // quantised trial step
  KC_COLSUM,          // W -= G/theta, b (and r -= (G p+)/theta where the z-update does not)
  KC_ZQU,             // fused z, q, u update of a hidden layer
  KC_ZLAST,           // z update of the last layer
  KC_SMALL,           // column sums of r_L; bias of a shard; sums of the CUDA-core products
  KC_AMAX,            // largest magnitude of a product's node-sized operand (for its power-of-two scaling)
  KC_PLANES,          // fp16 planes made or made again by a kernel of their own
  KC_COUNT
};
static const char *kclass_names[KC_COUNT] = {
    "gemm_resid", "gemm_gradp", "gemm_wg", "gemm_gradw", "gradw_reduce", "gemm_gp", "axpy",
    "quant_trial", "resid_colsum", "zqu", "zlast", "finalize", "absmax", "make_planes"};

// fp16 hi/lo planes of a matrix, in its own orientation and with its leading dimension, and the device word with the
// exponent of the power-of-two scaling they were made with.
struct Planes {
  __half *hi = nullptr, *lo = nullptr;
  int *exp = nullptr;
};
// One operand of a tensor-core product: its planes [rows][ld] (hi null: to be split first, from x), and, where the exponent was
// chosen before the largest magnitude was known, the word `check` with that magnitude, by which the product decides whether
// the planes are good or have to be made again from x.  int_mul > 0: hi holds small integers that are to be multiplied by
// int_mul (a quantised p = code * s, or the difference of two), there is no lo plane.
struct Operand {
  const float *x; int ld;
  const uint32_t *amax;             // for splitting x first (null: computed)
  const __half *hi = nullptr, *lo = nullptr;
  const int *exp = nullptr;
  const uint32_t *check = nullptr;
  float int_mul = 0.f;
  int uses = 1;                     // output tiles that read an element of it (and would each split it again)
};
static Operand int_operand(const __half *plane, int ld, float mul) {
  Operand o{nullptr, ld, nullptr};
  o.hi = plane; o.lo = plane; o.int_mul = mul;
  return o;
}
static Operand plane_operand(const float *x, int ld, const Planes &p, const uint32_t *check = nullptr) {
  return Operand{x, ld, check, p.hi, p.lo, p.exp, check};
}

// number of lanes for the concurrency across layers (measured on workload c2: 1 lane 241.8, 2 lanes 273.3 iterations/s)
#ifndef PDADMM_N_LANES
#define PDADMM_N_LANES 2
#endif

struct Layer {
  int n_in = 0, n_out = 0, ld_in = 0, ld_out = 0;
  float *p = nullptr;       // [N][ld_in]  (layer 1: X)
  float *W = nullptr;       // [n_out][ld_in]
  float *b = nullptr;       // [ld_out]
  float *z = nullptr, *r = nullptr;          // [N][ld_out]
  float *q = nullptr, *u = nullptr;          // [N][ld_out], hidden layers only
  bool q_stale = false;     // the stored q is older than z and u, which give it (c->q_implied)
  float *t = nullptr;       // [N][ld_in], l >= 2: u_{l-1} + rho (p_l - q_{l-1}), the product-free part of grad_p phi
  float *gradW = nullptr;   // [n_out][ld_in]
  // Tensor-core path: planes of W, of grad_W and of r (written by the z-step for the next p-gradient;
  // none if the device has no room: the products then split r first), of p_1 = X, which never changes; the exponent words
  // belong to finalize_tau_kernel / finalize_theta_kernel, which settle them before the planes are written
  Planes Wp, Gp, rp, xp;
  int *g_exp = nullptr;     // l >= 2: exponent of the next planes of g_l
  uint32_t *amax_W = nullptr;      // max|W|, bit pattern
  float *shift = nullptr;   // [ld_out] column means removed by the b-update
  // column sums of p_l (layer 1: X), how the last p-step changed them, and of r_l, which give the b-update; those of r as the z-update's
  // blocks left them, too
  double *p_sum = nullptr, *p_change = nullptr, *r_sum = nullptr, *r_slots = nullptr;
  int p_blocks = 1, r_blocks = 1;            // blocks of the kernels that leave them
  float *gp = nullptr;      // G p+ on its way to the z-update: the memory of q where that is not kept (c->q_implied), the last layer's own
  uint8_t *codes = nullptr; // [N][ld_in] codes of 1 byte (up to 256 levels) or 2 bytes, quantised mode, l >= 2
  __half *p_plane = nullptr; // [N][ld_in] the codes as fp16 integers: operand plane of p_l = code * scale (see int_operands)
  float scale = 1.0f;       // level spacing s_l of p_l
  float lo = 0.0f;          // smallest level of p_l: -(levels below zero) * s_l
  LayerScalars *sc = nullptr;
  // Largest magnitudes (bit patterns) of the two node-sized operands of this layer's products, kept by the kernels
  // that write them: amax_p covers every p_l written since the last tau of the layer, amax_r every r_l written
  // since its last theta -- upper bounds of the current maxima, which is all the power-of-two scaling needs.
  uint32_t *amax_p = nullptr, *amax_r = nullptr;
  // largest magnitudes of an iteration's g, W g, G and d: zero before the kernel that writes the matrix
  uint32_t *w_g = nullptr, *w_wg = nullptr, *w_G = nullptr, *w_d = nullptr;
  int *done = nullptr;             // [4] counters of finished blocks (trial, gradient sum, then products), zero between kernels
  int n_split = 1, k_chunk = 0;
  bool wide_W = false, wide_wg = false, wide_gp = false;      // wide tiles for the W-gradient, W g and G p (choose_wide)
};

struct Scratch {
  cudaStream_t st = nullptr;       // where its layers' kernels are queued
  cudaStream_t own = nullptr;      // the stream it owns (grouped: st is the main stream)
  float *s1 = nullptr;      // g, later G p+
  float *s2 = nullptr;      // W g, later W d
  float *p_new = nullptr;   // quantised trial
  float *d = nullptr;       // quantised trial
  uint8_t *codes_new = nullptr;
  __half *pn_plane = nullptr, *d_plane = nullptr;   // planes of the trial's codes and of their change (see int_operands)
  float *part = nullptr;    // partial tiles of grad_W
  double *slots = nullptr;  // per-block partial sums
  size_t n_slots = 0;
  double *p_slots = nullptr;       // column sums of p+ as the p-step's blocks left them
  double *red = nullptr;    // sums on their way through the reduction over shards (widest layer + 8 values)
  float *tail_ws = nullptr; // accumulators of the contraction slices of tail tiles (one tile per SM at most)
  int *tail_count = nullptr;
  uint32_t *amax_pool = nullptr;   // words for the largest magnitudes of product operands, handed out in stream order
  int amax_next = 0;
  // planes [N][ld] of node-sized operands, as wide as the widest matrix of the context.  pl0: of g, from the p-gradient to
  // W g; then of r after the p-step (or the accepted trial), up to the W-gradient.  pl1: of p after the p-step, up to G p+;
  // before that and outside iterations, of any operand that has to be split first.
  Planes pl0, pl1;
  int *a_exp = nullptr;
  size_t pl_cap = 0;               // elements each plane holds
  int *h_flag = nullptr;           // pinned word that receives the accept flag of the lane's quantised trial
  cudaEvent_t ev_flag = nullptr;   // recorded after the copy of that flag
};

struct ProfRec { int cls; cudaEvent_t e0, e1; double bytes, flops; };

}  // namespace pd

struct pdadmm_ctx {
  int device = 0;
  int64_t N = 0;                   // nodes this context owns
  int64_t N_total = 0, node_begin = 0;   // the whole graph; first owned node
  pdadmm_allreduce_fn reduce = nullptr;  // adds over the shards' contexts (null: this context holds every node)
  void *reduce_user = nullptr;
  int64_t comm_bytes = 0;
  int L = 0, d = 0, n_blocks = 0, n0 = 0, ld0 = 0, C = 0, levels = 0;
  int code_bytes = 1;              // 1 for up to 256 levels, else 2
  int neg_levels = 0;              // levels below zero
  float fixed_step = 0.f;          // > 0: the same level spacing for every layer
  bool quant_q = false;            // q_l is kept on the level set of p_{l+1} as well
  float slope = 0.f;               // f_l (see act_eval): [0, 1) = (leaky) ReLU with that slope for x <= 0, 2 = tanh, 3 = sigmoid
  float table_lo = 0.f, table_step = 0.f;   // lookup table of the z-update of a smooth activation: z_i = lo + i step
  int table_size = 0;
  bool table_even = false;         // see table_is_even
  bool ls_risk = false;            // R = least squares instead of cross-entropy
  float rho = 0, nu = 0;
  uint32_t flags = 0;
  int64_t nnz = 0;
  int *row_ptr = nullptr, *col_idx = nullptr;
  float *csr_val = nullptr;
  int *labels = nullptr;
  uint8_t *mask = nullptr;
  std::vector<pd::Layer> layers;
  pd::Scratch scr;                  // lane 0: the context's main stream and its scratch
  // Layer concurrency: the updates of different layers are independent inside each phase of an iteration, so
  // layer l's chain of kernels is queued on lane l mod n_lanes.  Every lane has its own stream and its own scratch
  // (product outputs, partial tiles, reduction slots), so that chains of different layers can overlap: the next
  // product starts on the SMs that the previous one has already left, and bandwidth-bound kernels run beside
  // tensor-bound ones.  `cur` is the lane that the host code is queueing on.
  std::vector<std::unique_ptr<pd::Scratch>> more_lanes;
  pd::Scratch *cur = &scr;
  // A problem small enough for scratch per layer is worked on in batches instead: every kernel is launched once for up to
  // MAX_GROUP layers, on the main stream.
  bool grouped = false;
  bool tail_split = true;           // large problems: products cut the tiles of a partly filled last round (launch_tc)
  int n_active = 1;                 // scratches in use: layer l works with number l mod n_active
  bool p_stale = false;             // p_l, l >= 2, exists as codes alone (integer operands): the fp32 values are older
  std::vector<cudaEvent_t> ev_p;    // [L]: p_l of this iteration is complete
  std::vector<cudaEvent_t> ev_lane; // [n_lanes]: fork / join
  bool r_valid = false;
  bool t_valid = false;             // every layer's t matches the stored u, p, q
  // q_l = f(z_l) + u_l/nu after every iteration (see zqu_kernel), unless it is kept on a level set: it is not stored then, and its
  // memory serves G p+.  After the caller has set z, q or u the stored q is read once (and written, so that it is the layer's q wherever
  // that iteration ends).
  bool q_free = false;              // the context may do without it
  bool q_implied = false;           // z and u give it now
  bool in_iteration = false;        // an iteration was begun and has not been queued to its end
  bool p_sums_valid = false, r_sums_valid = false;          // the column sums of p_l and of r_l are those of the stored values
  // Words that are zero between calls, one block so that one clear covers them: d_flag[0..3] (z_L solver non-convergence, expired
  // wait, non-finite sum, unused), the layers' `done` and w_* words, the tail counts of the lanes that cut tails.
  int *control = nullptr;
  size_t control_words = 0;
  int *d_flag = nullptr;
  // page-locked block (CTX_PINNED_BYTES): words 0..63 small read-backs, 64..127 the lanes' accept flags, from byte 1024 on
  // the results that kernels write themselves (objective, residuals, counts of pdadmm_predict)
  int *h_pinned = nullptr;
  double *h_results = nullptr;
  int *done = nullptr;              // device: finished blocks per layer of a read-out kernel, zero between launches
  unsigned long long *counts = nullptr;   // device: the four counts of pdadmm_predict, zero between calls
  int64_t launches = 0;
  cudaEvent_t ev_begin = nullptr, ev_end = nullptr;
  double last_step_ms = 0.0;
  bool profiling = false;
  std::vector<pd::ProfRec> prof;
  std::vector<cudaEvent_t> ev_pool;
  double prof_ms[pd::KC_COUNT] = {0}, prof_bytes[pd::KC_COUNT] = {0}, prof_flops[pd::KC_COUNT] = {0};
  int64_t prof_n[pd::KC_COUNT] = {0};
  std::vector<pd::DeviceBlock> allocs;   // from the device's pool: chunks and large arrays
  size_t bytes_handed_out = 0;      // device bytes handed out by dev_alloc so far
  char *arena_base = nullptr;       // current chunk
  size_t arena_cap = 0, arena_used = 0, arena_next = size_t(64) << 20;
  bool use_tc = true;               // dense products on the tensor cores
  // pdADMM-G-Q with at most 2048 levels: p_l = (code - levels below zero) * s_l, integers that are exact in fp16, so
  // the products whose operand is p_l (or d = p+ - p) take one plane of integers instead of a hi and a lo plane of
  // the values: two MMAs per product instead of three, a quarter of the operand bytes, no split pass
  bool int_operands = false;
  cudaGraphExec_t iter_graph = nullptr;   // one captured pdADMM-G iteration (no host round trips in it)
  int64_t iter_graph_launches = 0;
  bool graph_failed = false;
  // Iterations left in which scalings are still found (see check_planes): two per layer from the start, or from a tensor that was
  // set; what the first ones change travels one layer further with every second iteration.  They run eagerly if they have
  // work for check_planes that a replay of a later iteration would leave out (`wide`).
  int cold = 0;
  bool wide = false;
  int n_sms = 148;
  bool w_planes_valid = false;
  bool amax_p_valid = false;        // every layer's amax_p covers the stored p
  bool x_planes_valid = false;      // the planes of X match the stored X
  std::map<std::tuple<const void *, uint64_t, uint64_t, uint64_t>, CUtensorMap> tmaps;
};

namespace pd {

// Leading dimension of a matrix of n columns: a multiple of 32 floats (tile copies and the coalesced stores of the epilogues move
// whole 128-byte lines), or of 16 where that leaves out at least a twenty-fifth of the padded row (whole 32-byte sectors still, of
// the fp16 planes too): 2000 x 100 in rows of 112 instead of 128 0.1151 -> 0.1139 ms per iteration, 7013 x 333 in 336 instead of 352
// 0.455 -> 0.441; but 170 000 x 1000 in 1008 instead of 1024 20.7 -> 21.6.  A context that owns part of the nodes keeps
// whole lines: its gradients go over as rows of them.
static int row_ld(const pdadmm_ctx *c, int n) {
  const int a = round_up(n, 32), b = round_up(n, 16);
  return c->reduce == nullptr && 25 * (a - b) >= a ? b : a;
}

// ---- allocation bookkeeping -------------------------------------------------------------------------
// Device memory of a context.  Arrays of up to 64 MB are carved out of chunks (64 MB at first, doubling up to
// 1 GB), 256-byte aligned: a context has some twenty arrays per layer, and one allocation each made
// pdadmm_init spend most of its time in the allocator.  Larger arrays get a block of their own, so that
// a chunk never wastes more than one small array at its end.  destroy() returns everything to the device's pool.
// A chunk is cleared as a whole when it is taken (200 clears of small arrays cost the host 0.5 ms at c1's sizes).
constexpr size_t ARENA_MAX_ARRAY = size_t(64) << 20, ARENA_MAX_CHUNK = size_t(1) << 30;   // first chunk: arena_next
template <class T>
static int dev_alloc(pdadmm_ctx *c, T **ptr, size_t count, bool zero = true) {
  // slack: operand copies may read up to 31 floats past a matrix
  const size_t bytes = (count * sizeof(T) + 256 + 255) & ~size_t(255);
  char *p = nullptr;
  if (bytes <= ARENA_MAX_ARRAY && c->arena_used + bytes <= c->arena_cap) {
    p = c->arena_base + c->arena_used;
    c->arena_used += bytes;
  } else {
    const bool chunk = bytes <= ARENA_MAX_ARRAY;
    const size_t want = chunk ? std::max(bytes, c->arena_next) : bytes;
    DeviceBlock b;
    const cudaError_t e = device_pool(c->device).take(want, &b);
    if (e != cudaSuccess) return fail(PDADMM_ENOMEM, "cudaMalloc of %zu bytes failed: %s", want, cudaGetErrorString(e));
    c->allocs.push_back(b);
    p = (char *)b.p;
    if (chunk) {
      c->arena_base = p; c->arena_cap = b.bytes; c->arena_used = bytes;
      c->arena_next = std::min(ARENA_MAX_CHUNK, 2 * want);
    }
    if (chunk || zero) PD_CUDA(cudaMemsetAsync(p, 0, chunk ? b.bytes : bytes, c->scr.st));   // same stream as every kernel that uses it
  }
  c->bytes_handed_out += bytes;
  *ptr = (T *)p;
  return PDADMM_OK;
}

static inline int ew_grid(size_t n_items) {
  return (int)std::max<size_t>(1, std::min<size_t>(ceil_div((int64_t)n_items, EW_THREADS), 148 * 8));
}

// ---- sums over the shards' contexts ---------------------------------------------------------------------------
static int shard_sum(pdadmm_ctx *c, cudaStream_t st, void *buf, size_t count, int is_double, int op = 0) {
  if (c->reduce == nullptr) return PDADMM_OK;
  c->comm_bytes += (int64_t)(count * (is_double ? 8 : 4));
  const int rc = c->reduce(c->reduce_user, buf, count, is_double, op, (void *)st);
  if (rc != 0) return fail(PDADMM_ECUDA, "the reduction callback returned %d", rc);
  return PDADMM_OK;
}
// ---- profiling hooks ----------------------------------------------------------------------------------
static cudaEvent_t take_event(pdadmm_ctx *c) {
  cudaEvent_t e;
  if (!c->ev_pool.empty()) { e = c->ev_pool.back(); c->ev_pool.pop_back(); return e; }
  cudaEventCreate(&e);
  return e;
}
struct Launch {                    // brackets one kernel launch
  pdadmm_ctx *c; int cls; cudaStream_t st; double bytes, flops; cudaEvent_t e0 = nullptr;
  Launch(pdadmm_ctx *c_, int cls_, cudaStream_t st_, double bytes_, double flops_)
      : c(c_), cls(cls_), st(st_), bytes(bytes_), flops(flops_) {
    c->launches++;
    if (c->profiling) { e0 = take_event(c); cudaEventRecord(e0, st); }
  }
  ~Launch() {
    if (c->profiling) {
      cudaEvent_t e1 = take_event(c);
      cudaEventRecord(e1, st);
      c->prof.push_back({cls, e0, e1, bytes, flops});
    }
  }
};
static int prof_collect(pdadmm_ctx *c) {
  if (c->prof.empty()) return PDADMM_OK;
  PD_CUDA(cudaStreamSynchronize(c->scr.st));          // every lane has joined it
  for (auto &r : c->prof) {
    float ms = 0.f;
    cudaEventElapsedTime(&ms, r.e0, r.e1);
    c->prof_ms[r.cls] += ms; c->prof_n[r.cls]++; c->prof_bytes[r.cls] += r.bytes; c->prof_flops[r.cls] += r.flops;
    c->ev_pool.push_back(r.e0); c->ev_pool.push_back(r.e1);
  }
  c->prof.clear();
  return PDADMM_OK;
}

// ---- tensor maps -------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *, const cuuint64_t *,
                                  const cuuint64_t *, const cuuint32_t *, const cuuint32_t *, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
static EncodeTiledFn encode_tiled_fn() {
  static EncodeTiledFn fn = [] {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      p = nullptr;
    return (EncodeTiledFn)p;
  }();
  return fn;
}
// Operand tiles of the tensor-core products: 64 x 64 halves of a plane [outer][inner], 128-byte swizzle; elements outside the
// matrix read as zero.
static int get_tmap(pdadmm_ctx *c, const void *base, uint64_t inner, uint64_t outer, uint64_t ld, CUtensorMap *out) {
  auto key = std::make_tuple(base, inner, outer, ld);
  auto it = c->tmaps.find(key);
  if (it != c->tmaps.end()) { *out = it->second; return PDADMM_OK; }
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return fail(PDADMM_ECUDA, "cuTensorMapEncodeTiled is not available in this driver");
  cuuint64_t dims[2] = {inner, outer};
  cuuint64_t strides[1] = {ld * 2};
  cuuint32_t box[2] = {64u, 64u};
  cuuint32_t estr[2] = {1, 1};
  CUtensorMap m;
  const CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT16, 2, const_cast<void *>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(PDADMM_ECUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
  if (c->tmaps.size() > 4096) c->tmaps.clear();
  c->tmaps[key] = m;
  *out = m;
  return PDADMM_OK;
}

// Where the wide tiles of a product store: parts of 32 rows x 16 columns of a matrix [slice][rows][ld] (slices `stride` floats apart),
// 64-byte swizzle; what lies outside is clipped.
static int get_out_tmap(pdadmm_ctx *c, const float *base, uint64_t rows, uint64_t ld, uint64_t slices, uint64_t stride, CUtensorMap *out) {
  auto key = std::make_tuple((const void *)base, ~rows, ld, slices << 40 ^ stride);
  auto it = c->tmaps.find(key);
  if (it != c->tmaps.end()) { *out = it->second; return PDADMM_OK; }
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return fail(PDADMM_ECUDA, "cuTensorMapEncodeTiled is not available in this driver");
  cuuint64_t dims[3] = {ld, rows, slices};
  cuuint64_t strides[2] = {ld * 4, stride * 4};
  cuuint32_t box[3] = {(cuuint32_t)TC_WIDE_PART, 32u, 1u};
  cuuint32_t estr[3] = {1, 1, 1};
  CUtensorMap m;
  const CUresult r = fn(&m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<float *>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_64B, CU_TENSOR_MAP_L2_PROMOTION_NONE,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(PDADMM_ECUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
  if (c->tmaps.size() > 4096) c->tmaps.clear();
  c->tmaps[key] = m;
  *out = m;
  return PDADMM_OK;
}

// One layer's part of a product launch.
template <class Epi>
struct Prod {
  int M, N, K;
  Operand A, B;
  Epi epi;
  Scratch *s;                      // of the layer: room for planes that have to be made first
  double *slots = nullptr;         // one per tile and warp (null: no sum is wanted)
  int *done = nullptr;
  Step step{};
  int n_split = 1, k_chunk = 0;    // contraction slices, and their length
  size_t stride = 0;               // floats between the partial outputs of two slices
  bool wide = false;               // may run on wide tiles, and is to (see choose_wide)
};
// Products that this host thread has launched on the tensor cores: all, on wide tiles, with the last round's tiles cut
// (pdadmm_product_forms)
static thread_local int64_t product_forms[3] = {0, 0, 0};
template <int LAYOUT, class Epi, int ZERO, bool PAIR, bool WIDE>
static int launch_tc_form(pdadmm_ctx *c, cudaStream_t st, const TcGroup<Epi> &grp) {
  auto kern = gemm_tc_kernel<LAYOUT, Epi, ZERO, PAIR, WIDE>;
  // the attribute belongs to (kernel, device): one flag per device ordinal for this instantiation
  static bool configured[MAX_DEVICES] = {false};
  const int dev = c->device;
  if (dev < 0 || dev >= MAX_DEVICES || !configured[dev]) {
    // The kernel's warpgroups re-divide the registers the block is launched with; their shares were added up
    // against TC_REGS_LAUNCH per thread.  A build that launches with fewer would make an increase wait for ever:
    // refuse to launch it.
    cudaFuncAttributes attr;
    PD_CUDA(cudaFuncGetAttributes(&attr, kern));
    if (attr.numRegs != TC_REGS_LAUNCH)
      return fail(PDADMM_ECUDA, "tensor-core product kernel was built with %d registers per thread, %d expected",
                  attr.numRegs, TC_REGS_LAUNCH);
    PD_CUDA(cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, TC_SMEM_BYTES));
    if (dev >= 0 && dev < MAX_DEVICES) configured[dev] = true;
  }
  const int n_units = grp.unit_end[grp.n - 1];
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(PAIR ? 2 * std::min(n_units, c->n_sms / 2) : std::min(n_units, c->n_sms)));
  cfg.blockDim = dim3(TC_THREADS);
  cfg.dynamicSmemBytes = TC_SMEM_BYTES;
  cfg.stream = st;
  cudaLaunchAttribute a;
  a.id = cudaLaunchAttributeClusterDimension;
  a.val.clusterDim.x = 2; a.val.clusterDim.y = 1; a.val.clusterDim.z = 1;
  cfg.attrs = &a;
  cfg.numAttrs = PAIR ? 1 : 0;
  PD_CUDA(cudaLaunchKernelEx(&cfg, kern, grp));
  bool cut = false;
  for (int i = 0; i < grp.n; ++i) cut |= grp.l[i].tail_split > 1;
  product_forms[0] += 1;
  product_forms[1] += WIDE ? 1 : 0;
  product_forms[2] += cut ? 1 : 0;
  return PDADMM_OK;
}
// Whether products run on pairs of SMs: pairs halve the traffic of B, but a pair's tile has
// 256 rows.  So: where at least three quarters of the pairs get a tile, and padding M to 256 rows instead of 128 adds at most
// a tenth.  (20 000 x 500 x 500: 43.2 us in pairs, 45.5 us without; x 2000 x 2000: 399 against 457 us; 2000 x 100 x 100, 8
// pairs: 12.5 against 10.7 us.)
static bool worth_pairs(int n_sms, int64_t single, int64_t paired) { return paired * 10 <= single * 11 && (paired / 2) * 8 >= 3 * (int64_t)n_sms; }
template <class Epi>
static bool use_pairs(const pdadmm_ctx *c, const Prod<Epi> *v, int n) {
  int64_t single = 0, paired = 0;
  for (int i = 0; i < n; ++i) {
    const int64_t cols = ceil_div(v[i].N, TC_BN) * v[i].n_split;
    single += ceil_div(v[i].M, TC_BM) * cols;
    paired += 2 * ceil_div(v[i].M, 2 * TC_BM) * cols;
  }
  return worth_pairs(c->n_sms, single, paired);
}
// Whether some products [rows, columns, contraction of a slice, slices], worked on in one launch, run on wide tiles: the shorter
// estimate of the two.  The persistent grid takes the tiles in rounds; SM cycles per K block and at a tile's end, from traces of
// 20 000 x 500, 170 000 x 1000 and 90 000 x 2000: a block on its own 1560 and 2800, a pair 1080 and 2800, a pair with a wide
// tile 1500 and 8800 (its accumulate warps store the tile themselves); with two MMAs per product instead of three (integer
// operands) 1230, 830, 1130 and 6900 at the end.  A wide tile brings 64 KB per K block where two narrow ones bring 96.  By the
// estimate it wins from some six K blocks on, unless its columns are mostly padding or leave SMs idle; measured it wins from 16 on
// (170 000 x 1000 G p+: 1.04 -> 0.90 ms; 90 000 x 2000: 1.50 -> 1.30 ms; W-gradient of 20 000 x 500, 9 layers: 410 -> 330 us) and
// makes no difference at 8 (20 000 x 500, W g and G p+: 272 and 300 TFLOP/s either way), where the estimate says 7 %.  The norm-only product,
// which stores nothing, is estimated as one that stores.  The estimate has no cut of the last round's tiles along the contraction in it
// (launch_tc, single products), so where a form's last round is sparse it counts that round as a full one.
struct Shape { int64_t M, N, K, n_split; };
static bool choose_wide(int n_sms, const Shape *v, int n, bool ints, double *cost = nullptr) {
  double best[2];
  int64_t single = 0, paired = 0;
  for (int i = 0; i < n; ++i) {
    single += ceil_div(v[i].M, TC_BM) * ceil_div(v[i].N, TC_BN) * v[i].n_split;
    paired += 2 * ceil_div(v[i].M, 2 * TC_BM) * ceil_div(v[i].N, TC_BN) * v[i].n_split;
  }
  const bool pairs = worth_pairs(n_sms, single, paired);
  for (int wide = 0; wide < 2; ++wide) {
    const int rows = wide || pairs ? 2 * TC_BM : TC_BM, slots = wide || pairs ? n_sms / 2 : n_sms;
    const double per_block = wide ? (ints ? 1130 : 1500) : pairs ? (ints ? 830 : 1080) : ints ? 1230 : 1560;
    const double end = wide ? (ints ? 6900 : 8800) : 2800;
    double work = 0;
    int64_t units = 0;
    for (int i = 0; i < n; ++i) {
      const int64_t u = ceil_div(v[i].M, rows) * ceil_div(v[i].N, wide ? TC_WIDE : TC_BN) * v[i].n_split;
      units += u;
      work += (double)u * (per_block * ceil_div(v[i].K, TC_BK) + end);
    }
    best[wide] = work / units * ceil_div(units, slots);
  }
  if (cost) *cost = std::min(best[0], best[1]);
  return best[1] < best[0];
}
// op(A) is M x K, op(B) is N x K; A_MN: A is stored [K][M], B_MN: B is stored [K][N].  At most TC_MAX_GROUP products.
template <int LAYOUT, class Epi, int ZERO = 0>
static int launch_tc(pdadmm_ctx *c, cudaStream_t st, const Prod<Epi> *v, int n) {
  constexpr bool A_MN = (LAYOUT & TC_A_MN) != 0, B_MN = (LAYOUT & TC_B_MN) != 0;
  static_assert(sizeof(TcGroup<Epi>) <= 32000, "kernel parameters");
  TcGroup<Epi> grp;
  grp.n = n;
  grp.error = c->d_flag + 1;
  constexpr bool CAN_WIDE = Epi::kDirect;
  bool wide = CAN_WIDE;
  for (int i = 0; i < n; ++i) wide = wide && v[i].wide;
  const bool pair = wide || use_pairs(c, v, n);
  const int tile_n = wide ? TC_WIDE : TC_BN;
  int units = 0;
  for (int i = 0; i < n; ++i) {
    const Prod<Epi> &p = v[i];
    TcLayer<Epi> &y = grp.l[i];
    const uint64_t M = (uint64_t)p.M, N = (uint64_t)p.N, K = (uint64_t)p.K;
    PD_TRY(get_tmap(c, p.A.hi, A_MN ? M : K, A_MN ? K : M, (uint64_t)p.A.ld, &y.a));
    if (p.A.lo && p.A.lo != p.A.hi) PD_TRY(get_tmap(c, p.A.lo, A_MN ? M : K, A_MN ? K : M, (uint64_t)p.A.ld, &y.alo));
    else y.alo = y.a;
    PD_TRY(get_tmap(c, p.B.hi, B_MN ? N : K, B_MN ? K : N, (uint64_t)p.B.ld, &y.b));
    if (p.B.lo && p.B.lo != p.B.hi) PD_TRY(get_tmap(c, p.B.lo, B_MN ? N : K, B_MN ? K : N, (uint64_t)p.B.ld, &y.blo));
    else y.blo = y.b;
    if (wide && epi_stores<Epi>::value)
      PD_TRY(get_out_tmap(c, p.epi.C, M, (uint64_t)p.epi.ldc, (uint64_t)p.n_split, p.n_split > 1 ? p.stride : M * p.epi.ldc, &y.c));
    else
      y.c = y.a;
    y.M = p.M; y.N = p.N; y.K = p.K;
    y.k_chunk = p.n_split > 1 ? p.k_chunk : round_up(p.K, TC_BK);
    y.n_split = p.n_split;
    y.c_split_stride = p.stride;
    y.oa = TcOperand{p.A.exp, p.A.check, p.A.x, p.A.ld};
    y.ob = TcOperand{p.B.exp, p.B.check, p.B.x, p.B.ld};
    y.mul = p.A.int_mul > 0.f ? p.A.int_mul : (p.B.int_mul > 0.f ? p.B.int_mul : 1.f);
    y.epi = p.epi;
    y.slots = p.slots; y.done = p.done; y.step = p.step;
    y.tail_begin = 0; y.tail_split = 0; y.tail_ws = nullptr; y.tail_count = nullptr;
    const int tiles_n = (int)ceil_div(p.N, tile_n), tiles_mn = (int)ceil_div(p.M, pair ? 2 * TC_BM : TC_BM) * tiles_n, n_tiles = tiles_mn * p.n_split;
    y.tiles_n = TcDiv::of(tiles_n, tiles_mn);
    y.tiles_mn = TcDiv::of(tiles_mn, n_tiles);
    units += n_tiles;
    // The persistent grid works through the tiles in rounds; a last round that fills only part of the
    // SMs costs as much as a full one, so its tiles are cut along the contraction into as many slices as fit (at least 8 K
    // blocks per slice: parking and merging the slices of a tile costs about as much as four K blocks).  A product that only
    // wants its squared norm keeps whole tiles: it stores nothing that could be merged.
    const int slots = pair ? c->n_sms / 2 : c->n_sms, tail = n_tiles % slots;
    if (epi_stores<Epi>::value && c->tail_split && n == 1 && p.n_split == 1 && tail > 0 && p.s != nullptr && p.s->tail_ws != nullptr) {
      const int split = std::min(std::min(slots / tail, (int)ceil_div(p.K, TC_BK) / 8), 8);
      if (split > 1) {
        y.tail_begin = n_tiles - tail; y.tail_split = split;
        y.tail_ws = p.s->tail_ws; y.tail_count = p.s->tail_count;
        units = y.tail_begin + tail * split;
      }
    }
    grp.unit_end[i] = units;
  }
  if constexpr (CAN_WIDE) {
    if (wide) return launch_tc_form<LAYOUT, Epi, ZERO, true, true>(c, st, grp);
  }
  if (pair) return launch_tc_form<LAYOUT, Epi, ZERO, true, false>(c, st, grp);
  return launch_tc_form<LAYOUT, Epi, ZERO, false, false>(c, st, grp);
}

// ---- largest magnitudes of product operands ------------------------------------------------------------------
// Each tensor-core product scales its operands by powers of two taken from their largest magnitudes.  The words
// that receive them come from a pool that is cleared in stream order: at the start of every iteration (so that a
// captured iteration always uses the same words) and whenever it runs out.
constexpr int AMAX_POOL = 4096;
static int amax_reset(pdadmm_ctx *c, cudaStream_t st) {
  PD_CUDA(cudaMemsetAsync(c->cur->amax_pool, 0, AMAX_POOL * sizeof(uint32_t), st));
  c->cur->amax_next = 0;
  return PDADMM_OK;
}
// room for n more words that must stay valid together
static int amax_reserve(pdadmm_ctx *c, cudaStream_t st, int n) {
  if (c->cur->amax_next + n > AMAX_POOL) PD_TRY(amax_reset(c, st));
  return PDADMM_OK;
}
static uint32_t *amax_take(pdadmm_ctx *c) { return c->cur->amax_pool + c->cur->amax_next++; }
// max|x| of a matrix stored as n4 float4 values -> a fresh word
static uint32_t *amax_of(pdadmm_ctx *c, cudaStream_t st, const float *x, size_t n4) {
  uint32_t *w = amax_take(c);
  Launch l(c, KC_AMAX, st, 16.0 * (double)n4, 0);
  absmax_kernel<<<ew_grid(n4), EW_THREADS, 0, st>>>(x, n4, w);
  return w;
}

// planes of x [rows][ld] from the largest magnitude in *amax (lo_too: both planes)
static void split_rows(pdadmm_ctx *c, cudaStream_t st, const float *x, size_t rows, int cols, int ld, const uint32_t *amax,
                       const Planes &pl, bool lo_too = true) {
  const size_t n8 = rows * ld / 8;
  Launch l(c, KC_PLANES, st, (lo_too ? 8.0 : 6.0) * rows * cols, 0);
  rows_planes_kernel<<<dim3(ew_grid(n8)), 256, 0, st>>>(x, n8, amax, pl.exp, pl.hi, lo_too ? pl.lo : nullptr);
}
// Refused planes of a large matrix are made again by a kernel of their own instead of by the product (check_planes_kernel): always
// from 2^20 elements on; below, a launch that finds nothing to do costs more than it saves (2000 x 500, 6 layers: 237 us per
// iteration with it, 229 without), except in a context's first iterations, where maxima that were zero become something and
// no prediction holds, if many tiles of the product read each element and would split it again (CHECK_PLANES_USES reads;
// 500 x 2000, 4 layers: 0.86 ms for such an iteration, 0.37 so).
constexpr size_t CHECK_PLANES_FROM = size_t(1) << 20, CHECK_PLANES_USES = size_t(1) << 21;
static void check_planes(pdadmm_ctx *c, cudaStream_t st, size_t rows, const std::vector<Operand *> &ops) {
  Group<PlaneCheck> g;
  int n = 0;
  uint32_t n8_max = 0;
  for (Operand *o : ops) {
    const size_t e = rows * o->ld;
    if (!c->use_tc || o->hi == nullptr || o->check == nullptr || o->x == nullptr || (e < CHECK_PLANES_FROM && !(c->cold > 0 && e * o->uses >= CHECK_PLANES_USES))) continue;
    g.l[n++] = PlaneCheck{o->x, (uint32_t)(e / 8), o->check, o->exp, const_cast<__half *>(o->hi),
                          o->lo == o->hi ? nullptr : const_cast<__half *>(o->lo)};
    n8_max = std::max(n8_max, (uint32_t)(e / 8));
    o->x = nullptr;
  }
  if (n == 0) return;
  Launch l(c, KC_PLANES, st, 0, 0);
  check_planes_kernel<<<dim3((unsigned)std::max(1, ew_grid(n8_max) / n), (unsigned)n), 256, 0, st>>>(g);
}
static int alloc_planes(pdadmm_ctx *c, size_t n, Planes *pl, bool zero = true) {
  PD_TRY(dev_alloc(c, &pl->hi, n, zero));
  PD_TRY(dev_alloc(c, &pl->lo, n, zero));
  return dev_alloc(c, &pl->exp, 1);
}
// planes of W_l and its largest magnitude, after W was set
static int refresh_W_planes(pdadmm_ctx *c, Layer &ly, cudaStream_t st) {
  if (!c->use_tc) return PDADMM_OK;
  PD_CUDA(cudaMemsetAsync(ly.amax_W, 0, sizeof(uint32_t), st));
  const size_t n4 = (size_t)ly.n_out * ly.ld_in / 4;
  {
    Launch l(c, KC_AMAX, st, 16.0 * (double)n4, 0);
    absmax_kernel<<<ew_grid(n4), EW_THREADS, 0, st>>>(ly.W, n4, ly.amax_W);
  }
  split_rows(c, st, ly.W, (size_t)ly.n_out, ly.n_in, ly.ld_in, ly.amax_W, ly.Wp);
  return PDADMM_OK;
}

// ---- dense products --------------------------------------------------------------------------------------
// C[M][N] = A[M][K] * op(B) for several layers, fused epilogue.  B_MN = false: B is [N][K]; true: B is [K][N].  An operand A without
// planes is split into its layer's pl1 first (8 bytes per element; splitting inside the product, once per column tile, ran
// the MMAs at 0.6 of their speed).  bytes: what the epilogues move beside the operands and the output.
template <bool B_MN, class Epi>
static int gemm_nodes(pdadmm_ctx *c, int cls, cudaStream_t st, std::vector<Prod<Epi>> v, double extra_bytes) {
  if (v.empty()) return PDADMM_OK;
  double bytes = extra_bytes, flops = 0;
  for (const Prod<Epi> &p : v) {
    bytes += 4.0 * ((double)p.M * p.K + (double)p.N * p.K + (double)p.M * p.N);
    flops += 2.0 * p.M * p.N * p.K;
  }
  if (!c->use_tc) {
    for (const Prod<Epi> &p : v) {
      dim3 grid((unsigned)ceil_div(p.N, SG_BN), (unsigned)ceil_div(p.M, SG_BM));
      {
        Launch l(c, cls, st, bytes / v.size(), 2.0 * p.M * p.N * p.K);
        gemm_nt_kernel<B_MN, Epi><<<grid, SG_THREADS, 0, st>>>(p.M, p.N, p.K, p.A.x, p.A.ld, p.B.x, p.B.ld, p.epi, p.slots);
      }
      if (p.slots == nullptr) continue;
      Launch l(c, KC_SMALL, st, 8.0 * grid.x * grid.y, 0);
      finish_sum_kernel<<<1, FIN_THREADS, 0, st>>>(p.slots, (int)(grid.x * grid.y), p.step);
    }
    return PDADMM_OK;
  }
  for (Prod<Epi> &p : v) {
    if (p.A.hi != nullptr) continue;
    Scratch &sc = *p.s;
    if ((size_t)p.M * p.A.ld > sc.pl_cap || p.A.ld % 8) return fail(PDADMM_EINVAL, "operand does not fit the lane's planes");
    if (p.A.amax == nullptr) {
      PD_TRY(amax_reserve(c, st, 1));
      p.A.amax = amax_of(c, st, p.A.x, (size_t)p.M * p.A.ld / 4);
    }
    const Planes pl{sc.pl1.hi, sc.pl1.lo, sc.a_exp};
    split_rows(c, st, p.A.x, (size_t)p.M, p.K, p.A.ld, p.A.amax, pl, !epi_coarse<Epi>::value);
    p.A.hi = pl.hi; p.A.lo = pl.lo; p.A.exp = pl.exp; p.A.check = nullptr;
  }
  constexpr int LAYOUT = B_MN ? TC_B_MN : TC_NT;
  constexpr bool INT_FORM = std::is_same<Epi, EpiStoreSumsq>::value || std::is_same<Epi, EpiAddSumsq>::value;
  // operands of integers and others take different kernels
  const auto mid = std::stable_partition(v.begin(), v.end(), [](const Prod<Epi> &p) { return p.A.int_mul <= 0.f; });
  const int n = (int)(mid - v.begin()), n_int = (int)(v.end() - mid);
  if (n > 0) {
    Launch l(c, cls, st, bytes * n / (n + n_int), flops * n / (n + n_int));
    PD_TRY((launch_tc<LAYOUT, Epi>(c, st, v.data(), n)));
  }
  if (n_int > 0) {
    if constexpr (INT_FORM) {
      Launch l(c, cls, st, bytes * n_int / (n + n_int), flops * n_int / (n + n_int));
      PD_TRY((launch_tc<LAYOUT, Epi, 1>(c, st, v.data() + n, n_int)));
    } else {
      return fail(PDADMM_EINVAL, "no integer-operand form of this product is built");
    }
  }
  return PDADMM_OK;
}

// C parts [n_split][M][ldc] = A^T B over node slices, A = [K nodes][M], B = [K nodes][N], both as planes, for several layers
static int gemm_over_nodes(pdadmm_ctx *c, int cls, cudaStream_t st, std::vector<Prod<EpiStore>> v) {
  const auto mid = std::stable_partition(v.begin(), v.end(), [](const Prod<EpiStore> &p) { return p.B.int_mul <= 0.f; });
  const int n = (int)(mid - v.begin()), n_int = (int)(v.end() - mid);
  auto count = [&](int i0, int i1, double &bytes, double &flops) {
    bytes = flops = 0;
    for (int i = i0; i < i1; ++i) {
      bytes += 4.0 * ((double)v[i].K * v[i].N + (double)v[i].K * v[i].M);
      flops += 2.0 * v[i].K * v[i].N * v[i].M;
    }
  };
  double bytes, flops;
  if (n > 0) {
    count(0, n, bytes, flops);
    Launch k(c, cls, st, bytes, flops);
    PD_TRY((launch_tc<TC_A_MN | TC_B_MN, EpiStore>(c, st, v.data(), n)));
  }
  if (n_int > 0) {
    count(n, n + n_int, bytes, flops);
    Launch k(c, cls, st, bytes, flops);
    PD_TRY((launch_tc<TC_A_MN | TC_B_MN, EpiStore, 2>(c, st, v.data() + n, n_int)));
  }
  return PDADMM_OK;
}

// ---- pieces of one iteration -------------------------------------------------------------------------------

static Operand operand_W(const Layer &ly) { return plane_operand(ly.W, ly.ld_in, ly.Wp, ly.amax_W); }
// p_1 = X, which never changes (its planes are kept on the tensor-core path)
static Operand operand_X(const Layer &ly) { return plane_operand(ly.p, ly.ld_in, ly.xp); }
// r_l as the z-step left it
static Operand operand_r(const Layer &ly) {
  Operand o = plane_operand(ly.r, ly.ld_out, ly.rp, ly.amax_r);
  o.amax = ly.amax_r;
  return o;
}

// The layers of a batch are consecutive, at most MAX_GROUP, and share a stream; layer l uses scratch l mod the number of them.
typedef std::vector<int> Batch;
static Scratch &lane(pdadmm_ctx *c, int i) { return i == 0 ? c->scr : *c->more_lanes[i - 1]; }
static Scratch &scratch_of(pdadmm_ctx *c, int l) { return lane(c, l % c->n_active); }
static PlaneOut plane_out(pdadmm_ctx *c, const Planes &p) {
  return c->use_tc ? PlaneOut{p.hi, p.lo, p.exp} : PlaneOut{nullptr, nullptr, nullptr};
}
static Step make_step(pdadmm_ctx *c, Layer &ly, int kind) {
  Step t;
  t.kind = kind;
  t.sc = ly.sc; t.rho = c->rho; t.nu = c->nu; t.nonfinite = c->d_flag + 2;
  t.apply = kind != STEP_G2 && c->reduce == nullptr;     // a sharded context adds the sums over the shards first
  if (c->use_tc) { t.amax_p = ly.amax_p; t.amax_r = ly.amax_r; t.amax_W = ly.amax_W; }
  return t;
}
// The sums at `sums` are those of this shard: add them over the shards, then the step.
static int shard_step(pdadmm_ctx *c, cudaStream_t st, double *sums, size_t n, const Step &t) {
  if (c->reduce == nullptr) return PDADMM_OK;
  PD_TRY(shard_sum(c, st, sums, n, 1));
  run_step_kernel<<<1, 1, 0, st>>>(t);
  return PDADMM_OK;
}

// r_l = P_l W_l^T + b_l - z_l from scratch (only when the cached residual is not valid).
static int refresh_residual(pdadmm_ctx *c, Layer &ly, cudaStream_t st) {
  PD_CUDA(cudaMemsetAsync(ly.amax_r, 0, sizeof(uint32_t), st));
  EpiLinearResidual epi{ly.r, ly.ld_out, ly.b, ly.z, ly.amax_r};
  Operand P{ly.p, ly.ld_in, ly.amax_p};
  if (c->use_tc && ly.xp.hi != nullptr) P = operand_X(ly);
  PD_TRY((gemm_nodes<false, EpiLinearResidual>(c, KC_GEMM_RESID, st, {{(int)c->N, ly.n_out, ly.n_in, P, operand_W(ly), epi, &c->scr}},
                                               4.0 * c->N * ly.n_out)));
  if (!c->use_tc) {       // the CUDA-core product does not track the maximum of what it stores
    Launch l(c, KC_AMAX, st, 4.0 * c->N * ly.ld_out, 0);
    absmax_kernel<<<ew_grid((size_t)c->N * ly.ld_out / 4), EW_THREADS, 0, st>>>(ly.r, (size_t)c->N * ly.ld_out / 4, ly.amax_r);
  } else if (ly.rp.hi != nullptr) {
    split_rows(c, st, ly.r, (size_t)c->N, ly.n_out, ly.ld_out, ly.amax_r, ly.rp);
  }
  return PDADMM_OK;
}

// Layers 2..L (0-based l >= 1): g = nu r W + u_{l-1} + rho (p - q_{l-1}) -> s1, ||g||^2 ; W g -> s2, ||W g||^2 ; tau.
static int p_gradient_and_tau(pdadmm_ctx *c, cudaStream_t st, const Batch &batch) {
  const int N = (int)c->N;
  const bool norm_only = c->levels && c->use_tc;     // the quantised update only needs ||W g||^2 (for the first tau); its
                                                     // residual update uses W d
  std::vector<Operand> R, G;
  std::vector<Prod<EpiGradT>> grad;
  double bytes = 0;
  for (int l : batch) {
    Layer &ly = c->layers[l];
    Scratch &s = scratch_of(c, l);
    R.push_back(operand_r(ly));
    R.back().uses = (int)ceil_div(ly.n_in, TC_BN);
    // The epilogue that writes g writes its planes too (the hi plane alone for the norm-only product), scaled by an exponent
    // predicted from the previous iteration's max|g|: the true one is known only when the product has finished.
    EpiGradT epi{s.s1, ly.ld_in, ly.t, c->nu, c->use_tc ? ly.w_g : nullptr};
    if (c->use_tc) {
      epi.H = s.pl0.hi; epi.L = norm_only ? nullptr : s.pl0.lo; epi.h_exp = ly.g_exp;
      G.push_back(plane_operand(s.s1, ly.ld_in, Planes{s.pl0.hi, norm_only ? s.pl0.hi : s.pl0.lo, ly.g_exp}, ly.w_g));
    } else {
      G.push_back(Operand{s.s1, ly.ld_in, nullptr});
    }
    Prod<EpiGradT> p{N, ly.n_in, ly.n_out, R.back(), operand_W(ly), epi, &s, s.slots, ly.done + 2};
    p.step = make_step(c, ly, STEP_G2);
    grad.push_back(p);
    bytes += (c->use_tc ? (norm_only ? 6.0 : 8.0) : 4.0) * N * ly.n_in;
  }
  for (size_t i = 0; i < batch.size(); ++i) G[i].uses = (int)ceil_div(c->layers[batch[i]].n_out, TC_BN);
  auto check = [&](std::vector<Operand> &ops) {
    std::vector<Operand *> v;
    for (Operand &o : ops) v.push_back(&o);
    check_planes(c, st, (size_t)N, v);
  };
  check(R);
  for (size_t i = 0; i < batch.size(); ++i) grad[i].A = R[i];
  PD_TRY((gemm_nodes<true, EpiGradT>(c, KC_GEMM_GRADP, st, grad, bytes)));
  check(G);
  auto wg = [&](auto make_epi) -> int {
    std::vector<Prod<decltype(make_epi(0))>> v;
    for (size_t i = 0; i < batch.size(); ++i) {
      Layer &ly = c->layers[batch[i]];
      Scratch &s = scratch_of(c, batch[i]);
      Prod<decltype(make_epi(0))> p{N, ly.n_out, ly.n_in, G[i], operand_W(ly), make_epi(batch[i]), &s, s.slots + s.n_slots / 2, ly.done + 2};
      p.wide = ly.wide_wg;
      Step t = make_step(c, ly, STEP_TAU);
      if (c->use_tc) {
        t.w_in = ly.w_g; t.w_out = norm_only ? nullptr : ly.w_wg;
        t.exp_p = norm_only ? nullptr : s.pl1.exp; t.exp_r = s.pl0.exp; t.exp_g = ly.g_exp;
      }
      p.step = t;
      v.push_back(p);
    }
    PD_TRY((gemm_nodes<false>(c, KC_GEMM_WG, st, v, 0)));
    // ||g||^2 and ||W g||^2 are sums over nodes
    for (size_t i = 0; i < batch.size(); ++i) PD_TRY(shard_step(c, st, &c->layers[batch[i]].sc->sum_g2, 2, v[i].step));
    return PDADMM_OK;
  };
  if (norm_only) return wg([&](int l) { return EpiNormOnly{scratch_of(c, l).s2, c->layers[l].ld_out}; });
  return wg([&](int l) { return EpiStoreSumsq{scratch_of(c, l).s2, c->layers[l].ld_out, c->use_tc ? c->layers[l].w_wg : nullptr}; });
}

// Blocks of a kernel that sums columns, for each of the layers of its launch; at least four rows for every row subgroup of a block
// (2000 x 100, 9 layers: p-step 17.0 us with two, 14.9 so), fewer where that left SMs without a second block (few layers).
// The z-update gets two full rounds of what the SMs hold at 64 registers a thread, four for a layer on its own: 10 000 x 256, 5 layers 122 us,
// with 3.3 rounds 129; 90 000 x 2000 1.28 ms a layer, with two 1.33.  The p-step and the trial step get 16 per SM, the trial of a layer on its
// own 5 (one round: 170 000 x 1000 1.46 ms, 1.61 with 16).
static int sum_blocks(const pdadmm_ctx *c, int ld, int layers, bool z) {
  const RowShare share = row_share(ld);
  const int per_sm = z ? (layers > 1 ? 2 : 4) * (1024 / share.threads) : c->levels && layers == 1 ? 5 : 16;
  const int64_t blocks = std::max(1, per_sm * c->n_sms / std::max(layers, 1));
  int rows = 4;
  while (rows > 1 && layers * ceil_div(c->N, rows * share.n_sub) < 2 * c->n_sms) rows /= 2;
  return (int)std::max<int64_t>(1, std::min<int64_t>(blocks, ceil_div(c->N, rows * share.n_sub)));
}
static RowBlocks row_blocks(const pdadmm_ctx *c, int ld, int blocks, double *slots) {
  const RowShare s = row_share(ld);
  return RowBlocks{(int)c->N, ld, blocks, slots, s.cols_per_pass, s.n_sub};
}
static RowBlocks p_rows(const pdadmm_ctx *c, const Layer &ly, const Scratch &s) { return row_blocks(c, ly.ld_in, ly.p_blocks, s.p_slots); }
static RowBlocks r_rows(const pdadmm_ctx *c, const Layer &ly) { return row_blocks(c, ly.ld_out, ly.r_blocks, ly.r_slots); }

// pdADMM-G: p <- p - g/tau, r <- r - (W g)/tau, and the planes of both.
static void p_step_plain(pdadmm_ctx *c, cudaStream_t st, const Batch &batch) {
  Group<PStep> g;
  int n = 0, blocks = 0, threads = 0;
  double bytes = 0;
  for (int l : batch) {
    Layer &ly = c->layers[l];
    Scratch &s = scratch_of(c, l);
    const size_t n4r = (size_t)c->N * ly.ld_out / 4;
    // a thread has eight loads in flight if it gets four groups (2000 x 100: 9 layers 18.8 us with a group per thread, 14.7 so;
    // 7013 x 333, 6 layers: 80.9 and 71.5)
    const int nb = ew_grid((size_t)ceil_div((int64_t)n4r, 4));
    g.l[n] = PStep{ly.p, s.s1, p_rows(c, ly, s), ly.r, s.s2, (uint32_t)n4r, &ly.sc->inv_tau, plane_out(c, s.pl1),
                   plane_out(c, s.pl0), c->use_tc ? ly.amax_p : nullptr, c->use_tc ? ly.amax_r : nullptr, nb};
    blocks = std::max(blocks, g.l[n].p_rows.n_blocks + nb);
    threads = std::max(threads, row_share(ly.ld_in).threads);
    ++n;
    bytes += (c->use_tc ? 16.0 : 12.0) * c->N * (ly.n_in + ly.n_out);
  }
  Launch k(c, KC_AXPY, st, bytes, 0);
  pstep_kernel<<<dim3((unsigned)blocks, (unsigned)n), threads, 0, st>>>(g);
}

// pdADMM-G-Q: project p - g/tau on the level set, doubling tau until the stop condition holds.  Each trial ends
// with the accept flags on the host, which decides whether another trial is needed (the only host round
// trips of an iteration).
// One trial of some layers: trial p, d = trial p - p and its codes, W d with its squared norm, the accept test, the flag.
static int q_trial(pdadmm_ctx *c, cudaStream_t st, const Batch &batch) {
  const int N = (int)c->N;
  {
    Group<QuantTrial> g;
    int n = 0, blocks = 0, threads = 0;
    double bytes = 0;
    for (int l : batch) {
      Layer &ly = c->layers[l];
      Scratch &s = scratch_of(c, l);
      const RowBlocks rows = p_rows(c, ly, s);
      // with integer operands p+ and d exist as codes and planes of integers alone
      g.l[n++] = QuantTrial{s.s1, ly.sc, ly.scale, ly.lo, c->int_operands ? nullptr : s.p_new, c->int_operands ? nullptr : s.d, ly.codes,
                            s.codes_new, s.pn_plane, s.d_plane, rows, c->use_tc && !c->int_operands ? ly.amax_p : nullptr,
                            ly.w_d, s.slots, ly.done};
      blocks = std::max(blocks, rows.n_blocks);
      threads = std::max(threads, row_share(ly.ld_in).threads);
      bytes += (c->int_operands ? 8.0 + 2.0 * c->code_bytes : 12.0 + 2.0 * c->code_bytes) * N * ly.n_in;
    }
    Launch k(c, KC_QUANT, st, bytes, 0);
    const dim3 grid((unsigned)blocks, (unsigned)n);
    const bool wide = c->code_bytes == 2;
    if (c->int_operands && wide) quant_trial_kernel<true, true><<<grid, threads, 0, st>>>(g, c->levels, c->neg_levels);
    else if (c->int_operands) quant_trial_kernel<true, false><<<grid, threads, 0, st>>>(g, c->levels, c->neg_levels);
    else if (wide) quant_trial_kernel<false, true><<<grid, threads, 0, st>>>(g, c->levels, c->neg_levels);
    else quant_trial_kernel<false, false><<<grid, threads, 0, st>>>(g, c->levels, c->neg_levels);
  }
  // the trial's residual r + W d is written beside r (the two trade places when the trial is taken), with ||W d||^2;
  // max|r| takes the trial's values too, which keeps it an upper bound whether or not the trial is taken
  std::vector<Prod<EpiAddSumsq>> v;
  double bytes = 0;
  for (int l : batch) {
    Layer &ly = c->layers[l];
    Scratch &s = scratch_of(c, l);
    EpiAddSumsq epi{s.s2, ly.ld_out, ly.r, c->use_tc ? ly.amax_r : nullptr};
    if (c->use_tc) { epi.H = s.pl0.hi; epi.L = s.pl0.lo; epi.h_exp = s.pl0.exp; }      // planes of the trial's r for the W-gradient
    const Operand D = c->int_operands ? int_operand(s.d_plane, ly.ld_in, ly.scale)      // d = (new code - old code) s
                                      : Operand{s.d, ly.ld_in, c->use_tc ? ly.w_d : nullptr};
    Prod<EpiAddSumsq> p{N, ly.n_out, ly.n_in, D, operand_W(ly), epi, &s, s.slots + s.n_slots / 2, ly.done + 2};
    p.step = make_step(c, ly, STEP_TRIAL);
    p.step.w_in = c->use_tc && !c->int_operands ? ly.w_d : nullptr;
    p.step.host_flag = s.h_flag;
    *s.h_flag = 0;
    v.push_back(p);
    bytes += (c->use_tc ? 8.0 : 4.0) * N * ly.n_out;
  }
  PD_TRY((gemm_nodes<false>(c, KC_GEMM_WG, st, v, bytes)));
  for (size_t i = 0; i < batch.size(); ++i) PD_TRY(shard_step(c, st, &c->layers[batch[i]].sc->sum_d2, 2, v[i].step));
  PD_CUDA(cudaEventRecord(scratch_of(c, batch[0]).ev_flag, st));
  return PDADMM_OK;
}
// After the first trial of a batch was queued: wait for the flags, run further trials of the layers that say no, then take the
// trials: p, codes <- trial, r <- r + W d.
static int q_finish(pdadmm_ctx *c, cudaStream_t st, const Batch &batch, bool *hit_cap) {
  const int max_trials = 30;
  Batch open = batch;
  for (int trial = 0;; ++trial) {
    PD_CUDA(cudaEventSynchronize(scratch_of(c, open[0]).ev_flag));
    Batch refused;
    for (int l : open)
      if (!*scratch_of(c, l).h_flag) refused.push_back(l);
    if (refused.empty()) break;
    if (trial + 1 >= max_trials) { *hit_cap = true; break; }
    PD_TRY(q_trial(c, st, refused));
    open = refused;
  }
  for (int l : batch) {
    Layer &ly = c->layers[l];
    Scratch &s = scratch_of(c, l);
    if (!c->int_operands) std::swap(ly.p, s.p_new);
    std::swap(ly.codes, s.codes_new);
    std::swap(ly.p_plane, s.pn_plane);
    std::swap(ly.r, s.s2);                // r <- r + W d, written by the trial's product
  }
  if (c->int_operands) c->p_stale = true;
  return PDADMM_OK;
}

// Refused planes of grad_W are made again by the kernel that sums its slices where that is the quicker way: one block takes
// 0.12 us per 1000 elements, the product G p+ about 2.5 us per round of its tiles and K block; at least twice the time, and more than one round (the test costs
// the kernel's end half a microsecond, which 2000 x 100 does not get back).
static bool remade_with_sum(const pdadmm_ctx *c, const Layer &ly) {
  const size_t e = (size_t)ly.n_out * ly.ld_in;
  const int64_t rounds = ceil_div(ceil_div(c->N, TC_BM) * ceil_div(ly.n_out, TC_BN), c->n_sms);
  return c->use_tc && c->reduce == nullptr && e < CHECK_PLANES_FROM && rounds > 1 && (size_t)(rounds * ceil_div(ly.n_in, TC_BK)) * 10000 >= e;
}

// G = nu r^T p+ (contraction over nodes), theta, W <- W - G/theta, r <- r - (G p+)/theta,
// b <- b - mean_j r, shift = mean_j r.
static int w_and_b_step(pdadmm_ctx *c, cudaStream_t st, const Batch &batch) {
  const int N = (int)c->N;
  const bool fused = c->q_implied;                 // the z-update applies G p+
  // p+ (layer 1: X, which never changes; pdADMM-G: planes from the p-step; pdADMM-G-Q: p+ = code * s)
  std::vector<Operand> P, R;
  for (int l : batch) {
    Layer &ly = c->layers[l];
    Scratch &s = scratch_of(c, l);
    if (!c->use_tc) {
      P.push_back(Operand{ly.p, ly.ld_in, nullptr});
      R.push_back(Operand{ly.r, ly.ld_out, nullptr});
      continue;
    }
    P.push_back(l == 0 ? operand_X(ly) : c->int_operands ? int_operand(ly.p_plane, ly.ld_in, ly.scale)
                                                          : plane_operand(ly.p, ly.ld_in, s.pl1, ly.amax_p));
    R.push_back(l == 0 ? operand_r(ly) : plane_operand(ly.r, ly.ld_out, s.pl0, ly.amax_r));
    R.back().uses = (int)ceil_div(ly.n_in, TC_BN);
  }
  if (!c->use_tc) {
    for (int l : batch) {
      Layer &ly = c->layers[l];
      Scratch &s = scratch_of(c, l);
      dim3 grid((unsigned)ceil_div(ly.n_in, SG_BN), (unsigned)ceil_div(ly.n_out, SG_BM), (unsigned)ly.n_split);
      Launch k(c, KC_GEMM_GRADW, st, 4.0 * ((double)N * ly.n_in + (double)N * ly.n_out), 2.0 * N * ly.n_in * ly.n_out);
      gemm_tn_kernel<<<grid, SG_THREADS, 0, st>>>(ly.n_out, ly.n_in, N, ly.k_chunk, ly.r, ly.ld_out, ly.p, ly.ld_in, s.part, ly.ld_in);
    }
  } else {
    // both operands are node-major; the product contracts over the rows of their planes as they are
    std::vector<Operand *> to_check;
    std::vector<Prod<EpiStore>> v;
    for (size_t i = 0; i < batch.size(); ++i) {
      const int l = batch[i];
      Layer &ly = c->layers[l];
      Scratch &s = scratch_of(c, l);
      if (l == 0 || c->levels) to_check.push_back(&R[i]);       // (the p-step's planes are scaled by a bound)
      if (R[i].hi == nullptr) {                                 // no room was left for the planes of r
        const Planes pl{s.pl0.hi, s.pl0.lo, s.a_exp};
        split_rows(c, st, ly.r, (size_t)N, ly.n_out, ly.ld_out, ly.amax_r, pl);
        R[i] = plane_operand(ly.r, ly.ld_out, pl);
      }
      if (l > 0 && c->levels && !c->int_operands)               // p+ on a level set without integer planes
        split_rows(c, st, ly.p, (size_t)N, ly.n_in, ly.ld_in, ly.amax_p, s.pl1);
    }
    check_planes(c, st, (size_t)N, to_check);
    for (size_t i = 0; i < batch.size(); ++i) {
      Layer &ly = c->layers[batch[i]];
      Scratch &s = scratch_of(c, batch[i]);
      Prod<EpiStore> p{ly.n_out, ly.n_in, N, R[i], P[i], EpiStore{s.part, ly.ld_in}, &s};
      p.n_split = ly.n_split; p.k_chunk = ly.k_chunk; p.stride = (size_t)ly.n_out * ly.ld_in; p.wide = ly.wide_W;
      v.push_back(p);
    }
    PD_TRY(gemm_over_nodes(c, KC_GEMM_GRADW, st, v));
  }
  {
    Group<GradWSum> g;
    int n = 0, blocks = 0;
    double bytes = 0;
    for (int l : batch) {
      Layer &ly = c->layers[l];
      Scratch &s = scratch_of(c, l);
      const size_t n4 = (size_t)ly.n_out * ly.ld_in / 4;
      const int nb = ew_grid(n4);
      // the planes of G are scaled by a prediction, which the product G p+ checks; the parts of a sharded sum come first
      g.l[n++] = GradWSum{s.part, ly.n_split, (uint32_t)n4, ly.gradW, c->use_tc ? ly.w_G : nullptr,
                          c->reduce != nullptr ? PlaneOut{nullptr, nullptr, nullptr} : plane_out(c, ly.Gp), s.slots, ly.done + 1,
                          &ly.sc->sum_G2, nb, remade_with_sum(c, ly)};
      GradWSum &y = g.l[n - 1];
      y.totals[0] = GradWSum::Totals{s.p_slots, ly.p_sum, ly.p_change, l > 0 ? p_rows(c, ly, s).n_blocks : 0, ly.ld_in, l > 0 ? (int)ceil_div(ly.ld_in, TOTAL_COLS) : 0};
      y.totals[1] = GradWSum::Totals{ly.r_slots, ly.r_sum, nullptr, ly.r_blocks, ly.ld_out, (int)ceil_div(ly.ld_out, TOTAL_COLS)};
      blocks = std::max(blocks, nb + y.totals[0].n_blocks + y.totals[1].n_blocks);
      bytes += (4.0 * (ly.n_split + 1.0) + (c->use_tc ? 4.0 : 0.0)) * ly.n_out * ly.n_in;
    }
    Launch k(c, KC_GRADW_REDUCE, st, bytes, 0);
    reduce_gradW_kernel<<<dim3((unsigned)blocks, (unsigned)n), EW_THREADS, 0, st>>>(g, c->nu);
  }
  if (c->reduce != nullptr) {
    // nabla_W phi is a sum over nodes: add the shards' parts, then take the norm and the largest magnitude of the total
    for (int l : batch) {
      Layer &ly = c->layers[l];
      Scratch &s = scratch_of(c, l);
      const size_t n4 = (size_t)ly.n_out * ly.ld_in / 4;
      PD_TRY(shard_sum(c, st, ly.gradW, n4 * 4, 0));
      if (c->use_tc) PD_CUDA(cudaMemsetAsync(ly.w_G, 0, sizeof(uint32_t), st));
      sumsq_amax_kernel<<<ew_grid(n4), EW_THREADS, 0, st>>>(ly.gradW, n4, c->use_tc ? ly.w_G : nullptr, s.slots);
      reduce_slots_kernel<<<1, 256, 0, st>>>(s.slots, ew_grid(n4), 1, 1, &ly.sc->sum_G2);
      if (c->use_tc) split_rows(c, st, ly.gradW, (size_t)ly.n_out, ly.n_in, ly.ld_in, ly.w_G, ly.Gp);
    }
  }
  std::vector<Operand> G;
  std::vector<Operand *> to_check;
  for (int l : batch) {
    Layer &ly = c->layers[l];
    G.push_back(c->use_tc ? plane_operand(ly.gradW, ly.ld_in, ly.Gp, ly.w_G) : Operand{ly.gradW, ly.ld_in, nullptr});
    if (remade_with_sum(c, ly)) G.back().x = nullptr;
  }
  for (size_t i = 0; i < batch.size(); ++i) {
    const Layer &ly = c->layers[batch[i]];
    if (G[i].x == nullptr || (size_t)ly.n_out * ly.ld_in < CHECK_PLANES_FROM) continue;
    check_planes(c, st, (size_t)ly.n_out, {&G[i]});
  }
  {
    std::vector<Prod<EpiStoreSumsq>> v;
    for (size_t i = 0; i < batch.size(); ++i) {
      const int l = batch[i];
      Layer &ly = c->layers[l];
      Scratch &s = scratch_of(c, l);
      Prod<EpiStoreSumsq> p{N, ly.n_out, ly.n_in, P[i], G[i], EpiStoreSumsq{fused ? ly.gp : s.s1, ly.ld_out}, &s, s.slots + s.n_slots / 2, ly.done + 2};
      p.wide = ly.wide_gp;
      p.step = make_step(c, ly, STEP_THETA);
      if (c->use_tc) { p.step.w_in = ly.w_G; p.step.exp_W = ly.Wp.exp; p.step.exp_r = ly.rp.exp; p.step.exp_g = ly.Gp.exp; }
      v.push_back(p);
    }
    PD_TRY((gemm_nodes<false>(c, KC_GEMM_GP, st, v, 0)));
    // ||G p+||^2 is a sum over nodes (||G||^2 is the same on every shard already)
    for (size_t i = 0; i < batch.size(); ++i) PD_TRY(shard_step(c, st, &c->layers[batch[i]].sc->sum_Gp2, 1, v[i].step));
  }
  {
    Group<ThetaStep> g;
    int n = 0, blocks = 0;
    double bytes = 0;
    for (int l : batch) {
      Layer &ly = c->layers[l];
      Scratch &s = scratch_of(c, l);
      const size_t n4r = (size_t)N * ly.ld_out / 4;
      const int nbw = (int)ceil_div(ly.n_out, EW_THREADS / 32), nbr = fused ? 0 : ew_grid((size_t)ceil_div((int64_t)n4r, 4));
      g.l[n++] = ThetaStep{ly.W, ly.gradW, ly.n_out, ly.ld_in, c->use_tc ? ly.amax_W : nullptr, plane_out(c, ly.Wp),
                           ly.p_sum, ly.p_change, ly.r_sum, ly.b, ly.shift, c->reduce != nullptr ? s.red : nullptr, ly.sc, nbw,
                           ly.r, fused ? nullptr : s.s1, (uint32_t)n4r, nbr};
      blocks = std::max(blocks, nbw + nbr);
      bytes += (fused ? 0.0 : 12.0) * N * ly.n_out + (c->use_tc ? 16.0 : 12.0) * ly.n_out * ly.n_in;
    }
    {
      Launch k(c, KC_COLSUM, st, bytes, 0);
      theta_step_kernel<<<dim3((unsigned)blocks, (unsigned)n), EW_THREADS, 0, st>>>(g, 1.0 / (double)c->N_total);
    }
    if (c->reduce != nullptr) {
      // the sums run over all nodes: this shard's, added over the shards, then the mean over |V|
      for (int l : batch) {
        Layer &ly = c->layers[l];
        Scratch &s = scratch_of(c, l);
        PD_TRY(shard_sum(c, st, s.red, (size_t)ly.ld_out, 1));
        Launch k(c, KC_SMALL, st, 8.0 * ly.n_out, 0);
        finalize_bias_kernel<<<(unsigned)ceil_div(ly.n_out, EW_THREADS), EW_THREADS, 0, st>>>(s.red, ly.n_out, 1.0 / (double)c->N_total, ly.b, ly.shift);
      }
    }
  }
  return PDADMM_OK;
}

// z, q and u of hidden layers; needs p_{l+1} of this iteration.
static void zqu_step(pdadmm_ctx *c, cudaStream_t st, const Batch &batch) {
  Group<Zqu> g;
  int n = 0, blocks = 0, threads = 0;
  double bytes = 0;
  for (int l : batch) {
    Layer &ly = c->layers[l];
    const Layer &nx = c->layers[l + 1];
    const bool fused = c->q_implied;
    g.l[n++] = Zqu{ly.r, ly.z, fused ? ly.gp : nullptr, fused ? nullptr : ly.q, fused ? nullptr : ly.q, ly.u, nx.p, ly.shift, nx.t,
                   c->levels ? nx.codes : nullptr, nx.scale, nx.lo, r_rows(c, ly), ly.n_out, c->use_tc ? ly.amax_r : nullptr, plane_out(c, ly.rp), ly.sc};
    blocks = std::max(blocks, ly.r_blocks);
    threads = std::max(threads, row_share(ly.ld_out).threads);
    bytes += ((c->levels ? 28.0 + c->code_bytes : 32.0) + 4.0 + (fused ? 0.0 : 4.0) + (c->use_tc && ly.rp.hi ? 4.0 : 0.0)) * c->N * ly.n_out;
  }
  Launch k(c, KC_ZQU, st, bytes, 0);
  const ZquParams prm{c->rho, c->nu, c->slope, two_term(1.0, 2.0 + (double)c->slope * c->slope), c->quant_q ? (float)(c->levels - 1) : -1.0f, c->code_bytes == 2, c->table_lo,
                      c->table_step, c->table_size, c->table_even ? 1 : 0};
  const dim3 grid((unsigned)blocks, (unsigned)n);
  const bool general = !(c->q_implied && c->q_free);
  if (c->table_size > 0) {
    const size_t sh = c->table_size * sizeof(float);
    if (general) zqu_table_kernel<true><<<grid, threads, sh, st>>>(g, prm);
    else zqu_table_kernel<false><<<grid, threads, sh, st>>>(g, prm);
  } else if (c->levels) {
    if (general) zqu_kernel<true, true><<<grid, threads, 0, st>>>(g, prm);
    else zqu_kernel<true, false><<<grid, threads, 0, st>>>(g, prm);
  } else {
    if (general) zqu_kernel<false, true><<<grid, threads, 0, st>>>(g, prm);
    else zqu_kernel<false, false><<<grid, threads, 0, st>>>(g, prm);
  }
}
static void r_column_sums(pdadmm_ctx *c, cudaStream_t st, const Layer &ly) {
  Launch k(c, KC_SMALL, st, 4.0 * c->N * ly.n_out, 0);
  Group<ColSum> g;
  g.l[0] = ColSum{ly.r, r_rows(c, ly), nullptr};
  colsum_kernel<false><<<ly.r_blocks, row_share(ly.ld_out).threads, 0, st>>>(g, 0, 0);
}
static void zlast_step(pdadmm_ctx *c, cudaStream_t st) {
  Layer &ly = c->layers[c->L - 1];
  const int N = (int)c->N;
  {
    Launch k(c, KC_ZLAST, st, (c->use_tc ? 24.0 : 20.0) * N * ly.n_out, 0);
    launch_zlast(st, ly.r, ly.z, ly.shift, c->labels, c->mask, N, ly.n_out, ly.ld_out, (double)c->nu, c->d_flag,
                 c->use_tc ? ly.amax_r : nullptr, c->ls_risk ? 1 : 0, plane_out(c, ly.rp), c->q_implied ? ly.gp : nullptr, ly.sc);
  }
  r_column_sums(c, st, ly);
}

static int iterate_layers(pdadmm_ctx *c, bool *hit_cap) {
  const int S_all = 1 + (int)c->more_lanes.size();
  // Grouped: batches of up to S layers, one launch per kernel and batch, all on the main stream.  Otherwise one layer at a time,
  // layer l on lane l mod S; per-kernel timing wants one kernel at a time, a single lane then.
  const bool grouped = c->grouped;
  const int S = grouped || !c->profiling ? S_all : 1;
  c->n_active = S;
  const cudaStream_t main = c->scr.st;
  auto stream_of = [&](int l) { return grouped ? main : lane(c, l % S).st; };
  const bool many = !grouped && S > 1;
  // the other lanes start after everything queued on the main stream so far
  if (many) {
    PD_CUDA(cudaEventRecord(c->ev_lane[0], main));
    for (int i = 1; i < S; ++i) PD_CUDA(cudaStreamWaitEvent(lane(c, i).st, c->ev_lane[0], 0));
  }
  // p-update (layers 2..L, from the iterates of the previous iteration) and W-, b-update with the new p, batch by batch: the
  // scratch planes of r and p go from the one to the other.  The quantised p-update reads accept flags on the host after
  // every trial: the host queues a batch's gradient and first trial, and only then waits for the flags of the
  // batch that it queued on another lane before, so that the GPU always has other lanes' work while a flag travels.
  const int per_batch = grouped ? std::min(S, MAX_GROUP) : 1;
  std::vector<Batch> waiting(many ? S : 1);          // batch whose first trial is in flight on each lane
  auto finish = [&](int i) -> int {
    Batch b;
    b.swap(waiting[i]);
    if (b.empty()) return PDADMM_OK;
    Batch p;                                         // (layer 1 has no p-update)
    for (int l : b) if (l > 0) p.push_back(l);
    const cudaStream_t st = stream_of(b[0]);
    if (!p.empty()) PD_TRY(q_finish(c, st, p, hit_cap));
    if (many) for (int l : p) PD_CUDA(cudaEventRecord(c->ev_p[l], st));
    return w_and_b_step(c, st, b);
  };
  for (int l0 = 0; l0 < c->L; l0 += per_batch) {
    Batch b, p;
    for (int l = l0; l < std::min(c->L, l0 + per_batch); ++l) {
      b.push_back(l);
      if (l > 0) p.push_back(l);
    }
    const cudaStream_t st = stream_of(l0);
    const int slot = many ? l0 % S : 0;
    if (c->levels) PD_TRY(finish(slot));
    if (!p.empty()) {
      PD_TRY(p_gradient_and_tau(c, st, p));
      if (c->levels) {
        PD_TRY(q_trial(c, st, p));
        waiting[slot] = b;
        continue;
      }
      p_step_plain(c, st, p);
      if (many) for (int l : p) PD_CUDA(cudaEventRecord(c->ev_p[l], st));
    }
    PD_TRY(w_and_b_step(c, st, b));
  }
  const int n_batches = (int)ceil_div(c->L, per_batch);
  for (size_t i = 0; i < waiting.size(); ++i) PD_TRY(finish((int)((n_batches + i) % waiting.size())));    // the oldest first
  // z-, q-, u-update (q_l and u_l need p_{l+1} of this iteration, which another lane may have written)
  if (grouped) {
    // the last layer's Newton steps run beside the hidden layers' update
    const bool beside = S > 1 && !c->profiling && c->L > 1;
    const cudaStream_t other = beside ? c->more_lanes[0]->own : main;
    if (beside) {
      PD_CUDA(cudaEventRecord(c->ev_lane[0], main));
      PD_CUDA(cudaStreamWaitEvent(other, c->ev_lane[0], 0));
    }
    zlast_step(c, other);
    // up to three hidden layers one launch each: nothing to gain from a common one
    const int per = c->L - 1 > 3 ? MAX_GROUP : 1;
    for (int l0 = 0; l0 + 1 < c->L; l0 += per) {
      Batch b;
      for (int l = l0; l < std::min(c->L - 1, l0 + per); ++l) b.push_back(l);
      zqu_step(c, main, b);
    }
    if (beside) {
      PD_CUDA(cudaEventRecord(c->ev_lane[1], other));
      PD_CUDA(cudaStreamWaitEvent(main, c->ev_lane[1], 0));
    }
    return PDADMM_OK;
  }
  for (int l = 0; l < c->L; ++l) {
    const cudaStream_t st = stream_of(l);
    if (l + 1 == c->L) { zlast_step(c, st); break; }
    if (many) PD_CUDA(cudaStreamWaitEvent(st, c->ev_p[l + 1], 0));
    zqu_step(c, st, {l});
  }
  // join: the main stream continues after every lane
  for (int i = 1; many && i < S; ++i) {
    PD_CUDA(cudaEventRecord(c->ev_lane[i], lane(c, i).st));
    PD_CUDA(cudaStreamWaitEvent(main, c->ev_lane[i], 0));
  }
  return PDADMM_OK;
}
static void mark_q_stale(pdadmm_ctx *c) {
  for (int l = 0; l + 1 < c->L; ++l) c->layers[l].q_stale = true;
}
// An iteration with q_implied puts G p+ where q is, and may end early (a reduction over shards that fails): z and u give q before and
// after the z-update of every layer.
static void will_iterate(pdadmm_ctx *c) {
  if (c->q_implied) mark_q_stale(c);
  c->in_iteration = true;
}
static void iterated(pdadmm_ctx *c) {
  if (c->q_free) { c->q_implied = true; mark_q_stale(c); }
  c->in_iteration = false;
}
// What is derived from the tensors (the residual, t, planes and magnitudes, column sums) is formed again by the next call that needs it.
static void forget_derived(pdadmm_ctx *c) {
  c->r_valid = c->t_valid = c->w_planes_valid = c->amax_p_valid = c->r_sums_valid = c->p_sums_valid = false;
}
static int iterate_once(pdadmm_ctx *c, bool *hit_cap) {
  will_iterate(c);
  PD_TRY(iterate_layers(c, hit_cap));
  iterated(c);
  return PDADMM_OK;
}

}  // namespace pd

namespace pd {

// ---- construction ---------------------------------------------------------------------------------------------

static int check_config(const pdadmm_config *cfg) {
  if (!cfg) return fail(PDADMM_EINVAL, "config is null");
  if (cfg->n_nodes < 1 || cfg->n_nodes > (int64_t)INT32_MAX / 2) return fail(PDADMM_EINVAL, "n_nodes out of range");
  if (cfg->n_edges < 0 || (cfg->n_edges > 0 && (!cfg->edge_src || !cfg->edge_dst)))
    return fail(PDADMM_EINVAL, "edge list missing");
  if (cfg->feat_dim < 1 || !cfg->features) return fail(PDADMM_EINVAL, "features missing");
  if (cfg->n_hops < 0 || cfg->n_hops > 16) return fail(PDADMM_EINVAL, "n_hops must be in [0, 16]");
  if (cfg->n_layers < 1 || !cfg->layer_widths || !cfg->init_W) return fail(PDADMM_EINVAL, "layers missing");
  if (cfg->n_layers > 1024) return fail(PDADMM_EINVAL, "at most 1024 layers");
  if (cfg->n_classes < 2 || cfg->n_classes > ZL_MAX_C)
    return fail(PDADMM_EINVAL, "n_classes must be in [2, %d]", ZL_MAX_C);
  if (cfg->layer_widths[cfg->n_layers - 1] != cfg->n_classes)
    return fail(PDADMM_EINVAL, "last layer width must equal n_classes");
  for (int l = 0; l < cfg->n_layers; ++l) {
    if (cfg->layer_widths[l] < 1) return fail(PDADMM_EINVAL, "layer width %d is not positive", l + 1);
    if (!cfg->init_W[l]) return fail(PDADMM_EINVAL, "init_W[%d] is null", l);
  }
  if (!cfg->labels || !cfg->train_mask) return fail(PDADMM_EINVAL, "labels or mask missing");
  if (!(cfg->rho > 0.f) || !(cfg->nu > 0.f)) return fail(PDADMM_EINVAL, "rho and nu must be positive");
  if (cfg->quant_levels != 0 && (cfg->quant_levels < 2 || cfg->quant_levels > 65536))
    return fail(PDADMM_EINVAL, "quant_levels must be 0 or in [2, 65536]");
  if (cfg->quant_neg_levels < 0 || cfg->quant_neg_levels >= std::max(cfg->quant_levels, 1))
    return fail(PDADMM_EINVAL, "quant_neg_levels must be in [0, quant_levels)");
  if (cfg->quant_step < 0.f || (cfg->quant_neg_levels > 0 && !(cfg->quant_step > 0.f)))
    return fail(PDADMM_EINVAL, "quant_step must be >= 0, and > 0 when quant_neg_levels > 0");
  if (!(cfg->leaky_slope >= 0.f && cfg->leaky_slope < 1.f))
    return fail(PDADMM_EINVAL, "leaky_slope must be in [0, 1)");
  if (cfg->activation < 0 || cfg->activation > 2) return fail(PDADMM_EINVAL, "activation must be 0, 1 or 2");
  if (cfg->activation != 0) {
    if (cfg->leaky_slope != 0.f) return fail(PDADMM_EINVAL, "leaky_slope belongs to activation 0");
    if (cfg->table_size < 2 || cfg->table_size > 4096 || !(cfg->table_hi > cfg->table_lo))
      return fail(PDADMM_EINVAL, "a smooth activation needs table_size in [2, 4096] and table_lo < table_hi");
  }
  if ((cfg->flags & PDADMM_FLAG_QUANT_Q) && cfg->quant_levels == 0)
    return fail(PDADMM_EINVAL, "PDADMM_FLAG_QUANT_Q needs quant_levels >= 2");
  for (int64_t j = 0; j < cfg->n_nodes; ++j)
    if (cfg->labels[j] < 0 || cfg->labels[j] >= cfg->n_classes)
      return fail(PDADMM_EINVAL, "label of node %lld is outside [0, %d)", (long long)j, cfg->n_classes);
  return PDADMM_OK;
}

// Host -> device copies go through the context's stream, so that they are ordered with its kernels
// (the stream does not synchronise with the default stream).
static int upload_rows(pdadmm_ctx *c, cudaStream_t st, float *dst, int ld, const float *src, int width, int64_t rows) {
  return copy_rows(c->device, st, const_cast<float *>(src), dst, (size_t)ld * 4, (size_t)width * 4, (size_t)rows, false);
}

// Temporary device buffers of the CSR construction, carved out of one block that goes back when the builder returns.  The stream
// is waited for, not the device: that would wait for other threads' contexts too, and it is an error while one of them
// captures its iteration.
struct TempBuffers {
  int device;
  cudaStream_t st;
  std::vector<DeviceBlock> block;
  size_t used = 0;
  TempBuffers(int dev, cudaStream_t s) : device(dev), st(s) {}
  ~TempBuffers() { if (!block.empty()) { cudaStreamSynchronize(st); device_pool(device).give(block); } }
  static size_t room(size_t bytes) { return (std::max<size_t>(bytes, 16) + 255) & ~size_t(255); }
  int reserve(size_t bytes) {
    DeviceBlock b;
    const size_t want = (bytes + (size_t(2) << 20) - 1) & ~((size_t(2) << 20) - 1);
    const cudaError_t e = device_pool(device).take(want, &b);
    if (e != cudaSuccess) return fail(PDADMM_ENOMEM, "cudaMalloc of %zu bytes failed: %s", want, cudaGetErrorString(e));
    block.push_back(b);
    return PDADMM_OK;
  }
  template <class T>
  int get(T **out, size_t count) {
    const size_t bytes = room(count * sizeof(T));
    if (used + bytes > block[0].bytes) return fail(PDADMM_ENOMEM, "temporary buffers were reserved too small");
    *out = (T *)((char *)block[0].p + used);
    used += bytes;
    return PDADMM_OK;
  }
};

// Edge list (host) -> c->row_ptr, c->col_idx (device), c->nnz; c->csr_val is allocated, not filled.
static int build_csr(pdadmm_ctx *c, const pdadmm_config *cfg) {
  const int64_t N = c->N, E = cfg->n_edges;
  const size_t raw_cap = (size_t)(2 * E + N);
  if (raw_cap > (size_t)INT32_MAX) return fail(PDADMM_EINVAL, "more than 2^31-1 non-zeros");
  cudaStream_t st = c->scr.st;
  TempBuffers tmp(c->device, st);
  const size_t n4 = TempBuffers::room((size_t)N * 4 + 4);
  PD_TRY(tmp.reserve(2 * TempBuffers::room((size_t)E * 4) + 5 * n4 + 2 * TempBuffers::room(raw_cap * 4) + 1024));
  int *d_src, *d_dst, *deg, *cursor, *raw_ptr, *raw, *sorted, *len, *long_rows, *meta;
  unsigned long long *bad_edge;
  PD_TRY(tmp.get(&d_src, (size_t)E)); PD_TRY(tmp.get(&d_dst, (size_t)E));
  PD_TRY(tmp.get(&deg, (size_t)N)); PD_TRY(tmp.get(&cursor, (size_t)N)); PD_TRY(tmp.get(&len, (size_t)N));
  PD_TRY(tmp.get(&raw_ptr, (size_t)N + 1)); PD_TRY(tmp.get(&long_rows, (size_t)N));
  PD_TRY(tmp.get(&raw, raw_cap)); PD_TRY(tmp.get(&sorted, raw_cap));
  PD_TRY(tmp.get(&meta, 4)); PD_TRY(tmp.get(&bad_edge, 1));
  PD_TRY(dev_alloc(c, &c->row_ptr, (size_t)N + 1, false));
  PD_CUDA(cudaMemsetAsync(deg, 0, (size_t)N * 4, st));
  PD_CUDA(cudaMemsetAsync(cursor, 0, (size_t)N * 4, st));
  PD_CUDA(cudaMemsetAsync(len, 0, (size_t)N * 4, st));
  PD_CUDA(cudaMemsetAsync(meta, 0, 16, st));
  PD_CUDA(cudaMemsetAsync(bad_edge, 0xff, 8, st));
  const int e_grid = (int)std::max<int64_t>(1, ceil_div(E, 256)), r_grid = (int)ceil_div(N * 32, 256);
  if (E > 0) {
    PD_CUDA(cudaMemcpyAsync(d_src, cfg->edge_src, (size_t)E * 4, cudaMemcpyHostToDevice, st));
    PD_CUDA(cudaMemcpyAsync(d_dst, cfg->edge_dst, (size_t)E * 4, cudaMemcpyHostToDevice, st));
    edge_count_kernel<<<e_grid, 256, 0, st>>>(d_src, d_dst, (long long)E, (int)N, deg, meta, bad_edge);
  }
  exclusive_scan_kernel<<<1, 1024, 0, st>>>(deg, (int)N, 1, raw_ptr, meta);
  if (E > 0) edge_scatter_kernel<<<e_grid, 256, 0, st>>>(d_src, d_dst, (long long)E, (int)N, raw_ptr, cursor, raw);
  row_sort_warp_kernel<<<r_grid, 256, 0, st>>>(raw_ptr, (int)N, raw, sorted, len, long_rows, meta);
  row_sort_block_kernel<<<2 * c->n_sms, 1024, 0, st>>>(raw_ptr, raw, sorted, len, long_rows, meta);
  exclusive_scan_kernel<<<1, 1024, 0, st>>>(len, (int)N, 0, c->row_ptr, meta);
  int h_meta[4]; unsigned long long h_bad; int h_nnz;
  PD_CUDA(cudaMemcpyAsync(h_meta, meta, 16, cudaMemcpyDeviceToHost, st));
  PD_CUDA(cudaMemcpyAsync(&h_bad, bad_edge, 8, cudaMemcpyDeviceToHost, st));
  PD_CUDA(cudaMemcpyAsync(&h_nnz, c->row_ptr + N, 4, cudaMemcpyDeviceToHost, st));
  PD_CUDA(cudaStreamSynchronize(st));
  if (h_meta[0] == 1)
    return fail(PDADMM_EINVAL, "edge %llu = (%d, %d) is outside [0, %lld)", h_bad, cfg->edge_src[h_bad],
                cfg->edge_dst[h_bad], (long long)N);
  if (h_meta[0] == 2) return fail(PDADMM_EINVAL, "more than 2^31-1 non-zeros");
  if (h_meta[0] == 3) return fail(PDADMM_EINVAL, "a node has more than %d neighbours", CSR_MAX_ROW - 1);
  c->nnz = h_nnz;
  PD_TRY(dev_alloc(c, &c->col_idx, (size_t)c->nnz, false));
  PD_TRY(dev_alloc(c, &c->csr_val, (size_t)c->nnz, false));
  row_compact_kernel<<<r_grid, 256, 0, st>>>(raw_ptr, c->row_ptr, (int)N, sorted, c->col_idx);
  PD_CUDA(cudaGetLastError());
  PD_CUDA(cudaStreamSynchronize(st));     // the temporaries are released on return
  return PDADMM_OK;
}

// buffers of a lane's quantised trials: trial p, d, codes (they trade places with a layer's p and codes when a
// trial is taken, so all have one size), the pinned word and the event of the accept flag
static int alloc_trial_buffers(pdadmm_ctx *c, Scratch &s, size_t n) {
  if (!c->int_operands) {                                    // with integer operands p+ and d exist as codes and planes only
    PD_TRY(dev_alloc(c, &s.p_new, n));
    PD_TRY(dev_alloc(c, &s.d, n));
  }
  PD_TRY(dev_alloc(c, &s.codes_new, n * c->code_bytes));
  if (c->int_operands) {
    PD_TRY(dev_alloc(c, &s.pn_plane, n));
    PD_TRY(dev_alloc(c, &s.d_plane, n));
  }
  s.h_flag = c->h_pinned + 64 + (&s == &c->scr ? 0 : (int)c->more_lanes.size());
  PD_CUDA(device_pool(c->device).take_event(false, &s.ev_flag));
  return PDADMM_OK;
}

// Start of Algorithm 1 for layers first..L-1 (0-based) from the current p_first: b = 0, z_l = W_l p_l, q_l = f(z_l),
// p_{l+1} = q_l (projected in -Q mode, with the level spacing from max(q_l)), u = 0, r = 0.
static int feasible_start(pdadmm_ctx *c, int first) {
  const int64_t N = c->N;
  cudaStream_t st = c->scr.st;
  Scratch &s = c->scr;
  for (int l = first; l < c->L; ++l) {
    Layer &ly = c->layers[l];
    EpiStore epi{ly.z, ly.ld_out};
    PD_TRY(refresh_W_planes(c, ly, st));
    PD_CUDA(cudaMemsetAsync(ly.amax_p, 0, sizeof(uint32_t), st));
    absmax_kernel<<<ew_grid((size_t)N * ly.ld_in / 4), EW_THREADS, 0, st>>>(ly.p, (size_t)N * ly.ld_in / 4, ly.amax_p);
    Operand P{ly.p, ly.ld_in, ly.amax_p};
    if (l == 0 && c->use_tc) {
      split_rows(c, st, ly.p, (size_t)N, ly.n_in, ly.ld_in, ly.amax_p, ly.xp);
      P = operand_X(ly);
    }
    PD_TRY((gemm_nodes<false, EpiStore>(c, KC_GEMM_RESID, st, {{(int)N, ly.n_out, ly.n_in, P, operand_W(ly), epi, &c->scr}}, 0)));
    PD_CUDA(cudaMemsetAsync(ly.b, 0, (size_t)ly.ld_out * 4, st));
    PD_CUDA(cudaMemsetAsync(ly.shift, 0, (size_t)ly.ld_out * 4, st));
    PD_CUDA(cudaMemsetAsync(ly.r, 0, (size_t)N * ly.ld_out * 4, st));
    PD_CUDA(cudaMemsetAsync(ly.amax_r, 0, sizeof(uint32_t), st));
    if (l + 1 == c->L) break;
    PD_CUDA(cudaMemsetAsync(ly.u, 0, (size_t)N * ly.ld_out * 4, st));
    Layer &nx = c->layers[l + 1];
    const size_t n4 = (size_t)N * ly.ld_out / 4;
    const int grid = ew_grid(n4);
    float *bm = reinterpret_cast<float *>(s.slots);
    relu_max_kernel<<<grid, EW_THREADS, 0, st>>>(ly.z, ly.q, n4, c->slope, ly.n_out, (uint32_t)ly.ld_out / 4, bm);
    if (c->levels) {
      std::vector<float> hm(grid);
      PD_CUDA(cudaMemcpyAsync(hm.data(), bm, grid * sizeof(float), cudaMemcpyDeviceToHost, st));
      PD_CUDA(cudaStreamSynchronize(st));
      float mx = 0.f;
      for (float v : hm) mx = std::max(mx, v);
      if (c->reduce != nullptr) {            // the level spacing comes from the largest entry over all nodes
        PD_CUDA(cudaMemcpyAsync(s.red, &mx, 4, cudaMemcpyHostToDevice, st));
        PD_TRY(shard_sum(c, st, s.red, 1, 0, 1));
        PD_CUDA(cudaMemcpyAsync(&mx, s.red, 4, cudaMemcpyDeviceToHost, st));
        PD_CUDA(cudaStreamSynchronize(st));
      }
      nx.scale = c->fixed_step > 0.f ? c->fixed_step : (mx > 0.f ? mx / (float)(c->levels - 1) : 1.0f);
      nx.lo = -(float)c->neg_levels * nx.scale;
      quantize_kernel<<<ew_grid(n4 * 4), EW_THREADS, 0, st>>>(ly.q, n4 * 4, nx.scale, nx.lo, c->levels, nx.p, nx.codes,
                                                              c->code_bytes == 2);
      if (c->int_operands) codes_to_plane_kernel<<<ew_grid(n4), EW_THREADS, 0, st>>>(nx.codes, c->code_bytes == 2, c->neg_levels, n4, nx.p_plane);
      if (c->quant_q)      // start inside the level set: q_l = p_{l+1}
        PD_CUDA(cudaMemcpyAsync(ly.q, nx.p, n4 * 16, cudaMemcpyDeviceToDevice, st));
    } else {
      PD_CUDA(cudaMemcpyAsync(nx.p, ly.q, n4 * 16, cudaMemcpyDeviceToDevice, st));
    }
  }
  return PDADMM_OK;
}

static int take_ctx_pinned(pdadmm_ctx *c) {
  c->h_pinned = (int *)ctx_pinned_pool().take();
  if (!c->h_pinned) return fail(PDADMM_ENOMEM, "page-locked host memory is exhausted");
  c->h_results = (double *)((char *)c->h_pinned + 1024);
  return PDADMM_OK;
}

static int build(pdadmm_ctx *c, const pdadmm_config *cfg, const pdadmm_shard *shard) {
  const int64_t Ntot = cfg->n_nodes;
  const bool sharded = shard != nullptr && shard->allreduce != nullptr;
  const int64_t N = sharded ? shard->node_count : Ntot;
  const int64_t node0 = sharded ? shard->node_begin : 0;
  c->N_total = Ntot; c->node_begin = node0;
  if (sharded) { c->reduce = shard->allreduce; c->reduce_user = shard->user; }
  // the graph stage works on all nodes: c->N is the whole graph until X is built
  c->device = cfg->device; c->N = Ntot; c->L = cfg->n_layers; c->d = cfg->feat_dim; c->n_blocks = cfg->n_hops + 1;
  c->n0 = c->n_blocks * c->d; c->ld0 = row_ld(c, c->n0); c->C = cfg->n_classes; c->levels = cfg->quant_levels;
  c->neg_levels = cfg->quant_neg_levels; c->fixed_step = cfg->quant_step;
  c->code_bytes = cfg->quant_levels > 256 ? 2 : 1;
  c->quant_q = (cfg->flags & PDADMM_FLAG_QUANT_Q) != 0;
  c->slope = cfg->activation == 1 ? ACT_TANH : (cfg->activation == 2 ? ACT_SIGMOID : cfg->leaky_slope);
  if (cfg->activation != 0) {
    c->table_size = cfg->table_size;
    c->table_lo = cfg->table_lo;
    c->table_step = (cfg->table_hi - cfg->table_lo) / (float)(cfg->table_size - 1);      // single precision, like the candidates
    c->table_even = table_is_even(cfg->table_lo, cfg->table_hi, c->table_step);
  }
  c->ls_risk = (cfg->flags & PDADMM_FLAG_LEAST_SQUARES) != 0;
  c->rho = cfg->rho; c->nu = cfg->nu; c->flags = cfg->flags;
  c->q_free = !c->quant_q;
  c->use_tc = (cfg->flags & PDADMM_FLAG_SIMT_GEMM) == 0;
  c->int_operands = c->use_tc && c->levels >= 2 && c->levels <= 2048;
  PD_CUDA(cudaSetDevice(cfg->device));
  PD_CUDA(cudaDeviceGetAttribute(&c->n_sms, cudaDevAttrMultiProcessorCount, cfg->device));
  DevicePool &pool = device_pool(c->device);
  PD_CUDA(pool.take_stream(&c->scr.own));
  c->scr.st = c->scr.own;
  cudaStream_t st = c->scr.st;
  PD_TRY(take_ctx_pinned(c));
  PD_CUDA(pool.take_event(true, &c->ev_begin));
  PD_CUDA(pool.take_event(true, &c->ev_end));
  c->control_words = 4 + 8 * (size_t)c->L + (size_t)PDADMM_N_LANES * c->n_sms * 8;
  PD_TRY(dev_alloc(c, &c->control, c->control_words));
  c->d_flag = c->control;
  PD_TRY(dev_alloc(c, &c->done, OBJ_MAX_LAYERS + 1));
  PD_TRY(dev_alloc(c, &c->counts, 4));

  // graph: CSR pattern, values and sparse products all on the device
  PD_TRY(build_csr(c, cfg));
  adjacency_values_kernel<<<(int)ceil_div(Ntot * 32, 256), 256, 0, st>>>(c->row_ptr, c->col_idx, (int)Ntot, c->csr_val);
  PD_TRY(dev_alloc(c, &c->labels, (size_t)N, false));
  PD_TRY(dev_alloc(c, &c->mask, (size_t)N, false));
  PD_CUDA(cudaMemcpyAsync(c->labels, cfg->labels + node0, (size_t)N * 4, cudaMemcpyHostToDevice, st));
  PD_CUDA(cudaMemcpyAsync(c->mask, cfg->train_mask + node0, (size_t)N, cudaMemcpyHostToDevice, st));
  PD_CUDA(cudaStreamSynchronize(st));
  // X = [H, A~ H, A~^2 H, ...] for all nodes (a shard needs its neighbours' features, and theirs, ...); a shard then
  // keeps the rows of its own nodes
  float *x_full = nullptr;
  struct BlockLater {
    int device; cudaStream_t st; std::vector<DeviceBlock> b;
    ~BlockLater() { if (!b.empty()) { cudaStreamSynchronize(st); device_pool(device).give(b); } }
  } x_full_block{c->device, st, {}};
  if (sharded) {
    const size_t bytes = (size_t)Ntot * c->ld0 * 4 + 256;
    DeviceBlock b;
    if (pool.take(bytes, &b) != cudaSuccess) return fail(PDADMM_ENOMEM, "cudaMalloc of %zu bytes failed", bytes);
    x_full_block.b.push_back(b);
    x_full = (float *)b.p;
    PD_CUDA(cudaMemsetAsync(x_full, 0, bytes, st));
  }
  c->N = N;                                  // from here on: the nodes this context owns

  // layers
  c->layers.resize(c->L);
  int max_in = 0, max_out = 0;
  size_t max_part = 0;
  for (int l = 1; l < c->L; ++l) max_in = std::max(max_in, row_ld(c, cfg->layer_widths[l - 1]));
  for (int l = 0; l < c->L; ++l) max_out = std::max(max_out, row_ld(c, cfg->layer_widths[l]));
  for (int l = 0; l < c->L; ++l) {
    Layer &ly = c->layers[l];
    ly.n_in = l == 0 ? c->n0 : cfg->layer_widths[l - 1];
    ly.n_out = cfg->layer_widths[l];
    ly.ld_in = row_ld(c, ly.n_in); ly.ld_out = row_ld(c, ly.n_out);
    max_out = std::max(max_out, ly.ld_out);
    const size_t e_out = (size_t)N * ly.ld_out;
    // quantised mode: p_l and its codes trade places with the trial buffers, so all share one size
    const size_t e_in = (size_t)N * ((c->levels && l > 0) ? max_in : ly.ld_in);
    PD_TRY(dev_alloc(c, &ly.p, c->int_operands ? (size_t)N * ly.ld_in : e_in));
    if (l == 0)      // the features go first: their copy overlaps the clearing of everything allocated after them
      PD_TRY(upload_rows(c, st, sharded ? x_full : ly.p, ly.ld_in, cfg->features, c->d, Ntot));
    PD_TRY(dev_alloc(c, &ly.W, (size_t)ly.n_out * ly.ld_in));
    PD_TRY(dev_alloc(c, &ly.gradW, (size_t)ly.n_out * ly.ld_in));
    if (c->use_tc) {
      PD_TRY(alloc_planes(c, (size_t)ly.n_out * ly.ld_in, &ly.Wp));
      PD_TRY(alloc_planes(c, (size_t)ly.n_out * ly.ld_in, &ly.Gp));
      PD_TRY(dev_alloc(c, &ly.amax_W, 1));
      if (l == 0) PD_TRY(alloc_planes(c, (size_t)N * ly.ld_in, &ly.xp));
    }
    PD_TRY(dev_alloc(c, &ly.b, (size_t)ly.ld_out));
    PD_TRY(dev_alloc(c, &ly.shift, (size_t)ly.ld_out));
    PD_TRY(dev_alloc(c, &ly.p_sum, (size_t)ly.ld_in));
    PD_TRY(dev_alloc(c, &ly.p_change, (size_t)ly.ld_in));
    PD_TRY(dev_alloc(c, &ly.r_sum, (size_t)ly.ld_out));
    PD_TRY(dev_alloc(c, &ly.z, e_out));
    // quantised mode: r_l (l >= 2) trades places with the lane's buffer for the trial's r + W d, so all have one size
    PD_TRY(dev_alloc(c, &ly.r, (c->levels && l > 0) ? (size_t)N * max_out : e_out));
    if (l + 1 < c->L) { PD_TRY(dev_alloc(c, &ly.q, e_out)); PD_TRY(dev_alloc(c, &ly.u, e_out)); ly.gp = ly.q; }
    else if (c->q_free) PD_TRY(dev_alloc(c, &ly.gp, e_out));
    if (c->levels && l > 0) PD_TRY(dev_alloc(c, &ly.codes, e_in * c->code_bytes));
    if (c->int_operands && l > 0) PD_TRY(dev_alloc(c, &ly.p_plane, e_in));
    if (l > 0) PD_TRY(dev_alloc(c, &ly.t, (size_t)N * ly.ld_in));
    PD_TRY(dev_alloc(c, &ly.sc, 1));
    ly.done = c->control + 4 + 8 * l;
    ly.w_g = reinterpret_cast<uint32_t *>(ly.done + 4);
    ly.w_wg = ly.w_g + 1; ly.w_G = ly.w_g + 2; ly.w_d = ly.w_g + 3;
    if (l > 0) PD_TRY(dev_alloc(c, &ly.g_exp, 1));
    PD_TRY(dev_alloc(c, &ly.amax_p, 1));
    PD_TRY(dev_alloc(c, &ly.amax_r, 1));
    PD_TRY(upload_rows(c, st, ly.W, ly.ld_in, cfg->init_W[l], ly.n_in, ly.n_out));
  }
  // Scratch per layer, for working on the layers in batches, if it fits 4 GB for three layers at least; estimated from the two
  // fp32 matrices and the two pairs of planes, which are most of it.
  const size_t e_max = (size_t)N * std::max(max_in, max_out);
  const bool small = c->L > 1 && 3 * 16 * e_max <= (size_t(4) << 30);
  // Node slices of the W-gradient product (slices >= 256 nodes, at most 32): the count with the shortest estimated product
  // (choose_wide) and sum of the slices, which are written and read once more at 3000 bytes per SM cycle (6000 in L2).  Layers that are worked on
  // together have one common count.
  auto choose_slices = [&](int l0, int l1) {
    const int max_split = (int)std::max<int64_t>(1, std::min<int64_t>(32, ceil_div(N, 256)));
    int split = 1;
    double best = 0;
    for (int w = 1; w <= max_split; ++w) {
      const int64_t chunk = round_up((int)ceil_div(N, w), TC_BK), slices = ceil_div(N, chunk);
      Shape v[MAX_GROUP];
      double cost = 0, values = 0;
      for (int l = l0; l < l1; ++l) {
        v[l - l0] = Shape{c->layers[l].n_out, c->layers[l].n_in, chunk, slices};
        values += (double)c->layers[l].n_out * c->layers[l].ld_in;
      }
      choose_wide(c->n_sms, v, l1 - l0, c->int_operands, &cost);
      cost += 8.0 * values * slices / (4.0 * values * slices < 6e7 ? 6000.0 : 3000.0);
      if (w == 1 || cost < best) { best = cost; split = w; }
    }
    Shape vw[MAX_GROUP], vg[MAX_GROUP], vp[MAX_GROUP];
    int n = 0, n_wg = 0;
    for (int l = l0; l < l1; ++l, ++n) {
      const Layer &ly = c->layers[l];
      const int64_t chunk = round_up((int)ceil_div(N, split), TC_BK);
      vw[n] = Shape{ly.n_out, ly.n_in, chunk, ceil_div(N, chunk)};
      vp[n] = Shape{N, ly.n_out, ly.n_in, 1};
      if (l > 0) vg[n_wg++] = vp[n];
    }
    const bool ints = c->int_operands, wide_W = choose_wide(c->n_sms, vw, n, ints), wide_gp = choose_wide(c->n_sms, vp, n, ints);
    const bool wide_wg = n_wg > 0 && choose_wide(c->n_sms, vg, n_wg, ints);
    for (int l = l0; l < l1; ++l) {
      Layer &ly = c->layers[l];
      ly.wide_W = wide_W; ly.wide_gp = wide_gp; ly.wide_wg = wide_wg;
      ly.k_chunk = round_up((int)ceil_div(N, split), TC_BK);      // multiple of both kernels' K blocks
      ly.n_split = (int)ceil_div(N, ly.k_chunk);
      max_part = std::max(max_part, (size_t)ly.n_split * ly.n_out * ly.ld_in);
    }
  };
  // The CUDA-core products are one launch per layer anyway and gain from running beside each other: lanes, as many as 4 GB pay
  // for (3000 x 300, 4 layers: 0.94 ms per iteration on one stream, 0.39 on four).
  const bool batched = small && c->use_tc;
  for (int l = 0; l < c->L; l += batched ? MAX_GROUP : 1) choose_slices(l, std::min(c->L, l + (batched ? MAX_GROUP : 1)));
  // blocks of the kernels that sum columns (the counts of batches, whichever way the layers are queued: every way gives the same bits)
  const int per_launch = batched ? std::max(1, std::min(c->L - 1, MAX_GROUP)) : 1;       // (no p-step of layer 1, no z_L)
  size_t max_p_slots = 0;
  for (Layer &ly : c->layers) {
    ly.r_blocks = sum_blocks(c, ly.ld_out, per_launch, true);
    PD_TRY(dev_alloc(c, &ly.r_slots, (size_t)ly.r_blocks * ly.ld_out));
    ly.p_blocks = sum_blocks(c, ly.ld_in, per_launch, false);
    max_p_slots = std::max(max_p_slots, (size_t)ly.p_blocks * ly.ld_in);
  }
  // scratch
  Scratch &s = c->scr;
  const size_t bytes_before_scratch = c->bytes_handed_out;
  PD_TRY(dev_alloc(c, &s.s1, e_max));
  PD_TRY(dev_alloc(c, &s.s2, (size_t)N * max_out));
  if (c->levels) PD_TRY(alloc_trial_buffers(c, s, (size_t)N * max_in));
  PD_TRY(dev_alloc(c, &s.part, max_part));
  PD_TRY(dev_alloc(c, &s.p_slots, max_p_slots, false));
  s.n_slots = std::max<size_t>((size_t)c->n_sms * 4 * max_out, 8 * (size_t)ceil_div(N, SG_BM) * ceil_div(std::max(max_in, max_out), SG_BN) + 148 * 8 * 4);
  s.n_slots *= 2;                       // two halves: consecutive reductions of one layer use different halves
  PD_TRY(dev_alloc(c, &s.slots, s.n_slots));
  PD_TRY(dev_alloc(c, &s.red, (size_t)max_out + 8));
  if (c->use_tc) {
    if (!small) {                       // (small problems cut no tails)
      PD_TRY(dev_alloc(c, &s.tail_ws, (size_t)c->n_sms * TC_BM * TC_WIDE, false));
      s.tail_count = c->control + 4 + 8 * (size_t)c->L;
    }
    PD_TRY(dev_alloc(c, &s.amax_pool, (size_t)AMAX_POOL));
    s.pl_cap = e_max;
    PD_TRY(alloc_planes(c, s.pl_cap, &s.pl0));
    PD_TRY(alloc_planes(c, s.pl_cap, &s.pl1));
    PD_TRY(dev_alloc(c, &s.a_exp, 1));
  }

  // Further scratch: small problems are bound by the latency of their chain of launches, so their layers are worked on in
  // batches, every kernel launched once per batch; as much scratch as 4 GB pay for, at most one per layer.  Large ones keep two
  // lanes with a stream each (their scratch is gigabytes per lane, and more lanes gained nothing).
  const size_t lane_bytes = std::max<size_t>(c->bytes_handed_out - bytes_before_scratch, 1);
  const int affordable = (int)std::max<size_t>(2, (size_t(4) << 30) / lane_bytes);
  const bool one_lane = (cfg->flags & PDADMM_FLAG_ONE_LANE) != 0;
  c->tail_split = !small;
  c->grouped = batched && !one_lane;
  const int n_lanes = one_lane ? 1 : std::min(c->L, batched ? std::min(affordable, MAX_GROUP) : c->use_tc ? PDADMM_N_LANES : std::min(affordable, 64));
  for (int i = 1; i < n_lanes; ++i) {
    c->more_lanes.emplace_back(new Scratch());
    Scratch &x = *c->more_lanes.back();
    PD_CUDA(pool.take_stream(&x.own));
    x.st = c->grouped ? c->scr.st : x.own;
    PD_TRY(dev_alloc(c, &x.s1, e_max));
    PD_TRY(dev_alloc(c, &x.s2, (size_t)N * max_out));
    PD_TRY(dev_alloc(c, &x.part, max_part));
    PD_TRY(dev_alloc(c, &x.p_slots, max_p_slots, false));
    if (c->levels) PD_TRY(alloc_trial_buffers(c, x, (size_t)N * max_in));
    x.n_slots = s.n_slots;
    PD_TRY(dev_alloc(c, &x.slots, x.n_slots));
    PD_TRY(dev_alloc(c, &x.red, (size_t)max_out + 8));
    if (c->use_tc) {
      if (!small) {
        PD_TRY(dev_alloc(c, &x.tail_ws, (size_t)c->n_sms * TC_BM * TC_WIDE, false));
        x.tail_count = s.tail_count + (size_t)i * c->n_sms * 8;
      }
      x.pl_cap = s.pl_cap;
      PD_TRY(alloc_planes(c, x.pl_cap, &x.pl0));
      PD_TRY(alloc_planes(c, x.pl_cap, &x.pl1));
      PD_TRY(dev_alloc(c, &x.a_exp, 1));
    }
  }
  // Planes of r from one iteration to the next: worth their memory (the p-gradient's product would have to split
  // r first otherwise, 8 bytes per element), but nothing depends on them.  All or none, and at most 7/8 of what is free.
  if (c->use_tc) {
    size_t need = 0, free_bytes = 0, total = 0;
    for (int l = 0; l < c->L; ++l) need += (size_t)N * c->layers[l].ld_out * 4;
    const bool fits = need <= c->arena_cap - c->arena_used;            // (no question to the driver then, see DevicePool)
    if (!fits) PD_CUDA(cudaMemGetInfo(&free_bytes, &total));
    if (fits || need <= free_bytes / 8 * 7)
      for (int l = 0; l < c->L; ++l) PD_TRY(alloc_planes(c, (size_t)N * c->layers[l].ld_out, &c->layers[l].rp));
  }
  c->ev_p.resize(c->L);
  for (auto &e : c->ev_p) PD_CUDA(pool.take_event(false, &e));
  c->ev_lane.resize(std::max(n_lanes, 2));
  for (auto &e : c->ev_lane) PD_CUDA(pool.take_event(false, &e));

  // X = [H, A~ H, A~^2 H, ...] in the column blocks of p_1
  Layer &l0 = c->layers[0];
  {
    float *xb = sharded ? x_full : l0.p;
    for (int k = 1; k < c->n_blocks; ++k)
      launch_spmm(st, c->row_ptr, c->col_idx, c->csr_val, (int)Ntot, xb + (size_t)(k - 1) * c->d, xb + (size_t)k * c->d,
                  c->d, l0.ld_in);
    if (sharded)
      PD_CUDA(cudaMemcpyAsync(l0.p, x_full + (size_t)node0 * l0.ld_in, (size_t)N * l0.ld_in * 4, cudaMemcpyDeviceToDevice, st));
  }

  PD_TRY(feasible_start(c, 0));
  PD_CUDA(cudaStreamSynchronize(st));
  PD_CUDA(cudaGetLastError());
  c->r_valid = true;                        // z = W p + b exactly by construction, r = 0 (allocated as zero)
  c->w_planes_valid = true;
  c->amax_p_valid = true;
  c->x_planes_valid = true;
  c->q_implied = c->q_free;                 // q = f(z), u = 0
  c->r_sums_valid = true;                   // (allocated as zero, too)
  c->cold = 2 * c->L;
  for (const Layer &ly : c->layers)
    for (int i = 0; i < 2; ++i) {            // r_l and g_l: of an element, the column tiles of the product that reads it
      const size_t e = (size_t)N * (i ? ly.ld_in : ly.ld_out), uses = (size_t)ceil_div(i ? ly.n_out : ly.n_in, TC_BN);
      c->wide |= c->use_tc && e < CHECK_PLANES_FROM && e * uses >= CHECK_PLANES_USES;
    }
  c->launches = 0;
  c->comm_bytes = 0;
  return PDADMM_OK;
}

static void destroy(pdadmm_ctx *c) {
  if (!c) return;
  cudaSetDevice(c->device);
  for (int i = 0; i <= (int)c->more_lanes.size(); ++i) {            // everything of this context runs on streams of its own
    const cudaStream_t st = i == 0 ? c->scr.own : c->more_lanes[i - 1]->own;
    if (st != nullptr) cudaStreamSynchronize(st);
  }
  for (auto &r : c->prof) { cudaEventDestroy(r.e0); cudaEventDestroy(r.e1); }
  for (auto e : c->ev_pool) cudaEventDestroy(e);
  if (c->iter_graph) cudaGraphExecDestroy(c->iter_graph);
  DevicePool &pool = device_pool(c->device);
  pool.give(c->allocs);
  ctx_pinned_pool().give(c->h_pinned);
  pool.give_event(true, c->ev_begin);
  pool.give_event(true, c->ev_end);
  for (auto e : c->ev_p) pool.give_event(false, e);
  for (auto e : c->ev_lane) pool.give_event(false, e);
  for (int i = 0; i <= (int)c->more_lanes.size(); ++i) {
    pd::Scratch &x = i == 0 ? c->scr : *c->more_lanes[i - 1];
    pool.give_event(false, x.ev_flag);
    pool.give_stream(x.own);
  }
  delete c;
}

}  // namespace pd

// ======================================================================================================
// C ABI
// ======================================================================================================
using namespace pd;

extern "C" const char *pdadmm_last_error(void) { return err_text().c_str(); }

extern "C" int pdadmm_init(const pdadmm_config *cfg, pdadmm_ctx **out) { return pdadmm_init_sharded(cfg, nullptr, out); }

extern "C" int pdadmm_comm_bytes(pdadmm_ctx *c, int64_t *bytes) {
  if (!c || !bytes) return fail(PDADMM_EINVAL, "null argument");
  *bytes = c->comm_bytes;
  return PDADMM_OK;
}

extern "C" int pdadmm_init_sharded(const pdadmm_config *cfg, const pdadmm_shard *shard, pdadmm_ctx **out) {
  if (!out) return fail(PDADMM_EINVAL, "out is null");
  *out = nullptr;
  PD_TRY(check_config(cfg));
  if (shard != nullptr) {
    if (shard->node_begin < 0 || shard->node_count < 1 || shard->node_begin + shard->node_count > cfg->n_nodes)
      return fail(PDADMM_EINVAL, "shard [%lld, +%lld) is not inside the %lld nodes", (long long)shard->node_begin,
                  (long long)shard->node_count, (long long)cfg->n_nodes);
    if (shard->allreduce == nullptr && (shard->node_begin != 0 || shard->node_count != cfg->n_nodes))
      return fail(PDADMM_EINVAL, "a shard that is not the whole graph needs an allreduce callback");
  }
  int n_dev = 0;
  if (cudaGetDeviceCount(&n_dev) != cudaSuccess || n_dev == 0) {
    cudaGetLastError();
    return fail(PDADMM_ECUDA, "no CUDA device is available");
  }
  if (cfg->device < 0 || cfg->device >= n_dev || cfg->device >= MAX_DEVICES) return fail(PDADMM_EINVAL, "device %d does not exist", cfg->device);
  pdadmm_ctx *c = new (std::nothrow) pdadmm_ctx();
  if (!c) return fail(PDADMM_ENOMEM, "out of host memory");
  const int rc = guarded([&] { return build(c, cfg, shard); });
  if (rc != PDADMM_OK) { destroy(c); return rc; }
  *out = c;
  return PDADMM_OK;
}

static int refresh_p(pdadmm_ctx *c);
static int stored_q(pdadmm_ctx *c);

extern "C" int pdadmm_start_layers_from(pdadmm_ctx *c, int first_layer) {
  return guarded([&]() -> int {
    if (!c) return fail(PDADMM_EINVAL, "context is null");
    if (first_layer < 1 || first_layer > c->L) return fail(PDADMM_EINVAL, "first_layer must be in [1, %d]", c->L);
    PD_CUDA(cudaSetDevice(c->device));
    PD_TRY(refresh_p(c));
    PD_TRY(stored_q(c));
    PD_TRY(feasible_start(c, first_layer - 1));
    PD_CUDA(cudaStreamSynchronize(c->scr.st));
    PD_CUDA(cudaGetLastError());
    // the linear residual of the restarted layers is zero by construction; everything derived from the other tensors
    // (the residual of the kept layers, t, planes, largest magnitudes) is rebuilt by the next call that needs it
    forget_derived(c);
    return PDADMM_OK;
  });
}

extern "C" int pdadmm_product_forms(int64_t out[3]) {
  if (!out) return fail(PDADMM_EINVAL, "out is null");
  for (int i = 0; i < 3; ++i) out[i] = product_forms[i];
  return PDADMM_OK;
}

extern "C" int pdadmm_release_cached_memory(int device) {
  int n_dev = 0;
  if (cudaGetDeviceCount(&n_dev) != cudaSuccess || n_dev == 0) {
    cudaGetLastError();
    return fail(PDADMM_ECUDA, "no CUDA device is available");
  }
  if (device < 0 || device >= n_dev || device >= MAX_DEVICES) return fail(PDADMM_EINVAL, "device %d does not exist", device);
  PD_CUDA(cudaSetDevice(device));
  device_pool(device).trim();
  stage_pool().trim();
  ctx_pinned_pool().trim();
  return PDADMM_OK;
}

extern "C" int pdadmm_destroy(pdadmm_ctx *c) {
  destroy(c);
  return PDADMM_OK;
}

// p_l, l >= 2, from its codes where the fp32 values are older (integer operands)
static int refresh_p(pdadmm_ctx *c) {
  if (!c->p_stale) return PDADMM_OK;
  for (int l = 1; l < c->L; ++l) {
    Layer &ly = c->layers[l];
    const size_t n4 = (size_t)c->N * ly.ld_in / 4;
    codes_to_levels_kernel<<<ew_grid(n4), EW_THREADS, 0, c->scr.st>>>(ly.codes, c->code_bytes == 2, n4, ly.scale, ly.lo, ly.p);
  }
  PD_CUDA(cudaGetLastError());
  c->p_stale = false;
  c->amax_p_valid = false;          // no kernel of an iteration keeps max|p| of values that it does not write
  return PDADMM_OK;
}

// q of hidden layers first..last (0-based) as stored values, from z and u where these are newer
static int refresh_q(pdadmm_ctx *c, int first, int last) {
  for (int l = first; l <= last;) {
    Group<QOfZU> g;
    int n = 0;
    size_t n4_max = 0;
    double bytes = 0;
    for (; l <= last && n < MAX_GROUP; ++l) {
      Layer &ly = c->layers[l];
      if (!ly.q_stale) continue;
      g.l[n++] = QOfZU{ly.z, ly.u, ly.q, ly.n_out, (uint32_t)ly.ld_out / 4, (size_t)c->N * ly.ld_out / 4};
      n4_max = std::max(n4_max, g.l[n - 1].n4);
      bytes += 12.0 * c->N * ly.n_out;
      ly.q_stale = false;
    }
    if (n == 0) break;
    Launch k(c, KC_AXPY, c->scr.st, bytes, 0);
    q_of_z_and_u_kernel<<<dim3((unsigned)ew_grid(n4_max), (unsigned)n), EW_THREADS, 0, c->scr.st>>>(g, c->slope, c->nu);
  }
  PD_CUDA(cudaGetLastError());
  return PDADMM_OK;
}
// z, q or u is about to be set: q need not follow from the others any more
static int stored_q(pdadmm_ctx *c) {
  PD_TRY(refresh_q(c, 0, c->L - 2));
  c->q_implied = false;
  return PDADMM_OK;
}

// What products read beside the stored tensors: planes of W, largest magnitudes of p, planes of X.
static int ensure_operands(pdadmm_ctx *c) {
  if (!c->amax_p_valid || !c->t_valid || !c->r_valid) PD_TRY(refresh_p(c));
  if (!c->w_planes_valid) {
    for (auto &ly : c->layers) PD_TRY(refresh_W_planes(c, ly, c->scr.st));
    c->w_planes_valid = true;
  }
  // with integer operands max|p_l|, l >= 2, is read for a residual from scratch alone: not paid for after every look at p
  if (!c->amax_p_valid && (!c->int_operands || !c->r_valid || !c->x_planes_valid)) {
    for (auto &ly : c->layers) {
      const size_t n4 = (size_t)c->N * ly.ld_in / 4;
      PD_CUDA(cudaMemsetAsync(ly.amax_p, 0, sizeof(uint32_t), c->scr.st));
      Launch k(c, KC_AMAX, c->scr.st, 16.0 * n4, 0);
      absmax_kernel<<<ew_grid(n4), EW_THREADS, 0, c->scr.st>>>(ly.p, n4, ly.amax_p);
    }
    c->amax_p_valid = true;
  }
  if (!c->x_planes_valid && c->use_tc) {          // the planes of X follow the stored X
    Layer &l0 = c->layers[0];
    split_rows(c, c->scr.st, l0.p, (size_t)c->N, l0.n_in, l0.ld_in, l0.amax_p, l0.xp);
    c->x_planes_valid = true;
  }
  return PDADMM_OK;
}

static int ensure_residual(pdadmm_ctx *c) {
  PD_TRY(ensure_operands(c));
  if (!c->t_valid) {
    PD_TRY(refresh_q(c, 0, c->L - 2));
    for (int l = 1; l < c->L; ++l) {
      Layer &ly = c->layers[l];
      const Layer &pv = c->layers[l - 1];
      const size_t n4 = (size_t)c->N * ly.ld_in / 4;
      Launch k(c, KC_AXPY, c->scr.st, 16.0 * c->N * ly.n_in, 0);
      gradp_const_kernel<<<ew_grid(n4), EW_THREADS, 0, c->scr.st>>>(pv.u, ly.p, pv.q, c->rho, ly.t, n4);
    }
    c->t_valid = true;
  }
  if (c->r_valid) return PDADMM_OK;
  c->cold = 2 * c->L;
  for (int l = 0; l < c->L; ++l) PD_TRY(refresh_residual(c, c->layers[l], c->scr.st));
  c->r_valid = true;
  return PDADMM_OK;
}

// column sums that an iteration finds in place: of r, of p before its p-step
static int ensure_sums(pdadmm_ctx *c) {
  cudaStream_t st = c->scr.st;
  for (int l0 = 0; !c->r_sums_valid && l0 < c->L; l0 += MAX_GROUP) {
    Group<ColSum> g;
    int n = 0, blocks = 0, threads = 0;
    for (int l = l0; l < std::min(c->L, l0 + MAX_GROUP); ++l) {
      const Layer &ly = c->layers[l];
      g.l[n++] = ColSum{ly.r, r_rows(c, ly), nullptr};
      blocks = std::max(blocks, ly.r_blocks);
      threads = std::max(threads, row_share(ly.ld_out).threads);
    }
    Launch k(c, KC_SMALL, st, 0, 0);
    colsum_kernel<false><<<dim3((unsigned)blocks, (unsigned)n), threads, 0, st>>>(g, 0, 0);
  }
  c->r_sums_valid = true;
  if (c->p_sums_valid) return PDADMM_OK;
  if (!c->int_operands) PD_TRY(refresh_p(c));
  const int S = std::min(1 + (int)c->more_lanes.size(), MAX_GROUP);        // as many as have slots of their own
  for (int l0 = 0; l0 < c->L; l0 += S) {
    Group<ColSum> g;
    int n = 0, blocks = 0, threads = 0, ld = 0;
    for (int l = l0; l < std::min(c->L, l0 + S); ++l) {
      const Layer &ly = c->layers[l];
      g.l[n] = ColSum{ly.p, p_rows(c, ly, lane(c, n)), ly.p_sum, c->int_operands && l > 0 ? ly.codes : nullptr, ly.scale};
      blocks = std::max(blocks, g.l[n].rows.n_blocks);
      threads = std::max(threads, row_share(ly.ld_in).threads);
      ld = std::max(ld, ly.ld_in);
      ++n;
    }
    {
      Launch k(c, KC_SMALL, st, 0, 0);
      const dim3 grid((unsigned)blocks, (unsigned)n);
      if (c->int_operands) colsum_kernel<true><<<grid, threads, 0, st>>>(g, c->code_bytes == 2, c->neg_levels);
      else colsum_kernel<false><<<grid, threads, 0, st>>>(g, 0, 0);
    }
    Launch k(c, KC_SMALL, st, 0, 0);
    colsum_total_kernel<<<dim3((unsigned)ceil_div(ld, TOTAL_COLS), (unsigned)n), EW_THREADS, 0, st>>>(g);
  }
  PD_CUDA(cudaGetLastError());
  c->p_sums_valid = true;
  return PDADMM_OK;
}

static int finish_steps(pdadmm_ctx *c, bool hit_cap);

static int run_steps(pdadmm_ctx *c, int n_iters) {
  if (n_iters < 0) return fail(PDADMM_EINVAL, "n_iters is negative");
  PD_CUDA(cudaSetDevice(c->device));
  PD_CUDA(cudaEventRecord(c->ev_begin, c->scr.st));
  // The counters are zero already, unless a bounded wait expired in a product: its blocks then gave up between one arrival and
  // the last, and a count that starts from the leftover would take incomplete sums for complete ones.
  PD_CUDA(cudaMemsetAsync(c->control, 0, c->control_words * sizeof(int), c->scr.st));
  PD_TRY(ensure_residual(c));
  PD_TRY(ensure_sums(c));
  bool hit_cap = false;
  // pdADMM-G has no host decision inside an iteration, so after a first eager iteration the sequence of launches
  // is captured once into a CUDA graph and replayed; pointers and tensor maps never change in that mode.
  // pdADMM-G-Q reads the accept flag of every tau trial on the host, and per-kernel timing needs its events:
  // both stay eager.
  // A sharded context calls back for its sums over shards in the middle of an iteration: eager as well.
  const bool may_graph = c->levels == 0 && !c->profiling && !c->graph_failed && !(c->flags & PDADMM_FLAG_NO_GRAPH) &&
                         c->reduce == nullptr;
  int k = 0;
  for (; c->wide && c->cold > 0 && k < n_iters; ++k) {
    PD_TRY(iterate_once(c, &hit_cap));
    --c->cold;
  }
  // (the stored q is read in the first iteration after it was set: not the iteration that is captured)
  for (; c->q_free && !c->q_implied && k < n_iters; ++k) PD_TRY(iterate_once(c, &hit_cap));
  if (may_graph && c->iter_graph == nullptr && n_iters - k > 1) {
    PD_TRY(iterate_once(c, &hit_cap));
    ++k;
    const int64_t before = c->launches;
    cudaGraph_t g = nullptr;
    if (cudaStreamBeginCapture(c->scr.st, cudaStreamCaptureModeThreadLocal) == cudaSuccess) {
      const int rc = guarded([&] { return iterate_once(c, &hit_cap); });      // the capture has to be ended whatever happens
      const cudaError_t e = cudaStreamEndCapture(c->scr.st, &g);
      if (rc != PDADMM_OK || e != cudaSuccess || cudaGraphInstantiate(&c->iter_graph, g, 0) != cudaSuccess) {
        c->iter_graph = nullptr;
        c->graph_failed = true;
      }
      if (g) cudaGraphDestroy(g);
    } else {
      c->graph_failed = true;
    }
    cudaGetLastError();
    c->iter_graph_launches = c->launches - before;
    c->launches = before;                       // capturing launched nothing
  }
  for (; k < n_iters; ++k) {
    if (may_graph && c->iter_graph != nullptr) {
      will_iterate(c);
      PD_CUDA(cudaGraphLaunch(c->iter_graph, c->scr.st));
      iterated(c);
      c->launches += c->iter_graph_launches;
    } else {
      PD_TRY(iterate_once(c, &hit_cap));
    }
  }
  return finish_steps(c, hit_cap);
}

extern "C" int pdadmm_step(pdadmm_ctx *c, int n_iters) {
  if (!c) return fail(PDADMM_EINVAL, "context is null");
  const int rc = guarded([&] { return run_steps(c, n_iters); });
  // an iteration that was abandoned half way may have work on lanes that the main stream has not joined
  if (rc == PDADMM_ENOMEM || rc == PDADMM_ECUDA)
    for (auto &x : c->more_lanes) cudaStreamSynchronize(x->own);
  // and W and b are ahead of the residual, which the z-update brings after them
  if (c->in_iteration) forget_derived(c);
  c->in_iteration = false;
  return rc;
}

// What the iterations left in the error words.
static int finish_steps(pdadmm_ctx *c, bool hit_cap) {
  PD_CUDA(cudaMemcpyAsync(c->h_pinned + 8, c->d_flag, 3 * sizeof(int), cudaMemcpyDeviceToHost, c->scr.st));
  PD_CUDA(cudaEventRecord(c->ev_end, c->scr.st));
  PD_CUDA(cudaStreamSynchronize(c->scr.st));
  PD_CUDA(cudaGetLastError());
  {
    float ms = 0.f;
    PD_CUDA(cudaEventElapsedTime(&ms, c->ev_begin, c->ev_end));
    c->last_step_ms = ms;
  }
  if (c->profiling) PD_TRY(prof_collect(c));
  if (c->h_pinned[9] != 0) {
    // nothing derived from the tensors was finished either
    forget_derived(c);
    return fail(PDADMM_ETIMEOUT, "a bounded wait inside a tensor-core product expired");
  }
  if (c->h_pinned[10] != 0) return fail(PDADMM_ENUMERIC, "a non-finite value reached the gradient norms: the state holds NaN or Inf");
  if (c->h_pinned[8] != 0)
    return fail(PDADMM_ENOTCONV, "the last-layer z solver did not converge on %d nodes", c->h_pinned[8]);
  if (hit_cap) return fail(PDADMM_ENOTCONV, "the tau search of a quantised p-update reached its trial cap");
  return PDADMM_OK;
}

// The objective's sums of every layer (parts: OBJ_ALL or OBJ_RESIDUALS) into h_results[4 l ..], and with OBJ_ALL the risk
// into h_results[4 L]; returns when they are there.
constexpr int OBJ_MAX_BLOCKS = 592;          // per layer: four per SM
static int read_objective(pdadmm_ctx *c, int parts) {
  cudaStream_t st = c->scr.st;
  const int wide = c->code_bytes == 2;
  for (int l0 = 0; l0 < c->L; l0 += OBJ_MAX_LAYERS) {
    ObjLayers o;
    const int n = std::min(OBJ_MAX_LAYERS, c->L - l0);
    size_t n4_max = 0;
    for (int i = 0; i < n; ++i) {
      const Layer &ly = c->layers[l0 + i];
      const bool hidden = l0 + i + 1 < c->L;
      const Layer *nx = hidden ? &c->layers[l0 + i + 1] : nullptr;
      o.l[i] = ObjLayer{ly.r, ly.z, hidden ? ly.q : nullptr, hidden ? ly.u : nullptr, hidden ? nx->p : nullptr, hidden && c->levels ? nx->codes : nullptr,
                        (size_t)c->N * ly.ld_out / 4, hidden ? nx->scale : 0.f, hidden ? nx->lo : 0.f,
                         hidden && c->slope == ACT_SIGMOID ? ly.n_out : 0, (uint32_t)ly.ld_out / 4};
      n4_max = std::max(n4_max, o.l[i].n4);
    }
    // all layers side by side: the hidden ones, which are nearly all of the work, have one round of blocks, as many slots as the buffer holds
    const int n_hidden = std::max(1, l0 + n == c->L ? n - 1 : n);
    const size_t fit = std::min<size_t>(OBJ_MAX_BLOCKS, c->scr.n_slots / (4 * (size_t)n));
    const int per_layer = (int)std::max<size_t>(1, std::min(fit, std::min<size_t>((n4_max + EW_THREADS - 1) / EW_THREADS,
                                                                                  (size_t)(obj_blocks_per_sm(parts, c->table_size > 0) * c->n_sms / n_hidden))));
    const dim3 grid((unsigned)per_layer, (unsigned)n);
    double *out = c->h_results + 4 * (size_t)l0;
    auto launch = [&](auto parts_, auto implied, auto smooth) {
      objective_kernel<decltype(parts_)::value, decltype(implied)::value, decltype(smooth)::value>
          <<<grid, EW_THREADS, 0, st>>>(o, c->slope, c->nu, wide, c->scr.slots, c->done, out);
    };
    auto with = [&](auto parts_) {
      using T = std::true_type;
      using F = std::false_type;
      const bool smooth = c->table_size > 0;
      if (c->q_implied) { if (smooth) launch(parts_, T{}, T{}); else launch(parts_, T{}, F{}); }
      else { if (smooth) launch(parts_, F{}, T{}); else launch(parts_, F{}, F{}); }
    };
    if (parts == OBJ_ALL) with(std::integral_constant<int, OBJ_ALL>{});
    else with(std::integral_constant<int, OBJ_RESIDUALS>{});
  }
  if (parts == OBJ_ALL) {
    const Layer &ly = c->layers[c->L - 1];
    const int grid = (int)std::min<int64_t>(512, ceil_div(c->N, EW_THREADS));
    risk_kernel<<<grid, EW_THREADS, 0, st>>>(ly.z, c->labels, c->mask, (int)c->N, ly.n_out, ly.ld_out, c->scr.slots,
                                             c->ls_risk ? 1 : 0, c->done + OBJ_MAX_LAYERS, c->h_results + 4 * (size_t)c->L);
  }
  PD_CUDA(cudaGetLastError());
  PD_CUDA(cudaStreamSynchronize(st));
  return PDADMM_OK;
}

extern "C" int pdadmm_objective(pdadmm_ctx *c, double out[6]) {
  return guarded([&]() -> int {
    if (!c || !out) return fail(PDADMM_EINVAL, "null argument");
    PD_CUDA(cudaSetDevice(c->device));
    PD_TRY(ensure_residual(c));
    cudaStream_t st = c->scr.st;
    PD_TRY(read_objective(c, OBJ_ALL));
    double lin = 0, act = 0, dual = 0, pen = 0, R = c->h_results[4 * (size_t)c->L];
    for (int l = 0; l < c->L; ++l) {
      const double *h = c->h_results + 4 * (size_t)l;
      lin += h[0]; act += h[1]; dual += h[2]; pen += h[3];
    }
    if (c->reduce != nullptr) {                 // every component is a sum over nodes
      double h[5] = {R, lin, act, dual, pen};
      PD_CUDA(cudaMemcpyAsync(c->scr.red, h, sizeof h, cudaMemcpyHostToDevice, st));
      PD_TRY(shard_sum(c, st, c->scr.red, 5, 1));
      PD_CUDA(cudaMemcpyAsync(h, c->scr.red, sizeof h, cudaMemcpyDeviceToHost, st));
      PD_CUDA(cudaStreamSynchronize(st));
      R = h[0]; lin = h[1]; act = h[2]; dual = h[3]; pen = h[4];
    }
    out[0] = R; out[1] = 0.5 * c->nu * lin; out[2] = 0.5 * c->nu * act; out[3] = dual; out[4] = 0.5 * c->rho * pen;
    out[5] = out[0] + out[1] + out[2] + out[3] + out[4];
    return PDADMM_OK;
  });
}

extern "C" int pdadmm_predict(pdadmm_ctx *c, float *logits_out, int32_t *pred_out, int64_t counts_out[4]) {
  return guarded([&]() -> int {
    if (!c) return fail(PDADMM_EINVAL, "context is null");
    PD_CUDA(cudaSetDevice(c->device));
    cudaStream_t st = c->scr.st;
    PD_TRY(ensure_operands(c));
    // forward pass with the constraints enforced: activations alternate between the two scratch matrices
    const int N = (int)c->N;
    const float *in = c->layers[0].p;
    float *bufs[2] = {c->scr.s1, c->scr.s2};
    float *out = nullptr;
    const uint32_t *w_in = nullptr;            // max|activations| of the layer's input
    if (c->use_tc) {
      PD_TRY(amax_reset(c, st));               // one word per layer output, all from one pass through the pool
      w_in = c->layers[0].amax_p;
    }
    for (int l = 0; l < c->L; ++l) {
      Layer &ly = c->layers[l];
      out = bufs[l & 1];
      uint32_t *w_out = nullptr;
      if (c->use_tc) w_out = amax_take(c);
      EpiBiasAct epi{out, ly.ld_out, ly.b, l + 1 < c->L ? 1 : 0, c->slope, w_out};
      Operand P{in, ly.ld_in, w_in};
      if (l == 0 && c->use_tc) P = operand_X(ly);
      PD_TRY((gemm_nodes<false, EpiBiasAct>(c, KC_GEMM_RESID, st, {{N, ly.n_out, ly.n_in, P, operand_W(ly), epi, &c->scr}}, 0)));
      w_in = w_out;
      in = out;
    }
    const Layer &last = c->layers[c->L - 1];
    int *d_pred = reinterpret_cast<int *>(bufs[c->L & 1]);              // the scratch matrix the logits are not in
    unsigned long long *h_counts = reinterpret_cast<unsigned long long *>(c->h_results);
    argmax_kernel<<<(int)std::min<int64_t>(1184, ceil_div(N, EW_THREADS)), EW_THREADS, 0, st>>>(
        out, c->labels, c->mask, N, last.n_out, last.ld_out, d_pred, c->counts, c->done, c->d_flag + 1, h_counts);
    PD_CUDA(cudaGetLastError());
    const size_t row = (size_t)last.n_out * 4, lg_bytes = logits_out ? (size_t)N * row : 0, pr_bytes = pred_out ? (size_t)N * 4 : 0;
    const bool staged = lg_bytes + pr_bytes <= STAGE_BYTES && !(logits_out && is_direct(logits_out)) && !(pred_out && is_direct(pred_out));
    char *stage = staged ? (char *)stage_pool().take() : nullptr;
    if (stage != nullptr) {       // small: everything packed into one page-locked block, one wait for the whole call
      cudaError_t e = cudaSuccess;
      if (logits_out) e = launch_pack(st, out, (size_t)last.ld_out * 4, row, (size_t)N, stage);
      if (pred_out && e == cudaSuccess) e = launch_pack(st, d_pred, pr_bytes, pr_bytes, 1, stage + lg_bytes);
      const cudaError_t w = cudaStreamSynchronize(st);
      if (e == cudaSuccess) e = w;
      if (e == cudaSuccess) {
        if (logits_out) memcpy(logits_out, stage, lg_bytes);
        if (pred_out) memcpy(pred_out, stage + lg_bytes, pr_bytes);
      }
      stage_pool().give(stage);
      PD_CUDA(e);
    } else {
      if (logits_out) PD_TRY(copy_rows(c->device, st, logits_out, out, (size_t)last.ld_out * 4, row, (size_t)N, true));
      if (pred_out) PD_TRY(copy_rows(c->device, st, pred_out, d_pred, pr_bytes, pr_bytes, 1, true));
      PD_CUDA(cudaStreamSynchronize(st));
    }
    if (counts_out)
      for (int i = 0; i < 4; ++i) counts_out[i] = (int64_t)h_counts[i];
    if (h_counts[4]) {
      PD_CUDA(cudaMemsetAsync(c->control, 0, c->control_words * sizeof(int), st));
      return fail(PDADMM_ETIMEOUT, "a bounded wait inside a tensor-core product expired");
    }
    return PDADMM_OK;
  });
}

extern "C" int pdadmm_residuals(pdadmm_ctx *c, double *per_layer_sq, int n) {
  return guarded([&]() -> int {
    if (!c) return fail(PDADMM_EINVAL, "context is null");
    if (n != c->L - 1 || (n > 0 && !per_layer_sq)) return fail(PDADMM_EINVAL, "n must be L-1 = %d", c->L - 1);
    PD_CUDA(cudaSetDevice(c->device));
    PD_TRY(ensure_residual(c));
    if (n > 0) PD_TRY(read_objective(c, OBJ_RESIDUALS));
    for (int l = 0; l + 1 < c->L; ++l) per_layer_sq[l] = c->h_results[4 * (size_t)l + 3];
    if (c->reduce != nullptr && n > 0) {
      if ((size_t)n > 8 + (size_t)c->layers[0].ld_out) return fail(PDADMM_EINVAL, "too many layers for the reduction buffer");
      PD_CUDA(cudaMemcpyAsync(c->scr.red, per_layer_sq, (size_t)n * 8, cudaMemcpyHostToDevice, c->scr.st));
      PD_TRY(shard_sum(c, c->scr.st, c->scr.red, (size_t)n, 1));
      PD_CUDA(cudaMemcpyAsync(per_layer_sq, c->scr.red, (size_t)n * 8, cudaMemcpyDeviceToHost, c->scr.st));
      PD_CUDA(cudaStreamSynchronize(c->scr.st));
    }
    return PDADMM_OK;
  });
}

// ---- tensors in and out -------------------------------------------------------------------------------------
struct TensorRef { void *ptr; size_t rows, width, ld, elem; bool settable; };

static int locate(pdadmm_ctx *c, int kind, int layer, TensorRef *t) {
  const int L = c->L;
  auto need = [&](int lo, int hi) {
    return (layer >= lo && layer <= hi) ? PDADMM_OK
                                        : fail(PDADMM_EINVAL, "layer %d is outside [%d, %d] for tensor kind %d", layer, lo, hi, kind);
  };
  const size_t N = (size_t)c->N;
  switch (kind) {
    case PDADMM_T_X: { Layer &y = c->layers[0]; *t = {y.p, N, (size_t)y.n_in, (size_t)y.ld_in, 4, true}; return PDADMM_OK; }
    case PDADMM_T_P: { PD_TRY(need(1, L)); Layer &y = c->layers[layer - 1]; *t = {y.p, N, (size_t)y.n_in, (size_t)y.ld_in, 4, true}; return PDADMM_OK; }
    case PDADMM_T_W: { PD_TRY(need(1, L)); Layer &y = c->layers[layer - 1]; *t = {y.W, (size_t)y.n_out, (size_t)y.n_in, (size_t)y.ld_in, 4, true}; return PDADMM_OK; }
    case PDADMM_T_B: { PD_TRY(need(1, L)); Layer &y = c->layers[layer - 1]; *t = {y.b, 1, (size_t)y.n_out, (size_t)y.ld_out, 4, true}; return PDADMM_OK; }
    case PDADMM_T_Z: { PD_TRY(need(1, L)); Layer &y = c->layers[layer - 1]; *t = {y.z, N, (size_t)y.n_out, (size_t)y.ld_out, 4, true}; return PDADMM_OK; }
    case PDADMM_T_Q: { PD_TRY(need(1, L - 1)); Layer &y = c->layers[layer - 1]; *t = {y.q, N, (size_t)y.n_out, (size_t)y.ld_out, 4, true}; return PDADMM_OK; }
    case PDADMM_T_U: { PD_TRY(need(1, L - 1)); Layer &y = c->layers[layer - 1]; *t = {y.u, N, (size_t)y.n_out, (size_t)y.ld_out, 4, true}; return PDADMM_OK; }
    case PDADMM_T_CODES: {
      if (!c->levels) return fail(PDADMM_EINVAL, "codes exist only in quantised mode");
      PD_TRY(need(2, L)); Layer &y = c->layers[layer - 1];
      *t = {y.codes, N, (size_t)y.n_in, (size_t)y.ld_in, (size_t)c->code_bytes, false}; return PDADMM_OK;
    }
    case PDADMM_T_TAU: { PD_TRY(need(2, L)); *t = {&c->layers[layer - 1].sc->tau, 1, 1, 1, 8, false}; return PDADMM_OK; }
    case PDADMM_T_THETA: { PD_TRY(need(1, L)); *t = {&c->layers[layer - 1].sc->theta, 1, 1, 1, 8, false}; return PDADMM_OK; }
    case PDADMM_T_TRIALS: { PD_TRY(need(2, L)); *t = {&c->layers[layer - 1].sc->trials, 1, 1, 1, 4, false}; return PDADMM_OK; }
    case PDADMM_T_CSR_ROWPTR: *t = {c->row_ptr, 1, (size_t)c->N_total + 1, (size_t)c->N_total + 1, 4, false}; return PDADMM_OK;
    case PDADMM_T_CSR_COLIDX: *t = {c->col_idx, 1, (size_t)c->nnz, (size_t)c->nnz, 4, false}; return PDADMM_OK;
    case PDADMM_T_CSR_VAL: *t = {c->csr_val, 1, (size_t)c->nnz, (size_t)c->nnz, 4, false}; return PDADMM_OK;
    default: return fail(PDADMM_EINVAL, "unknown tensor kind %d", kind);
  }
}

extern "C" int pdadmm_get_tensor(pdadmm_ctx *c, int kind, int layer, void *host_dst, size_t bytes) {
  return guarded([&]() -> int {
    if (!c || !host_dst) return fail(PDADMM_EINVAL, "null argument");
    PD_CUDA(cudaSetDevice(c->device));
    if (kind == PDADMM_T_QSCALE) {
      if (layer < 2 || layer > c->L || bytes != 4) return fail(PDADMM_EINVAL, "QSCALE: layer in [2, L], 4 bytes");
      memcpy(host_dst, &c->layers[layer - 1].scale, 4);
      return PDADMM_OK;
    }
    TensorRef t;
    PD_TRY(locate(c, kind, layer, &t));
    if (bytes != t.rows * t.width * t.elem)
      return fail(PDADMM_EINVAL, "tensor kind %d layer %d has %zu bytes, caller passed %zu", kind, layer,
                  t.rows * t.width * t.elem, bytes);
    if (kind == PDADMM_T_P) PD_TRY(refresh_p(c));
    if (kind == PDADMM_T_Q) PD_TRY(refresh_q(c, layer - 1, layer - 1));
    return copy_rows(c->device, c->scr.st, host_dst, t.ptr, t.ld * t.elem, t.width * t.elem, t.rows, true);
  });
}

// pdADMM-G-Q: the kernels read p_l (l >= 2, paper numbering) as its codes, so the two must always agree: the codes
// are taken from p_l and p_l becomes the levels of those codes (the same bits if it was on the level set already).
static int project_p_on_its_levels(pdadmm_ctx *c, int layer) {
  Layer &y = c->layers[layer - 1];
  const size_t n = (size_t)c->N * y.ld_in;
  quantize_kernel<<<ew_grid(n), EW_THREADS, 0, c->scr.st>>>(y.p, n, y.scale, y.lo, c->levels, y.p, y.codes, c->code_bytes == 2);
  if (c->int_operands) codes_to_plane_kernel<<<ew_grid(n / 4), EW_THREADS, 0, c->scr.st>>>(y.codes, c->code_bytes == 2, c->neg_levels, n / 4, y.p_plane);
  PD_CUDA(cudaGetLastError());
  PD_CUDA(cudaStreamSynchronize(c->scr.st));
  c->r_valid = c->r_sums_valid = c->p_sums_valid = false;
  c->amax_p_valid = false;
  c->t_valid = false;
  return PDADMM_OK;
}

extern "C" int pdadmm_set_tensor(pdadmm_ctx *c, int kind, int layer, const void *host_src, size_t bytes) {
  return guarded([&]() -> int {
    if (!c || !host_src) return fail(PDADMM_EINVAL, "null argument");
    PD_CUDA(cudaSetDevice(c->device));
    if (kind == PDADMM_T_QSCALE) {
      if (layer < 2 || layer > c->L || bytes != 4) return fail(PDADMM_EINVAL, "QSCALE: layer in [2, L], 4 bytes");
      float v;
      memcpy(&v, host_src, 4);
      if (!(v > 0.f)) return fail(PDADMM_EINVAL, "QSCALE must be positive");
      PD_TRY(refresh_p(c));
      c->layers[layer - 1].scale = v;
      c->layers[layer - 1].lo = -(float)c->neg_levels * v;
      if (c->levels) PD_TRY(project_p_on_its_levels(c, layer));       // p_l moves to the new level set
      return PDADMM_OK;
    }
    TensorRef t;
    if (kind == PDADMM_T_P) PD_TRY(refresh_p(c));
    PD_TRY(locate(c, kind, layer, &t));
    if (!t.settable) return fail(PDADMM_EINVAL, "tensor kind %d is read-only", kind);
    if (bytes != t.rows * t.width * t.elem)
      return fail(PDADMM_EINVAL, "tensor kind %d layer %d has %zu bytes, caller passed %zu", kind, layer,
                  t.rows * t.width * t.elem, bytes);
    if (kind == PDADMM_T_Z || kind == PDADMM_T_Q || kind == PDADMM_T_U) PD_TRY(stored_q(c));
    PD_TRY(copy_rows(c->device, c->scr.st, const_cast<void *>(host_src), t.ptr, t.ld * t.elem, t.width * t.elem, t.rows, false));
    if (kind == PDADMM_T_X || kind == PDADMM_T_P || kind == PDADMM_T_W || kind == PDADMM_T_B || kind == PDADMM_T_Z)
      c->r_valid = c->r_sums_valid = false;
    if (kind == PDADMM_T_X || kind == PDADMM_T_P) c->p_sums_valid = false;
    if (kind == PDADMM_T_W) c->w_planes_valid = false;
    if (kind == PDADMM_T_X || kind == PDADMM_T_P) c->amax_p_valid = false;
    if (kind == PDADMM_T_X || (kind == PDADMM_T_P && layer == 1)) c->x_planes_valid = false;
    if (kind == PDADMM_T_P || kind == PDADMM_T_Q || kind == PDADMM_T_U) c->t_valid = false;
    if (kind == PDADMM_T_P && c->levels && layer >= 2) PD_TRY(project_p_on_its_levels(c, layer));
    return PDADMM_OK;
  });
}

// ---- stand-alone entry points for single kernels ------------------------------------------------------------------
extern "C" int pdadmm_quantize(int device, const float *x, size_t n, float scale, float lo, int levels, void *codes_out,
                               float *p_out) {
  if (!x && n) return fail(PDADMM_EINVAL, "x is null");
  if (levels < 2 || levels > 65536 || !(scale > 0.f)) return fail(PDADMM_EINVAL, "levels in [2,65536], scale > 0");
  const size_t code_bytes = levels > 256 ? 2 : 1;
  if (n == 0) return PDADMM_OK;
  PD_CUDA(cudaSetDevice(device));
  float *dx = nullptr, *dp = nullptr;
  uint8_t *dc = nullptr;
  int rc = PDADMM_OK;
  auto body = [&]() -> int {
    PD_CUDA(cudaMalloc((void **)&dx, n * 4));
    PD_CUDA(cudaMalloc((void **)&dp, n * 4));
    PD_CUDA(cudaMalloc((void **)&dc, n * code_bytes));
    PD_CUDA(cudaMemcpy(dx, x, n * 4, cudaMemcpyHostToDevice));
    quantize_kernel<<<ew_grid(n), EW_THREADS>>>(dx, n, scale, lo, levels, dp, dc, code_bytes == 2);
    PD_CUDA(cudaGetLastError());
    PD_CUDA(cudaDeviceSynchronize());
    if (p_out) PD_CUDA(cudaMemcpy(p_out, dp, n * 4, cudaMemcpyDeviceToHost));
    if (codes_out) PD_CUDA(cudaMemcpy(codes_out, dc, n * code_bytes, cudaMemcpyDeviceToHost));
    return PDADMM_OK;
  };
  rc = body();
  cudaFree(dx); cudaFree(dp); cudaFree(dc);
  return rc;
}

extern "C" int pdadmm_spmm(int device, int64_t n_rows, const int32_t *row_ptr, const int32_t *col_idx, const float *val,
                           const float *x, int32_t width, float *y_out) {
  if (n_rows < 0 || width < 1 || !row_ptr || !y_out || !x) return fail(PDADMM_EINVAL, "bad argument");
  if (n_rows == 0) return PDADMM_OK;
  if (n_rows > INT32_MAX / 2) return fail(PDADMM_EINVAL, "too many rows");
  if (row_ptr[0] != 0) return fail(PDADMM_EINVAL, "row_ptr[0] must be 0");
  for (int64_t i = 0; i < n_rows; ++i)
    if (row_ptr[i + 1] < row_ptr[i]) return fail(PDADMM_EINVAL, "row_ptr decreases at row %lld", (long long)i);
  const int64_t nnz = row_ptr[n_rows];
  if (nnz > 0 && (!col_idx || !val)) return fail(PDADMM_EINVAL, "col_idx or val is null");
  for (int64_t e = 0; e < nnz; ++e)
    if (col_idx[e] < 0 || col_idx[e] >= n_rows) return fail(PDADMM_EINVAL, "column index %lld out of range", (long long)e);
  PD_CUDA(cudaSetDevice(device));
  int *drp = nullptr, *dci = nullptr;
  float *dv = nullptr, *dx = nullptr, *dy = nullptr;
  auto body = [&]() -> int {
    PD_CUDA(cudaMalloc((void **)&drp, (n_rows + 1) * 4));
    PD_CUDA(cudaMalloc((void **)&dci, std::max<int64_t>(nnz, 1) * 4));
    PD_CUDA(cudaMalloc((void **)&dv, std::max<int64_t>(nnz, 1) * 4));
    PD_CUDA(cudaMalloc((void **)&dx, (size_t)n_rows * width * 4));
    PD_CUDA(cudaMalloc((void **)&dy, (size_t)n_rows * width * 4));
    PD_CUDA(cudaMemcpy(drp, row_ptr, (n_rows + 1) * 4, cudaMemcpyHostToDevice));
    if (nnz) {
      PD_CUDA(cudaMemcpy(dci, col_idx, nnz * 4, cudaMemcpyHostToDevice));
      PD_CUDA(cudaMemcpy(dv, val, nnz * 4, cudaMemcpyHostToDevice));
    }
    PD_CUDA(cudaMemcpy(dx, x, (size_t)n_rows * width * 4, cudaMemcpyHostToDevice));
    launch_spmm(0, drp, dci, dv, (int)n_rows, dx, dy, width, width);
    PD_CUDA(cudaGetLastError());
    PD_CUDA(cudaDeviceSynchronize());
    PD_CUDA(cudaMemcpy(y_out, dy, (size_t)n_rows * width * 4, cudaMemcpyDeviceToHost));
    return PDADMM_OK;
  };
  const int rc = body();
  cudaFree(drp); cudaFree(dci); cudaFree(dv); cudaFree(dx); cudaFree(dy);
  return rc;
}

extern "C" int pdadmm_matmul(int device, int mode, int M, int N, int K, const float *A, const float *B, float *C,
                             double *sumsq, uint32_t flags) {
  return guarded([&]() -> int {
    if (mode < 0 || mode > 2 || M < 1 || N < 1 || K < 1 || !A || !B || !C || device >= MAX_DEVICES) return fail(PDADMM_EINVAL, "bad argument");
    PD_CUDA(cudaSetDevice(device));
    pdadmm_ctx *c = new (std::nothrow) pdadmm_ctx();
    if (!c) return fail(PDADMM_ENOMEM, "out of host memory");
    c->device = device;
    c->use_tc = (flags & PDADMM_FLAG_SIMT_GEMM) == 0;
    auto body = [&]() -> int {
      PD_CUDA(cudaDeviceGetAttribute(&c->n_sms, cudaDevAttrMultiProcessorCount, device));
      PD_CUDA(device_pool(device).take_stream(&c->scr.own));
      c->scr.st = c->scr.own;
      cudaStream_t st = c->scr.st;
      PD_TRY(dev_alloc(c, &c->d_flag, 4));
      if (c->use_tc) {
        PD_TRY(dev_alloc(c, &c->scr.tail_ws, (size_t)c->n_sms * TC_BM * TC_WIDE, false));
        PD_TRY(dev_alloc(c, &c->scr.tail_count, (size_t)c->n_sms * 8));
      }
      // operand shapes as stored: rows x cols
      const int a_rows = mode == 2 ? K : M, a_cols = mode == 2 ? M : K;
      const int b_rows = mode == 0 ? N : K, b_cols = mode == 0 ? K : N;
      const int lda = round_up(a_cols, 8), ldb = round_up(b_cols, 8), ldc = round_up(N, 4);
      float *dA, *dB, *dC, *part = nullptr;
      double *slots;
      Planes Ap, Bp;
      PD_TRY(dev_alloc(c, &dA, (size_t)a_rows * lda));
      PD_TRY(dev_alloc(c, &dB, (size_t)b_rows * ldb));
      PD_TRY(dev_alloc(c, &dC, (size_t)M * ldc));
      const int n_slots = 16 * (int)(ceil_div(M, 128) * ceil_div(N, 128)) + 2048;
      PD_TRY(dev_alloc(c, &slots, (size_t)n_slots));
      PD_TRY(upload_rows(c, st, dA, lda, A, a_cols, a_rows));
      PD_TRY(upload_rows(c, st, dB, ldb, B, b_cols, b_rows));
      Operand oA{dA, lda, nullptr}, oB{dB, ldb, nullptr};
      if (c->use_tc) {        // planes of both operands as they are stored
        PD_TRY(dev_alloc(c, &c->scr.amax_pool, (size_t)AMAX_POOL));
        PD_TRY(alloc_planes(c, (size_t)a_rows * lda, &Ap));
        PD_TRY(alloc_planes(c, (size_t)b_rows * ldb, &Bp));
        PD_TRY(amax_reserve(c, st, 2));
        split_rows(c, st, dA, (size_t)a_rows, a_cols, lda, amax_of(c, st, dA, (size_t)a_rows * lda / 4), Ap);
        split_rows(c, st, dB, (size_t)b_rows, b_cols, ldb, amax_of(c, st, dB, (size_t)b_rows * ldb / 4), Bp);
        oA = plane_operand(dA, lda, Ap);
        oB = plane_operand(dB, ldb, Bp);
      }
      double *res = slots + n_slots - 1;
      int *done;
      PD_TRY(dev_alloc(c, &done, 1));
      Step step;
      step.kind = STEP_SUM; step.sum = res;
      EpiStoreSumsq epi{dC, ldc};
      if (mode == 0) {
        Prod<EpiStoreSumsq> p{M, N, K, oA, oB, epi, &c->scr, slots, done, step};
        const Shape shape{M, N, K, 1};
        p.wide = choose_wide(c->n_sms, &shape, 1, false);
        PD_TRY((gemm_nodes<false, EpiStoreSumsq>(c, KC_GEMM_WG, st, {p}, 0)));
      } else if (mode == 1) {
        Prod<EpiStoreSumsq> p{M, N, K, oA, oB, epi, &c->scr, slots, done, step};
        const Shape shape{M, N, K, 1};
        p.wide = choose_wide(c->n_sms, &shape, 1, false);
        PD_TRY((gemm_nodes<true, EpiStoreSumsq>(c, KC_GEMM_WG, st, {p}, 0)));
      } else {
        const int split = (int)std::max<int64_t>(1, std::min<int64_t>(8, ceil_div(K, 64)));
        const int k_chunk = round_up((int)ceil_div(K, split), TC_BK);
        const int n_split = (int)ceil_div(K, k_chunk);
        PD_TRY(dev_alloc(c, &part, (size_t)n_split * M * ldc));
        if (!c->use_tc) {
          dim3 grid((unsigned)ceil_div(N, SG_BN), (unsigned)ceil_div(M, SG_BM), (unsigned)n_split);
          gemm_tn_kernel<<<grid, SG_THREADS, 0, st>>>(M, N, K, k_chunk, dA, lda, dB, ldb, part, ldc);
        } else {
          Prod<EpiStore> p{M, N, K, oA, oB, EpiStore{part, ldc}, &c->scr};
          p.n_split = n_split; p.k_chunk = k_chunk; p.stride = (size_t)M * ldc;
          const Shape shape{M, N, k_chunk, n_split};
          p.wide = choose_wide(c->n_sms, &shape, 1, false);
          PD_TRY(gemm_over_nodes(c, KC_GEMM_GRADW, st, {p}));
        }
        const size_t n4 = (size_t)M * ldc / 4;
        Group<GradWSum> g;
        g.l[0] = GradWSum{part, n_split, (uint32_t)n4, dC, nullptr, PlaneOut{nullptr, nullptr, nullptr}, slots, done, res, ew_grid(n4), 0, {}};
        reduce_gradW_kernel<<<dim3((unsigned)ew_grid(n4), 1u), EW_THREADS, 0, st>>>(g, 1.0f);
      }
      double h = 0;
      PD_CUDA(cudaMemcpyAsync(&h, res, 8, cudaMemcpyDeviceToHost, st));
      PD_TRY(copy_rows(device, st, C, dC, (size_t)ldc * 4, (size_t)N * 4, (size_t)M, true));
      int err = 0;
      PD_CUDA(cudaMemcpyAsync(&err, c->d_flag + 1, 4, cudaMemcpyDeviceToHost, st));
      PD_CUDA(cudaStreamSynchronize(st));
      PD_CUDA(cudaGetLastError());
      if (sumsq) *sumsq = h;
      if (err) return fail(PDADMM_ETIMEOUT, "a bounded wait inside a tensor-core product expired");
      return PDADMM_OK;
    };
    const int rc = body();
    destroy(c);
    return rc;
  });
}

// ---- self-test of the bounded waits ------------------------------------------------------------------------------
namespace pd {
// One warp waits, with the products' own wait routine, on an mbarrier that nothing ever arrives at.  The wait gives up
// after `limit_cycles`, raises the block's abort flag, and the block reports through the same error word as the
// products and returns by itself.
__global__ void bounded_wait_selftest_kernel(long long limit_cycles, int *error, long long *waited) {
  __shared__ uint64_t bar;
  __shared__ int abort_word;
  volatile int *abort_flag = &abort_word;
  if (threadIdx.x == 0) {
    *abort_flag = 0;
    ptx::mbar_init(&bar, 1);
    ptx::fence_barrier_init();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    const long long t0 = clock64();
    const bool ok = ptx::mbar_wait(&bar, 0, abort_flag, limit_cycles);
    *waited = clock64() - t0;
    if (!ok) atomicExch(error, 1);
  }
}
}  // namespace pd

extern "C" int pdadmm_selftest_bounded_wait(int device, long long limit_cycles, long long *waited_cycles) {
  if (limit_cycles < 1 || limit_cycles > 100000000ll) return fail(PDADMM_EINVAL, "limit_cycles must be in [1, 1e8]");
  PD_CUDA(cudaSetDevice(device));
  int *d_err = nullptr;
  auto body = [&]() -> int {
    PD_CUDA(cudaMalloc((void **)&d_err, 16));
    PD_CUDA(cudaMemset(d_err, 0, 16));
    bounded_wait_selftest_kernel<<<1, 32>>>(limit_cycles, d_err, reinterpret_cast<long long *>(d_err) + 1);
    PD_CUDA(cudaGetLastError());
    PD_CUDA(cudaDeviceSynchronize());
    long long h[2] = {0, 0};
    PD_CUDA(cudaMemcpy(h, d_err, 16, cudaMemcpyDeviceToHost));
    if (waited_cycles) *waited_cycles = h[1];
    if ((int)h[0] != 0) return fail(PDADMM_ETIMEOUT, "a bounded device-side wait expired after %lld cycles", h[1]);
    return PDADMM_OK;
  };
  const int rc = body();
  cudaFree(d_err);
  return rc;
}

// The words of a context as blocks that gave up in the middle of their products leave them (the error word set, counters between
// one arrival and the last, largest magnitudes of no number), then what pdadmm_step does after its last iteration.
extern "C" int pdadmm_selftest_expired_wait(pdadmm_ctx *c) {
  return guarded([&]() -> int {
    if (!c) return fail(PDADMM_EINVAL, "context is null");
    PD_CUDA(cudaSetDevice(c->device));
    std::vector<int> words(c->control_words, 1);
    words[0] = words[2] = 0;
    for (int l = 0; l < c->L; ++l)
      for (int i = 4; i < 8; ++i) words[4 + 8 * (size_t)l + i] = 0x7fc00000;
    PD_CUDA(cudaEventRecord(c->ev_begin, c->scr.st));
    PD_CUDA(cudaMemcpyAsync(c->control, words.data(), words.size() * sizeof(int), cudaMemcpyHostToDevice, c->scr.st));
    PD_CUDA(cudaStreamSynchronize(c->scr.st));
    return finish_steps(c, false);
  });
}

// ---- timing ----------------------------------------------------------------------------------------------------
extern "C" int pdadmm_profile(pdadmm_ctx *c, int enable) {
  return guarded([&]() -> int {
    if (!c) return fail(PDADMM_EINVAL, "context is null");
    PD_CUDA(cudaSetDevice(c->device));
    PD_TRY(prof_collect(c));
    for (int k = 0; k < KC_COUNT; ++k) { c->prof_ms[k] = 0; c->prof_n[k] = 0; c->prof_bytes[k] = 0; c->prof_flops[k] = 0; }
    c->profiling = enable != 0;
    return PDADMM_OK;
  });
}
extern "C" int pdadmm_profile_classes(void) { return KC_COUNT; }
extern "C" const char *pdadmm_profile_name(int k) { return (k >= 0 && k < KC_COUNT) ? kclass_names[k] : ""; }
extern "C" int pdadmm_profile_read(pdadmm_ctx *c, int k, double *ms, int64_t *launches, double *bytes, double *flops) {
  return guarded([&]() -> int {
    if (!c || k < 0 || k >= KC_COUNT) return fail(PDADMM_EINVAL, "bad argument");
    PD_TRY(prof_collect(c));
    if (ms) *ms = c->prof_ms[k];
    if (launches) *launches = c->prof_n[k];
    if (bytes) *bytes = c->prof_bytes[k];
    if (flops) *flops = c->prof_flops[k];
    return PDADMM_OK;
  });
}
extern "C" int pdadmm_time_augmentation(pdadmm_ctx *c, int reps, double *ms_per_hop, double *bytes_per_hop) {
  if (!c || reps < 1 || reps > 1000 || !ms_per_hop) return fail(PDADMM_EINVAL, "bad argument");
  if (c->n_blocks < 2) return fail(PDADMM_EINVAL, "the input has a single block: no sparse product to time");
  if (c->N != c->N_total) return fail(PDADMM_EINVAL, "a sharded context keeps only its own rows of X");
  PD_CUDA(cudaSetDevice(c->device));
  Layer &l0 = c->layers[0];
  cudaStream_t st = c->scr.st;
  // the first hop again, block 0 -> block 1 of X: the same kernel on the same data writes the same bits
  launch_spmm(st, c->row_ptr, c->col_idx, c->csr_val, (int)c->N, l0.p, l0.p + c->d, c->d, l0.ld_in);
  PD_CUDA(cudaEventRecord(c->ev_begin, st));
  for (int i = 0; i < reps; ++i)
    launch_spmm(st, c->row_ptr, c->col_idx, c->csr_val, (int)c->N, l0.p, l0.p + c->d, c->d, l0.ld_in);
  PD_CUDA(cudaEventRecord(c->ev_end, st));
  PD_CUDA(cudaStreamSynchronize(st));
  PD_CUDA(cudaGetLastError());
  float ms = 0.f;
  PD_CUDA(cudaEventElapsedTime(&ms, c->ev_begin, c->ev_end));
  *ms_per_hop = ms / reps;
  if (bytes_per_hop) *bytes_per_hop = (double)c->nnz * (8.0 + 4.0 * c->d) + 8.0 * (double)c->N * c->d;
  return PDADMM_OK;
}
extern "C" int pdadmm_last_step_ms(pdadmm_ctx *c, double *ms) {
  if (!c || !ms) return fail(PDADMM_EINVAL, "null argument");
  *ms = c->last_step_ms;
  return PDADMM_OK;
}
extern "C" int pdadmm_launches(pdadmm_ctx *c, int64_t *count) {
  if (!c || !count) return fail(PDADMM_EINVAL, "null argument");
  *count = c->launches;
  return PDADMM_OK;
}

#include "no_alloc.cuh"
