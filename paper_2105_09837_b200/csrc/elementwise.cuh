// Elementwise, reduction and per-node kernels of one pdADMM-G / pdADMM-G-Q iteration.
//
// All matrices are node-major [N][ld] float32 with ld a multiple of 4 and zero padding columns,
// so a matrix is processed as a flat array of N*ld/4 float4 values.  Every operation below maps
// zero padding to zero padding.  Sums are accumulated per block in double precision and written
// to a slot per block; a single-block kernel adds the slots in index order, so results do not
// depend on scheduling.
#pragma once

#include <cuda_fp16.h>

#include <algorithm>
#include <cmath>
#include <type_traits>

#include "common.cuh"
#include "planes.cuh"
#include "scalars.cuh"

namespace pd {

constexpr int EW_THREADS = 256;

// ---- largest magnitude of an array (see commit_amax) ---------------------------------------------
__global__ void __launch_bounds__(EW_THREADS)
absmax_kernel(const float *__restrict__ x, size_t n4, uint32_t *__restrict__ word) {
  uint32_t m = 0u;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x)
    m = max(m, abs_bits(reinterpret_cast<const float4 *>(x)[i]));
  commit_amax(m, word);
}

// Kernels of an iteration work on several layers at a time: blocks (x, y) = part x of layer y of the group.  What a layer's
// blocks do, and the order of its sums, depends on the layer alone.
constexpr int MAX_GROUP = 16;
template <class T> struct Group { T l[MAX_GROUP]; };
// The last block of a layer to arrive (`done`: zero before and after the kernel) has every slot that the others wrote.
__device__ __forceinline__ bool last_block(int *done, int n_blocks, int *sh) {
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    *sh = atomicAdd(done, 1) == n_blocks - 1;
    if (*sh) *done = 0;
  }
  __syncthreads();
  if (!*sh) return false;
  __threadfence();
  return true;
}

__device__ __forceinline__ float4 ld4(const float *p, size_t i) { return reinterpret_cast<const float4 *>(p)[i]; }
__device__ __forceinline__ float4 ld4f(const float *p, size_t i) { return reinterpret_cast<const float4 *>(p)[i]; }
__device__ __forceinline__ void st4(float *p, size_t i, float4 v) { reinterpret_cast<float4 *>(p)[i] = v; }
// Of group i of a matrix with rows of `groups` groups of four, the columns that are not padding; the group with the others at zero.  For
// what does not map zero to zero: f = sigmoid.
__device__ __forceinline__ int columns_inside(size_t i, uint32_t groups, int width) { return width - 4 * (int)(i % groups); }
__device__ __forceinline__ float4 keep_columns(float4 v, int inside) {
  return make_float4(inside > 0 ? v.x : 0.f, inside > 1 ? v.y : 0.f, inside > 2 ? v.z : 0.f, inside > 3 ? v.w : 0.f);
}

// ---- final, fixed-order reduction of per-block slots -------------------------------------------
// out[j] = sum_i slots[i * stride + j], j < n_out, i < n_slots.  One block of 256 threads: thread t adds the
// slots t, t+256, ... in that order, then the 256 partial sums are combined in a fixed tree, so the result
// does not depend on scheduling.
__global__ void __launch_bounds__(256)
reduce_slots_kernel(const double *__restrict__ slots, int n_slots, int stride, int n_out, double *__restrict__ out) {
  __shared__ double sh[256];
  for (int j = 0; j < n_out; ++j) {
    double s = 0.0;
    for (int i = threadIdx.x; i < n_slots; i += 256) s += slots[(size_t)i * stride + j];
    sh[threadIdx.x] = s;
    __syncthreads();
    for (int w = 128; w > 0; w >>= 1) {
      if (threadIdx.x < w) sh[threadIdx.x] += sh[threadIdx.x + w];
      __syncthreads();
    }
    if (threadIdx.x == 0) out[j] = sh[0];
    __syncthreads();
  }
}

// Quantisation to m uniform levels lo, lo + s, ... (Eq. "update p quantized", elementwise argmin):
// code = clamp(floor((x - lo)/s + 1/2), 0, m-1), value = lo + float(code) * s, every operation rounded once.
// The quotient comes from the rounded reciprocal, inv = 1/s, and two corrections by the exact remainder (Markstein 1990: a
// quotient within one unit in the last place, corrected once more with the correctly rounded reciprocal, is the correctly
// rounded one), floor from the sum with 2^23: with a division and conversions per element the trial kernel was bound
// by arithmetic (20 000 x 500, 9 layers, 256 levels: 255 us, 187 so; 170 000 x 1000: 529 and 364).  Spacings outside
// [1e-20, 1e20] are divided by.
struct Quantiser { float s, inv, lo, top; bool divide; };
__device__ __forceinline__ Quantiser make_quantiser(float s, float lo, float top) {
  return Quantiser{s, __frcp_rn(s), lo, top, !(s >= 1e-20f && s <= 1e20f)};
}
// the code as a float (an integer in [0, 65535]) and as an integer
__device__ __forceinline__ float quantise_code(const Quantiser &k, float x, unsigned &code) {
  const float d = __fsub_rn(x, k.lo);
  float q;
  if (k.divide) {
    q = __fdiv_rn(d, k.s);
  } else {
    const float q0 = __fmul_rn(d, k.inv);
    const float q1 = __fmaf_rn(__fmaf_rn(-q0, k.s, d), k.inv, q0);
    const float q2 = __fmaf_rn(__fmaf_rn(-q1, k.s, d), k.inv, q1);
    q = fabsf(q0) < 1e6f ? q2 : q0;                      // beyond: only the side counts (the products could overflow); NaN: code 0
  }
  const float v = fminf(fmaxf(__fadd_rn(q, 0.5f), 0.0f), k.top);
  const float t = __fadd_rn(v, 8388608.0f), n = __fsub_rn(t, 8388608.0f);      // n: nearest integer
  const bool above = n > v;
  code = (__float_as_uint(t) & 0x7fffffu) - (above ? 1u : 0u);
  return above ? n - 1.0f : n;
}
__device__ __forceinline__ float quantize_one(const Quantiser &k, float x, unsigned &code) {
  return __fadd_rn(k.lo, __fmul_rn(quantise_code(k, x, code), k.s));
}
// an integer below 2^23 as a float
__device__ __forceinline__ float float_of(unsigned i) { return __fsub_rn(__uint_as_float(0x4B000000u | i), 8388608.0f); }

// Four consecutive values of a quantised matrix from its codes: lo + code * s, rounded as quantize_one rounds them,
// i.e. bit for bit the stored values (1 or 2 bytes read per value instead of 4).
__device__ __forceinline__ float4 levels_of4(const void *__restrict__ codes, int wide_codes, size_t i, float s, float lo) {
  float c0, c1, c2, c3;
  if (wide_codes) {
    const ushort4 o = reinterpret_cast<const ushort4 *>(codes)[i];
    c0 = o.x; c1 = o.y; c2 = o.z; c3 = o.w;
  } else {
    const uchar4 o = reinterpret_cast<const uchar4 *>(codes)[i];
    c0 = o.x; c1 = o.y; c2 = o.z; c3 = o.w;
  }
  return make_float4(__fadd_rn(lo, __fmul_rn(c0, s)), __fadd_rn(lo, __fmul_rn(c1, s)), __fadd_rn(lo, __fmul_rn(c2, s)),
                     __fadd_rn(lo, __fmul_rn(c3, s)));
}

// Planes of a matrix that a kernel writes beside the fp32 values, for a later tensor-core product: the exponent was chosen
// before the kernel started (a bound or a prediction, see tc_planes_usable).  hi == nullptr: none are wanted.
struct PlaneOut { __half *hi, *lo; const int *exp; };
__device__ __forceinline__ void store_planes4(const PlaneOut &o, size_t i, float4 v, float scale) {
  uint2 h, l;
  tc_split4(v, scale, h, l);
  reinterpret_cast<uint2 *>(o.hi)[i] = h;
  reinterpret_cast<uint2 *>(o.lo)[i] = l;
}

// ---- blocks of rows -------------------------------------------------------------------------------
// Kernels that sum a matrix's columns beside what they do.  A block works on n_sub rows at a time and goes on to those n_blocks n_sub
// rows further (all blocks together walk through the matrix: with a run of rows of its own for every block the z-update of
// 20 000 x 500, 9 layers, took 5 to 8 % longer with 8-bit codes).  A thread owns a group of 4 columns (float4; several groups if the rows are
// longer than 1024) of one of the rows, so its sums stay in registers; the row subgroups' sums are combined in subgroup
// order, then written to slots[block][ld].
struct RowBlocks { int n_rows, ld, n_blocks; double *slots; int cols_per_pass, n_sub; };
// How a block's threads share rows of ld values: n_sub rows of cols_per_pass groups at a time, as many as leave the fewest lanes of the
// block's warps idle (rows of 352: 88 groups, 176 of 192 threads; with blocks of 256 the z-update of 7013 x 333 took 121 us, 103 of
// the previous pass without sums).
struct RowShare { int cols_per_pass, n_sub, threads; };
inline RowShare row_share(int ld) {
  const int groups = ld / 4, passes = (groups + EW_THREADS - 1) / EW_THREADS, cols = (groups + passes - 1) / passes;
  RowShare best{cols, 1, (cols + 31) / 32 * 32};
  for (int k = 2; k * cols <= EW_THREADS; ++k) {
    const int t = (k * cols + 31) / 32 * 32;
    if ((int64_t)k * cols * best.threads >= (int64_t)best.n_sub * cols * t) best = RowShare{cols, k, t};
  }
  return best;
}
// at(first float4, stride, count, column group, sums[4]) for every thread's column group; sh: EW_THREADS * 4 doubles.  All threads
// take part.
template <class F>
__device__ __forceinline__ void row_block_sums(const RowBlocks &y, int block, double *sh, F &&at) {
  const int n_groups = y.ld >> 2, cols_per_pass = y.cols_per_pass, n_sub = y.n_sub;
  const int sub = threadIdx.x / cols_per_pass, c0 = threadIdx.x % cols_per_pass;
  const int row0 = block * n_sub + sub, step = y.n_blocks * n_sub, n = row0 < y.n_rows ? (y.n_rows - row0 + step - 1) / step : 0;
  double *out = y.slots + (size_t)block * y.ld;
  if (sub < n_sub) {
    for (int cg = c0; cg < n_groups; cg += cols_per_pass) {
      double sum[4] = {0, 0, 0, 0};
      at((uint32_t)row0 * (uint32_t)n_groups + (uint32_t)cg, (uint32_t)step * (uint32_t)n_groups, n, cg, sum);
      double *dst = (n_sub > 1 ? sh + (size_t)sub * y.ld : out) + 4 * cg;
#pragma unroll
      for (int e = 0; e < 4; ++e) dst[e] = sum[e];
    }
  }
  if (n_sub > 1) {
    __syncthreads();
    for (int c = threadIdx.x; c < y.ld; c += blockDim.x) {
      double t = 0.0;
      for (int k = 0; k < n_sub; ++k) t += sh[(size_t)k * y.ld + c];
      out[c] = t;
    }
  }
}
__device__ __forceinline__ void add4(double (&s)[4], float4 v) {
  s[0] += (double)v.x; s[1] += (double)v.y; s[2] += (double)v.z; s[3] += (double)v.w;
}
// column sums of a stored matrix (X, the last layer's r; r and p after the start or after the caller has set a tensor)
struct ColSum { const float *x; RowBlocks rows; double *out; const void *codes /* may be null: read instead of x */; float scale; };
// CODES: of a p that the products read as integers, (code - neg_levels) scale, as quant_trial_kernel sums the next p (the fp32 values are
// rounded from it: the difference of two sums would not be zero where p does not change).
template <bool CODES>
__global__ void __launch_bounds__(EW_THREADS)
colsum_kernel(const __grid_constant__ Group<ColSum> group, int wide_codes, int neg_levels) {
  __shared__ double sh[EW_THREADS * 4];
  const ColSum &y = group.l[blockIdx.y];
  if ((int)blockIdx.x >= y.rows.n_blocks) return;
  const float *__restrict__ x = y.x;
  const void *__restrict__ codes = y.codes;
  row_block_sums(y.rows, (int)blockIdx.x, sh, [&](uint32_t i, uint32_t stride, int n, int, double (&sum)[4]) {
    if (CODES && codes != nullptr) {
      const int rows = n;
      unsigned up[4] = {0, 0, 0, 0};
#pragma unroll 4
      for (; n > 0; --n, i += stride) {
        if (wide_codes) {
          const uint2 w = reinterpret_cast<const uint2 *>(codes)[i];
          up[0] += w.x & 0xffffu; up[1] += w.x >> 16; up[2] += w.y & 0xffffu; up[3] += w.y >> 16;
        } else {
          const uint32_t w = reinterpret_cast<const uint32_t *>(codes)[i];
          up[0] += w & 0xffu; up[1] += (w >> 8) & 0xffu; up[2] += (w >> 16) & 0xffu; up[3] += w >> 24;
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) sum[e] = (double)y.scale * ((double)up[e] - (double)rows * neg_levels);
      return;
    }
#pragma unroll 4
    for (; n > 0; --n, i += stride) add4(sum, ld4(x, i));
  });
}
// The slots' totals of TOTAL_COLS columns, the first column at c0: total of column c0 + thread, valid in the block's first TOTAL_COLS
// threads.  Slot group g = thread / TOTAL_COLS adds the slots g, g + 16, ..., the groups are added in group order.
constexpr int TOTAL_COLS = 16, TOTAL_GROUPS = EW_THREADS / TOTAL_COLS;
__device__ __forceinline__ double slot_total(const double *__restrict__ slots, int n_slots, int ld, int c0, double (*sh)[TOTAL_COLS + 1]) {
  const int g = threadIdx.x / TOTAL_COLS, k0 = threadIdx.x % TOTAL_COLS, c = c0 + k0;
  double s = 0.0;
  for (int i0 = g; c < ld && i0 < n_slots; i0 += 16 * TOTAL_GROUPS) {      // sixteen loads on their way, the last ones too
    double v[16];
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = i0 + k * TOTAL_GROUPS < n_slots ? slots[(size_t)(i0 + k * TOTAL_GROUPS) * ld + c] : 0.0;
#pragma unroll
    for (int k = 0; k < 16; ++k) s += v[k];
  }
  sh[g][k0] = s;
  __syncthreads();
  double t = 0.0;
  if (g == 0)
    for (int k = 0; k < TOTAL_GROUPS; ++k) t += sh[k][k0];
  return t;
}
__global__ void __launch_bounds__(EW_THREADS)
colsum_total_kernel(const __grid_constant__ Group<ColSum> group) {
  __shared__ double sh[TOTAL_GROUPS][TOTAL_COLS + 1];
  const ColSum &y = group.l[blockIdx.y];
  const int c0 = (int)blockIdx.x * TOTAL_COLS, c = c0 + (int)threadIdx.x;
  const double t = slot_total(y.rows.slots, y.rows.n_blocks, y.rows.ld, c0, sh);
  if (threadIdx.x < TOTAL_COLS && c < y.rows.ld) y.out[c] = t;
}

// ---- p-step of pdADMM-G ----------------------------------------------------------------------------
// p+ = p - g/tau  (Eq. "update p") and the matching update of the linear residual, r <- r - (W g)/tau, in one launch (the
// elements of p first, then those of r), with the planes of both for the W-gradient and G p+.  16 bytes per element and
// matrix: read 8, write 4 and the planes 4.  (Separate passes that split r and p again cost 8 bytes more each, and the
// products that took them fp32 ran at 0.6 of their speed.)
struct PStep {
  float *p; const float *g; RowBlocks p_rows;        // with the column sums of p+ (for the b-update)
  float *r; const float *wg; uint32_t n4r;
  const float *inv_tau;
  PlaneOut pp, rp;
  uint32_t *amax_p, *amax_r;          // receive max|p|, max|r| (see commit_amax); may be null
  int n_blocks_r;                     // blocks of r, after those of p
};
__global__ void __launch_bounds__(EW_THREADS)
pstep_kernel(const __grid_constant__ Group<PStep> group) {
  __shared__ double sh[EW_THREADS * 4];
  const PStep &y = group.l[blockIdx.y];
  const int block = (int)blockIdx.x - y.p_rows.n_blocks;
  if (block >= y.n_blocks_r) return;
  const float a = *y.inv_tau;
  uint32_t m = 0u;
  // four groups per pass: eight loads in flight per thread
  auto pass = [&](float *__restrict__ out, const float *__restrict__ x, uint32_t i0, uint32_t step, int n, const PlaneOut &o, float scale, double *sum) {
    float4 v[4], w[4];
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (k < n) { v[k] = ld4(out, i0 + k * step); w[k] = ld4(x, i0 + k * step); }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      if (k >= n) continue;
      v[k].x = fmaf(-a, w[k].x, v[k].x); v[k].y = fmaf(-a, w[k].y, v[k].y);
      v[k].z = fmaf(-a, w[k].z, v[k].z); v[k].w = fmaf(-a, w[k].w, v[k].w);
      st4(out, i0 + k * step, v[k]);
      if (o.hi != nullptr) store_planes4(o, i0 + k * step, v[k], scale);
      if (sum != nullptr) { sum[0] += (double)v[k].x; sum[1] += (double)v[k].y; sum[2] += (double)v[k].z; sum[3] += (double)v[k].w; }
      m = max(m, abs_bits(v[k]));
    }
  };
  if (block < 0) {
    const float scale = y.pp.hi != nullptr ? tc_scale_of(*y.pp.exp) : 1.f;
    row_block_sums(y.p_rows, (int)blockIdx.x, sh, [&](uint32_t i, uint32_t stride, int n, int, double (&sum)[4]) {
      for (; n > 0; n -= 4, i += 4 * stride) pass(y.p, y.g, i, stride, n, y.pp, scale, sum);
    });
    if (y.amax_p != nullptr) commit_amax(m, y.amax_p);
    return;
  }
  const float scale = y.rp.hi != nullptr ? tc_scale_of(*y.rp.exp) : 1.f;
  const uint32_t stride = y.n_blocks_r * blockDim.x;
  for (uint32_t i = block * blockDim.x + threadIdx.x; i < y.n4r; i += 4 * stride)
    pass(y.r, y.wg, i, stride, (int)((y.n4r - i + stride - 1) / stride), y.rp, scale, nullptr);
  if (y.amax_r != nullptr) commit_amax(m, y.amax_r);
}

// ---- quantised trial step ------------------------------------------------------------------------
// x = p - g/tau; p_new = nearest level; d = p_new - p; codes; per-block sum of d^2.
// p lies on the level set, p = lo + code * scale bit for bit (quantize_one), so it is read as its 1- or 2-byte codes
// instead of as 4-byte values.
struct QuantTrial {
  const float *g; LayerScalars *sc; float scale, lo;
  float *p_new, *d /* may be null */;
  const void *codes_old; void *codes;      // of p; of p_new
  __half *pn_plane;                        // the new codes, counted from the level zero, as fp16 integers: operand plane of
                                           // p_new = (code - neg_levels) * scale; may be null
  __half *d_plane;                         // new code - old code as fp16 integers (operand plane of d)
  RowBlocks rows;                          // with the column sums of p_new (for the b-update)
  uint32_t *amax_p /* max|p_new|, may be null */, *amax_d /* max|d| */;
  double *slots; int *done;
};
// INTS: with integer planes (p+ and d exist as codes and planes of integers alone); WIDE: codes of two bytes.
template <bool INTS, bool WIDE>
__global__ void __launch_bounds__(EW_THREADS, INTS ? 5 : 3)
quant_trial_kernel(const __grid_constant__ Group<QuantTrial> group, int levels, int neg_levels) {
  __shared__ double red[EW_THREADS / 32];
  __shared__ double sh[EW_THREADS * 4];
  __shared__ int is_last;
  const QuantTrial &y = group.l[blockIdx.y];
  if ((int)blockIdx.x >= y.rows.n_blocks) return;
  const float scale = y.scale, lo = y.lo, inv_tau = y.sc->inv_tau, neg = (float)neg_levels;
  const Quantiser quant = make_quantiser(scale, lo, (float)(levels - 1));
  double ss = 0.0;
  unsigned long long steps2 = 0;                  // with integer planes d = (new code - old code) s: the sum of the squared integers
  uint32_t mp = 0u, md = 0u;
  row_block_sums(y.rows, (int)blockIdx.x, sh, [&](uint32_t i, uint32_t stride, int rows, int, double (&sum)[4]) {
    const float *__restrict__ g = y.g;
    const void *__restrict__ codes_old = y.codes_old;
    void *__restrict__ codes = y.codes;
    __half *__restrict__ pn_plane = y.pn_plane, *__restrict__ d_plane = y.d_plane;
    unsigned levels_up[4] = {0, 0, 0, 0};         // sums of the codes
#pragma unroll 2
    for (int n = rows; n > 0; --n, i += stride) {
      const float4 gv = ld4(g, i);
      unsigned o[4], c[4];
      if (WIDE) {
        const uint2 w = reinterpret_cast<const uint2 *>(codes_old)[i];
        o[0] = w.x & 0xffffu; o[1] = w.x >> 16; o[2] = w.y & 0xffffu; o[3] = w.y >> 16;
      } else {
        const uint32_t w = reinterpret_cast<const uint32_t *>(codes_old)[i];
        o[0] = w & 0xffu; o[1] = (w >> 8) & 0xffu; o[2] = (w >> 16) & 0xffu; o[3] = w >> 24;
      }
      const float gx[4] = {gv.x, gv.y, gv.z, gv.w};
      float of[4], cf[4], pv[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        of[e] = float_of(o[e]);
        pv[e] = __fadd_rn(lo, __fmul_rn(of[e], scale));
        cf[e] = quantise_code(quant, fmaf(-inv_tau, gx[e], pv[e]), c[e]);
      }
      if (WIDE)            // more than 256 levels: 16-bit codes
        reinterpret_cast<uint2 *>(codes)[i] = make_uint2(c[0] | c[1] << 16, c[2] | c[3] << 16);
      else
        reinterpret_cast<uint32_t *>(codes)[i] = c[0] | c[1] << 8 | c[2] << 16 | c[3] << 24;
      if constexpr (INTS) {
        // integers up to 2048 are exact in fp16: the planes hold the codes (counted from the level zero) and their change
        const __half2 a0 = __floats2half2_rn(cf[0] - neg, cf[1] - neg), a1 = __floats2half2_rn(cf[2] - neg, cf[3] - neg);
        const __half2 e0 = __floats2half2_rn(cf[0] - of[0], cf[1] - of[1]), e1 = __floats2half2_rn(cf[2] - of[2], cf[3] - of[3]);
        reinterpret_cast<uint2 *>(pn_plane)[i] = make_uint2(*reinterpret_cast<const uint32_t *>(&a0), *reinterpret_cast<const uint32_t *>(&a1));
        reinterpret_cast<uint2 *>(d_plane)[i] = make_uint2(*reinterpret_cast<const uint32_t *>(&e0), *reinterpret_cast<const uint32_t *>(&e1));
        uint32_t sq = 0;                          // at most 4 * 2047^2
#pragma unroll
        for (int e = 0; e < 4; ++e) { const int d = (int)c[e] - (int)o[e]; sq += (uint32_t)(d * d); levels_up[e] += c[e]; }
        steps2 += sq;
      } else {
        float nv[4], dv[4];
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          nv[e] = __fadd_rn(lo, __fmul_rn(cf[e], scale));
          dv[e] = nv[e] - pv[e];
          ss += (double)dv[e] * dv[e];
          sum[e] += (double)nv[e];
          mp = max(mp, abs_bits(nv[e])); md = max(md, abs_bits(dv[e]));
        }
        st4(y.p_new, i, make_float4(nv[0], nv[1], nv[2], nv[3]));
        st4(y.d, i, make_float4(dv[0], dv[1], dv[2], dv[3]));
      }
    }
    if constexpr (INTS) {                         // p_new = (code - neg) s
#pragma unroll
      for (int e = 0; e < 4; ++e) sum[e] = (double)scale * ((double)levels_up[e] - (double)rows * neg_levels);
    }
  });
  if (INTS) ss = (double)scale * (double)scale * (double)steps2;
  if (!INTS && y.amax_p != nullptr) { commit_amax(mp, y.amax_p); commit_amax(md, y.amax_d); }
  const double tot = block_sum_any(ss, red);
  if (threadIdx.x == 0) y.slots[blockIdx.x] = tot;
  if (!last_block(y.done, y.rows.n_blocks, &is_last)) return;
  double v = 0.0;
  for (int i = threadIdx.x; i < y.rows.n_blocks; i += blockDim.x) v += __ldcg(y.slots + i);
  v = block_sum_any(v, red);
  if (threadIdx.x == 0) y.sc->sum_d2 = v;
}

// Plain projection of an array (initial forward pass, pdadmm_quantize, pdadmm_set_tensor).
__global__ void __launch_bounds__(EW_THREADS)
quantize_kernel(const float *x, size_t n, float scale, float lo, int levels, float *p_out /* may be x itself */,
                void *__restrict__ codes_out, int wide_codes) {
  const Quantiser quant = make_quantiser(scale, lo, (float)(levels - 1));
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    unsigned c;
    const float v = quantize_one(quant, x[i], c);
    if (p_out) p_out[i] = v;
    if (codes_out) {
      if (wide_codes) reinterpret_cast<uint16_t *>(codes_out)[i] = (uint16_t)c;
      else reinterpret_cast<uint8_t *>(codes_out)[i] = (uint8_t)c;
    }
  }
}

// ---- operand planes of a quantised p from its codes ------------------------------------------------------------
// p = (code - neg_levels) s with at most 2048 levels: the fp16 plane of the integers is the whole operand (the products
// multiply by s).
__global__ void __launch_bounds__(EW_THREADS)
codes_to_plane_kernel(const void *__restrict__ codes, int wide_codes, int neg_levels, size_t n4, __half *__restrict__ plane) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    float c0, c1, c2, c3;
    if (wide_codes) {
      const ushort4 o = reinterpret_cast<const ushort4 *>(codes)[i];
      c0 = o.x; c1 = o.y; c2 = o.z; c3 = o.w;
    } else {
      const uchar4 o = reinterpret_cast<const uchar4 *>(codes)[i];
      c0 = o.x; c1 = o.y; c2 = o.z; c3 = o.w;
    }
    const float j = (float)neg_levels;
    const __half2 a = __floats2half2_rn(c0 - j, c1 - j), b = __floats2half2_rn(c2 - j, c3 - j);
    reinterpret_cast<uint2 *>(plane)[i] = make_uint2(*reinterpret_cast<const uint32_t *>(&a), *reinterpret_cast<const uint32_t *>(&b));
  }
}
// p itself from its codes, for whoever wants the values (pdadmm_get_tensor, a residual from scratch).
__global__ void __launch_bounds__(EW_THREADS)
codes_to_levels_kernel(const void *__restrict__ codes, int wide_codes, size_t n4, float s, float lo, float *__restrict__ p) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x)
    st4(p, i, levels_of4(codes, wide_codes, i, s, lo));
}

// ---- sums that no product completed ---------------------------------------------------------------------------
// The CUDA-core products leave one slot per block: fixed-order sum by one block (thread t adds slots t, t + FIN_THREADS, ...),
// then the step.
constexpr int FIN_THREADS = 256;
__global__ void __launch_bounds__(FIN_THREADS)
finish_sum_kernel(const double *__restrict__ slots, int n, Step step) {
  __shared__ double red[FIN_THREADS / 32];
  double v = 0.0;
  for (int i = threadIdx.x; i < n; i += FIN_THREADS) v += slots[i];
  v = block_sum<FIN_THREADS>(v, red);
  if (threadIdx.x == 0) finish_step(step, v);
}
// A context that owns part of the nodes: the step after its sums were added over the shards.
__global__ void run_step_kernel(Step step) { run_step(step); }

// ---- planes of a stored matrix -----------------------------------------------------------------------
// x [rows][ld] fp32 -> hi, lo [rows][ld] halves (the padding columns, zero in x, come out as zero), scaled by the exponent of
// max|x|, which goes to *exp_out: for operands whose planes no kernel wrote (the start, after pdadmm_set_tensor, the
// prediction's activations).  A thread converts eight consecutive values.
__global__ void __launch_bounds__(256)
rows_planes_kernel(const float *__restrict__ x, size_t n8, const uint32_t *__restrict__ amax, int *__restrict__ exp_out,
                   __half *__restrict__ hi, __half *__restrict__ lo /* may be null */) {
  const int e = tc_scale_exp(*amax);
  if (blockIdx.x == 0 && threadIdx.x == 0) *exp_out = e;
  const float scale = tc_pow2(e);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n8; i += (size_t)gridDim.x * blockDim.x) {
    uint4 h, l;
    tc_split8(reinterpret_cast<const float4 *>(x)[2 * i], reinterpret_cast<const float4 *>(x)[2 * i + 1], scale, h, l);
    reinterpret_cast<uint4 *>(hi)[i] = h;
    if (lo != nullptr) reinterpret_cast<uint4 *>(lo)[i] = l;
  }
}

// Planes whose exponent was chosen before the largest magnitude was known, in front of a product of a large matrix: normally
// nothing to do; if the scaling turned out unusable they are made again, with the exponent of *amax (which is what the product
// assumes then; *exp stays as it is).  (Inside the product, per output tile, it would take 5 to 10 times the product: a
// few such iterations at the start of a context of 20 000 x 500 cost more than all these launches.)
struct PlaneCheck { const float *x; uint32_t n8; const uint32_t *amax; const int *exp; __half *hi, *lo /* may be null */; };
__global__ void __launch_bounds__(256)
check_planes_kernel(const __grid_constant__ Group<PlaneCheck> group) {
  const PlaneCheck &y = group.l[blockIdx.y];
  if (tc_planes_usable(*y.amax, *y.exp)) return;
  const float scale = tc_pow2(tc_scale_exp(*y.amax));
  for (uint32_t i = blockIdx.x * 256u + threadIdx.x; i < y.n8; i += gridDim.x * 256u) {
    uint4 h, l;
    tc_split8(reinterpret_cast<const float4 *>(y.x)[2 * (size_t)i], reinterpret_cast<const float4 *>(y.x)[2 * (size_t)i + 1], scale, h, l);
    reinterpret_cast<uint4 *>(y.hi)[i] = h;
    if (y.lo != nullptr) reinterpret_cast<uint4 *>(y.lo)[i] = l;
  }
}

// ---- reduction of the split partial tiles of grad_W, scaling by nu, ||grad_W||^2 ------------------
// `remake`: if the predicted scaling of the planes turned out unusable (the first iterations of a context), the layer's last
// block makes them again with the exponent of *amax.  It costs one block 30 us for 500 x 500 and 130 us for 1000 x 1000, nothing
// otherwise; left to the product G p+, every output tile splits G again: 0.85 ms more per layer at 60 000 x 1000, 0.1 ms at
// 20 000 x 500 (remade_with_sum says when).  Larger matrices have check_planes_kernel.
struct GradWSum {
  const float *part; int n_split; uint32_t n4;
  float *G;
  uint32_t *amax /* max|G|, may be null */; PlaneOut planes;
  double *slots; int *done; double *sum /* ||G||^2 */; int n_blocks, remake;
  // Blocks after these: totals of the column sums of p+ (and their change) and of r, TOTAL_COLS columns each, which the W-step takes
  struct Totals { const double *slots; double *out, *change /* may be null */; int n_slots, ld, n_blocks; } totals[2];
};
__global__ void __launch_bounds__(EW_THREADS)
reduce_gradW_kernel(const __grid_constant__ Group<GradWSum> group, float nu) {
  __shared__ double red[EW_THREADS / 32];
  __shared__ int is_last;
  __shared__ double sh[TOTAL_GROUPS][TOTAL_COLS + 1];
  const GradWSum &y = group.l[blockIdx.y];
  int block = (int)blockIdx.x - y.n_blocks;
  if (block >= 0) {
    const int which = block < y.totals[0].n_blocks ? 0 : 1;
    if (which == 1) block -= y.totals[0].n_blocks;
    const GradWSum::Totals &t = y.totals[which];
    if (block >= t.n_blocks) return;
    const double v = slot_total(t.slots, t.n_slots, t.ld, TOTAL_COLS * block, sh);
    const int c = TOTAL_COLS * block + (int)threadIdx.x;
    if (threadIdx.x < TOTAL_COLS && c < t.ld) {
      if (t.change != nullptr) t.change[c] = v - t.out[c];
      t.out[c] = v;
    }
    return;
  }
  const float scale = y.planes.hi != nullptr ? tc_scale_of(*y.planes.exp) : 1.f;
  const float *__restrict__ part = y.part;
  const int n_split = y.n_split;
  double ss = 0.0;
  uint32_t m = 0u;
  for (uint32_t i = blockIdx.x * EW_THREADS + threadIdx.x; i < y.n4; i += y.n_blocks * EW_THREADS) {
    float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int s = 0; s < n_split; ++s) {
      const float4 v = ld4(part + (size_t)s * y.n4 * 4, i);
      a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
    }
    a.x *= nu; a.y *= nu; a.z *= nu; a.w *= nu;
    ss += (double)a.x * a.x + (double)a.y * a.y + (double)a.z * a.z + (double)a.w * a.w;
    st4(y.G, i, a);
    if (y.planes.hi != nullptr) store_planes4(y.planes, i, a, scale);
    m = max(m, abs_bits(a));
  }
  if (y.amax != nullptr) commit_amax(m, y.amax);        // the product G p+ checks the planes' scaling with it
  const double tot = block_sum<EW_THREADS>(ss, red);
  if (threadIdx.x == 0) y.slots[blockIdx.x] = tot;
  if (!last_block(y.done, y.n_blocks, &is_last)) return;
  const uint32_t top = y.remake ? __ldcg(y.amax) : 0u;           // (on its way while the slots are added)
  const bool usable = !y.remake || tc_planes_usable(top, *y.planes.exp);
  double v = 0.0;
  for (int i = threadIdx.x; i < y.n_blocks; i += EW_THREADS) v += __ldcg(y.slots + i);
  v = block_sum<EW_THREADS>(v, red);
  if (threadIdx.x == 0) *y.sum = v;
  if (usable) return;
  const float again = tc_pow2(tc_scale_exp(top));
#pragma unroll 8
  for (uint32_t i = threadIdx.x; i < y.n4; i += EW_THREADS)
    store_planes4(y.planes, i, __ldcg(reinterpret_cast<const float4 *>(y.G) + i), again);
}

// ---- what follows theta: W+ and b+ ----------------------------------------------------------------------------
// W+ = W - G/theta  (Eq. "update W"), with the planes of W+: a warp per row of W.  b+ = b - mean_j r  (Eq. "update b" with the step
// 1/(nu N), i.e. the exact minimiser), where r is the linear residual after the p- and the W-step:
//     sum_j r = sum_j (r as the last z-update left it) + W (sum_j p+ - sum_j p) - (G sum_j p+)/theta,
// from column sums that the kernels writing r and p kept, in double precision; the warp has the row of W and of G.  shift is the mean,
// which the z-update subtracts.  The sum of r is that of the stored values, so what the rounding of this iteration's products leaves
// of the mean is taken out by the next one.  (From sums of z and W+ p+ + b instead it piles up: the products round towards zero,
// 2e-7 of their size.)  Sums of r - (G p+)/theta itself took a pass of 12 bytes per element of r, 185 us of 2.9 ms at 20 000 x 500,
// 10 layers, and a launch more; the z-update applies G p+ now.
// `sums`: a context that owns part of the nodes leaves its part of the sum there instead (finalize_bias_kernel follows).
// `gp`: where G p+ is not left to the z-update, further blocks do r <- r - (G p+)/theta.
struct ThetaStep {
  float *W; const float *G; int n_out, ld;
  uint32_t *amax_W /* may be null */; PlaneOut Wp;
  const double *p_sum, *p_change, *r_sum;
  float *b, *shift;
  double *sums /* may be null */;
  const LayerScalars *sc;
  int n_blocks_w;
  float *r; const float *gp /* may be null */; uint32_t n4r; int n_blocks_r;
};
__global__ void __launch_bounds__(EW_THREADS)
theta_step_kernel(const __grid_constant__ Group<ThetaStep> group, double inv_n) {
  const ThetaStep &y = group.l[blockIdx.y];
  const float a = y.sc->inv_theta;
  if ((int)blockIdx.x < y.n_blocks_w) {
    const int row = (int)blockIdx.x * (EW_THREADS / 32) + (int)(threadIdx.x >> 5), lane = threadIdx.x & 31;
    const float scale = y.Wp.hi != nullptr ? tc_scale_of(*y.Wp.exp) : 1.f;
    uint32_t m = 0u;
    double dot = 0.0;
    if (row < y.n_out) {
      const float bias = y.b[row];
      const double rs = y.r_sum[row];
      const int n4 = y.ld >> 2;
#pragma unroll 2
      for (int k = lane; k < n4; k += 32) {
        const size_t i = (size_t)row * n4 + k;
        float4 v = ld4(y.W, i);
        const float4 g = ld4(y.G, i);
        const double2 p0 = reinterpret_cast<const double2 *>(y.p_sum)[2 * k], p1 = reinterpret_cast<const double2 *>(y.p_sum)[2 * k + 1];
        const double2 c0 = reinterpret_cast<const double2 *>(y.p_change)[2 * k], c1 = reinterpret_cast<const double2 *>(y.p_change)[2 * k + 1];
        dot += ((double)v.x * c0.x + (double)v.y * c0.y) + ((double)v.z * c1.x + (double)v.w * c1.y);
        dot -= (double)a * (((double)g.x * p0.x + (double)g.y * p0.y) + ((double)g.z * p1.x + (double)g.w * p1.y));
        v.x = fmaf(-a, g.x, v.x); v.y = fmaf(-a, g.y, v.y); v.z = fmaf(-a, g.z, v.z); v.w = fmaf(-a, g.w, v.w);
        st4(y.W, i, v);
        if (y.Wp.hi != nullptr) store_planes4(y.Wp, i, v, scale);
        m = max(m, abs_bits(v));
      }
      dot = warp_sum(dot);
      if (lane == 0) {
        const double sum = rs + dot;
        if (y.sums != nullptr) {
          y.sums[row] = sum;
        } else {
          const float mean = (float)(sum * inv_n);
          y.shift[row] = mean;
          y.b[row] = bias - mean;
        }
      }
    }
    if (y.amax_W != nullptr) commit_amax(m, y.amax_W);        // the next W-step bounds W by it
    return;
  }
  const int block = (int)blockIdx.x - y.n_blocks_w;
  if (block >= y.n_blocks_r) return;
#pragma unroll 4
  for (uint32_t i = block * EW_THREADS + threadIdx.x; i < y.n4r; i += y.n_blocks_r * EW_THREADS) {
    float4 v = ld4(y.r, i);
    const float4 g = ld4(y.gp, i);
    v.x = fmaf(-a, g.x, v.x); v.y = fmaf(-a, g.y, v.y); v.z = fmaf(-a, g.z, v.z); v.w = fmaf(-a, g.w, v.w);
    st4(y.r, i, v);
  }
}

// sum of squares (one slot per block) and largest magnitude of a weight-sized matrix
__global__ void __launch_bounds__(EW_THREADS)
sumsq_amax_kernel(const float *__restrict__ G, size_t n4, uint32_t *__restrict__ amax, double *__restrict__ slots) {
  __shared__ double red[EW_THREADS / 32];
  double ss = 0.0;
  uint32_t m = 0u;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    const float4 a = ld4(G, i);
    ss += (double)a.x * a.x + (double)a.y * a.y + (double)a.z * a.z + (double)a.w * a.w;
    m = max(m, abs_bits(a));
  }
  if (amax != nullptr) commit_amax(m, amax);
  const double tot = block_sum<EW_THREADS>(ss, red);
  if (threadIdx.x == 0) slots[blockIdx.x] = tot;
}

// The same from sums that were added over the contexts of all nodes.
__global__ void __launch_bounds__(EW_THREADS)
finalize_bias_kernel(const double *__restrict__ sums, int width, double inv_n, float *__restrict__ b, float *__restrict__ shift) {
  const int c = blockIdx.x * EW_THREADS + threadIdx.x;
  if (c >= width) return;
  const float m = (float)(sums[c] * inv_n);
  shift[c] = m;
  b[c] -= m;
}

// ---- z-, q-, u-update of a hidden layer, fused ----------------------------------------------------
// a = W+ p+ + b+ = (r - (G p+)/theta - shift) + z.  z+ by the ReLU closed form of Eq. "update z" (better of the two
// half-line minimisers; a tie keeps the non-positive one; slope > 0: leaky ReLU f(x) = slope x for x <= 0, whose
// minimiser on z <= 0 is (a + slope q + z)/(2 + slope^2)), q+ by Eq. "update q" (q_top >= 0: projected onto
// the level set of p_{l+1}, the variant at the end of Sec. "Quantization Extension"), residual p_{l+1} - q+,
// u+ by Eq. "update u", the linear residual of the next iteration r = a - z+, t_{l+1} = u+ + rho (p_{l+1} - q+),
// the part of the next p-gradient that does not involve a product, and the column sums of that r for the next b-update.
//
// q is not kept: the minimiser of the q-subproblem satisfies u+ = nu (q+ - f(z+))  (Lemma "q_opt"), so q = f(z) + u/nu, and
//     u+ = nu/(rho + nu) (rho (p - f(z+)) + u),   q+ = f(z+) + u+/nu
// with relative errors of a few roundings of their terms, the cancelling difference p - q+ of u + rho (p - q+) avoided.  `q` is read
// only in the first iteration after a caller has set z, q or u (which need not satisfy it), and written then; its memory holds G p+ otherwise.
// 40 bytes per element with that, 56 with q, and r - (G p+)/theta as a pass before: 20 000 x 500, 9 layers 825 us in two
// kernels.  A q on the level set does not satisfy it: q_out is written and read.
struct Zqu {
  float *r, *z; const float *gp /* null: r has it */; const float *q /* null: from z and u */; float *q_out /* null: not kept */;
  float *u; const float *p_next, *shift; float *t_next;
  const void *codes_next;                 // pdADMM-G-Q: codes of p_next, read instead of it
  float q_scale, q_lo; RowBlocks rows; int width;
  uint32_t *amax_r;                       // max|r| (see commit_amax); may be null
  PlaneOut rp;                            // planes of r for the coming p-gradient
  const LayerScalars *sc;
};
// x * (num/den), the factor to two terms: a rounded one is the same error in the same direction for every element and iteration.  (With
// fl(1/3), which is 3e-8 high, the distance of b from the 64-bit oracle was 7.2e-6 and 1.00e-5 in two forms of the q-update, the first
// biased the other way, after 40 iterations of 1500 x 256, 6 layers; 7.6e-7 so, and half to nine tenths elsewhere.)
struct TwoTerm { float hi, lo; };
__host__ __device__ constexpr TwoTerm two_term(double num, double den) {
  return TwoTerm{(float)(num / den), (float)(num / den - (double)(float)(num / den))};
}
__device__ __forceinline__ float times(float x, TwoTerm f) { return fmaf(x, f.hi, f.lo != 0.0f ? x * f.lo : 0.0f); }
struct ZquParams { float rho, nu, slope; TwoTerm inv_neg /* 1/(2 + slope^2) */; float q_top; int wide_codes; float t_lo, t_step; int T, table_even; };
// what follows z+ = zz with f = f(z+): q, u and t
template <bool LEVELS>                      // LEVELS: q may be kept on a level set
struct QuUpdate {
  float rho, nu, inv_nu, inv_rn, u_factor, q_top;
  Quantiser quant;
  __device__ __forceinline__ QuUpdate(const ZquParams &p, float q_scale, float q_lo)
      : rho(p.rho), nu(p.nu), inv_nu(1.0f / p.nu), inv_rn(1.0f / (p.rho + p.nu)), u_factor(p.nu / (p.rho + p.nu)), q_top(p.q_top),
        quant(LEVELS ? make_quantiser(q_scale, q_lo, p.q_top) : Quantiser{}) {}
  __device__ __forceinline__ void operator()(float f, float p, float u, float &qn, float &un, float &tn) const {
    if (LEVELS && q_top >= 0.0f) {
      unsigned code;
      qn = quantize_one(quant, (rho * p + u + nu * f) * inv_rn, code);
      un = fmaf(rho, p - qn, u);
    } else {
      un = u_factor * fmaf(rho, p - f, u);
      qn = fmaf(un, inv_nu, f);
    }
    tn = fmaf(rho, p - qn, un);
  }
};
// GENERAL: q is read, or kept, or G p+ is in r already.  (One kernel for all took 74 registers, three blocks per SM.)
template <bool CODES, bool GENERAL>
__global__ void __launch_bounds__(EW_THREADS, GENERAL ? 3 : 4)
zqu_kernel(const __grid_constant__ Group<Zqu> group, const __grid_constant__ ZquParams prm) {
  __shared__ double sh[EW_THREADS * 4];
  const Zqu &y = group.l[blockIdx.y];
  if ((int)blockIdx.x >= y.rows.n_blocks) return;
  float *__restrict__ r = y.r, *__restrict__ z = y.z, *__restrict__ q_out = y.q_out, *__restrict__ u = y.u, *__restrict__ t_next = y.t_next;
  const float *q_in = GENERAL ? y.q : nullptr;     // (may be q_out)
  const float *__restrict__ gp = y.gp, *__restrict__ p_next = y.p_next;
  const void *__restrict__ codes_next = y.codes_next;
  const float slope = prm.slope, q_scale = y.q_scale, q_lo = y.q_lo, theta = !GENERAL || gp != nullptr ? y.sc->inv_theta : 0.f;
  const float scale = y.rp.hi != nullptr ? tc_scale_of(*y.rp.exp) : 1.f;
  const QuUpdate<GENERAL> update(prm, q_scale, q_lo);
  constexpr TwoTerm third = two_term(1.0, 3.0);
  const TwoTerm inv_neg = prm.inv_neg;
  uint32_t mr = 0u;
  row_block_sums(y.rows, (int)blockIdx.x, sh, [&](uint32_t i, uint32_t stride, int n, int cg, double (&sum)[4]) {
    const float4 sh4 = ld4(y.shift, cg);
    for (; n > 0; --n, i += stride) {
      float4 rv = ld4(r, i);
      const float4 zv = ld4(z, i), uv = ld4(u, i);
      float4 gv = make_float4(0.f, 0.f, 0.f, 0.f), qv = gv;
      if (!GENERAL || gp != nullptr) gv = ld4(gp, i);
      if (GENERAL && q_in != nullptr) qv = ld4(q_in, i);
      const float4 pv = CODES ? levels_of4(codes_next, prm.wide_codes, i, q_scale, q_lo) : ld4(p_next, i);
      float4 zn, qn, un, rn, tn;
#define PD_ZQU(f)                                                                   \
      {                                                                             \
        const float zo = zv.f, qo = GENERAL && q_in != nullptr ? qv.f : fmaf(uv.f, update.inv_nu, zo > 0.0f ? zo : slope * zo); \
        const float a = (fmaf(-theta, gv.f, rv.f) - sh4.f) + zo;                    \
        const float zneg = fminf(times(fmaf(slope, qo, a) + zo, inv_neg), 0.0f);    \
        const float zpos = fmaxf(times((a + qo) + zo, third), 0.0f);                \
        const float qneg = qo - slope * zneg;                                       \
        const float fneg = (zneg - a) * (zneg - a) + qneg * qneg + (zneg - zo) * (zneg - zo); \
        const float fpos = (zpos - a) * (zpos - a) + (qo - zpos) * (qo - zpos) + (zpos - zo) * (zpos - zo); \
        const float zz = fpos < fneg ? zpos : zneg;                                 \
        update(zz > 0.0f ? zz : slope * zz, pv.f, uv.f, qn.f, un.f, tn.f);          \
        zn.f = zz; rn.f = a - zz;                                                   \
      }
      PD_ZQU(x) PD_ZQU(y) PD_ZQU(z) PD_ZQU(w)
#undef PD_ZQU
      st4(z, i, zn); st4(u, i, un); st4(r, i, rn); st4(t_next, i, tn);
      if (GENERAL && q_out != nullptr) st4(q_out, i, qn);
      if (y.rp.hi != nullptr) store_planes4(y.rp, i, rn, scale);
      add4(sum, rn);
      mr = max(mr, abs_bits(rn));
    }
  });
  if (y.amax_r != nullptr) commit_amax(mr, y.amax_r);
}

// ---- the same for a smooth activation: z-update by lookup table ---------------------------------------------
// f = tanh or sigmoid has no closed-form z-update; the paper recommends a lookup table (remark after Eq. "update z").
// The table holds T equally spaced candidates z_i = lo + i h with f(z_i); z+ is the candidate with the smallest
// (z - a)^2 + (q - f(z))^2 + (z - z^k)^2 (the first one if equal), element by element.  q, u, r, t as in zqu_kernel.
// Dynamic shared memory: T floats, f(z_i).
// Columns from the layer's width on are left at zero: the best candidate for a = q = z = 0 need not be zero (a table of 300 candidates from
// -6 to 6 has none there, and f(0) = 1/2 for sigmoid), and t of the padding would enter ||g||^2 and with it tau.
//
// The candidate is found without trying them all.  The second derivative of the objective is
// 4 + 2 f'^2 - 2 f'' (q - f) >= c = 4 - 2 max|f''| (|q| + 1), so for c > 0 (|q| < 1.59 for tanh, < 19.7 for sigmoid) the
// values on the grid are convex and a walk downhill from any candidate ends at the smallest; two Newton steps from the
// midpoint of a and z^k leave it a step or two to walk.  In floating point the smallest COMPUTED value could still lie
// elsewhere: with a relative error of at most 5 eps per value (all terms are positive) and an error d of the tabulated f,
// a candidate j >= 2 steps beyond the end of the walk is larger by at least
// c h^2 j (j - 1) / 2 - (10 j + 11) eps g - 4 (j + 1) sqrt(g) d, which is positive for every j >= 2 if it is for j = 2:
// c h^2 > 31 eps g + 12 sqrt(g) d.  Elements that fail the test (and NaN) try all candidates as before, so the result is the same
// bit for bit.  10 000 x 256, 513 candidates: 474 us with all candidates tried, 35 us so.
// All this for candidates that lie where they should: z_i = fl(lo + fl(i h)) is up to 3 eps max|z| off, and the room left in the
// constants of the test (8 %) covers 0.25 % of h at every candidate.  A table whose spacing is below 1200 eps max|z| (one far from zero: lo = 1000, 1010
// wide, 4096 candidates; never one that reaches from -x to x) is searched as a whole (table_is_even, on the host).
inline bool table_is_even(float lo, float hi, float step) {
  return (double)step >= 1200.0 * 5.9604644775390625e-8 * std::max(std::fabs((double)lo), std::fabs((double)hi));
}
__device__ __forceinline__ float table_h(float z, float f, float a, float q, float zk) {
  const float d0 = z - a, d1 = q - f, d2 = z - zk;
  return fmaf(d0, d0, fmaf(d1, d1, d2 * d2));
}
__device__ __forceinline__ void table_best(const float *__restrict__ f_sh, int T, float lo, float step, bool even, float act, float a,
                                           float q, float zk, float &z_best, float &f_best) {
  auto z_at = [&](int i) { return __fadd_rn(lo, __fmul_rn((float)i, step)); };
  auto h_at = [&](int i) { return table_h(z_at(i), f_sh[i], a, q, zk); };
  const bool th = act == ACT_TANH;
  const float c = 4.0f - 2.0f * (th ? 0.77f : 0.0963f) * (fabsf(q) + 1.0f);
  const float m = 0.5f * (a + zk), inv_step = 1.0f / step, top = (float)(T - 1);
  if (even && c > 0.1f && fabsf(m) < 1e30f) {
    float x = fminf(fmaxf((m - lo) * inv_step, 0.0f), top);
#pragma unroll
    for (int n = 0; n < 2; ++n) {
      const int i = __float2int_rn(x);
      const float f = f_sh[i], z = z_at(i);
      const float df = th ? 1.0f - f * f : f * (1.0f - f);
      x = (float)i - (2.0f * (z - m) - df * (q - f)) / fmaf(df, df, 2.0f) * inv_step;
      x = fminf(fmaxf(x, 0.0f), top);
    }
    int k = __float2int_rn(x);
    float hk = h_at(k);
    for (;;) {                                      // to the left while not larger: the first one if equal
      if (k == 0) break;
      const float v = h_at(k - 1);
      if (!(v <= hk)) break;
      --k; hk = v;
    }
    for (;;) {                                      // after a move the left neighbour is the larger one
      if (k == T - 1) break;
      const float v = h_at(k + 1);
      if (!(v < hk)) break;
      ++k; hk = v;
    }
    if (c * step * step > 2e-6f * hk + 4e-6f * sqrtf(hk)) {
      z_best = z_at(k); f_best = f_sh[k];
      return;
    }
  }
  float best = 3.0e38f;
  z_best = 0.f; f_best = 0.f;
  for (int i = 0; i < T; ++i) {
    const float v = h_at(i);
    if (v < best) { best = v; z_best = z_at(i); f_best = f_sh[i]; }
  }
}
template <bool GENERAL>
__global__ void __launch_bounds__(EW_THREADS, GENERAL ? 3 : 4)
zqu_table_kernel(const __grid_constant__ Group<Zqu> group, const __grid_constant__ ZquParams prm) {
  __shared__ double sh[EW_THREADS * 4];
  const Zqu &y = group.l[blockIdx.y];
  if ((int)blockIdx.x >= y.rows.n_blocks) return;
  float *__restrict__ r = y.r, *__restrict__ z = y.z, *__restrict__ q_out = y.q_out, *__restrict__ u = y.u, *__restrict__ t_next = y.t_next;
  const float *q_in = GENERAL ? y.q : nullptr;
  const float *__restrict__ gp = y.gp, *__restrict__ p_next = y.p_next;
  const void *__restrict__ codes_next = y.codes_next;
  const float act = prm.slope, q_scale = y.q_scale, q_lo = y.q_lo, theta = !GENERAL || gp != nullptr ? y.sc->inv_theta : 0.f;
  const float inv_step = 1.0f / prm.t_step, top = (float)(prm.T - 1);
  const float t_lo = prm.t_lo, t_step = prm.t_step;
  const int T = prm.T;
  const bool even = prm.table_even != 0;
  extern __shared__ float table_sh[];              // f(z_i)
  for (int i = threadIdx.x; i < T; i += blockDim.x) table_sh[i] = act_eval(__fadd_rn(t_lo, __fmul_rn((float)i, t_step)), act);
  __syncthreads();
  const QuUpdate<GENERAL> update(prm, q_scale, q_lo);
  const float scale = y.rp.hi != nullptr ? tc_scale_of(*y.rp.exp) : 1.f;
  uint32_t mr = 0u;
  row_block_sums(y.rows, (int)blockIdx.x, sh, [&](uint32_t i, uint32_t stride, int n, int cg, double (&sum)[4]) {
    const float4 sh4 = ld4(y.shift, cg);
    for (; n > 0; --n, i += stride) {
      float4 rv = ld4(r, i);
      const float4 zv = ld4(z, i), uv = ld4(u, i);
      if (!GENERAL || gp != nullptr) {
        const float4 gv = ld4(gp, i);
        rv.x = fmaf(-theta, gv.x, rv.x); rv.y = fmaf(-theta, gv.y, rv.y); rv.z = fmaf(-theta, gv.z, rv.z); rv.w = fmaf(-theta, gv.w, rv.w);
      }
      const float4 pv = codes_next != nullptr ? levels_of4(codes_next, prm.wide_codes, i, q_scale, q_lo) : ld4(p_next, i);
      const float a[4] = {(rv.x - sh4.x) + zv.x, (rv.y - sh4.y) + zv.y, (rv.z - sh4.z) + zv.z, (rv.w - sh4.w) + zv.w};
      const float zo[4] = {zv.x, zv.y, zv.z, zv.w}, uo[4] = {uv.x, uv.y, uv.z, uv.w}, pn[4] = {pv.x, pv.y, pv.z, pv.w};
      float qo[4];
      if (GENERAL && q_in != nullptr) {
        const float4 qv = ld4(q_in, i);
        qo[0] = qv.x; qo[1] = qv.y; qo[2] = qv.z; qo[3] = qv.w;
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          // f(z): from the table, as z is one of its candidates (except at the start)
          const int k = __float2int_rn(fminf(fmaxf((zo[e] - t_lo) * inv_step, 0.0f), top));
          const float f = __fadd_rn(t_lo, __fmul_rn((float)k, t_step)) == zo[e] ? table_sh[k] : act_eval(zo[e], act);
          qo[e] = fmaf(uo[e], update.inv_nu, f);
        }
      }
      float zn[4], fn[4], qn[4], un[4], rn[4], tn[4];
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        table_best(table_sh, T, t_lo, t_step, even, act, a[e], qo[e], zo[e], zn[e], fn[e]);
        update(fn[e], pn[e], uo[e], qn[e], un[e], tn[e]);
        rn[e] = a[e] - zn[e];
      }
      if (4 * cg + 4 > y.width) {
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (4 * cg + e >= y.width) zn[e] = qn[e] = un[e] = rn[e] = tn[e] = 0.f;
      }
      const float4 r4 = make_float4(rn[0], rn[1], rn[2], rn[3]);
      st4(z, i, make_float4(zn[0], zn[1], zn[2], zn[3])); st4(u, i, make_float4(un[0], un[1], un[2], un[3]));
      if (GENERAL && q_out != nullptr) st4(q_out, i, make_float4(qn[0], qn[1], qn[2], qn[3]));
      if (y.rp.hi != nullptr) store_planes4(y.rp, i, r4, scale);
      st4(r, i, r4); st4(t_next, i, make_float4(tn[0], tn[1], tn[2], tn[3]));
      add4(sum, r4);
      mr = max(mr, abs_bits(r4));
    }
  });
  if (y.amax_r != nullptr) commit_amax(mr, y.amax_r);
}
// q = f(z) + u/nu, for whoever wants the values
struct QOfZU { const float *z, *u; float *q; int width; uint32_t groups /* of 4 columns in a row */; size_t n4; };
__global__ void __launch_bounds__(EW_THREADS)
q_of_z_and_u_kernel(const __grid_constant__ Group<QOfZU> group, float slope, float nu) {
  const QOfZU &y = group.l[blockIdx.y];
  const float inv_nu = 1.0f / nu;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < y.n4; i += (size_t)gridDim.x * blockDim.x) {
    const float4 zv = ld4(y.z, i), uv = ld4(y.u, i);
    st4(y.q, i, keep_columns(make_float4(fmaf(uv.x, inv_nu, act_eval(zv.x, slope)), fmaf(uv.y, inv_nu, act_eval(zv.y, slope)),
                                         fmaf(uv.z, inv_nu, act_eval(zv.z, slope)), fmaf(uv.w, inv_nu, act_eval(zv.w, slope))),
                             columns_inside(i, y.groups, y.width)));
  }
}

// ---- z-update of the last layer -------------------------------------------------------------------
// a = (r - (G p+)/theta - shift) + z.  Labelled node: z+ = argmin CE(z; y) + (nu/2)||z - a||^2
// (Eq. "update zl"), the unique root of softmax(z) - e_y + nu (z - a) = 0, by damped Newton with the
// Hessian diag(s) + nu I - s s^T inverted through the rank-one update formula; double precision
// inside, since nu is small and the Hessian is close to singular along (1,..,1).  Unlabelled: z+ = a.
// The search starts from the stored z, the root for the previous a, where the gradient is nu (a_old - a) alone; where that does
// not converge (an a that moved by 1e4 at nu = 1e-6) it starts again from a.
//
// G lanes share a node, two classes each, everything in registers, sums by shuffles; the loop is common to the warp and has
// one evaluation per turn: a group whose trial point is accepted takes the gradient there from the exponentials it just
// computed and sets out on the next step, another one halves its step.  (One thread per node with the C-long arrays in
// local memory, two sets of exponentials per step and a start from a: 170 000 x 40 1150 us, 20 000 x 10 31 us.)
constexpr int ZL_MAX_C = 64;
template <int G>
__global__ void __launch_bounds__(128)
zlast_kernel(float *__restrict__ r, float *__restrict__ z, const float *__restrict__ shift,
             const int *__restrict__ labels, const uint8_t *__restrict__ mask, int n_rows, int C, int ld,
             double nu, int *__restrict__ not_converged, uint32_t *__restrict__ amax_r /* max|r|, may be null */,
             int least_squares /* R = 1/2 ||z - e_y||^2: z+ = (e_y + nu a)/(1 + nu) */, PlaneOut rp,
             const float *__restrict__ gp /* null: r has it */, const LayerScalars *sc) {
  const int j = (int)((blockIdx.x * (size_t)blockDim.x + threadIdx.x) / G), lane = threadIdx.x % G;
  const bool row = j < n_rows;
  const size_t at = (size_t)(row ? j : n_rows - 1) * ld + 2 * lane;          // (may lie beyond the row: every access is guarded by in[])
  const int c0 = 2 * lane;
  const bool in[2] = {c0 < C, c0 + 1 < C};
  auto sum = [&](double v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o, G);
    return v;
  };
  auto top = [&](double v) {
#pragma unroll
    for (int o = G / 2; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o, G));
    return v;
  };
  double a[2] = {0.0, 0.0}, x[2] = {0.0, 0.0};
#pragma unroll
  for (int i = 0; i < 2; ++i)
    if (in[i]) {
      const float rv = gp != nullptr ? fmaf(-sc->inv_theta, gp[at + i], r[at + i]) : r[at + i];
      x[i] = (double)z[at + i];
      a[i] = (double)((rv - shift[c0 + i]) + z[at + i]);
    }
  const bool labelled = row && mask[j];
  const int y = labelled ? labels[j] : -1;
  const double e[2] = {c0 == y ? 1.0 : 0.0, c0 + 1 == y ? 1.0 : 0.0};
  if (least_squares) {
#pragma unroll
    for (int i = 0; i < 2; ++i) x[i] = labelled ? (e[i] + nu * a[i]) / (1.0 + nu) : a[i];
  } else {
    if (!labelled) { x[0] = a[0]; x[1] = a[1]; }
    bool done = !labelled, resolvable = false;
    double d[2] = {0.0, 0.0}, t = 0.0, fx = 0.0, slope = 0.0;
    int steps = 0;
    bool from_a = false;
    while (__any_sync(0xffffffffu, !done)) {
      const double v[2] = {x[0] + t * d[0], x[1] + t * d[1]};
      const double m = top(fmax(in[0] ? v[0] : -1e300, in[1] ? v[1] : -1e300));
      const double ex[2] = {in[0] ? exp(v[0] - m) : 0.0, in[1] ? exp(v[1] - m) : 0.0};
      const double se = sum(ex[0] + ex[1]);
      const double rest = sum(0.5 * nu * ((v[0] - a[0]) * (v[0] - a[0]) + (v[1] - a[1]) * (v[1] - a[1])) - (e[0] * v[0] + e[1] * v[1]));
      const double f = m + log(se) + rest;
      const bool accept = !resolvable || f <= fx + 1e-4 * t * slope || t < 1e-12;
      // gradient, Newton step and slope at v; used if v is accepted
      double g[2], mi[2], s[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        s[i] = ex[i] / se;
        g[i] = in[i] ? s[i] - e[i] + nu * (v[i] - a[i]) : 0.0;
        mi[i] = 1.0 / (s[i] + nu);
      }
      const double gmax = top(fmax(fabs(g[0]), fabs(g[1])));
      const double s_mg = sum(s[0] * mi[0] * g[0] + s[1] * mi[1] * g[1]), s_ms = sum(s[0] * mi[0] * s[0] + s[1] * mi[1] * s[1]);
      const double k = s_mg / (1.0 - s_ms);
      const double nd[2] = {-(mi[0] * g[0] + mi[0] * s[0] * k), -(mi[1] * g[1] + mi[1] * s[1] * k)};
      const double ns = sum(g[0] * nd[0] + g[1] * nd[1]);
      if (!done) {
        if (accept) {
          x[0] = v[0]; x[1] = v[1]; fx = f;
          d[0] = nd[0]; d[1] = nd[1]; slope = ns; t = 1.0;
          resolvable = -slope > 1e-9 * (1.0 + fabs(fx));
          if (gmax <= 1e-10) done = true;
          else if (++steps >= 100 && !from_a) {
            from_a = true;
            x[0] = a[0]; x[1] = a[1];
            steps = 0; t = 0.0; resolvable = false;
          } else if (steps >= 100) {
            done = true;
            if (lane == 0) atomicAdd(not_converged, 1);
          }
        } else {
          t *= 0.5;
        }
      }
    }
  }
  uint32_t mr = 0u;
  if (row) {
    float rn[2] = {0.f, 0.f};
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      if (!in[i]) continue;
      const float zn = (float)x[i];
      z[at + i] = zn;
      rn[i] = (float)(a[i] - (double)zn);
      r[at + i] = rn[i];
      mr = max(mr, abs_bits(rn[i]));
    }
    if (rp.hi != nullptr && in[0]) {
      const float scale = tc_scale_of(*rp.exp);
      float h0, l0, h1, l1;
      tc_split(rn[0], scale, h0, l0);
      tc_split(rn[1], scale, h1, l1);
      *reinterpret_cast<uint32_t *>(rp.hi + at) = tc_pack(h0, h1);
      *reinterpret_cast<uint32_t *>(rp.lo + at) = tc_pack(l0, l1);
    }
  }
  if (amax_r != nullptr) commit_amax(mr, amax_r);
}
inline void launch_zlast(cudaStream_t st, float *r, float *z, const float *shift, const int *labels, const uint8_t *mask, int n_rows,
                         int C, int ld, double nu, int *not_converged, uint32_t *amax_r, int least_squares, const PlaneOut &rp,
                         const float *gp, const LayerScalars *sc) {
  auto go = [&](auto G) {
    constexpr int g = decltype(G)::value;
    zlast_kernel<g><<<(int)ceil_div((int64_t)n_rows * g, 128), 128, 0, st>>>(r, z, shift, labels, mask, n_rows, C, ld, nu, not_converged,
                                                                            amax_r, least_squares, rp, gp, sc);
  };
  if (C <= 8) go(std::integral_constant<int, 4>{});
  else if (C <= 16) go(std::integral_constant<int, 8>{});
  else if (C <= 32) go(std::integral_constant<int, 16>{});
  else go(std::integral_constant<int, 32>{});
}

// t = u + rho (p - q) from the stored iterates (after the start or after the caller has set a tensor); the same
// operations as in zqu_kernel, so both give the same bits.
__global__ void __launch_bounds__(EW_THREADS)
gradp_const_kernel(const float *__restrict__ u, const float *__restrict__ p, const float *__restrict__ q, float rho,
                   float *__restrict__ t, size_t n4) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    const float4 uv = ld4(u, i), pv = ld4(p, i), qv = ld4(q, i);
    float4 tv;
    tv.x = fmaf(rho, pv.x - qv.x, uv.x); tv.y = fmaf(rho, pv.y - qv.y, uv.y);
    tv.z = fmaf(rho, pv.z - qv.z, uv.z); tv.w = fmaf(rho, pv.w - qv.w, uv.w);
    st4(t, i, tv);
  }
}

// ---- elementwise helpers of the initial forward pass ---------------------------------------------
__global__ void __launch_bounds__(EW_THREADS)
relu_max_kernel(const float *__restrict__ z, float *__restrict__ q, size_t n4, float slope, int width, uint32_t groups, float *__restrict__ block_max) {
  __shared__ float red[EW_THREADS / 32];
  float m = 0.0f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n4; i += (size_t)gridDim.x * blockDim.x) {
    float4 v = ld4(z, i);
    v.x = act_eval(v.x, slope); v.y = act_eval(v.y, slope); v.z = act_eval(v.z, slope); v.w = act_eval(v.w, slope);
    v = keep_columns(v, columns_inside(i, groups, width));
    m = fmaxf(m, fmaxf(fmaxf(v.x, v.y), fmaxf(v.z, v.w)));
    st4(q, i, v);
  }
  m = warp_max(m);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = m;
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int i = 1; i < EW_THREADS / 32; ++i) m = fmaxf(m, red[i]);
    block_max[blockIdx.x] = m;
  }
}

// ---- objective pieces of all layers ---------------------------------------------------------------
// Blocks (x, y): part x of layer y; sums r^2, (q - f(z))^2, u (p_next - q), (p_next - q)^2 (u == nullptr: only r^2), one
// slot of four per block; the block of a layer that finishes last (one counter per layer, back to zero afterwards) adds
// the layer's slots in block order and writes the four sums to out[4 y ..] -- page-locked host memory, so that the whole
// read-out is one launch and one wait.  Two launches, a copy and a wait per layer before: 22 launches and 11 waits on
// ten layers of 2000 x 100 took 307 us, and scalar loads with an fp32 p_next kept the wide layers at 2.3 TB/s.
// `parts`: OBJ_ALL, or OBJ_RESIDUALS for the last sum alone.
// 16-byte loads, p_next as its codes in pdADMM-G-Q (the same bits).
constexpr int OBJ_MAX_LAYERS = 40;           // layers per launch: their pointers travel as a kernel argument
enum : int { OBJ_ALL = 0, OBJ_RESIDUALS = 1 };
constexpr int obj_blocks_per_sm(int parts, bool smooth) { return parts == OBJ_ALL || smooth ? 4 : 6; }      // resident ones, which is what a launch has
struct ObjLayer { const float *r, *z, *q, *u /* null: only r^2 */, *p_next; const void *codes_next; size_t n4; float scale, lo; int width /* 0: padding adds nothing */; uint32_t groups /* of 4 columns in a row */; };
struct ObjLayers { ObjLayer l[OBJ_MAX_LAYERS]; };
__device__ __forceinline__ void add_sq4(double &s, float4 v) {
  const double a = v.x, b = v.y, c = v.z, d = v.w;
  s += (a * a + b * b) + (c * c + d * d);
}
// IMPLIED: q from z and u (every layer's, see zqu_kernel).  SMOOTH: f = tanh or sigmoid, whose evaluation would otherwise stand between the
// loads.  A thread has the loads of two groups on their way, and the blocks are one round of what the SMs hold.  Bound by memory: 16 bytes per
// element, the residuals alone 12 (q is not stored: 8 with it).  60 000 x 1000, 4 layers: objective 460 us, residuals 350; with f in its
// general form between the loads of one group 705 and 363, with a stored q and 20 bytes 552 and 246.
template <int PARTS, bool IMPLIED, bool SMOOTH>
__global__ void __launch_bounds__(EW_THREADS, obj_blocks_per_sm(PARTS, SMOOTH))
objective_kernel(const __grid_constant__ ObjLayers layers, float slope, float nu, int wide_codes, double *slots, int *counters,
                 double *out) {
  __shared__ double red[EW_THREADS / 32];
  __shared__ int last;
  const ObjLayer &y = layers.l[blockIdx.y];
  double s[4] = {0, 0, 0, 0};
  const float inv_nu = 1.0f / nu;
  const size_t stride = (size_t)gridDim.x * blockDim.x;
  auto f = [&](float x) { return SMOOTH ? act_eval(x, slope) : x > 0.0f ? x : slope * x; };
  constexpr int U = 2;
  for (size_t i0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i0 < y.n4; i0 += U * stride) {
    if (y.u == nullptr) {
      if (PARTS == OBJ_ALL)
        for (size_t i = i0; i < y.n4 && i < i0 + U * stride; i += stride) add_sq4(s[0], ld4(y.r, i));
      continue;
    }
    float4 rv[U], zv[U], uv[U], qv[U], pv[U];
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const size_t i = i0 + k * stride;
      if (i >= y.n4) continue;
      if (PARTS == OBJ_ALL) rv[k] = ld4(y.r, i);
      if (PARTS == OBJ_ALL || IMPLIED) { zv[k] = ld4(y.z, i); uv[k] = ld4(y.u, i); }
      if (!IMPLIED) qv[k] = ld4(y.q, i);
      pv[k] = y.codes_next != nullptr ? levels_of4(y.codes_next, wide_codes, i, y.scale, y.lo) : ld4(y.p_next, i);
    }
#pragma unroll
    for (int k = 0; k < U; ++k) {
      const size_t i = i0 + k * stride;
      if (i >= y.n4) continue;
      float4 fv = make_float4(0.f, 0.f, 0.f, 0.f);
      if (PARTS == OBJ_ALL || IMPLIED) fv = make_float4(f(zv[k].x), f(zv[k].y), f(zv[k].z), f(zv[k].w));
      if (IMPLIED) qv[k] = make_float4(fmaf(uv[k].x, inv_nu, fv.x), fmaf(uv[k].y, inv_nu, fv.y), fmaf(uv[k].z, inv_nu, fv.z), fmaf(uv[k].w, inv_nu, fv.w));
      if (SMOOTH && y.width > 0) {           // f(0) is not zero: q = f(z) + u/nu of the padding isn't either
        const int inside = columns_inside(i, y.groups, y.width);
        fv = keep_columns(fv, inside);
        qv[k] = keep_columns(qv[k], inside);
        pv[k] = keep_columns(pv[k], inside);
      }
#define PD_OBJ(e)                                                                       \
      {                                                                                 \
        const double q = qv[k].e, res = (double)pv[k].e - q;                            \
        if (PARTS == OBJ_ALL) {                                                         \
          const double d = q - (double)fv.e;                                            \
          s[1] += d * d; s[2] += (double)uv[k].e * res;                                 \
        }                                                                               \
        s[3] += res * res;                                                              \
      }
      if (PARTS == OBJ_ALL) add_sq4(s[0], rv[k]);
      PD_OBJ(x) PD_OBJ(y) PD_OBJ(z) PD_OBJ(w)
#undef PD_OBJ
    }
  }
  double *mine = slots + ((size_t)blockIdx.y * gridDim.x + blockIdx.x) * 4;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    if (PARTS == OBJ_RESIDUALS && k < 3) continue;
    const double t = block_sum<EW_THREADS>(s[k], red);
    if (threadIdx.x == 0) mine[k] = t;
  }
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(counters + blockIdx.y, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  for (int k = 0; k < 4; ++k) {
    if (PARTS == OBJ_RESIDUALS && k < 3) continue;
    double v = 0.0;
    for (int i = threadIdx.x; i < (int)gridDim.x; i += EW_THREADS) v += __ldcg(slots + ((size_t)blockIdx.y * gridDim.x + i) * 4 + k);
    const double t = block_sum<EW_THREADS>(v, red);
    if (threadIdx.x == 0) out[4 * blockIdx.y + k] = t;
  }
  if (threadIdx.x == 0) counters[blockIdx.y] = 0;
}

// R(z_L; y): sum over masked nodes of -z_y + logsumexp(z), or of 1/2 ||z - e_y||^2 (least_squares).
// One thread per node, one slot per block; the block that finishes last adds the slots in block order into *out
// (page-locked host memory) and clears the counter.
__global__ void __launch_bounds__(EW_THREADS)
risk_kernel(const float *__restrict__ z, const int *__restrict__ labels, const uint8_t *__restrict__ mask,
            int n_rows, int C, int ld, double *slots, int least_squares, int *counter, double *out) {
  __shared__ double red[EW_THREADS / 32];
  __shared__ int last;
  double acc = 0.0;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n_rows; j += gridDim.x * blockDim.x) {
    if (!mask[j]) continue;
    const float *zj = z + (size_t)j * ld;
    if (least_squares) {
      double sq = 0.0;
      for (int c = 0; c < C; ++c) {
        const double d = (double)zj[c] - (c == labels[j] ? 1.0 : 0.0);
        sq += d * d;
      }
      acc += 0.5 * sq;
      continue;
    }
    double m = zj[0];
    for (int c = 1; c < C; ++c) m = fmax(m, (double)zj[c]);
    double se = 0.0;
    for (int c = 0; c < C; ++c) se += exp((double)zj[c] - m);
    acc += m + log(se) - (double)zj[labels[j]];
  }
  const double t = block_sum<EW_THREADS>(acc, red);
  if (threadIdx.x == 0) {
    slots[blockIdx.x] = t;
    __threadfence();
    last = atomicAdd(counter, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double v = 0.0;
  for (int i = threadIdx.x; i < (int)gridDim.x; i += EW_THREADS) v += __ldcg(slots + i);
  v = block_sum<EW_THREADS>(v, red);
  if (threadIdx.x == 0) { *out = v; *counter = 0; }
}

// Predicted class of every node: the largest of its C logits, the first one among equals.  counts[0..3] (zero before and
// after) gather: correct and total over the nodes with mask = 1, correct and total over the others; the block that
// finishes last moves them, and the products' error word, to out[0..4] (page-locked host memory).
__global__ void __launch_bounds__(EW_THREADS)
argmax_kernel(const float *__restrict__ z, const int *__restrict__ labels, const uint8_t *__restrict__ mask, int n_rows,
              int C, int ld, int *__restrict__ pred, unsigned long long *counts, int *counter, const int *error,
              unsigned long long *out) {
  __shared__ int last;
  unsigned long long c_in = 0, n_in = 0, c_out = 0, n_out = 0;
  for (int j = blockIdx.x * blockDim.x + threadIdx.x; j < n_rows; j += gridDim.x * blockDim.x) {
    const float *zj = z + (size_t)j * ld;
    int best = 0;
    float vbest = zj[0];
    for (int c = 1; c < C; ++c) {
      const float v = zj[c];
      if (v > vbest) { vbest = v; best = c; }
    }
    pred[j] = best;
    const bool hit = best == labels[j];
    if (mask[j]) { ++n_in; c_in += hit; } else { ++n_out; c_out += hit; }
  }
  // integer sums: the order of the atomics does not matter
  c_in = warp_sum_u64(c_in); n_in = warp_sum_u64(n_in); c_out = warp_sum_u64(c_out); n_out = warp_sum_u64(n_out);
  if ((threadIdx.x & 31) == 0) {
    if (n_in) { atomicAdd(counts + 0, c_in); atomicAdd(counts + 1, n_in); }
    if (n_out) { atomicAdd(counts + 2, c_out); atomicAdd(counts + 3, n_out); }
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = atomicAdd(counter, 1) == (int)gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  if (threadIdx.x < 4) {
    out[threadIdx.x] = __ldcg(counts + threadIdx.x);
    counts[threadIdx.x] = 0ull;
  }
  if (threadIdx.x == 4) out[4] = (unsigned long long)(unsigned)*error;
  if (threadIdx.x == 0) *counter = 0;
}

}  // namespace pd
