// fp32-accurate dense products on the sm_100a tensor cores.
//
// Every product C = A * B is issued as three fp16 MMAs on a scaled two-term split of the operands,
//     xs = x * 2^e                      (e per matrix, from max|x|, so that max|xs| lies in [2^14, 2^15))
//     x_hi = xs rounded to 11 significant bits      (exact in fp16 down to 2^-14)
//     x_lo = (xs - x_hi) * 2^11, rounded to fp16    (xs - x_hi is exact in fp32; the factor keeps it out of the
//                                                    fp16 subnormals, so the pair carries 22 bits down to 2^-14
//                                                    and at least 11 bits down to 2^-25 of the scaled range)
//     A * B ~= 2^-(eA+eB) [ A_hi B_hi + 2^-11 (A_hi B_lo + A_lo B_hi) ]      (the dropped lo*lo term is 2^-24 relative)
// Products of two 11-bit numbers are exact in the fp32 accumulator, so the split is as accurate as the same
// split on tf32 operands at twice the tensor-core rate and half the shared-memory footprint per operand.
//
// Both operands are read as planes (hi, lo) in the orientation in which their matrix is stored, by TMA: the tensor cores
// take an operand whose contraction index is contiguous (K-major: a matrix of nodes contracted over its columns) as well as
// one whose output index is contiguous (MN-major: the contraction over the nodes, and W in r W), so nothing is ever
// transposed, and the kernels that write a matrix write its planes beside it.  Such a kernel does not know the
// largest magnitude of what it writes and takes the exponent from a bound or a prediction (TcOperand::exp); the product
// compares it with the largest magnitude that was then seen, and if the scaling turns out unusable two spare warps build
// that operand's planes from the fp32 matrix instead of loading them (rare, slower, same result; large matrices get a
// kernel that does it beforehand, see check_planes_kernel).
//
// One thread issues tcgen05.mma; completion is tracked with mbarriers.  Eight accumulate warps read each K block's main term
// from tensor memory and add it to register accumulators; a finished tile goes through shared memory to eight epilogue
// warps, which apply the fused operations and store it while the next tile is accumulated.  (With one set of warps for
// both, the loads and stores of the epilogue had 16 KB in flight per SM and the tensor pipe waited for them: 9 layers of
// 20 000 x 500 x 500, r W with its epilogue 533 us.)
//
// Tile: 128 x 128 outputs per block, 64-deep K blocks.  What bounds the product is the traffic between L2 and the SMs
// (10.6 TB/s measured, whatever the number of planes): a block on its own loads A and B planes of 64 KB per K block for
// three times 2 MFLOP.  So two neighbouring SMs work as a pair on 256 x 128 outputs (tcgen05 cta_group::2): each loads the
// planes of its own 128 rows of A and of half of the 128 columns of B, 48 KB, and the tensor cores read the other half
// from the neighbour's shared memory.  No copy is multicast.  Products with few rows run one block per tile.
// Wide tiles (256 x 256 per pair, choose_wide says when) bring 64 KB per K block for twice the work, two thirds of the traffic:
// the W-gradient of 20 000 x 500 (9 layers) 410 -> 330 us, of 90 000 x 2000 (8 layers) 9.3 -> 7.6 ms, 1370 TFLOP/s of MMAs at
// 1.4 GHz under the power limit.  Two accumulators of 256 columns fill tensor memory, so the correction terms share the main
// term's: they come first, and the first MMA of the main term scales their sum by 2^-11 (relative error 1.5e-7 to 2.2e-7 either
// way, a hundredth less with the shared one).  A tile's 128 KB of sums per block leave neither registers nor shared memory for
// epilogue warps: the accumulate warps store it themselves, in bulk copies (with ordinary stores the end of a tile took
// 10 000 cycles instead of 6500), so the form is built for products that store their sums as they are.  Tried: a finished tile parked
// in tensor memory and stored between the K blocks of the next one (x W^T of 20 000 x 500, 9 layers: 560 us against 325).
// Every wait is bounded; a wait that expires raises an error word in global memory and the CTA drains and exits.
#pragma once

#include <cuda_fp16.h>

#include <type_traits>

#include "common.cuh"
#include "planes.cuh"
#include "scalars.cuh"
#include "gemm_simt.cuh"   // epilogue functors
#include "tc_ptx.cuh"

namespace pd {

// Operands that are MN-major (output index contiguous) where the others are K-major.
enum : int { TC_NT = 0, TC_A_MN = 1, TC_B_MN = 2 };
constexpr int TC_BM = 128, TC_BN = 128, TC_BK = 64;
constexpr int TC_KSTEPS = TC_BK / 16;                          // MMAs (K = 16) per pair of planes and K block
constexpr int TC_FLUSH = 1;                                    // K blocks per read-out of the main accumulator
constexpr int TC_PLANE_BYTES = 128 * TC_BK * 2;                // 16 KB: one 128 x 64 fp16 operand plane
constexpr int TC_BOX_BYTES = 64 * TC_BK * 2;                   // 8 KB: what one TMA load brings, 64 x 64
constexpr int TC_SPACE = 14 * TC_PLANE_BYTES;                  // 224 KB: stages and finished tile
constexpr int TC_MAX_STAGES = 8;
// Five warpgroups (register budgets are set per warpgroup): 0 = TMA warp, MMA warp and two warps that split operands when
// a scaling was unusable; 1, 2 = the accumulate warps: a warp can only reach its own 32-lane quarter of tensor memory, so
// warp w owns the rows of quarter w mod 4 and columns 64 (w / 4) .. +63 of the tile, 64 accumulators per thread; 3, 4 = the
// epilogue warps, each with an accumulate warp to serve.
// Registers: the block is launched with 640 x 96 = 61440; warpgroup 0 keeps 56 per thread, the accumulate warps take 120, the
// epilogue warps 88: 128 (56 + 2 x 120 + 2 x 88) = 60416, so every increase is satisfiable.
constexpr int TC_SPLIT0 = 2, TC_SPLIT_WARPS = 2;               // first splitting warp
constexpr int TC_ACC0 = 4, TC_EPI0 = 12;                       // first accumulate warp, first epilogue warp
constexpr int TC_THREADS = 640;
constexpr int TC_ACC_WARPS = 8;
constexpr int TC_REGS_LAUNCH = 96, TC_REGS_CTRL = 56, TC_REGS_ACC = 120, TC_REGS_EPI = 88;
static_assert(TC_THREADS * TC_REGS_LAUNCH <= 65536, "register file");
static_assert(128 * (TC_REGS_CTRL + 2 * TC_REGS_ACC + 2 * TC_REGS_EPI) <= TC_THREADS * TC_REGS_LAUNCH,
              "the warpgroups' register shares exceed what the block is launched with: an increase would wait for ever");
constexpr int TC_ACC_BUFS = 3;                                 // main-term accumulator tiles in tensor memory
constexpr int TC_TMEM_COLS = 512;                              // 3 main tiles, 1 correction tile
constexpr uint32_t TC_COL_CORR = TC_ACC_BUFS * TC_BN;          // first column of the correction tile
constexpr int TC_TILE_BYTES = 8 * 32 * 64 * 4;                 // finished tile: 8 warps x 32 rows x 64 columns
// Wide tiles (pairs of SMs, 256 x 256): sixteen accumulate warps, 64 accumulators per thread, that store their piece themselves, in
// parts of 32 rows x 16 columns through 2 KB of shared memory each; two accumulators of 256 columns in tensor memory.
constexpr int TC_WIDE = 256, TC_WIDE_WARPS = 16, TC_WIDE_PART = 16;
constexpr int TC_WIDE_PART_BYTES = 32 * TC_WIDE_PART * 4;
constexpr int TC_WIDE_REGS_CTRL = 64, TC_WIDE_REGS_ACC = 104;
static_assert(128 * (TC_WIDE_REGS_CTRL + 4 * TC_WIDE_REGS_ACC) <= TC_THREADS * TC_REGS_LAUNCH, "register shares of the wide form");
constexpr int TC_SMEM_BYTES = TC_SPACE + 1024 /* alignment slack */ + 512 /* barriers */;
static_assert(8 * (3 * TC_MAX_STAGES + 2 * TC_ACC_BUFS + 3 + 2 * TC_ACC_WARPS) + 24 <= 512, "barriers");
// How many parts a finished tile is handed over in (none if nothing is stored).  In one part it takes 64 KB; in two, one after
// the other through 32 KB, it leaves room for one more stage if a stage holds four planes.  Two parts for the contraction
// over the nodes, which is long and stores little: 100 000 x 500 x 500, 8 layers: 395 us against 444.  For the other products, whose
// contraction is a layer's width, the second part holds up the accumulate warps: x W^T 468 us against 453.
__host__ __device__ constexpr int tc_parts(int layout, bool stores) { return !stores ? 0 : layout == (TC_A_MN | TC_B_MN) ? 2 : 1; }

// Epilogues store their result unless they say otherwise (kStore = false).
template <class Epi, class = void> struct epi_stores { static constexpr bool value = true; };
template <class Epi> struct epi_stores<Epi, std::enable_if_t<!Epi::kStore>> { static constexpr bool value = false; };
// An epilogue that wants nothing but the sum of squares of the product may say kCoarse = true: the product is then
// issued as the main term A_hi B_hi alone (one MMA instead of three).  Each term then carries an independent relative
// rounding of 2^-11 instead of 2^-22; over the 1e6..1e9 squares of the sum these average out to far below the
// single-precision accuracy of the sum itself.
template <class Epi, class = void> struct epi_coarse { static constexpr bool value = false; };
template <class Epi> struct epi_coarse<Epi, std::enable_if_t<Epi::kCoarse>> { static constexpr bool value = true; };
// An epilogue whose sum of squares is that of the product itself, not of what it stores, says kSumsqOfAcc = true.
template <class Epi, class = void> struct epi_sumsq_acc { static constexpr bool value = false; };
template <class Epi> struct epi_sumsq_acc<Epi, std::enable_if_t<Epi::kSumsqOfAcc>> { static constexpr bool value = true; };
// An epilogue with a word for the largest magnitude of what it stores says kAmax = true.
template <class Epi, class = void> struct epi_amax { static constexpr bool value = false; };
template <class Epi> struct epi_amax<Epi, std::enable_if_t<Epi::kAmax>> { static constexpr bool value = true; };
// An epilogue that also leaves its result as planes for a later product (H, L [rows][ldc], scaled by 2^(*h_exp); L may be
// null: only the hi plane is wanted; H may be null: none are) says kPlanes = true.
template <class Epi, class = void> struct epi_planes { static constexpr bool value = false; };
template <class Epi> struct epi_planes<Epi, std::enable_if_t<Epi::kPlanes>> { static constexpr bool value = true; };

// What the kernel has to know about an operand beside its tensor maps.
struct TcOperand {
  const int *exp = nullptr;        // exponent the planes were made with; null: 0 (integer planes)
  const uint32_t *amax = nullptr;  // bit pattern of max|x| as seen by now; null: the planes are known to be good
  const float *x = nullptr;        // the fp32 matrix (read only if the planes are refused), leading dimension ld; null: refused
                                   // planes were made again beforehand, with the exponent of amax (check_planes_kernel)
  int ld = 0;
};

// One launch works on the same product of several layers, whose output tiles form one sequence of work units: a small
// problem's layers fill the GPU together, and a large one has one partly filled last round instead of one per layer.
constexpr int TC_MAX_GROUP = 16;
// Division by a number known on the host: the quotient is the high word of n * inv, inv = ceil(2^32 / d), where that is exact for every
// n that occurs (n d < 2^32; inv = 0 otherwise).  (Three divisions per tile and role took 650 cycles.)
struct TcDiv {
  int d; uint32_t inv;
  static TcDiv of(int d, int64_t n_max) { return TcDiv{d, n_max * d < (int64_t(1) << 32) && d > 1 ? (uint32_t)(((int64_t(1) << 32) + d - 1) / d) : 0u}; }
  __device__ __forceinline__ int operator()(int n) const { return d == 1 ? n : inv != 0u ? (int)__umulhi((uint32_t)n, inv) : n / d; }
};
template <class Epi>
struct TcLayer {
  CUtensorMap a, alo, b, blo;      // planes of the operands
  CUtensorMap c;                   // wide tiles: the output, all slices' rows one after the other
  int M, N, K;            // output rows, output columns, contraction length
  int k_chunk;            // contraction slice (multiple of TC_BK); K rounded up if not split
  int n_split;            // number of contraction slices; slice z writes its own partial output
  size_t c_split_stride;  // elements between the partial outputs of consecutive slices
  TcOperand oa, ob;
  float mul;              // factor applied to the result after the power-of-two scalings (integer operands, see ZERO)
  Epi epi;
  // Sums of squares (Epi::kSumsq and slots != null): one slot per 128-row tile, column tile and accumulate warp, written by
  // whichever block has the tile; the block that completes the layer (`done`, zero before and after) adds them in index order
  // and passes the sum to `step`.  Neither depends on how the tiles were shared out.  (One arrival per block and layer: an
  // arrival per tile and warp held up the epilogue by 3 us a tile.)
  double *slots;
  int *done;
  Step step;
  // Tail balancing (one layer, n_split == 1): output tiles from tail_begin on are cut into tail_split contraction
  // slices, one work unit each, so that the last, partly filled round of the persistent grid is shorter.
  // A slice leaves its accumulators in tail_ws; the warp that finds itself last (tail_count) adds the slices
  // in slice order and runs the epilogue.  tail_split <= 1 switches this off.
  int tail_begin, tail_split;
  TcDiv tiles_n, tiles_mn;                // column tiles, output tiles
  // Pieces of 32 rows x 64 columns, one per accumulate warp: 8 of a block's tile, 16 of a pair's, 32 of a pair's wide one.  A round has n_sms
  // units of blocks or n_sms / 2 of pairs and a cut takes at least two of them, so n_sms * 8 counts are enough (n_sms / 4 wide tiles).
  float *tail_ws;         // [tiles from tail_begin][tail_split][pieces][64][32] floats
  int *tail_count;        // [tiles from tail_begin][pieces], zero before and after every launch
};
template <class Epi>
struct TcGroup {
  int n;
  int unit_end[TC_MAX_GROUP];      // work units of a layer and of those before it (side by side: walking through the layers'
                                   // descriptions cost a miss in the constant cache each, half of a small launch's start)
  int *error;             // set to 1 if a bounded wait expired
  TcLayer<Epi> l[TC_MAX_GROUP];
};

// LAYOUT bit 0: A is MN-major, bit 1: B is MN-major.  Tensor maps: planes of A (a = hi, alo = lo) and of B.
//   K-major:  matrix [output index][contraction index];  MN-major: matrix [contraction index][output index];
//   boxes of 64 x 64 either way: 64 output indices (rows) x 64 values, or 64 rows x 64 output indices
// PAIR: clusters of two blocks, each pair one tile of 256 x 128 outputs: block `rank` of the pair holds rows 128 rank .. +127
// of A, of the accumulators and of the output, and columns 64 rank .. +63 of B.  Block 0 issues the MMAs of both; its
// barriers collect what both blocks loaded and read out.
//
// Persistent: the grid has at most one block per SM and the blocks (pairs) take the output tiles in rounds, upwards in even
// rounds and downwards in odd ones (column tile fastest, so that neighbouring blocks share the streamed operand in L2): the
// first layer's contraction is often several times as long, and the blocks that began with it get nothing of a partly filled
// second round.  All roles keep running counters over K blocks, so the producer prefetches the next tile while the current one
// is in its epilogue.
//
// The tensor cores add into their fp32 accumulator with truncation, which costs about 2^-24 of the
// accumulator per MMA and always in the same direction.  To keep fp32-class accuracy the main term
// A_hi B_hi is accumulated in tensor memory for ONE K block only (4 MMAs): after each block the accumulate
// warps read it out and add it to a register accumulator with round-to-nearest, while the MMAs of the next
// blocks fill the other buffers.  The two correction terms are 2^-11 of the main term, so they are summed over
// the whole contraction in a tile of their own and added once at the end.
//
// ZERO: bit 0 = the lo plane of A is identically zero, bit 1 = the lo plane of B is.  An operand of
// pdADMM-G-Q that lies on a level set {c s} (the quantised p, or the difference of two of them) is the spacing s times
// a small integer, and integers up to 2048 are exact in one fp16 plane: its plane holds the integers, there is no lo
// plane to load and no MMA for it (two MMAs per product instead of three), and mul = s restores the values.
template <int LAYOUT, class Epi, int ZERO, bool PAIR, bool WIDE>
__global__ void __maxnreg__(TC_REGS_LAUNCH)
gemm_tc_kernel(const __grid_constant__ TcGroup<Epi> grp) {
  constexpr bool A_MN = (LAYOUT & TC_A_MN) != 0, B_MN = (LAYOUT & TC_B_MN) != 0, COARSE = epi_coarse<Epi>::value || ZERO == 3;
  // which lo planes are loaded and used (a product that only wants its squared norm uses neither, and lets the main
  // term accumulate in tensor memory over 8 K blocks: the truncation of that accumulation, 2e-6 relative, does not matter to a
  // norm that only starts a search; over the whole contraction it was 1e-5 at 1000 values)
  constexpr bool A_LO = !(ZERO & 1) && !COARSE, B_LO = !(ZERO & 2) && !COARSE;
  constexpr int FLUSH = COARSE ? 8 : TC_FLUSH;        // K blocks per read-out of the main accumulator
  constexpr int A_PLANES = A_LO ? 2 : 1, B_PLANES = B_LO ? 2 : 1;
  static_assert(PAIR || !WIDE, "wide tiles are those of pairs");
  constexpr int CG = PAIR ? 2 : 1, WARPS = CG * TC_ACC_WARPS, TILE_M = PAIR ? 2 * TC_BM : TC_BM, TILE_N = WIDE ? TC_WIDE : TC_BN;
  constexpr int BN = TILE_N / CG, B_PLANE_BYTES = BN * TC_BK * 2;    // B held by this block
  constexpr int STAGE_BYTES = A_PLANES * TC_PLANE_BYTES + B_PLANES * B_PLANE_BYTES;
  constexpr bool STORES = epi_stores<Epi>::value;
  constexpr int PARTS = tc_parts(LAYOUT, STORES);
  constexpr int STAGE_SPACE = TC_SPACE - (WIDE ? (STORES ? TC_WIDE_WARPS * TC_WIDE_PART_BYTES : 0) : PARTS > 0 ? TC_TILE_BYTES / PARTS : 0);
  constexpr int STAGES = STAGE_SPACE / STAGE_BYTES < TC_MAX_STAGES ? STAGE_SPACE / STAGE_BYTES : TC_MAX_STAGES;
  constexpr int B_OFF = A_PLANES * TC_PLANE_BYTES;            // stage: A_hi, A_lo, B_hi, B_lo (those that exist)
  extern __shared__ uint8_t smem_raw[];
  uint8_t *smem = reinterpret_cast<uint8_t *>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t *tr_base = smem + STAGE_SPACE;
  uint64_t *bars = reinterpret_cast<uint64_t *>(smem + TC_SPACE);
  uint64_t *full_bar = bars, *empty_bar = bars + STAGES;
  constexpr int BUFS = WIDE ? TC_TMEM_COLS / TC_WIDE : TC_ACC_BUFS, READERS = WIDE ? TC_WIDE_WARPS : TC_ACC_WARPS;
  uint64_t *acc_full = bars + 2 * STAGES, *acc_empty = acc_full + BUFS;
  uint64_t *corr_empty = acc_empty + BUFS, *drain_bar = corr_empty + 1, *team_bar = drain_bar + 1, *split_bar = team_bar + 1;
  uint64_t *done_full = split_bar + STAGES, *done_empty = done_full + TC_ACC_WARPS;     // one pair per accumulate warp
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(done_empty + TC_ACC_WARPS);
  volatile int *abort_flag = reinterpret_cast<volatile int *>(tmem_slot + 1);
  volatile int *skip_flag = abort_flag + 1;           // an earlier block gave up: this one does no work
  // wide: the layers that the block completed, but for the last one; set when every layer but the last is counted
  int *layers_done = reinterpret_cast<int *>(tmem_slot + 3);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = PAIR ? ptx::cluster_rank() : 0u;
  const int unit0 = (int)(PAIR ? blockIdx.x >> 1 : blockIdx.x), unit_step = (int)(PAIR ? gridDim.x >> 1 : gridDim.x);
  const int n_units = grp.unit_end[grp.n - 1];
  auto unit_of = [&](int round) { return round & 1 ? (round + 1) * unit_step - 1 - unit0 : round * unit_step + unit0; };

  if (threadIdx.x == 0) {
    for (int s = 0; s < STAGES; ++s) {
      ptx::mbar_init(&full_bar[s], 1);
      ptx::mbar_init(&empty_bar[s], 1);
      ptx::mbar_init(&split_bar[s], CG * TC_SPLIT_WARPS);
    }
    for (int b = 0; b < BUFS; ++b) {
      ptx::mbar_init(&acc_full[b], 1);
      ptx::mbar_init(&acc_empty[b], CG * READERS);
    }
    ptx::mbar_init(corr_empty, CG * TC_ACC_WARPS);
    ptx::mbar_init(drain_bar, 1);
    ptx::mbar_init(team_bar, READERS);
    for (int w = 0; w < TC_ACC_WARPS; ++w) {
      ptx::mbar_init(&done_full[w], 1);
      ptx::mbar_init(&done_empty[w], 1);
    }
    *abort_flag = 0;
    layers_done[0] = layers_done[1] = 0;
    ptx::fence_barrier_init();
  }
  if (warp == 1) ptx::tmem_alloc<CG>(tmem_slot, TC_TMEM_COLS);
  // Scaling exponents of every layer's operands (written by earlier kernels of the stream), and whether the planes made with
  // them are usable; only of layers this block works on: the step of a finished layer may already have changed the words of
  // the others.
  __shared__ int lay_exp[TC_MAX_GROUP][2];
  __shared__ double team_scratch[1 + READERS];
  __shared__ int lay_split[TC_MAX_GROUP];             // bit 0: A has to be split here, bit 1: B has
  __shared__ int lay_left[TC_MAX_GROUP];              // wide: accumulate warps that have left the layer
  if (warp == 2 && lane < grp.n) {
    const TcLayer<Epi> &y = grp.l[lane];
    const int begin = lane > 0 ? grp.unit_end[lane - 1] : 0, end = grp.unit_end[lane];
    bool has_unit = false;
    for (int k = begin / unit_step; k * unit_step < end && !has_unit; ++k) has_unit = unit_of(k) >= begin && unit_of(k) < end;
    lay_split[lane] = lay_left[lane] = 0;
    if (has_unit) {
      const int ea = y.oa.exp ? *y.oa.exp : 0, eb = y.ob.exp ? *y.ob.exp : 0;
      const uint32_t ma = y.oa.amax ? *y.oa.amax : 0u, mb = y.ob.amax ? *y.ob.amax : 0u;
      const bool good_a = y.oa.amax == nullptr || tc_planes_usable(ma, ea), good_b = y.ob.amax == nullptr || tc_planes_usable(mb, eb);
      // (a matrix of zeros is good whatever its exponent, that of no prediction included: any factor will do then)
      lay_exp[lane][0] = !good_a ? tc_scale_exp(ma) : ea < -100 || ea > 100 ? 0 : ea;
      lay_exp[lane][1] = !good_b ? tc_scale_exp(mb) : eb < -100 || eb > 100 ? 0 : eb;
      lay_split[lane] = (!good_a && y.oa.x != nullptr ? 1 : 0) | (!good_b && y.ob.x != nullptr ? 2 : 0);
    }
  }
  if (warp == 3 && lane == 0) {
    // One thread reads the error word for the whole block, so that all warps take the same path: every block still
    // allocates and releases its tensor memory and passes both block-wide barriers.
    *skip_flag = *reinterpret_cast<volatile int *>(grp.error) != 0;
    int g = 0;
    while (g + 1 < grp.n && unit0 >= grp.unit_end[g]) ++g;
    ptx::prefetch_tmap(&grp.l[g].a);
    ptx::prefetch_tmap(&grp.l[g].b);
    if (A_LO) ptx::prefetch_tmap(&grp.l[g].alo);
    if (B_LO) ptx::prefetch_tmap(&grp.l[g].blo);
    if (WIDE && STORES) ptx::prefetch_tmap(&grp.l[g].c);
  }
  ptx::tc_fence_before_sync();
  if constexpr (PAIR) ptx::cluster_sync();          // the barriers of both blocks are in place
  else __syncthreads();
  ptx::tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_slot;

  // Work unit -> its layer, row and column tile origin, first and number of K blocks, contraction slice; a unit is an output
  // tile or, in the tail, one contraction slice of an output tile.  Units are visited in ascending order.
  struct Tile { int g = 0, m0, n0, k_begin, n_kb, z, out, slice; };
  auto locate = [&](int unit, Tile &t) {
    while (unit >= grp.unit_end[t.g]) ++t.g;
    const TcLayer<Epi> &y = grp.l[t.g];
    if (t.g > 0) unit -= grp.unit_end[t.g - 1];
    t.out = unit; t.slice = -1;
    if (y.tail_split > 1 && unit >= y.tail_begin) {
      t.out = y.tail_begin + (unit - y.tail_begin) / y.tail_split;
      t.slice = (unit - y.tail_begin) % y.tail_split;
    }
    t.z = y.n_split == 1 ? 0 : y.tiles_mn(t.out);
    const int rem = t.out - t.z * y.tiles_mn.d, row = y.tiles_n(rem);
    t.m0 = row * TILE_M + (int)rank * TC_BM;       // of this block
    t.n0 = (rem - row * y.tiles_n.d) * TILE_N;
    t.k_begin = t.z * y.k_chunk;
    const int k_end = min(y.K, t.k_begin + y.k_chunk);
    t.n_kb = (max(k_end - t.k_begin, 0) + TC_BK - 1) / TC_BK;
    if (t.slice >= 0) {
      const int kb0 = t.slice * t.n_kb / y.tail_split, kb1 = (t.slice + 1) * t.n_kb / y.tail_split;
      t.k_begin += kb0 * TC_BK;
      t.n_kb = kb1 - kb0;
    }
  };

  auto n_slots = [](const TcLayer<Epi> &y) { return (y.M + TC_BM - 1) / TC_BM * ((y.N + TC_BN - 1) / TC_BN) * TC_ACC_WARPS; };
  // Adds this block's finished units of a layer to its count; 1 if that completes it.  What the caller waited for -- the sums and
  // maxima of every accumulate warp -- comes before the count.
  auto count_units = [&](int g, int visited) {
    const int units = (grp.unit_end[g] - (g > 0 ? grp.unit_end[g - 1] : 0)) * CG;
    __threadfence();
    return atomicAdd(grp.l[g].done, visited) + visited == units ? 1 : 0;
  };

  // Register budgets per warpgroup (every warp of a warpgroup executes the same instruction; the choice is
  // block-uniform, so a block that skips its work leaves the budgets alone).
  const bool skip = PAIR ? ptx::ld_cluster_int(ptx::cluster_addr(const_cast<int *>(skip_flag), 0)) != 0 : *skip_flag != 0;
  if (skip) {
    // nothing: do not queue work behind a block whose bounded wait expired
  } else if (warp < TC_ACC0) {
    ptx::setmaxnreg_dec<WIDE ? TC_WIDE_REGS_CTRL : TC_REGS_CTRL>();
    if (warp == 0) {
      // -------------------------------------------------------------- TMA producer (one lane)
      if (lane == 0) {
        int s = 0, it = 0;
        uint32_t ph = 1;                                // phase of the stage's previous use
        bool ok = true, any_split = false;
        for (int g = 0; g < grp.n; ++g) any_split |= lay_split[g] != 0;
        // `boxes` boxes of 64 output indices from o0 on
        auto load = [&](uint8_t *dst, const CUtensorMap *map, bool mn, int o0, int k0, int boxes) {
          const uint32_t bar = PAIR ? ptx::cluster_addr(&full_bar[s], 0) : ptx::smem_u32(&full_bar[s]);
          for (int i = 0; i < boxes; ++i)
            ptx::tma_load_2d<CG>(dst + i * TC_BOX_BYTES, map, mn ? o0 + 64 * i : k0, mn ? k0 : o0 + 64 * i, bar);
        };
        Tile t;
        for (int round = 0, unit = unit0; unit < n_units && ok; unit = unit_of(++round)) {
          locate(unit, t);
          const TcLayer<Epi> &y = grp.l[t.g];
          const bool split_a = lay_split[t.g] & 1, split_b = lay_split[t.g] & 2;
          const uint32_t tx = CG * (uint32_t)((split_a ? 0 : A_PLANES * TC_PLANE_BYTES) + (split_b ? 0 : B_PLANES * B_PLANE_BYTES));
          for (int kb = 0; kb < t.n_kb; ++kb, ++it) {
            if (it >= STAGES && !ptx::mbar_wait(&empty_bar[s], ph, abort_flag)) { ok = false; break; }
            uint8_t *st = smem + s * STAGE_BYTES;
            const int k0 = t.k_begin + kb * TC_BK;
            const int nb = t.n0 + (int)rank * BN;          // columns of B that this block loads
            if (rank == 0 && !any_split) ptx::mbar_expect_tx(&full_bar[s], tx);       // the bytes of both blocks
            if (!split_a) {
              load(st, &y.a, A_MN, t.m0, k0, 2);
              if (A_LO) load(st + TC_PLANE_BYTES, &y.alo, A_MN, t.m0, k0, 2);
            }
            if (!split_b) {
              load(st + B_OFF, &y.b, B_MN, nb, k0, BN / 64);
              if (B_LO) load(st + B_OFF + B_PLANE_BYTES, &y.blo, B_MN, nb, k0, BN / 64);
            }
            if (rank == 0 && any_split) {
              // what the splitting warps of both blocks have written comes before this arrival
              if (!ptx::mbar_wait(&split_bar[s], ph ^ 1u, abort_flag)) { ok = false; break; }
              if (PAIR) ptx::fence_cluster();
              ptx::mbar_expect_tx(&full_bar[s], tx);
            }
            if (++s == STAGES) { s = 0; ph ^= 1u; }
          }
        }
        if (*abort_flag && rank == 0) {
          // copies in flight must land before shared memory is released (block 1 of a pair is held by the cluster barrier at
          // the end).  A barrier that the splitting warps or the other block feed as well may never complete: its copies
          // are waited for until the limit of the wait.
          for (int j = max(it - STAGES, 0); j < it; ++j)      // (a stage that never got its arrival runs into the limit)
            ptx::mbar_wait(&full_bar[j % STAGES], (j / STAGES) & 1, abort_flag, 200000000ll, false);
        }
      }
    } else if (warp == 1) {
      // -------------------------------------------------------------- MMA issuer
      // The whole warp walks through the K blocks and one elected lane issues: everything an MMA needs then sits in uniform
      // registers.  (With a single lane running this loop, every descriptor word went through a vector register first: 416
      // cycles per K block on top of 72 per MMA.)
      if (rank == 0) {
        constexpr uint32_t idesc = ptx::idesc_f16(TILE_M, TILE_N, A_MN, B_MN);
        const uint32_t d_corr = tmem_base + TC_COL_CORR;        // (not of a wide tile)
        // descriptors with a constant high word; the low word of stage 0 advances by whole stages and K steps (16 values of
        // the contraction index: 32 bytes of every row if K-major, 16 rows if MN-major)
        const uint32_t hi_w = ptx::smem_desc_hi();
        const uint32_t lo_a0 = ptx::smem_desc_lo(ptx::smem_u32(smem), A_MN, TC_BOX_BYTES);
        const uint32_t lo_b0 = ptx::smem_desc_lo(ptx::smem_u32(smem) + B_OFF, B_MN, TC_BOX_BYTES);
        constexpr uint32_t step_a = (A_MN ? 2048u : 32u) >> 4, step_b = (B_MN ? 2048u : 32u) >> 4;
        constexpr uint32_t plane_a = TC_PLANE_BYTES >> 4, plane_b = B_PLANE_BYTES >> 4;
        bool ok = true;
        int splits = 0;
        for (int g = 0; g < grp.n; ++g) splits |= lay_split[g];
        const bool any_split = __any_sync(0xffffffffu, splits != 0);
        // running state: stage s with phase bit sp, accumulator buffer b with phase bit bp (of its *previous* use)
        int s = 0, b = 0, ti = 0, used = 0;
        uint32_t sp = 0, bp = 1;
        Tile t;
        for (int unit = unit0; unit < n_units && ok; unit = unit_of(++ti)) {
          locate(unit, t);
          const int n_kb = t.n_kb;
          for (int kb = 0; kb < n_kb; ++kb) {
            const bool first = kb % FLUSH == 0, last = kb % FLUSH == FLUSH - 1 || kb == n_kb - 1;
            bool good = ptx::mbar_wait(&full_bar[s], sp, abort_flag);
            if (first && used >= BUFS) good = good && ptx::mbar_wait(&acc_empty[b], bp, abort_flag);
            ok = __all_sync(0xffffffffu, good);
            if (!ok) break;
            if (PAIR && any_split) ptx::fence_cluster();
            ptx::tc_fence_after_sync();
            const uint32_t la = lo_a0 + (uint32_t)s * (STAGE_BYTES >> 4), lb = lo_b0 + (uint32_t)s * (STAGE_BYTES >> 4);
            const uint32_t d = tmem_base + (uint32_t)(b * TILE_N);
            auto desc_a = [&](int kk, bool lo) { return ptx::smem_desc(hi_w, la + (lo ? plane_a : 0u) + kk * step_a); };
            auto desc_b = [&](int kk, bool lo) { return ptx::smem_desc(hi_w, lb + (lo ? plane_b : 0u) + kk * step_b); };
            const bool corr_busy = !COARSE && !WIDE && kb == 0 && ti > 0;
            if (corr_busy) {
              // The correction tile still holds the previous output tile until the accumulate warps have read it:
              // the main-term MMAs of this block, which do not touch it, go first and keep the tensor pipe busy
              // while that read finishes.
              if (ptx::elect_one()) {
#pragma unroll
                for (int kk = 0; kk < TC_KSTEPS; ++kk) ptx::mma_f16<CG, ptx::A_ONCE>(d, desc_a(kk, false), desc_b(kk, false), idesc, kk > 0);
              }
              ok = __all_sync(0xffffffffu, ptx::mbar_wait(corr_empty, (ti - 1) & 1, abort_flag));
              if (!ok) break;
              ptx::tc_fence_after_sync();
            }
            if (ptx::elect_one()) {
              if constexpr (WIDE && !COARSE) {
                // into one accumulator: the correction terms first, which are small; the first MMA of the main term scales their
                // sum by 2^-11
#pragma unroll
                for (int kk = 0; kk < TC_KSTEPS; ++kk) {
                  if (A_LO) ptx::mma_f16<CG, ptx::A_ONCE>(d, desc_a(kk, true), desc_b(kk, false), idesc, kk > 0);
                  if (B_LO) ptx::mma_f16<CG, ptx::A_ONCE>(d, desc_a(kk, false), desc_b(kk, true), idesc, A_LO || kk > 0);
                }
                ptx::mma_f16_scaled<CG>(d, desc_a(0, false), desc_b(0, false), idesc);
#pragma unroll
                for (int kk = 1; kk < TC_KSTEPS; ++kk) ptx::mma_f16<CG, ptx::A_ONCE>(d, desc_a(kk, false), desc_b(kk, false), idesc, true);
              } else if (corr_busy) {
#pragma unroll
                for (int kk = 0; kk < TC_KSTEPS; ++kk) {
                  // the first correction MMA of a tile overwrites the tile, every later one accumulates
                  if (B_LO) ptx::mma_f16<CG, ptx::A_ONCE>(d_corr, desc_a(kk, false), desc_b(kk, true), idesc, kk > 0);
                  if (A_LO) ptx::mma_f16<CG, ptx::A_ONCE>(d_corr, desc_a(kk, true), desc_b(kk, false), idesc, B_LO || kk > 0);
                }
              } else {
#pragma unroll
                for (int kk = 0; kk < TC_KSTEPS; ++kk) {
                  if constexpr (COARSE) {
                    ptx::mma_f16<CG, ptx::A_ONCE>(d, desc_a(kk, false), desc_b(kk, false), idesc, !first || kk > 0);
                  } else {
                    // A_hi serves two MMAs in a row: the second takes it from the collector
                    ptx::mma_f16<CG, B_LO ? ptx::A_KEEP : ptx::A_ONCE>(d, desc_a(kk, false), desc_b(kk, false), idesc, !first || kk > 0);
                    if (B_LO) ptx::mma_f16<CG, ptx::A_AGAIN>(d_corr, desc_a(kk, false), desc_b(kk, true), idesc, kb > 0 || kk > 0);
                    if (A_LO) ptx::mma_f16<CG, ptx::A_ONCE>(d_corr, desc_a(kk, true), desc_b(kk, false), idesc, B_LO || kb > 0 || kk > 0);
                  }
                }
              }
              ptx::mma_commit<CG>(&empty_bar[s]);          // stage can be refilled once these MMAs have read it
              if (last) ptx::mma_commit<CG>(&acc_full[b]);      // the group's partial product is complete
            }
            if (last) {
              ++used;
              if (++b == BUFS) { b = 0; bp ^= 1u; }
            }
            if (++s == STAGES) { s = 0; sp ^= 1u; }
          }
        }
        if (!ok) {
          // after an abandoned wait: let the MMAs already issued finish before tensor memory is released
          if (ptx::elect_one()) ptx::mma_commit<CG>(drain_bar, false);
          ptx::mbar_wait(drain_bar, 0, abort_flag, 200000000ll, false);
        }
      }
    } else {
      // -------------------------------------------------------------- planes of a refused operand (two warps)
      // Once a layer of this block needs them, they and the producer go through every stage together: a waiter that lags by
      // more than one phase of a barrier would take an earlier completion of the same parity for its own.
      const int t = threadIdx.x - 32 * TC_SPLIT0;
      auto split_tile = [&](const TcOperand &o, bool mn, bool lo_too, float scale, uint8_t *dst, int boxes, int o0, int k0, int n_outer, int n_k) {
        // K-major: 64 or 128 rows of 8 chunks, inner = contraction; MN-major: 64 rows of 8 or 16 chunks, inner = output index
        const int rows = mn ? n_k - k0 : n_outer - o0, chunks = mn ? 8 * boxes : 8, inner0 = mn ? o0 : k0;
        const float *src = o.x + (size_t)(mn ? k0 : o0) * o.ld + inner0;
#pragma unroll 4
        for (int i = t; i < 512 * boxes; i += 32 * TC_SPLIT_WARPS) {
          const int r = i / chunks, c = i % chunks;
          float4 x0 = make_float4(0.f, 0.f, 0.f, 0.f), x1 = x0;
          if (r < rows) {                      // rows are padded with zeros to ld, a multiple of 4
            if (inner0 + 8 * c + 4 <= o.ld) x0 = *reinterpret_cast<const float4 *>(src + (size_t)r * o.ld + 8 * c);
            if (inner0 + 8 * c + 8 <= o.ld) x1 = *reinterpret_cast<const float4 *>(src + (size_t)r * o.ld + 8 * c + 4);
          }
          uint4 h, l;
          tc_split8(x0, x1, scale, h, l);
          const uint32_t off = (uint32_t)(c >> 3) * TC_BOX_BYTES + (uint32_t)r * 128u + (((uint32_t)(c & 7) ^ (uint32_t)(r & 7)) << 4);
          *reinterpret_cast<uint4 *>(dst + off) = h;
          if (lo_too) *reinterpret_cast<uint4 *>(dst + boxes * TC_BOX_BYTES + off) = l;
        }
      };
      // Wide tiles: warp 3 counts the tiles of a layer that the block has no further unit of, once the accumulate warps have arrived,
      // and notes the layers that this completes; the accumulate warps add those layers' slots at the end.  (With the accumulate
      // warps counting, and waiting for one another, at every change of layer the tensor cores stood still; with warp 3
      // adding the slots as well one block became the last of every layer, one after the other.)
      // A count for each layer, not a barrier: the accumulate warps may be several layers ahead, and ahead of one another (by the two
      // accumulators, which is two layers where a layer's tile is one read-out), so that in a common count the arrivals of warps that
      // are ahead would stand for those of one that has not written its sums yet.
      int visited = 0;
      auto leave = [&](int g) {
        const long long t0 = clock64();
        while (*reinterpret_cast<volatile int *>(lay_left + g) < TC_WIDE_WARPS) {
          if (*abort_flag) return false;
          if (clock64() - t0 > 1000000000ll) { *abort_flag = 1; return false; }
          __nanosleep(100);
        }
        if (lane == 0 && count_units(g, visited)) layers_done[0] |= 1 << g;
        return true;
      };
      int s = 0, it = 0;
      uint32_t ph = 1;
      bool ok = true, any_split = false;
      for (int g = 0; g < grp.n; ++g) any_split |= lay_split[g] != 0;
      const bool counts = WIDE && Epi::kSumsq && warp == 3 && grp.n > 1;
      Tile u;
      for (int round = 0, unit = unit0; unit < n_units && ok && (counts || any_split); unit = unit_of(++round)) {
        int g_before = u.g;
        locate(unit, u);
        if (round == 0) g_before = u.g;
        const TcLayer<Epi> &y = grp.l[u.g];
        const int split = lay_split[u.g];
        const float scale_a = tc_pow2(lay_exp[u.g][0]), scale_b = tc_pow2(lay_exp[u.g][1]);
        for (int kb = 0; any_split && kb < u.n_kb; ++kb, ++it) {
          ok = it < STAGES || ptx::mbar_wait(&empty_bar[s], ph, abort_flag);
          if (!__all_sync(0xffffffffu, ok)) { ok = false; break; }
          uint8_t *st = smem + s * STAGE_BYTES;
          const int k0 = u.k_begin + kb * TC_BK;
          if (split & 1) split_tile(y.oa, A_MN, A_LO, scale_a, st, 2, u.m0, k0, y.M, y.K);
          if (split & 2) split_tile(y.ob, B_MN, B_LO, scale_b, st + B_OFF, BN / 64, u.n0 + (int)rank * BN, k0, y.N, y.K);
          if (split != 0) {
            ptx::fence_proxy_async_smem();
            if (PAIR) ptx::fence_cluster();
          }
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive_cluster(ptx::cluster_addr(&split_bar[s], 0));      // (every stage: the phases stay in step)
          if (++s == STAGES) { s = 0; ph ^= 1u; }
        }
        if (ok && counts) {
          // (the accumulate warps finish the layer before during the first tile of the next one, for which nothing may be left
          // to do here)
          if (u.g != g_before) {
            ok = grp.l[g_before].slots == nullptr || __all_sync(0xffffffffu, leave(g_before));
            visited = 0;
          }
          ++visited;
        }
      }
      if (counts && ok && lane == 0) {
        __threadfence_block();
        *reinterpret_cast<volatile int *>(layers_done + 1) = 1;
      }
    }
  } else if constexpr (WIDE) {
    // ---------------------------------------------------------------- wide tiles
    ptx::setmaxnreg_inc<TC_WIDE_REGS_ACC>();
    // Accumulate warp aw: rows of quarter aw mod 4, columns 64 (aw / 4) .. +63 of every tile of the block.
    const int aw = warp - TC_ACC0, quarter = warp & 3, col_base = 64 * (aw >> 2), lane_base = quarter * 32;
    float *buf = reinterpret_cast<float *>(tr_base + (size_t)aw * TC_WIDE_PART_BYTES);
    bool ok = true;
    Tile t;
    int visited = 0;                                   // units of layer t.g that this block has finished
    // The accumulate warps among themselves, bounded like every other wait.
    uint32_t team_ph = 0;
    auto team_sync = [&]() {
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(team_bar);
      const bool there = ptx::mbar_wait(team_bar, team_ph, abort_flag);
      team_ph ^= 1u;
      return __all_sync(0xffffffffu, there) != 0;
    };
    // The block has no further unit: add the slots of every layer that it completed, the last one with this.
    auto leave_last = [&](int g_last) {
      if (!Epi::kSumsq) return;
      volatile int *mask_sh = reinterpret_cast<volatile int *>(team_scratch);
      volatile double *part = team_scratch + 1;
      if (!team_sync()) return;
      if (aw == 0 && lane == 0) {
        int mask = grp.l[g_last].slots != nullptr && count_units(g_last, visited) ? 1 << g_last : 0;
        if (grp.n > 1) {
          const long long t0 = clock64();
          while (*reinterpret_cast<volatile int *>(layers_done + 1) == 0 && !*abort_flag)
            if (clock64() - t0 > 1000000000ll) *abort_flag = 1;
          __threadfence();
          mask |= *reinterpret_cast<volatile int *>(layers_done);
        }
        *mask_sh = *abort_flag ? 0 : mask;
      }
      if (!team_sync()) return;
      const int mask = *mask_sh;
      for (int g = 0; mask >> g; ++g) {
        if (!(mask >> g & 1)) continue;
        const TcLayer<Epi> &y = grp.l[g];
        __threadfence();
        const int n = n_slots(y);
        double v = 0.0;
#pragma unroll 16
        for (int i = aw * 32 + lane; i < n; i += 32 * TC_WIDE_WARPS) v += __ldcg(y.slots + i);
        v = warp_sum(v);
        if (lane == 0) part[aw] = v;
        if (!team_sync()) return;
        if (aw == 0 && lane == 0) {
          double sum = 0.0;
          for (int w = 0; w < TC_WIDE_WARPS; ++w) sum += part[w];
          *y.done = 0;
          finish_step(y.step, sum);
        }
        if (!team_sync()) return;
      }
    };
    auto put_sum = [&](const TcLayer<Epi> &y, double v) {
      v = warp_sum(v);
      const int tiles_n = (y.N + TC_BN - 1) / TC_BN, tile = t.n0 / TC_BN + (aw >> 3);
      if (lane == 0 && t.m0 < y.M && tile < tiles_n) y.slots[((size_t)(t.m0 / TC_BM) * tiles_n + tile) * TC_ACC_WARPS + (aw & 7)] = v;
    };
    int b = 0;
    uint32_t ph = 0;                                   // phase of acc_full[b]
    const uint32_t tm_lane = tmem_base + ((uint32_t)lane_base << 16) + (uint32_t)col_base;
    for (int round = 0, unit = unit0; unit < n_units && ok; unit = unit_of(++round)) {
      const int g_before = t.g;
      locate(unit, t);
      if (round > 0 && t.g != g_before) {
        visited = 0;
        if (Epi::kSumsq && grp.l[g_before].slots != nullptr) {
          __syncwarp();
          if (lane == 0) {
            __threadfence_block();
            atomicAdd(lay_left + g_before, 1);
          }
        }
      }
      ++visited;
      const TcLayer<Epi> &y = grp.l[t.g];
      const int n_grp = (t.n_kb + FLUSH - 1) / FLUSH;    // read-outs of an accumulator for this tile
      uint64_t acc[32];                                  // columns 2 j, 2 j + 1 in acc[j]
#pragma unroll
      for (int j = 0; j < 32; ++j) acc[j] = 0ull;
      for (int g = 0; g < n_grp; ++g) {
        ok = __all_sync(0xffffffffu, ptx::mbar_wait(&acc_full[b], ph, abort_flag));
        if (!ok) break;
        ptx::tc_fence_after_sync();
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          uint32_t v[16];
          ptx::tmem_ld16(tm_lane + (uint32_t)(b * TC_WIDE + 16 * c), v);
          ptx::tmem_ld_wait(v);
          if (c == 3) {
            // the accumulator is given back (one arrival per warp on block 0's barrier, whose MMA warp waits) as soon as its last
            // columns are in registers
            ptx::tc_fence_before_sync();
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive_cluster(ptx::cluster_addr(&acc_empty[b], 0));
          }
#pragma unroll
          for (int j = 0; j < 8; ++j) acc[8 * c + j] = ptx::add_f2(acc[8 * c + j], ptx::pack_f2(v[2 * j], v[2 * j + 1]));
        }
        if (++b == BUFS) { b = 0; ph ^= 1u; }
      }
      if (!ok) break;
      {
        // undo the operand scalings (an exact factor, or two where one would leave the range)
        const int e = lay_exp[t.g][0] + lay_exp[t.g][1], e1 = e >= -120 && e <= 120 ? e : e / 2, e2 = e - e1;
        const uint32_t u1 = __float_as_uint(tc_pow2(-e1)), u2 = __float_as_uint(tc_pow2(-e2));
        const uint64_t w1 = ptx::pack_f2(u1, u1), w2 = ptx::pack_f2(u2, u2);
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = ptx::mul_f2(acc[j], w1);
        if (e2 != 0) {
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] = ptx::mul_f2(acc[j], w2);
        }
        if constexpr (ZERO != 0) {
          const uint64_t mul = ptx::pack_f2(__float_as_uint(y.mul), __float_as_uint(y.mul));
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] = ptx::mul_f2(acc[j], mul);
        }
      }
      if (STORES && t.slice >= 0) {
        // contraction slice of a tail tile: park the piece; the last warp to arrive adds the slices, in slice order
        constexpr int PIECES = CG * TC_WIDE_WARPS;
        const int t_idx = t.out - y.tail_begin, piece = (int)rank * TC_WIDE_WARPS + aw;
        float4 *part = reinterpret_cast<float4 *>(y.tail_ws) + ((size_t)t_idx * y.tail_split * PIECES + piece) * 512 + lane;
        constexpr size_t SLICE = (size_t)PIECES * 512;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          float4 v;
          ptx::unpack_f2(acc[2 * j], v.x, v.y);
          ptx::unpack_f2(acc[2 * j + 1], v.z, v.w);
          part[t.slice * SLICE + j * 32] = v;
        }
        __syncwarp();
        int prev = 0;
        if (lane == 0) {
          __threadfence();             // of the whole warp's parked values
          prev = atomicAdd(y.tail_count + t_idx * PIECES + piece, 1);
        }
        prev = __shfl_sync(0xffffffffu, prev, 0);
        if (prev != y.tail_split - 1) continue;
        __threadfence();
        if (lane == 0) y.tail_count[t_idx * PIECES + piece] = 0;
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = 0ull;
        for (int sl = 0; sl < y.tail_split; ++sl) {
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float4 v = __ldcg(part + sl * SLICE + j * 32);
            acc[2 * j] = ptx::add_f2(acc[2 * j], ptx::pack_f2(__float_as_uint(v.x), __float_as_uint(v.y)));
            acc[2 * j + 1] = ptx::add_f2(acc[2 * j + 1], ptx::pack_f2(__float_as_uint(v.z), __float_as_uint(v.w)));
          }
        }
      }
      // Parts of 32 rows x 16 columns, a row per lane, go into the warp's buffer (16-byte groups XOR-ed as the copy's 64-byte swizzle
      // wants them, which is free of bank conflicts) and out by a bulk copy; rows and columns outside the matrix are clipped.
      // Columns up to the leading dimension are written: those from N on come out as exact zeros, which keeps the padding of every
      // matrix zero.  The sum of squares and the largest magnitude (rows and columns outside hold exact zeros) are taken while a
      // copy reads the buffer: one after the other the end of a tile took 8000 cycles, of which the MMAs run ahead 3000.
      const int row0 = t.m0 + lane_base;
      uint64_t s2[4] = {0ull, 0ull, 0ull, 0ull};
      uint32_t mx = 0u;
      const bool wants_sum = Epi::kSumsq && y.slots != nullptr;
      bool wants_max = false;
      if constexpr (epi_amax<Epi>::value) wants_max = y.epi.amax != nullptr;
#pragma unroll
      for (int p = 0; p < 4; ++p) {
        if constexpr (STORES) {
          const int col = t.n0 + col_base + TC_WIDE_PART * p;
          ptx::bulk_wait_read();                       // (of the lane that copied) the buffer is free again
          __syncwarp();
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            float4 v;
            ptx::unpack_f2(acc[8 * p + 2 * j], v.x, v.y);
            ptx::unpack_f2(acc[8 * p + 2 * j + 1], v.z, v.w);
            reinterpret_cast<float4 *>(buf)[lane * 4 + (j ^ ((lane >> 1) & 3))] = v;
          }
          ptx::fence_proxy_async_smem();
          __syncwarp();
          if (lane == 0 && row0 < y.M && col < y.epi.ldc) {
            ptx::tma_store_3d(&y.c, buf, col, row0, t.z);
            ptx::bulk_commit();
          }
        }
        if (Epi::kSumsq && wants_sum) {
#pragma unroll
          for (int j = 0; j < 8; ++j) s2[j & 3] = ptx::fma_f2(acc[8 * p + j], acc[8 * p + j], s2[j & 3]);
        }
        if constexpr (epi_amax<Epi>::value) {
          if (wants_max) {
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              float a0, a1;
              ptx::unpack_f2(acc[8 * p + j], a0, a1);
              mx = __vimax3_u32(mx, abs_bits(a0), abs_bits(a1));
            }
          }
        }
      }
      if (Epi::kSumsq && wants_sum) {
        float s4[8];
#pragma unroll
        for (int j = 0; j < 4; ++j) ptx::unpack_f2(s2[j], s4[2 * j], s4[2 * j + 1]);
        put_sum(y, (((double)s4[0] + (double)s4[1]) + ((double)s4[2] + (double)s4[3])) + (((double)s4[4] + (double)s4[5]) + ((double)s4[6] + (double)s4[7])));
      }
      if constexpr (epi_amax<Epi>::value) {
        if (wants_max) commit_amax(mx, y.epi.amax);      // the output is an operand of a later product
      }
    }
    if (STORES) ptx::bulk_wait_all();                 // before shared memory goes, and before the sums are announced
    __syncwarp();
    if (ok) leave_last(t.g);
  } else {
    // Accumulate warp aw and epilogue warp aw: rows of quarter aw mod 4, columns col_base .. +63 of every tile of the block.
    const bool accumulates = warp < TC_EPI0;
    const int aw = warp - (accumulates ? TC_ACC0 : TC_EPI0), quarter = warp & 3, col_base = 64 * (aw >> 2);
    const int lane_base = quarter * 32, piece = (int)rank * TC_ACC_WARPS + aw;
    // The warp pair's piece of the finished tile (or one half of its rows after the other): row i at 16 i, its 16 float4 groups
    // with the group index XOR-ed by (i mod 8), so that both sides (a lane per row; 16 lanes per row) are free of bank conflicts.
    constexpr int PART_ROWS = PARTS == 2 ? 16 : 32, PART_F4 = PART_ROWS * 16;
    float4 *tr = reinterpret_cast<float4 *>(tr_base) + (size_t)aw * PART_F4;
    bool ok = true;
    Tile t;
    int visited = 0;                                   // units of layer t.g that this block has finished
    // The eight warps that know the sums of squares (the epilogue warps; the accumulate warps if nothing is stored), bounded
    // like every other wait.
    uint32_t team_ph = 0;
    auto team_sync = [&]() {
      __syncwarp();
      if (lane == 0) ptx::mbar_arrive(team_bar);
      const bool there = ptx::mbar_wait(team_bar, team_ph, abort_flag);
      team_ph ^= 1u;
      return __all_sync(0xffffffffu, there) != 0;
    };
    // The block has no further unit of layer g: if every unit of the layer is finished with this, add the slots.
    auto leave = [&](int g) {
      const TcLayer<Epi> &y = grp.l[g];
      if (!Epi::kSumsq || y.slots == nullptr || visited == 0) return true;
      constexpr int n_threads = 32 * TC_ACC_WARPS;
      const int tid = aw * 32 + lane;
      volatile int *last = reinterpret_cast<volatile int *>(team_scratch);
      volatile double *part = team_scratch + 1;
      if (!team_sync()) return false;
      if (tid == 0) {
        const int units = (grp.unit_end[g] - (g > 0 ? grp.unit_end[g - 1] : 0)) * CG;
        __threadfence();                 // the team's sums and maxima, which its arrivals put before this, come before the count
        const int before = atomicAdd(y.done, visited);
        *last = before + visited == units;
      }
      if (!team_sync()) return false;
      if (*last != 0) {
        __threadfence();
        const int n = n_slots(y);
        double v = 0.0;
#pragma unroll 4
        for (int i = tid; i < n; i += n_threads) v += __ldcg(y.slots + i);
        v = warp_sum(v);
        if (lane == 0) part[aw] = v;
        if (!team_sync()) return false;
        if (tid == 0) {
          double sum = 0.0;
          for (int i = 0; i < TC_ACC_WARPS; ++i) sum += part[i];
          *y.done = 0;
          finish_step(y.step, sum);
        }
      }
      visited = 0;
      return team_sync();                              // the scratch is free again
    };
    auto put_sum = [&](const TcLayer<Epi> &y, double v) {
      v = warp_sum(v);
      const int tiles_n = (y.N + TC_BN - 1) / TC_BN;
      if (lane == 0) y.slots[((size_t)(t.m0 / TC_BM) * tiles_n + t.n0 / TC_BN) * TC_ACC_WARPS + aw] = v;
    };
    if (accumulates) {
      ptx::setmaxnreg_inc<TC_REGS_ACC>();
      // ------------------------------------------------------------ accumulate
      int b = 0;
      uint32_t ph = 0, handed = 0;                     // phase of acc_full[b]; parts handed over so far
      for (int round = 0, unit = unit0; unit < n_units && ok; unit = unit_of(++round)) {
        const int g_before = t.g;
        locate(unit, t);
        if (!STORES) {
          if (t.g != g_before && !leave(g_before)) { ok = false; break; }
          ++visited;
        }
        const TcLayer<Epi> &y = grp.l[t.g];
        const int n_grp = (t.n_kb + FLUSH - 1) / FLUSH;   // read-outs of the main accumulator for this tile
        uint64_t acc[32];                             // columns 2 j, 2 j + 1 in acc[j]
#pragma unroll
        for (int j = 0; j < 32; ++j) acc[j] = 0ull;
        // acc += tile (or tile * 2^-11).  The tile is given back (one arrival per warp on `done` of block 0, whose MMA thread
        // waits) as soon as its last columns are in registers.
        auto add_tile = [&](uint32_t col, auto plain, uint64_t *done) {
          const uint32_t src = tmem_base + ((uint32_t)lane_base << 16) + col + (uint32_t)col_base;
          uint32_t v[32];
          auto add = [&](int h) {
            const uint64_t w = ptx::pack_f2(0x3A000000u, 0x3A000000u);       // 2^-11 twice
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const uint64_t x = ptx::pack_f2(v[2 * j], v[2 * j + 1]);
              acc[16 * h + j] = decltype(plain)::value ? ptx::add_f2(acc[16 * h + j], x) : ptx::fma_f2(w, x, acc[16 * h + j]);
            }
          };
          ptx::tmem_ld32(src, v);
          ptx::tmem_ld_wait(v);
          add(0);
          ptx::tmem_ld32(src + 32u, v);
          ptx::tmem_ld_wait(v);
          ptx::tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) ptx::mbar_arrive_cluster(ptx::cluster_addr(done, 0));
          add(1);
        };
        for (int g = 0; g < n_grp && ok; ++g) {
          ok = ptx::mbar_wait(&acc_full[b], ph, abort_flag);
          if (!ok) break;
          ptx::tc_fence_after_sync();
          add_tile((uint32_t)(b * TC_BN), std::true_type{}, &acc_empty[b]);
          if (++b == TC_ACC_BUFS) { b = 0; ph ^= 1u; }
        }
        if (!ok) break;
        if (t.n_kb > 0) {
          // correction terms: complete once the last block's commit has arrived (it covers every earlier MMA)
          if constexpr (!COARSE) add_tile(TC_COL_CORR, std::false_type{}, corr_empty);
          // undo the operand scalings (two exact factors, so that neither leaves the range on its own)
          const int e = lay_exp[t.g][0] + lay_exp[t.g][1], e1 = e / 2, e2 = e - e1;
          const uint32_t u1 = __float_as_uint(tc_pow2(-e1)), u2 = __float_as_uint(tc_pow2(-e2));
          const uint64_t w1 = ptx::pack_f2(u1, u1), w2 = ptx::pack_f2(u2, u2);
#pragma unroll
          for (int j = 0; j < 32; ++j) acc[j] = ptx::mul_f2(ptx::mul_f2(acc[j], w1), w2);
          if constexpr (ZERO != 0) {
            const uint64_t mul = ptx::pack_f2(__float_as_uint(y.mul), __float_as_uint(y.mul));
#pragma unroll
            for (int j = 0; j < 32; ++j) acc[j] = ptx::mul_f2(acc[j], mul);
          }
        }
        if constexpr (!STORES) {
          // only the squared norm: straight from the registers (rows and columns outside the matrix hold exact zeros)
          uint64_t s2[2] = {0ull, 0ull};
#pragma unroll
          for (int j = 0; j < 32; ++j) s2[j & 1] = ptx::fma_f2(acc[j], acc[j], s2[j & 1]);
          float s4[4];
          ptx::unpack_f2(s2[0], s4[0], s4[1]);
          ptx::unpack_f2(s2[1], s4[2], s4[3]);
          if (y.slots != nullptr && t.m0 < y.M) put_sum(y, ((double)s4[0] + (double)s4[1]) + ((double)s4[2] + (double)s4[3]));
        } else {
          // hand the piece over; the epilogue warp has finished with the previous one
#pragma unroll
          for (int h = 0; h < PARTS; ++h) {
            ok = ok && __all_sync(0xffffffffu, ptx::mbar_wait(&done_empty[aw], (handed & 1u) ^ 1u, abort_flag));
            if (!ok) break;
            ++handed;
            if (PARTS == 1 || (lane >> 4) == h) {
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                float4 v;
                ptx::unpack_f2(acc[2 * j], v.x, v.y);
                ptx::unpack_f2(acc[2 * j + 1], v.z, v.w);
                tr[(lane & (PART_ROWS - 1)) * 16 + (j ^ (lane & 7))] = v;
              }
            }
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&done_full[aw]);
          }
          if (!ok) break;
        }
      }
      if (!STORES && ok) leave(t.g);
    } else {
      ptx::setmaxnreg_dec<TC_REGS_EPI>();
      // ------------------------------------------------------------ epilogue
      // The warp walks over its 32 rows two at a time: lanes 16 k .. +15 take row 2 step + k, 4 consecutive columns per lane, so
      // that every access is two runs of 256 bytes.  The loads of eight steps are issued together (rows past the end are
      // clamped, their results dropped).
      if constexpr (STORES) {
        uint32_t taken = 0;
        for (int round = 0, unit = unit0; unit < n_units && ok; unit = unit_of(++round)) {
          const int g_before = t.g;
          locate(unit, t);
          if (t.g != g_before && !leave(g_before)) { ok = false; break; }
          ++visited;
          const TcLayer<Epi> &y = grp.l[t.g];
          const Epi epi = y.epi;
          const int row0 = t.m0 + lane_base + (lane >> 4), col = t.n0 + col_base + 4 * (lane & 15);
          // columns up to the leading dimension are written: those from N on come out as exact zeros (zero-filled
          // operand rows, zero padding of the epilogue inputs), which keeps the padding of every matrix zero
          const bool col_in = col < epi.ldc;
          if (t.m0 + lane_base + lane < y.M) {          // this lane's row of the epilogue inputs, on its way to L2
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const int c = t.n0 + col_base + h * 32;
              if (c < epi.ldc) epi.prefetch(t.m0 + lane_base + lane, c);
            }
          }
          // the inputs of the first eight steps are on their way before the tile is complete
          float4 in[8][Epi::kInputs > 0 ? Epi::kInputs : 1];
          auto load_inputs = [&](int s0) {
#pragma unroll
            for (int i = 0; i < 8; ++i)
              if constexpr (!Epi::kDirect) epi.load(min(row0 + 2 * (s0 + i), y.M - 1), col, in[i]);
          };
          float h_scale = 0.f;               // scaling of the planes of the result, if they are wanted
          if constexpr (epi_planes<Epi>::value) {
            if (epi.H != nullptr) h_scale = tc_scale_of(*epi.h_exp);
          }
          if (col_in) load_inputs(0);
          float *C = epi.C + (size_t)t.z * y.c_split_stride;
          float ssf = 0.f;
          uint32_t mx = 0u;                  // largest magnitude stored by this thread
          auto wait_part = [&]() { return __all_sync(0xffffffffu, ptx::mbar_wait(&done_full[aw], taken++ & 1u, abort_flag)) != 0; };
          auto release_part = [&]() {
            __syncwarp();
            if (lane == 0) ptx::mbar_arrive(&done_empty[aw]);
          };
          auto at = [&](int i) { const int r = 2 * i + (lane >> 4); return r * 16 + ((lane & 15) ^ (r & 7)); };     // step i of a part
          // eight steps, value i from get(i), whose inputs have been loaded
          auto finish_half = [&](int h, auto get) {
            if (!col_in) return;
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const int row = row0 + 16 * h + 2 * i;
              float4 o = get(i);
              if (row >= y.M) continue;
              if constexpr (epi_sumsq_acc<Epi>::value) ssf = fmaf(o.x, o.x, fmaf(o.y, o.y, fmaf(o.z, o.z, fmaf(o.w, o.w, ssf))));
              if constexpr (!Epi::kDirect) o = epi.apply(col, o, in[i]);
              if (Epi::kSumsq && !epi_sumsq_acc<Epi>::value) ssf = fmaf(o.x, o.x, fmaf(o.y, o.y, fmaf(o.z, o.z, fmaf(o.w, o.w, ssf))));
              *reinterpret_cast<float4 *>(C + (size_t)row * epi.ldc + col) = o;
              if constexpr (epi_planes<Epi>::value) {
                if (epi.H != nullptr) {
                  uint2 hi, lo;
                  tc_split4(o, h_scale, hi, lo);
                  *reinterpret_cast<uint2 *>(epi.H + (size_t)row * epi.ldc + col) = hi;
                  if (epi.L != nullptr) *reinterpret_cast<uint2 *>(epi.L + (size_t)row * epi.ldc + col) = lo;
                }
              }
              if constexpr (epi_amax<Epi>::value) mx = max(mx, abs_bits(o));
            }
          };
          const int t_idx = t.out - y.tail_begin;
          bool whole = t.slice < 0;
          if (!whole) {
            // contraction slice of a tail tile: park the piece; the last warp to arrive sums the slices
            float4 *mine = reinterpret_cast<float4 *>(y.tail_ws) + ((size_t)(t_idx * y.tail_split + t.slice) * WARPS + piece) * 512;
#pragma unroll 1
            for (int h = 0; h < PARTS && ok; ++h) {
              ok = wait_part();
              if (!ok) break;
#pragma unroll 4
              for (int j = 0; j < PART_F4 / 32; ++j) mine[h * PART_F4 + j * 32 + lane] = tr[j * 32 + lane];
              release_part();
            }
            if (!ok) break;
            __syncwarp();
            int prev = 0;
            if (lane == 0) {
              __threadfence();             // of the whole warp's parked values
              prev = atomicAdd(y.tail_count + t_idx * WARPS + piece, 1);
            }
            prev = __shfl_sync(0xffffffffu, prev, 0);
            whole = prev == y.tail_split - 1;
            if (whole) {
              __threadfence();
              if (lane == 0) y.tail_count[t_idx * WARPS + piece] = 0;
            }
          }
          if (whole) {
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
              if (h > 0 && col_in) load_inputs(8);
              if (t.slice >= 0) {
                const float4 *part = reinterpret_cast<const float4 *>(y.tail_ws) + ((size_t)t_idx * y.tail_split * WARPS + piece) * 512 + h * 256;
                finish_half(h, [&](int i) {
                  float4 a = make_float4(0.f, 0.f, 0.f, 0.f);
                  for (int sl = 0; sl < y.tail_split; ++sl) {
                    const float4 v = __ldcg(part + (size_t)sl * WARPS * 512 + at(i));
                    a.x += v.x; a.y += v.y; a.z += v.z; a.w += v.w;
                  }
                  return a;
                });
                continue;
              }
              if (h == 0 || PARTS == 2) ok = wait_part();
              if (!ok) break;
              const float4 *src = tr + (PARTS == 2 ? 0 : h * 256);
              finish_half(h, [&](int i) { return src[at(i)]; });
              if (h == 1 || PARTS == 2) release_part();
            }
            if (!ok) break;
            if constexpr (epi_amax<Epi>::value) {
              if (epi.amax != nullptr) commit_amax(mx, epi.amax);      // the output is an operand of a later product
            }
            if (Epi::kSumsq && y.slots != nullptr && t.m0 < y.M) put_sum(y, (double)ssf);
          }
        }
        if (ok) leave(t.g);
      }
    }
  }
  ptx::tc_fence_before_sync();
  // neither block of a pair leaves while the other may still arrive on its barriers or read its shared memory
  if constexpr (PAIR) ptx::cluster_sync();
  else __syncthreads();
  if (warp == 1) {
    ptx::tc_fence_after_sync();
    ptx::tmem_dealloc<CG>(tmem_base, TC_TMEM_COLS);
  }
  if (threadIdx.x == 0 && *abort_flag) atomicExch(grp.error, 1);
}

}  // namespace pd
