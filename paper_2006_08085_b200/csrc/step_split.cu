// DeTAG step with the polynomial P = P_K(M) applied on the fifth-generation tensor cores in exact integer arithmetic,
// for gossip matrices with 48 < n <= 256 whose distinct 32 x 32 blocks of P fit in shared memory.  Its other kernel, step_rows.cu,
// takes the others and what it is faster at (rows_ok in detag_api.cu): left here are the DeTAG step of 65 to 96 workers and D-PSGD of theirs
// with sparse polynomials, long vectors up to 64, the longest of 97 to 128 with the printed timing, long ones of block-circulant matrices beyond 128.
//
// AG_K(z) = P z.  The float64 tensor path (mma m8n8k4) bounds this product at 64 multiply-adds per clock and SM, which
// for n = 100 is 3.3 times and for a dense n = 256 eight times the time of the step's HBM traffic.  Here both operands
// are split into five balanced base-256 digits:
//     z_j = 2^-s sum_k Z_kj 256^k   (39 bits and sign, one power of two s per coordinate and array, from the largest |z_j|)
//     P_ij = 2^-r_i sum_l P_lij 256^l   (the same per output worker, split once by the host)
// and the products of digits are summed by tcgen05.mma kind::i8 into 32-bit integers, exactly.  The fifteen digit pairs
// with k + l >= 4 are kept, one accumulator per k + l.  What is dropped is, for an output of m terms, some 2^-38 sqrt(m) of
// its largest weight times the coordinate's largest operand: 1e-11 .. 1e-12 of the result in the 2-norm.
//
// That scale is the coordinate's; an output that reads no operand near the largest must not inherit its error.  The host
// therefore chooses groups of inputs such that every output gives every input of one of the groups at least `theta` of its
// largest weight (split_guard in split_poly.cpp).  If the largest operand of each group is at least tau of the coordinate's largest,
// every sum of magnitudes sum_j |P_ij z_j| is at least theta tau of largest weight times largest operand, and
// tau = 2^-12 sqrt(m) / theta keeps the error below 2^-24 of that sum by more than five standard deviations (largest found on
// rings, tori and random graphs of 36 .. 256 workers, magnitudes spread in various ways: a fifth of it).  A coordinate that fails the test - or holds infinities, NaN or values outside
// the scalable range - is summed in float64: the warp that owns it takes its 32 coordinates through the float64 tensor path,
// from the operands, which stay staged that long.  Operands drawn alike fail less than once in a thousand coordinates.
//
// A unit of work is a slab of 64 coordinates.  Rows 0..63 of the MMA's M = 128 are the model digits of the slab's
// coordinates, rows 64..127 its tracker digits, so one instruction serves both arrays: A [128][32 workers] from tensor
// memory, where the threads that split the operands put it (thread = row = tensor memory lane), B the stacked digit planes
// of a block of P in shared memory, D the accumulators of an output chunk side by side.  An MMA with M = 128 and K = 32
// bytes takes 68 cycles for any N up to 128 (measured: N = 16, 32, 64, 96, 128, from tensor or shared memory alike), so a
// digit of z meets all planes it is kept with in one: five MMAs (N = 160 .. 32) per block of 32 x 32 weights, digit k with
// the planes 4 .. 4 - k, whose accumulators are neighbours.  Two chunks of 32 output workers are in flight, one beyond 128
// workers.  A thread that reads an accumulator owns one coordinate and consecutive workers: the four workers of a Philox
// call are its own and shared-memory rows are read 32 coordinates at a time, without conflicts and without swizzle.
//
// Roles: 4 or 8 splitting warps; F groups of 4 finishing warps that take 16 workers (a unit) in turn; one thread each for
// the MMAs, the x, y loads (one slab, handed back block by block while it is split), the g, a, c loads (R stages of 16
// workers per finishing group, overwritten with g', x', y') and the stores.  Model and tracker sums of a coordinate sit in
// different warps (lanes 64 apart): each of the two finishes eight of the sixteen workers and hands the sums of the other
// eight over, through the stage slots of its own eight whose g and a it has already taken into registers.  All sums are
// taken at the start, so that the accumulators are free again before the noise, the gradient and the fold.
// Blocks of P without a digit (rings, tori with few rounds) are skipped; equal blocks (circulant and block-circulant matrices) are
// kept once.
//
// Bound by the issue slots and the latency of what the six warps of a scheduler do, at a dense n = 256 by the MMAs, which take
// turns with splitting and with reading the one accumulator there is room for.  us per step, the float64 kernels this one
// replaced -> now: 100 workers, d = 2 M 3518 -> 1880 (step_rows.cu 1670 .. 1800); 256-ring at K = 196, d = 200 k 1940 -> 607; 16 x 16 torus, d = 500 k
// 8992 -> 1470.  (Four digits and four accumulators took 1680, 566 and 1420 when this took 2060, 640 and 1640, but left 2^-31 of the
// coordinate's largest operand in every result.)  From those figures it came by fewer instructions in the finishing and more
// registers for it: the scale of a coordinate sits in the number that joins the sums, a row's scale is one factor of x~ - alpha y~
// and one of the fold, doubles are handed over whole, digits, normals and gradients are made in packed float32, and the issuing
// warps give 48 registers each to the finishing ones, without which the former changes do not pay (100 workers 2100 us).
// With every coordinate in float64: 100 workers, K = 2, d = 1 M 1040 -> 4730; the torus 1570 -> 8710 - P comes from L2 and the slab is
// held.
//
// Measured without gain (us for the 1880 of 100 workers; the torus; the ring): digits and their places handed over block by
// block 1915, 1550, 680 (the splitting takes issue slots from the MMAs it then runs beside); an MMA warp per accumulator 1955; the
// normals between model update and gradient instead of before the other warp's sums 1915.
// Every wait is bounded but the allocation of tensor memory, which waits for kernels that do not depend on this
// one.
#include <cuda.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <utility>

#include "chain.cuh"
#include "detag_internal.h"
#include "digits.cuh"
#include "noise.cuh"
#include "packed.cuh"
#include "pipeline.cuh"
#include "tensor_memory.cuh"
#include "tma.cuh"

namespace detag {

namespace {

constexpr int kPS = 64;             // coordinates per slab
constexpr int kPChunk = 32;         // workers per block of P and of the staged slab
constexpr int kPUnit = 16;          // workers a finishing group takes at a time
constexpr int kPDigits = 5;         // of z and of P; also accumulators: digit pairs with k + l = 8, 7, 6, 5, 4
constexpr int kPBlockBytes = kPDigits * kPChunk * kPChunk;  // one block of P: the digit planes 4, 3, 2, 1, 0
constexpr int kPTileFloats = kPChunk * kPS;          // 32 rows of x or y
constexpr int kPStageFloats = kPUnit * kPS;          // one array of one unit
constexpr int kPStageBytes = 3 * kPStageFloats * 4;  // g | a | c  ->  g' | x' | y'
constexpr int kPScaleSlots = 4;     // slabs whose scales are kept: see the splitting warps
constexpr int kPMaxGroups = 4, kPMaxStages = 2, kPMaxBlocks = 8;
// Splitting and finishing warps.  Up to 128 workers two groups of four share the blocks of a slab: its splitting is a
// serial chain (largest value, then digits) that one group needed 5.6 k cycles for at n = 48, as long as the slab's HBM
// time (such worker counts have left for step_dense.cu since; 64 workers 213 -> 185 us, d = 400 k).  Beyond, a slab's other stages take longer than its splitting, and the warps finish instead.
__host__ __device__ constexpr int split_warps(bool big) { return big ? 4 : 8; }
__host__ __device__ constexpr int finish_groups(bool big) { return big ? 4 : 3; }
constexpr int kPThreads = 24 * 32;  // both: split_warps + 4 finish_groups + 4
constexpr int kTmemColumns = 512, kPAccColumns = kPDigits * kPChunk;
// Tensor memory: digits of a slab (forty columns per block of 32 workers) and accumulators.  Two accumulators, i.e. four
// units in flight, hide the finishing warps' way from one unit to the next and come before a second slab's digits.
__host__ __device__ constexpr int digit_buffers(int nb) { return nb <= 2 ? 2 : 1; }
__host__ __device__ constexpr int accumulators(bool big) { return big ? 1 : 2; }
static_assert(digit_buffers(2) * 40 * 2 + accumulators(false) * kPAccColumns <= kTmemColumns &&
                  digit_buffers(4) * 40 * 4 + accumulators(false) * kPAccColumns <= kTmemColumns &&
                  digit_buffers(8) * 40 * 8 + accumulators(true) * kPAccColumns <= kTmemColumns,
              "tensor memory plan");
constexpr size_t kPCtrlBytes = 640, kPSmemLimit = 232448;

struct SplitMaps {
  CUtensorMap x, y;        // boxes {64 coordinates, 32 workers}
  CUtensorMap g, a, c;     // boxes {64, 16}
  CUtensorMap xs, ys, gs;  // boxes {64, 16}, ending on a 16-byte boundary: stores
};
static_assert(sizeof(SplitMaps) <= sizeof(TensorMapSet), "tensor map storage");

struct SplitTables {
  const uint4* blocks;     // distinct blocks of P, digit planes in core-matrix order
  const int* row_exp;      // exponent of each output worker's scale
  // P itself, for what stays in float64: [input worker, padded to 32][output worker, padded to 16], or, if the blocks of P
  // depend on their distance only, [input worker][output workers 0 .. 31]
  const double* poly_t;
  int circulant;
  int num_blocks;
  int nb;                  // 32-worker blocks per side
  const uint8_t* guard;    // guard_groups x guard_size inputs
  int guard_groups, guard_size;  // size 2 or a multiple of 4
  float guard_tau;
  uint64_t id[8];          // [output chunk], a byte per input block: distinct block, 255: no digit of it is set
  uint8_t reach[8];        // [output chunk], a bit per input block: some entry of P itself is not zero
};

struct SplitPlan {
  int groups, stages;
  size_t blocks_at, e_at, guard_at, scale_at, ctrl_at, bytes;
};

// Shared memory: x, y of a slab (whole blocks of 32 rows) | blocks of P | g, a, c stages | groups of the guard | row
// scales, scales, flags, maxima (two splitting groups only) | barriers.
inline SplitPlan plan_for(int nb, int num_blocks, int guard_entries, int groups, int stages) {
  SplitPlan s{};
  s.groups = groups;
  s.stages = stages;
  s.blocks_at = static_cast<size_t>(nb) * 2 * kPTileFloats * 4;
  s.e_at = s.blocks_at + static_cast<size_t>(num_blocks) * kPBlockBytes;
  s.guard_at = s.e_at + static_cast<size_t>(groups) * stages * kPStageBytes;
  s.scale_at = s.guard_at + static_cast<size_t>(guard_entries + 3) / 4 * 16;
  s.ctrl_at = s.scale_at + 256 * 8 + kPScaleSlots * 128 * 2 + kPScaleSlots * 4 * 4 + (nb <= 4 ? 4 * 128 * 8 : 0);
  s.bytes = s.ctrl_at + kPCtrlBytes;
  return s;
}

// Finishing groups and their stages: as many as fit, two stages before a fourth group (bytes = 0: nothing fits).
inline SplitPlan split_plan(int nb, int num_blocks, int guard_entries) {
  constexpr int tries[4][2] = {{4, 2}, {3, 2}, {4, 1}, {3, 1}};
  for (const auto& t : tries) {
    if (t[0] > finish_groups(nb > 4)) continue;
    const SplitPlan s = plan_for(nb, num_blocks, guard_entries, t[0], t[1]);
    if (s.bytes <= kPSmemLimit) return s;
  }
  return SplitPlan{};
}

// Eight joined sums of this thread's coordinate from the accumulators at `acc` (whole warp).
template <bool kBig>
__device__ __forceinline__ void take_sums(uint32_t acc, int magic_hi, double magic, double (&out)[8]) {
  int hi[8], s6[8], s5[8], s4[8];
  {
    int s7[8];
    tmem_load8(acc, hi);
    tmem_load8(acc + kPChunk, s7);
    tmem_wait_load();
#pragma unroll
    for (int u = 0; u < 8; ++u) hi[u] = hi[u] * 256 + s7[u];
  }
  tmem_load8(acc + 2 * kPChunk, s6);
  tmem_load8(acc + 3 * kPChunk, s5);
  tmem_load8(acc + 4 * kPChunk, s4);
  tmem_wait_load();
#pragma unroll
  for (int u = 0; u < 8; ++u) out[u] = join_sums<kBig>(hi[u], s6[u], s5[u] + ((s4[u] + 128) >> 8), magic_hi, magic);
}

// Largest magnitude of a block's 32 staged rows (those beyond n are zeros), with what came before.
__device__ __forceinline__ float block_max(const float* src, float top) {
#pragma unroll
  for (int r = 0; r < 32; r += 8) {
    const float m = max_abs3(max_abs3(src[r * kPS], src[(r + 1) * kPS], src[(r + 2) * kPS]),
                             max_abs3(src[(r + 3) * kPS], src[(r + 4) * kPS], src[(r + 5) * kPS]),
                             max_abs3(src[(r + 6) * kPS], src[(r + 7) * kPS], 0.f));
    top = max_abs3(top, m, m);
  }
  return top;
}

// Digits of a block's 32 workers (zeros beyond n): digit 0 in w0, digit k in words 8 (k - 1) .. 8 k - 1 of w.  No test per row:
// the splitting is a serial chain, and so its loads and chains overlap.
__device__ __forceinline__ void block_digits(const float* src, float scale, uint32_t (&w)[32], uint32_t (&w0)[8]) {
#pragma unroll
  for (int u = 0; u < 8; ++u) {
    uint32_t d[5];
    four_digits(src + 4 * u * kPS, kPS, scale, d);
    w0[u] = d[0];
#pragma unroll
    for (int k = 1; k < 5; ++k) w[8 * (k - 1) + u] = d[k];
  }
}

// kMode: kModeDetag or kModeDpsgd.  kWide: the gradient in float64 (the precision of the rounds kernel, in whose place
// the call runs) instead of float32 at the rounded model (the other tensor-path kernels').  kBig: n > 128.
template <int kMode, bool kWide, bool kBig>
__global__ void __launch_bounds__(kPThreads, 1)
step_split_kernel(const StepParams p, const __grid_constant__ SplitMaps maps, const __grid_constant__ SplitTables tb,
                  const __grid_constant__ SplitPlan plan) {
  constexpr int kSplitWarps = split_warps(kBig), kMmaWarp = kSplitWarps, kLoadXYWarp = kMmaWarp + 1, kLoadEWarp = kMmaWarp + 2, kStoreWarp = kMmaWarp + 3,
                kFinishWarp = kMmaWarp + 4;
  constexpr int kAccs = accumulators(kBig);
  extern __shared__ __align__(128) unsigned char smem[];
  float* const xy_mem = reinterpret_cast<float*>(smem);                    // [block][x | y][32 rows][64]
  float* const e_mem = reinterpret_cast<float*>(smem + plan.e_at);
  int* const guard = reinterpret_cast<int*>(smem + plan.guard_at);          // [group][guard_size]
  double* const row_scale = reinterpret_cast<double*>(smem + plan.scale_at);  // a power of two per output worker
  short* const scales = reinterpret_cast<short*>(row_scale + 256);         // [slot][128 rows]
  unsigned* const flags = reinterpret_cast<unsigned*>(scales + kPScaleSlots * 128);  // [slot][lane quarter]: rows in float64
  float2* const maxima = reinterpret_cast<float2*>(flags + kPScaleSlots * 4);  // [slab parity][splitting group][128 rows]
  uint64_t* const xy_full = reinterpret_cast<uint64_t*>(smem + plan.ctrl_at);
  uint64_t* const xy_empty = xy_full + 1;                                  // [block]
  uint64_t* const dig_full = xy_empty + kPMaxBlocks;
  uint64_t* const dig_empty = dig_full + 2;
  // [group][parity of its unit count]: with three groups both chunks in flight may hold a unit of the same group, and a
  // parity wait must not find its barrier two phases ahead
  uint64_t* const acc_full = dig_empty + 2;
  uint64_t* const acc_empty = acc_full + 2 * kPMaxGroups;                  // [accumulator]
  uint64_t* const e_full = acc_empty + 2;                           // [group][stage], like the next two
  uint64_t* const e_empty = e_full + kPMaxGroups * kPMaxStages;
  uint64_t* const out_ready = e_empty + kPMaxGroups * kPMaxStages;
  uint64_t* const pair_bar = out_ready + kPMaxGroups * kPMaxStages;        // [group][warp pair][written, read]
  uint64_t* const drained = pair_bar + kPMaxGroups * 4;
  uint64_t* const max_ready = drained + 1;
  unsigned* const finished = reinterpret_cast<unsigned*>(max_ready + 1);     // [finishing warp]: units done
  uint32_t* const tmem_slot = finished + 4 * kPMaxGroups;
  static_assert((1 + kPMaxBlocks + 6 + 2 * kPMaxGroups + 3 * kPMaxGroups * kPMaxStages + 4 * kPMaxGroups + 2) * 8 + (4 * kPMaxGroups + 1) * 4 <= kPCtrlBytes,
                "barrier area");

  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform for the compiler
  const int n = p.n, nb = tb.nb, groups = plan.groups, stages = plan.stages;
  const unsigned limit = p.spin_limit;
  const bool aligned = (s_addr(smem) & 127u) == 0;  // the TMA tiles and core matrices need it
  {
    const uint4* src = tb.blocks;
    uint4* dst = reinterpret_cast<uint4*>(smem + plan.blocks_at);
    for (int e = tid; e < tb.num_blocks * (kPBlockBytes / 16); e += blockDim.x) dst[e] = src[e];
    for (int e = tid; e < 256; e += blockDim.x) row_scale[e] = __hiloint2double((1023 + (e < n ? tb.row_exp[e] : 0)) << 20, 0);
    for (int e = tid; e < tb.guard_groups * tb.guard_size; e += blockDim.x)  // as offsets into a coordinate's staged column
      guard[e] = tb.guard[e] / kPChunk * (2 * kPTileFloats) + tb.guard[e] % kPChunk * kPS;
  }
  if (tid == 0) {
    bar_init(xy_full, 1);
    for (int b = 0; b < kPMaxBlocks; ++b) bar_init(&xy_empty[b], 4);
    for (int s = 0; s < 2; ++s) {
      bar_init(&dig_full[s], kSplitWarps);
      bar_init(&dig_empty[s], 1);
      bar_init(&acc_empty[s], 8);
    }
    for (int s = 0; s < 2 * kPMaxGroups; ++s) bar_init(&acc_full[s], 1);
    for (int s = 0; s < kPMaxGroups * kPMaxStages; ++s) {
      bar_init(&e_full[s], 1);
      bar_init(&e_empty[s], 1);
      bar_init(&out_ready[s], 4);
    }
    for (int s = 0; s < kPMaxGroups * 4; ++s) bar_init(&pair_bar[s], 2);
    bar_init(drained, 1);
    bar_init(max_ready, kSplitWarps);
    for (int w = 0; w < 4 * kPMaxGroups; ++w) finished[w] = 0;
    fence_barrier_init();
    if (!aligned) atomicExch(p.status, 2);
  }
  if (warp == kMmaWarp) tmem_alloc(tmem_slot, kTmemColumns);
  fence_async_shared();
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  chain_wait();
  chain_next();
  constexpr uint32_t tmem = 0;  // all 512 columns are this CTA's: they start at address 0
  if (tid == 0 && *tmem_slot != 0) atomicExch(p.status, 2);

  // Tensor memory: digits 4 .. 1 of a slab in 32 columns per block (digit k in the eight from 8 (k - 1) on), digit 0 in
  // eight per block, the accumulators behind all buffers of both: weight 8, 7, 6, 5, 4 in 32 columns each.
  const int dig_buffers = kBig ? 1 : digit_buffers(nb);
  const uint32_t low_column = tmem + dig_buffers * 32 * nb, acc_column = tmem + dig_buffers * 40 * nb;

  // this CTA takes slabs blockIdx.x, blockIdx.x + gridDim.x, ...; chunk q = slab number * nb + output chunk,
  // unit v = slab number * units + half chunk
  const int my_slabs = aligned && *tmem_slot == 0 && blockIdx.x < p.num_slabs
                           ? static_cast<int>((p.num_slabs - blockIdx.x + gridDim.x - 1) / gridDim.x) : 0;
  const int units = (n + kPUnit - 1) / kPUnit, total = my_slabs * units;
  auto slab_col = [&](int k) { return (static_cast<long long>(blockIdx.x) + static_cast<long long>(k) * gridDim.x) * kPS; };
  auto warp_wait = [&](uint64_t* bar, int phase) {  // every lane polls the same barrier: no broadcast of the verdict
    return __all_sync(0xffffffffu, bar_wait(bar, phase & 1, limit));
  };

  // Registers from the warps that only issue to those that finish: of the 768 x 80 the block is launched with, 80 per splitting
  // thread, 32 per issuing thread and 96 (88 beyond 128 workers) per finishing thread.
  constexpr int kFinishRegisters = kBig ? 88 : 96;
  static_assert(kSplitWarps * 80 + 4 * 32 + (24 - kSplitWarps - 4) * kFinishRegisters <= 24 * 80, "register split");
  if (warp >= kFinishWarp) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kFinishRegisters));
  } else if (warp >= kSplitWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 32;");
  }
  if (warp < kSplitWarps) {
    // ---------------------------------------------------------------- splitting warps: thread = row of A = tensor memory lane
    const int part = warp >> 2, quarter = warp & 3;
    const bool tracker = quarter >= 2;
    const int row = quarter * 32 + lane, coord = (quarter & 1) * 32 + lane;
    const uint32_t lane_base = static_cast<uint32_t>(quarter) << 21;
    const bool idle = kMode == kModeDpsgd && tracker;  // D-PSGD has no tracker: its rows of A are never read back
    const float* const col = xy_mem + (tracker ? kPTileFloats : 0) + coord;
    const int first = part == 0 ? 0 : nb / 2, last = kBig || part == 1 ? nb : nb / 2;  // blocks of this group
    bool ok = true;
    for (int k = 0; k < my_slabs && ok; ++k) {
      const int buf = dig_buffers == 2 ? k & 1 : 0, use = dig_buffers == 2 ? k >> 1 : k, slot = k % kPScaleSlots;
      ok = warp_wait(xy_full, k);
      if (!ok) break;
      // largest magnitude, and the smallest of the largest magnitudes of the guard's groups
      float top_f = 0.f, low_f = __uint_as_float(0x7f800000u);
      if (!idle) {
        for (int b = first; b < last; ++b) {
          top_f = block_max(col + b * (2 * kPTileFloats), top_f);
        }
        low_f = group_low<int4, int2>([&](int at) { return col[at]; }, guard, tb.guard_groups, tb.guard_size, kBig ? 0 : part, kBig ? 1 : 2);
      }
      if (!kBig) {  // the other group's blocks
        float2* const mx = maxima + (k & 1) * 256 + row;  // read again two slabs later, behind the next hand-over
        mx[part * 128] = make_float2(top_f, low_f);
        __syncwarp();
        if (lane == 0) bar_arrive(max_ready);
        ok = warp_wait(max_ready, k);
        if (!ok) break;
        const float2 other = mx[(part ^ 1) * 128];
        top_f = max_abs3(top_f, other.x, other.x);
        low_f = fminf(low_f, other.y);
      }
      const unsigned top = __float_as_uint(top_f);
      // as float bits: not finite, too small for the scale; an output may read nothing near the largest operand
      const bool exact = top >= 0x7f800000u || (top != 0 && (top < kSmallest || low_f < tb.guard_tau * top_f));
      const int e = top == 0 || exact ? 30 : static_cast<int>((top + kRoundUp) >> 23) - 127;  // all |z| < 2^(e+1)
      const float scale = __uint_as_float(static_cast<unsigned>(157 - e) << 23);              // 2^(30 - e)
      const unsigned exact_lanes = __ballot_sync(0xffffffffu, exact);
      const bool any_exact = exact_lanes != 0;
      if (use > 0) ok = warp_wait(&dig_empty[buf], use - 1);
      if (!ok) break;
      tmem_fence_after();
      // The slot was last read for slab k - 4: a finishing group reads a unit's scales before it releases the
      // accumulators, and the MMAs of slab k - 2 (complete: dig_empty) came after that release for all units of k - 4 (two
      // slabs have at least as many chunks as there are accumulators).
      if (part == 0) {
        scales[slot * 128 + row] = static_cast<short>(exact ? 0 : e - 6);
        if (lane == 0) flags[slot * 4 + quarter] = exact_lanes;
      }
      for (int b = first; b < last; ++b) {
        if (!idle) {
          uint32_t w[32], w0[8];
          block_digits(col + b * (2 * kPTileFloats), scale, w, w0);
          tmem_store32(lane_base + tmem + (buf * nb + b) * 32, w);
          tmem_store8(lane_base + low_column + (buf * nb + b) * 8, w0);
        }
        __syncwarp();
        if (lane == 0 && !any_exact) bar_arrive(&xy_empty[b]);  // the loads of the next slab follow block by block
      }
      tmem_wait_store();
      tmem_fence_before();
      __syncwarp();
      if (lane == 0) bar_arrive(&dig_full[buf]);
      if (any_exact) {  // the finishing warps read these rows' operands themselves: keep the slab until they are done with it
        if (lane < 4 * groups)  // a lane per finishing warp
          ok = count_wait_relaxed(&finished[lane], static_cast<unsigned>(((k + 1) * units - (lane >> 2) + groups - 1) / groups), limit);
        ok = __all_sync(0xffffffffu, ok);
        asm volatile("fence.acq_rel.cta;" ::: "memory");
        if (lane == 0)
          for (int b = first; b < last && ok; ++b) bar_arrive(&xy_empty[b]);
        __syncwarp();
      }
    }
    if (!ok && lane == 0) atomicExch(p.status, 1);
  } else if (warp >= kFinishWarp) {
    // ---------------------------------------------------------------- finishing warps
    const int t = (warp - kFinishWarp) >> 2, quarter = warp & 3;
    const bool second = quarter >= 2;  // reads the tracker rows; finishes workers 8..15 of every sixteen
    const int pair = quarter & 1, coord = pair * 32 + lane, mine = second ? 8 : 0;
    const uint32_t acc_lane = acc_column + (static_cast<uint32_t>(quarter) << 21);
    float* const e_group = e_mem + static_cast<size_t>(t) * stages * (kPStageBytes / 4) + coord;
    uint64_t* const written = &pair_bar[4 * t + 2 * pair];
    uint64_t* const taken = written + 1;
    const double alpha = p.alpha;
    const float sigma = static_cast<float>(p.sigma);
    const bool noisy = p.sigma != 0.0, at_start = p.grad_at_start != 0;
    const long long d_tma = p.d & ~3LL;  // columns below this are written by the TMA stores
    int k = 0, h = t, st = 0, st_phase = 0, m = 0;
    while (h >= units) {
      h -= units;
      ++k;
    }
    bool ok = true;
    for (int v = t; v < total && t < groups; v += groups, ++m) {
      const int a = (k * nb + (h >> 1)) & (kAccs - 1);
      ok = warp_wait(&acc_full[2 * t + (m & 1)], m >> 1) && warp_wait(&e_full[t * kPMaxStages + st], st_phase);
      if (!ok) break;
      tmem_fence_after();
      const int slot = k % kPScaleSlots;
      const unsigned exact_lanes = flags[slot * 4 + quarter];
      const long long j = slab_col(k) + coord;
      const int w0 = kPUnit * h + mine;  // first of this thread's eight workers
      float* const sg = e_group + st * (kPStageBytes / 4) + mine * kPS;
      float* const sa = sg + kPStageFloats;
      float* const sc = sa + kPStageFloats;
      float gold[8], av[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        gold[u] = sg[u * kPS];
        av[u] = sa[u * kPS];
      }
      // ---- sums of sixteen workers, but for the factor of their rows: eight handed to the other warp of the pair, eight kept.
      // A handed double lies across this warp's part of two rows, so that half a warp's are 128 bytes in a row.
      double own[8];
      const double magic = __hiloint2double(0x43380000 + scales[slot * 128 + (second ? 64 : 0) + coord] * (1 << 20), 0);
      const int magic_hi = __double2hiint(magic);
      double* const box = reinterpret_cast<double*>(e_mem + (static_cast<size_t>(t) * stages + st) * (kPStageBytes / 4) + pair * 32 + (lane >> 4) * kPS) + (lane & 15);
      double* const my_box = box + mine * (kPS / 2);
      auto box_at = [](int u) { return (u >> 2) * (kPStageFloats / 2) + (u & 3) * kPS; };
      __syncwarp();  // every lane has taken its g and a out
      if (exact_lanes == 0) {
        const uint32_t acc = acc_lane + a * kPAccColumns + (h & 1) * kPUnit;
        if (kMode != kModeDpsgd || !second) {
          double give[8];
          take_sums<kBig>(acc + (mine ^ 8), magic_hi, magic, give);
#pragma unroll
          for (int u = 0; u < 8; ++u) my_box[box_at(u)] = give[u];
        }
        take_sums<kBig>(acc + mine, magic_hi, magic, own);
      } else {
        // Some row of this warp was not split: all 32 in float64, from the operands themselves.
        const float* const z = xy_mem + (second ? kPTileFloats : 0) + pair * 32;
        float* const hi_word = sg - lane;  // this warp's part of the mailbox, [worker][coordinate]
        float* const lo_word = sa - lane;
        const int c = h >> 1, pitch = tb.circulant ? kPChunk : units * kPUnit;
        const double* const columns = tb.poly_t + (tb.circulant ? kPUnit * (h & 1) : kPUnit * h);
        bool finite = true;
        // 1 / the row's scale
        auto unscale = [&](int row) { return __hiloint2double((2046 << 20) - __double2hiint(row_scale[row]), 0); };
        // Products on the float64 tensor path: four tiles of eight coordinates (M) by eight output workers (N)
#pragma unroll
        for (int half = 0; half < 2; ++half) {
          const int to = half == 0 ? mine : mine ^ 8;
          double sum[4][2] = {{0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}, {0.0, 0.0}};
          for (int b = 0; b < nb; ++b) {
            if ((tb.reach[c] >> b & 1) == 0) continue;  // a zero block of P
            const int pb = !tb.circulant ? b : b >= c ? b - c : b - c + nb;  // block row 0 holds them all
            const double* const pw = columns + static_cast<size_t>(32 * pb + (lane & 3)) * pitch + to + (lane >> 2);
            const float* const zb = z + b * (2 * kPTileFloats) + (lane & 3) * kPS + (lane >> 2);
            double w[8];  // P comes from L2: all of a block's at once
#pragma unroll
            for (int s = 0; s < 8; ++s) w[s] = __ldg(pw + static_cast<size_t>(4 * s) * pitch);
#pragma unroll
            for (int s = 0; s < 8; ++s)
#pragma unroll
              for (int i = 0; i < 4; ++i) dmma(sum[i], static_cast<double>(zb[4 * s * kPS + 8 * i]), w[s]);
          }
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 2; ++e) {
              const int at = (2 * (lane & 3) + e) * kPS + 8 * i + (lane >> 2);
              hi_word[at] = __int_as_float(__double2hiint(sum[i][e]));
              lo_word[at] = __int_as_float(__double2loint(sum[i][e]));
            }
          __syncwarp();
          double take[8];
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const double v = __hiloint2double(__float_as_int(sg[u * kPS]), __float_as_int(sa[u * kPS]));
            finite = finite && (__double2hiint(v) & 0x7ff00000) != 0x7ff00000;
            take[u] = v * unscale(kPUnit * h + to + u);
          }
          __syncwarp();
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            if (half == 0) {
              own[u] = take[u];
            } else {
              my_box[box_at(u)] = take[u];
            }
          }
        }
        if (__any_sync(0xffffffffu, !finite)) {
          // Infinities or NaN among the operands: a lane sums its own coordinate, without the zeros of P, which the products
          // above turn into NaN.
#pragma unroll
          for (int half = 0; half < 2; ++half) {
            const int to = half == 0 ? mine : mine ^ 8;
            double sum[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
            for (int b = 0; b < nb; ++b) {
              if ((tb.reach[c] >> b & 1) == 0) continue;
              const int pb = !tb.circulant ? b : b >= c ? b - c : b - c + nb;
              for (int w = 0; w < 32; ++w) {
                const double zw = static_cast<double>(z[b * (2 * kPTileFloats) + w * kPS + lane]);
                const double* const pw = columns + static_cast<size_t>(32 * pb + w) * pitch + to;
#pragma unroll
                for (int u = 0; u < 8; ++u)
                  if (pw[u] != 0.0) sum[u] = fma(pw[u], zw, sum[u]);
              }
            }
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const double scaled = sum[u] * unscale(kPUnit * h + to + u);
              if (half == 0) {
                own[u] = scaled;
              } else {
                my_box[box_at(u)] = scaled;
              }
            }
          }
        }
      }
      tmem_fence_before();
      __syncwarp();
      if (lane == 0) {
        bar_arrive(written);
        bar_arrive(&acc_empty[a]);
        if (h + 1 == units && (h & 1) == 0) bar_arrive(&acc_empty[a]);  // there is no other half of this chunk
      }
      // ---- normals of this thread's eight workers, while the other warp arrives
      float xi[8];
      if (noisy) {
        const unsigned long long jn = static_cast<unsigned long long>(p.coord_offset + j);
        normal_eight(p.round_key, jn, static_cast<uint32_t>(w0 >> 2), p.t_noise, sigma, xi);
      } else {
#pragma unroll
        for (int u = 0; u < 8; ++u) xi[u] = 0.f;
      }
      // gradient point of Algorithm 2 as printed: the model the step started from, still in global memory - this unit's rows are
      // stored after this
      float start[8];
      if (at_start) {
#pragma unroll
        for (int u = 0; u < 8; ++u) start[u] = w0 + u < n && j < p.d ? p.x[static_cast<long long>(w0 + u) * p.ld + j] : 0.f;
      }
      ok = warp_wait(written, m);
      if (!ok) break;
      const double* const other_box = box + (mine ^ 8) * (kPS / 2);
      if (kMode != kModeDpsgd && p.y_obs != nullptr) {  // optional observer: the gossiped tracker
#pragma unroll
        for (int u = 0; u < 8; ++u)
          if (w0 + u < n && j < p.d)
            p.y_obs[static_cast<long long>(w0 + u) * p.ld + j] = static_cast<float>((second ? own[u] : other_box[box_at(u)]) * row_scale[w0 + u]);
      }
      // ---- gossiped model and tracker, model update, y~ - g
      double yg[8];
      float at[8], go[8], xo[8], yo[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const double other = (kMode != kModeDpsgd || second) ? other_box[box_at(u)] : 0.0;
        const double factor = row_scale[w0 + u];  // a power of two: its products are exact
        const double xt = second ? other : own[u], yt = second ? own[u] : other, gd = static_cast<double>(gold[u]);
        const double xd = kMode == kModeDpsgd ? fma(-alpha, gd, xt * factor) : fma(-alpha, yt, xt) * factor;
        yg[u] = fma(yt, factor, -gd);
        xo[u] = static_cast<float>(xd);
        at[u] = at_start ? start[u] : xo[u];
        if (kWide) own[u] = at_start ? static_cast<double>(at[u]) : xd;
      }
      // ---- gradient and fold
#pragma unroll
      for (int u = 0; u < 8; u += 2) {
        const float c0 = sc[u * kPS], c1 = sc[(u + 1) * kPS];
        if (kWide) {
          go[u] = static_cast<float>(fma(static_cast<double>(av[u]), own[u] - static_cast<double>(c0), static_cast<double>(xi[u])));
          go[u + 1] = static_cast<float>(fma(static_cast<double>(av[u + 1]), own[u + 1] - static_cast<double>(c1), static_cast<double>(xi[u + 1])));
        } else {
          unpack2(fma2(pack2(av[u], av[u + 1]), sub2(pack2(at[u], at[u + 1]), pack2(c0, c1)), pack2(xi[u], xi[u + 1])), go[u], go[u + 1]);
        }
#pragma unroll
        for (int e = 0; e < 2; ++e) yo[u + e] = static_cast<float>(yg[u + e] + static_cast<double>(go[u + e]));
      }
      __syncwarp();
      if (lane == 0) bar_arrive(taken);
      ok = warp_wait(taken, m);
      if (!ok) break;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        sg[u * kPS] = go[u];
        sa[u * kPS] = xo[u];
        if (kMode != kModeDpsgd) sc[u * kPS] = yo[u];
      }
      if (j >= d_tma && j < p.d) {  // TMA clips a store at 16-byte granularity: the last d % 4 columns are written here
        for (int u = 0; u < 8 && w0 + u < n; ++u) {
          const long long off = static_cast<long long>(w0 + u) * p.ld + j;
          p.g[off] = sg[u * kPS];
          p.x[off] = sa[u * kPS];
          if (kMode != kModeDpsgd) p.y[off] = sc[u * kPS];
        }
      }
      fence_async_shared();  // results visible to the TMA stores
      __syncwarp();
      if (lane == 0) {
        bar_arrive(&out_ready[t * kPMaxStages + st]);
        // relaxed: what a reader of the count waits for, this unit's reads of x and y, went into the results above
        *const_cast<volatile unsigned*>(&finished[warp - kFinishWarp]) = static_cast<unsigned>(m + 1);
      }
      if (++st == stages) {
        st = 0;
        ++st_phase;
      }
      h += groups;
      while (h >= units) {
        h -= units;
        ++k;
      }
    }
    if (!ok && lane == 0) atomicExch(p.status, 1);
  } else if (warp == kMmaWarp) {
    // ---------------------------------------------------------------- MMAs
    // The whole warp walks the loop, one lane issues: operands computed in uniform control flow stay in uniform registers
    // (issued from inside a one-lane branch each MMA cost 127 cycles, eight times its time on the tensor cores).
    const uint64_t b_base = mma_operand(s_addr(smem + plan.blocks_at), 256, 128);
    const bool leader = lane == 0;
    bool ok = true;
    int q = 0, t = 0, turn = 0;  // t, turn: group of the next unit and the parity of how many it has had
    auto hand_over = [&]() {     // the group waits for all MMAs issued so far
      mma_commit(&acc_full[2 * t + turn], leader);
      if (++t == groups) {
        t = 0;
        turn ^= 1;
      }
    };
    for (int k = 0; k < my_slabs && ok; ++k) {
      const int buf = dig_buffers == 2 ? k & 1 : 0, use = dig_buffers == 2 ? k >> 1 : k;
      ok = warp_wait(&dig_full[buf], use);
      for (int c = 0; c < nb && ok; ++c, ++q) {
        if (q >= kAccs) ok = warp_wait(&acc_empty[q & (kAccs - 1)], q / kAccs - 1);
        if (!ok) break;
        tmem_fence_after();
        const uint32_t acc = acc_column + (q & (kAccs - 1)) * kPAccColumns;
        unsigned add = 0;  // the first product of an accumulator clears it
        uint64_t ids = tb.id[c];
        uint32_t z = tmem + buf * nb * 32, z0 = low_column + buf * nb * 8;
        for (int kb = 0; kb < nb; ++kb, ids >>= 8, z += 32, z0 += 8) {
          const uint32_t id = static_cast<uint32_t>(ids) & 0xffu;
          if (id == 0xffu) continue;
          const uint64_t b = b_base + id * (kPBlockBytes / 16);
          // digit k of z with the planes 4 .. 4 - k of P -> weights 4 + k .. 4
          mma_i8(acc, z + 24, b, mma_i8_desc(5 * kPChunk), add, leader);
          mma_i8(acc + kPChunk, z + 16, b, mma_i8_desc(4 * kPChunk), 1u, leader);
          mma_i8(acc + 2 * kPChunk, z + 8, b, mma_i8_desc(3 * kPChunk), 1u, leader);
          mma_i8(acc + 3 * kPChunk, z, b, mma_i8_desc(2 * kPChunk), 1u, leader);
          mma_i8(acc + 4 * kPChunk, z0, b, mma_i8_desc(kPChunk), 1u, leader);
          add = 1;
        }
        hand_over();
        if (2 * c + 1 < units) hand_over();
      }
      if (ok) mma_commit(&dig_empty[buf], leader);
    }
    if (!ok) {  // nothing may be in flight when the tensor memory is given back
      if (leader) atomicExch(p.status, 1);
      mma_commit(drained, leader);
      warp_wait(drained, 0);
    }
  } else if (warp == kLoadXYWarp) {
    if (lane == 0) {
      const unsigned bytes = (kMode == kModeDpsgd ? 1u : 2u) * nb * kPTileFloats * 4u;
      int k = 0;
      bool ok = true;
      for (; k < my_slabs && ok; ++k) {
        if (p.stall_after >= 0 && static_cast<long long>(k) * units >= p.stall_after) break;  // self test: the loads stop
        const int col = static_cast<int>(slab_col(k));
        for (int b = 0; b < nb; ++b) {
          if (k > 0) ok = bar_wait(&xy_empty[b], (k - 1) & 1, limit);
          if (!ok) break;
          if (b == 0) bar_expect_tx(xy_full, bytes);
          float* dst = xy_mem + b * (2 * kPTileFloats);
          tile_load(dst, &maps.x, col, 32 * b, xy_full);
          if (kMode != kModeDpsgd) tile_load(dst + kPTileFloats, &maps.y, col, 32 * b, xy_full);
        }
      }
      if (!ok) atomicExch(p.status, 1);
      if (k > 0) bar_wait(xy_full, (k - 1) & 1, limit);  // nothing in flight when the CTA leaves (bounded)
    }
    __syncwarp();
  } else if (warp == kLoadEWarp) {
    if (lane == 0) {
      int v = 0, k = 0, h = 0, t = 0, st = 0, phase = 0;  // group and stage of unit v; phase = uses of the stage so far
      bool ok = true;
      for (; v < total; ++v) {
        if (p.stall_after >= 0 && v >= p.stall_after) break;
        const int s = t * kPMaxStages + st;
        if (phase > 0) ok = bar_wait(&e_empty[s], (phase - 1) & 1, limit);
        if (!ok) break;
        float* dst = e_mem + static_cast<size_t>(t * stages + st) * (kPStageBytes / 4);
        const int col = static_cast<int>(slab_col(k));
        bar_expect_tx(&e_full[s], kPStageBytes);
        tile_load(dst, &maps.g, col, kPUnit * h, &e_full[s]);
        tile_load(dst + kPStageFloats, &maps.a, col, kPUnit * h, &e_full[s]);
        tile_load(dst + 2 * kPStageFloats, &maps.c, col, kPUnit * h, &e_full[s]);
        if (++t == groups) {
          t = 0;
          if (++st == stages) {
            st = 0;
            ++phase;
          }
        }
        if (++h == units) {
          h = 0;
          ++k;
        }
      }
      if (!ok) atomicExch(p.status, 1);
      for (int back = 1; back <= groups * stages && back <= v; ++back) {
        const int z = v - back, u = z / groups;
        bar_wait(&e_full[(z % groups) * kPMaxStages + u % stages], (u / stages) & 1, limit);
      }
    }
    __syncwarp();
  } else if (warp == kStoreWarp) {
    if (lane == 0) {
      int k = 0, h = 0, t = 0, st = 0, phase = 0;
      for (int v = 0; v < total; ++v) {
        const int s = t * kPMaxStages + st;
        if (!bar_wait(&out_ready[s], phase & 1, limit)) {
          atomicExch(p.status, 1);
          break;
        }
        const float* src = e_mem + static_cast<size_t>(t * stages + st) * (kPStageBytes / 4);  // now g' | x' | y'
        const long long col = slab_col(k);
        if (col < (p.d & ~3LL)) {
          tile_store(&maps.gs, static_cast<int>(col), kPUnit * h, src);
          tile_store(&maps.xs, static_cast<int>(col), kPUnit * h, src + kPStageFloats);
          if (kMode != kModeDpsgd) tile_store(&maps.ys, static_cast<int>(col), kPUnit * h, src + 2 * kPStageFloats);
        }
        store_commit();
        store_wait_read();  // the stage may be refilled now
        bar_arrive(&e_empty[s]);
        if (++t == groups) {
          t = 0;
          if (++st == stages) {
            st = 0;
            ++phase;
          }
        }
        if (++h == units) {
          h = 0;
          ++k;
        }
      }
      store_wait_all();
    }
    __syncwarp();
  }
  tmem_fence_before();
  __syncthreads();
  if (warp == kMmaWarp) {
    tmem_fence_after();
    tmem_free(tmem, kTmemColumns);
  }
}

typedef void (*SplitKernel)(const StepParams, const SplitMaps, const SplitTables, const SplitPlan);

template <bool kBig>
SplitKernel pick_split(const StepParams& p, bool wide) {
  if (p.mode == kModeDpsgd)
    return wide ? step_split_kernel<kModeDpsgd, true, kBig> : step_split_kernel<kModeDpsgd, false, kBig>;
  return wide ? step_split_kernel<kModeDetag, true, kBig> : step_split_kernel<kModeDetag, false, kBig>;
}

}  // namespace

// Digits of P: distinct 32 x 32 blocks, their table and the rows' exponents.  `poly`: the n x n matrix, or (circulant: the
// blocks depend on their distance only) its first 32 rows.  Leaves `out` empty when the kernel does not take the matrix:
// n outside 33 .. 256, an entry or a row that cannot be scaled, too many distinct blocks.
void split_polynomial(int n, const std::vector<double>& poly, bool circulant, SplitPoly& out) {
  out = SplitPoly{};
  if (n <= 32 || n > 256 || encode_tiled_fn() == nullptr) return;
  const int nb = (n + kPChunk - 1) / kPChunk, rows = circulant ? kPChunk : n, wide = nb * kPChunk;
  std::vector<int64_t> digits;
  std::vector<int32_t> row_exp;
  if (!split_digits(n, poly, rows, wide, digits, row_exp)) return;
  digits.resize(static_cast<size_t>(circulant ? 1 : nb) * kPChunk * wide, 0);
  SplitPoly made{};
  split_guard(n, poly, rows, made);
  std::vector<unsigned char> blocks;
  std::memset(made.id, 255, sizeof made.id);
  std::vector<unsigned char> block(kPBlockBytes);
  constexpr int plane = kPChunk * kPChunk;  // bytes
  for (int c = 0; c < (circulant ? 1 : nb); ++c)
    for (int kb = 0; kb < nb; ++kb) {
      int64_t any = 0;
      for (int i = c * kPChunk; i < std::min((c + 1) * kPChunk, rows); ++i)
        for (int j = kb * kPChunk; j < std::min((kb + 1) * kPChunk, n); ++j)
          if (poly[static_cast<size_t>(i) * n + j] != 0.0) made.reach[c] |= static_cast<unsigned char>(1u << kb);
      for (int r = 0; r < kPChunk; ++r) {
        const int64_t* src = &digits[(static_cast<size_t>(c) * kPChunk + r) * wide + kb * kPChunk];
        // planes 4 .. 0 of core matrices of 8 rows x 16 bytes, the two of a row group side by side
        unsigned char* at = &block[(r / 8) * 256 + (r % 8) * 16];
        for (int w = 0; w < kPChunk; ++w) {
          any |= src[w];
          for (int l = 0; l < kPDigits; ++l)
            at[(kPDigits - 1 - l) * plane + (w / 16) * 128 + w % 16] = static_cast<unsigned char>(src[w] >> (8 * l));
        }
      }
      if (any == 0) continue;
      const int have = static_cast<int>(blocks.size() / kPBlockBytes);
      int hit = 0;
      while (hit < have && std::memcmp(&blocks[static_cast<size_t>(hit) * kPBlockBytes], block.data(), kPBlockBytes) != 0) ++hit;
      if (hit == have) {
        if (split_plan(nb, have + 1, static_cast<int>(made.guard.size())).bytes == 0) return;
        blocks.insert(blocks.end(), block.begin(), block.end());
      }
      made.id[c * 8 + kb] = static_cast<unsigned char>(hit);
    }
  if (circulant)
    for (int c = 1; c < nb; ++c)
      for (int kb = 0; kb < nb; ++kb) {
        made.id[c * 8 + kb] = made.id[(kb - c + nb) % nb];
        made.reach[c] |= static_cast<unsigned char>((made.reach[0] >> ((kb - c + nb) % nb) & 1) << kb);
      }
  const size_t pitch = circulant ? kPChunk : static_cast<size_t>((n + kPUnit - 1) / kPUnit) * kPUnit;
  made.poly.assign(wide * pitch, 0.0);
  for (int i = 0; i < rows; ++i)
    for (int j = 0; j < n; ++j) made.poly[j * pitch + i] = poly[static_cast<size_t>(i) * n + j];
  made.weights.swap(blocks);
  made.row_exp.swap(row_exp);
  made.circulant = circulant;
  out = std::move(made);
}

bool build_maps_split(const StepParams& p, TensorMapSet* out) {
  SplitMaps& m = *reinterpret_cast<SplitMaps*>(out->bytes);
  const float* y = p.mode == kModeDpsgd ? p.x : p.y;  // D-PSGD has no tracker: those maps are never used
  if (!make_map(&m.x, p.x, p.n, p.d, p.ld, kPChunk, kPS) || !make_map(&m.y, y, p.n, p.d, p.ld, kPChunk, kPS) ||
      !make_map(&m.g, p.g, p.n, p.d, p.ld, kPUnit, kPS) || !make_map(&m.a, p.a, p.n, p.d, p.ld, kPUnit, kPS) ||
      !make_map(&m.c, p.c, p.n, p.d, p.ld, kPUnit, kPS))
    return false;
  const long long d_tma = p.d & ~3LL;  // the stores' tensor ends on a 16-byte boundary
  if (d_tma > 0 && (!make_map(&m.xs, p.x, p.n, d_tma, p.ld, kPUnit, kPS) ||
                    !make_map(&m.ys, y, p.n, d_tma, p.ld, kPUnit, kPS) || !make_map(&m.gs, p.g, p.n, d_tma, p.ld, kPUnit, kPS)))
    return false;
  if (d_tma == 0) m.xs = m.ys = m.gs = m.x;  // never used
  return true;
}

int launch_step_split(StepParams p, const TensorMapSet& maps, const SplitPoly& poly, const SplitDevice& dev, bool wide,
                      int sm_count, cudaStream_t stream) {
  if (p.mode == kModeExternal || poly.weights.empty()) return static_cast<int>(cudaErrorInvalidValue);
  p.S = kPS;
  p.num_slabs = (p.d + kPS - 1) / kPS;
  SplitTables tb{};
  tb.blocks = static_cast<const uint4*>(dev.weights);
  tb.row_exp = dev.row_exp;
  tb.poly_t = dev.poly;
  tb.guard = dev.guard;
  tb.guard_size = poly.guard_size;
  tb.guard_groups = static_cast<int>(poly.guard.size()) / poly.guard_size;
  tb.guard_tau = poly.guard_tau;
  tb.circulant = poly.circulant ? 1 : 0;
  tb.num_blocks = static_cast<int>(poly.weights.size() / kPBlockBytes);
  tb.nb = (p.n + kPChunk - 1) / kPChunk;
  std::memcpy(tb.id, poly.id, sizeof tb.id);
  std::memcpy(tb.reach, poly.reach, sizeof tb.reach);
  const SplitPlan plan = split_plan(tb.nb, tb.num_blocks, static_cast<int>(poly.guard.size()));
  const SplitKernel kernel = p.n > 128 ? pick_split<true>(p, wide) : pick_split<false>(p, wide);
  const int e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), static_cast<int>(plan.bytes));
  if (e != 0) return e;
  const long long grid = p.num_slabs < sm_count ? p.num_slabs : sm_count;
  if (grid <= 0) return 0;
  return launch_chained(kernel, static_cast<unsigned>(grid), kPThreads, plan.bytes, stream, p, *reinterpret_cast<const SplitMaps*>(maps.bytes), tb, plan);
}

}  // namespace detag
