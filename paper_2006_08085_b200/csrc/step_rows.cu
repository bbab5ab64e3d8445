// DeTAG step with the polynomial P = P_K(M) in exact integer arithmetic on the fifth-generation tensor cores, like step_split.cu (whose
// head explains the digits, the scales and the test that sends a coordinate to float64), with the output workers as lanes: any matrix
// of 49 to 256 workers, caller-written gradients up to 192.
//
// A unit of work is a chunk of 32 coordinates.  A of the MMA is a digit plane of P (128 output workers x 32 inputs), B the digits
// of the chunk's models and trackers, 64 columns per digit, digit by digit: plane l meets the digits 4 - l .. 4 in one instruction (N up to
// 256; five digits take two), whose sums all start at the same column of the accumulators, weight 4 first.  Six instructions per
// 32 inputs serve 128 output workers and both arrays; with coordinates as lanes it is twenty for the same chunk.  Up to 128 workers P
// stays in tensor memory (160 of its columns beside 320 of accumulators); beyond, two halves of the outputs take turns on the accumulators,
// four tiles of P stay in tensor memory - of a block-circulant matrix four that both halves use, half of all there is to do - and the
// others come from L2 through a ring, whole tiles of five planes at a time where there is room for two (waiting for single planes
// the MMA warp took 290 .. 440 cycles each; without the four, 256-ring, K = 40, d = 19 k 119 -> 85 us).
//
// A lane has model and tracker sums of its worker, eight coordinates in a row: the element-wise tail is its own, reads and writes
// shared memory in 16-byte pieces (128-byte swizzle, no conflicts), and a Philox call's four workers are four neighbouring lanes, which
// draw two coordinates each and transpose.  No hand-over between warps, unlike step_split.cu.
//
// Roles: 8 splitting warps (a column of B and a quarter of the workers per thread; maxima exchanged through shared memory), 16 finishing
// warps (four groups of eight coordinates on the four lane quarters), one warp each for the MMAs, for x and y, for g, a, c and the results,
// for the planes of P.  Up to 64 workers the lanes hold them twice and half of the groups take every other chunk.  Of 65 to 96 workers a lane
// quarter, which only one of the SM's schedulers reaches, has nothing to finish; there that scheduler's warps do the splitting (96
// workers, d = 1 M 801 -> 782 us).
//
// Caller-written gradients: y + (g_new - g) is split as the float32 sum and what it rounds off, normalised where the three cancel (a loop of
// its own for each: with the choice inside the unrolled one 100 workers, d = 1 M 862 -> 930 us); g' = g_new is stored from the staged rows.
//
// Bound by issue slots and latency of the finishing warps (136 instructions per worker-coordinate of 128 lanes, 0.6 of the slots), by
// the power cap (1.5 .. 1.7 GHz on long vectors), and beyond a row pitch of 2 MB by rows travelling in pieces of 128 bytes: loads
// and stores alone then reach 0.68 of the copy rate (0.85 below that pitch), where 256-byte pieces reach 0.84.  us per step,
// step_split.cu -> here: 100 workers, d = 2 k 13.0 -> 9.4, 20 k 31.8 -> 26.0, 300 k 283 -> 262, 1 M 938 -> 859; 128, 40 k 53.2 -> 42.7, 1 M 1063 -> 1044;
// D-PSGD of 128, 1 M 966 -> 828; 256-ring, K = 40, d = 4 k 34.6 -> 21.9, 60 k 263 -> 233; rounds -> here: 144, K = 6, d = 500 k 3396 -> 984, 256
// 5327 -> 1680 (waiting for P; all of it at hand would be 1250); caller-written gradients, 100 workers, d = 1 M 3177 -> 862, 20 k 76 -> 27.
//
// Measured without gain: asking for 256-byte pieces in L2 ahead of the loads 917 -> 1200 us (128 workers, loads and stores alone); sums
// read sixteen columns at a time 966 -> 1043 (spills); normals drawn before the sums, or by half of the groups before, 1690 -> 1815, 1905
// (100 workers, d = 2 M); two buffers of digits and one stage 1690 -> 1786; a lane per slot of the ring, single planes 1166 -> 1187 (144).
// Every wait is bounded but the allocation of tensor memory, which waits for kernels that do not depend on this one.
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

constexpr int kPS = 32;             // coordinates per chunk
constexpr int kPBlock = 32;         // workers per k-step of the MMA (32 bytes)
constexpr int kPRows = 128;         // output workers per MMA
constexpr int kPGroup = 8;          // coordinates a finishing warp takes
constexpr int kPDigits = 5;         // of z and of P; also accumulators: digit pairs with k + l = 4 .. 8
constexpr int kPColumns = 2 * kPS;  // of an accumulator: model, tracker
constexpr int kPPlaneBytes = kPRows * kPBlock;                   // one digit plane of 128 x 32 weights
constexpr int kPDigitBytes = kPColumns * kPBlock;                // one digit of 32 workers: [8 coordinates][model | tracker][of them][32 bytes]
constexpr int kPBlockBytes = kPDigits * kPDigitBytes;
constexpr int kPSplitWarps = 8, kPFinishWarps = 16;
constexpr int kPMmaWarp = kPSplitWarps, kPLoadXYWarp = kPMmaWarp + 1, kPTailWarp = kPMmaWarp + 2,
              kPFinishWarp = kPMmaWarp + 4;  // the one before it fetches P
constexpr int kPThreads = (kPSplitWarps + 4 + kPFinishWarps) * 32;
// Registers: 72 per thread at launch; what the issuing and the splitting warps give up goes to the finishing ones.
constexpr int kPLaunchRegisters = 72, kPSplitRegisters = 48, kPIssueRegisters = 24, kPFinishRegisters = 96;
static_assert(kPSplitWarps * kPSplitRegisters + 4 * kPIssueRegisters + kPFinishWarps * kPFinishRegisters <= kPThreads / 32 * kPLaunchRegisters,
              "register split");
// Tensor memory: the accumulators; up to 128 workers the digit planes of P, eight columns each, behind them.
constexpr int kPTmemColumns = 512, kPPolyColumn = kPDigits * kPColumns;
static_assert(kPPolyColumn + 4 * kPDigits * 8 <= kPTmemColumns, "tensor memory plan");
constexpr int kPScaleSlots = 4;     // chunks whose scales are kept: see the splitting warps
constexpr int kPMaxBuffers = 3, kPMaxRing = 8;
constexpr size_t kPCtrlBytes = 512, kPSmemLimit = 232448;

struct RowsMaps {
  CUtensorMap x, y;        // boxes {32 coordinates, 32 nb workers}
  CUtensorMap g, a, c;     // boxes {32, 128 (or all) workers}, 128-byte swizzle; caller-written gradients: g, g_new like x
  CUtensorMap xs, ys, gs;  // the same, ending on a 16-byte boundary: stores
};
static_assert(sizeof(RowsMaps) <= sizeof(TensorMapSet), "tensor map storage");

struct RowsTables {
  const unsigned char* tiles;  // [output half][input block][digit plane 4 .. 0][rows x 32 bytes in core-matrix order]
  const int* row_exp;      // exponent of each output worker's scale
  // P itself, for what stays in float64: [output worker][input worker, padded to 32], or, if the blocks of P depend on their
  // distance only, its first 32 rows
  const double* poly;
  int circulant;
  int nb;                  // blocks of 32 input workers
  const uint8_t* guard;    // guard_groups x guard_size inputs
  int guard_groups, guard_size;  // size 2 or a multiple of 4
  float guard_tau;
  RowsTiles use;           // beyond 128 workers: which tiles, in which order, from where
  int plane_bytes[2], half_at;  // [output half]: a plane of the rows there are; where the second half's tiles begin
  uint8_t reach[8];        // [32 outputs], a bit per input block: some entry of P itself is not zero
};

struct RowsPlan {
  int raws, digs, stages;        // buffers of x and y, of digits, of g, a, c
  int ring, unit;                // slots for planes of P (0: they are in tensor memory), planes in one
  int rows;                      // of a stage
  int ins, outs;                 // arrays of x and y (and the gradients of the caller), of a stage
  int chunk_shift;               // log2 of the chunks a block takes next to one another
  int raw_at, dig_at, ring_at, scale_at, exp_at, max_at, guard_at, ctrl_at, bytes;
};

// Bytes of a digit plane of 32 inputs for the output workers there are in a half; up to 128 workers planes are whole.
inline int plane_bytes(int n, int half) { return n <= kPRows ? kPPlaneBytes : (std::min(n - kPRows * half, kPRows) + 7) / 8 * 256; }

inline int stage_rows(int n) { return std::min(kPRows, (n + kPBlock - 1) / kPBlock * kPBlock); }

// Shared memory: g, a, c stages | x, y of a chunk | its digits | planes of P | scales and flags | row exponents | maxima | groups
// of the guard | barriers.  1 KiB of slack aligns the whole.
inline RowsPlan plan_for(int n, int mode, int guard_entries, int raws, int digs, int stages, int ring, int unit) {
  const int nb = (n + kPBlock - 1) / kPBlock;
  RowsPlan s{};
  s.raws = raws;
  s.digs = digs;
  s.stages = stages;
  s.ring = ring;
  s.unit = unit;
  s.rows = stage_rows(n);
  s.ins = mode == kModeExternal ? 4 : 2;
  s.outs = mode == kModeExternal ? 2 : 3;
  s.raw_at = stages * s.outs * s.rows * kPS * 4;
  s.dig_at = s.raw_at + raws * s.ins * nb * kPBlock * kPS * 4;
  s.ring_at = s.dig_at + digs * nb * kPBlockBytes;
  s.scale_at = s.ring_at + ring * unit * kPPlaneBytes;
  s.exp_at = s.scale_at + kPScaleSlots * (kPColumns + 2) * 4;
  s.max_at = s.exp_at + 256 * 4;
  s.guard_at = s.max_at + 2 * 4 * kPColumns * 8;
  s.ctrl_at = s.guard_at + (guard_entries + 15) / 16 * 16;
  s.bytes = s.ctrl_at + static_cast<int>(kPCtrlBytes) + 1024;
  return s;
}

// The largest of these that fits (bytes = 0: none); what is left over beyond 128 workers goes to the planes of P.
inline RowsPlan rows_plan(int n, int mode, int guard_entries) {
  constexpr int one[4][3] = {{3, 2, 3}, {2, 2, 2}, {2, 1, 2}, {2, 1, 1}};
  constexpr int two[2][3] = {{2, 1, 1}, {1, 1, 1}};
  if (n <= kPRows) {
    for (const auto& t : one) {
      if (n <= 64 && t[2] < 2) continue;  // two sets of warps take stages in turn
      const RowsPlan s = plan_for(n, mode, guard_entries, t[0], t[1], t[2], 0, 0);
      if (static_cast<size_t>(s.bytes) <= kPSmemLimit) return s;
    }
    return RowsPlan{};
  }
  for (const auto& t : two) {
    const int left = (static_cast<int>(kPSmemLimit) - plan_for(n, mode, guard_entries, t[0], t[1], t[2], 0, 0).bytes) / kPPlaneBytes;
    // whole tiles, if there is room for two; else two planes at a time
    const int unit = left >= 2 * kPDigits ? kPDigits : 2, ring = std::min(left / unit, kPMaxRing);
    if (left >= (t[0] == 1 ? 4 : 2 * kPDigits)) return plan_for(n, mode, guard_entries, t[0], t[1], t[2], ring, unit);
  }
  return RowsPlan{};
}

// `bytes` (a multiple of 16) from global to shared memory, both 16-byte aligned.
__device__ __forceinline__ void bytes_load(void* dst, const void* src, unsigned bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(s_addr(dst)), "l"(src), "r"(bytes),
               "r"(s_addr(bar))
               : "memory");
}

// Joined sums of this thread's output worker from the accumulators at `acc` on (whole warp): its eight
// coordinates, model or tracker.  `magic_hi`: of these; `row_power`: the row's exponent in the same place.
template <bool kTwo>
__device__ __forceinline__ void take_sums(uint32_t acc, const int* magic_hi, int row_power, double* out) {
  constexpr int kCount = 8;
  int hi[kCount], low[kCount], s6[kCount];
  {
    int s7[kCount];
    tmem_load8(acc + 4 * kPColumns, hi);
    tmem_load8(acc + 3 * kPColumns, s7);
    tmem_wait_load();
#pragma unroll
    for (int u = 0; u < kCount; ++u) hi[u] = hi[u] * 256 + s7[u];
  }
  {
    int s5[kCount];
    tmem_load8(acc, low);
    tmem_load8(acc + kPColumns, s5);
    tmem_wait_load();
#pragma unroll
    for (int u = 0; u < kCount; ++u) low[u] = s5[u] + ((low[u] + 128) >> 8);
  }
  tmem_load8(acc + 2 * kPColumns, s6);
  tmem_wait_load();
#pragma unroll
  for (int u = 0; u < kCount; u += 4) {
    const int4 four = *reinterpret_cast<const int4*>(magic_hi + u);
    const int m[4] = {four.x, four.y, four.z, four.w};
#pragma unroll
    for (int v = 0; v < 4; ++v) {
      const int magic = m[v] + row_power;
      out[u + v] = join_sums<kTwo>(hi[u + v], s6[u + v], low[u + v], magic, __hiloint2double(magic, 0));
    }
  }
}

// A warp's 32 output workers x 8 coordinates in float64, from the operands themselves: of the model for bits 0 .. 7 of `which`, of the
// tracker (kFold: with the caller's gradients, y + g_new - g) for bits 8 .. 15.  z: [array][input worker][32] at
// the first of the coordinates.  poly: rows of P of these workers (circulant: of the first 32, block `b` of whose columns is block
// (b + c) mod nb here).  Products on the float64 tensor path: four tiles of eight output workers (M) by eight columns (N), either the bits
// that are set, of both arrays (exact_columns), or all eight coordinates of both (100 workers, K = 6, d = 300 k, spread over six decades
// 729 -> 577 us, 256, K = 8, 200 k, over four 1787 -> 1423; not with the caller's gradients, where it costs the splitting warps 263 -> 277, 100
// workers, d = 300 k).
// Rare, and so out of the way of the main path's registers, on which its own tell all the same: with sixteen entries of P in flight
// instead of eight the main path took 1824 us for 1651 (100 workers, d = 2 M), with the columns in the same function 1656 for 1645, in one to
// choose from 1678, with what the two share in functions of its own 1673.  Bound by the latency of P from L2: with every coordinate here 100
// workers, K = 2, d = 1 M 888 -> 3900 us (with an array at a time a third more).
__device__ __noinline__ void exact_columns(const float* z, const double* poly, unsigned which, int circulant, int c, int nb, unsigned reach, double* out) {
  const int lane = threadIdx.x & 31, pitch = nb * kPBlock;
  const int stride = nb * kPBlock * kPS;
  auto weights = [&](int b) {  // this lane's entry of the first tile and k-step
    const int pb = !circulant ? b : b >= c ? b - c : b - c + nb;
    return poly + static_cast<size_t>(lane >> 2) * pitch + kPBlock * pb + (lane & 3);
  };
  bool finite = true;
  // lane l has tiles' rows l / 4, columns 2 (l % 4) + e; it wants row l, i.e. row l % 8 of tile l / 8
  auto hand_over = [&](const double (&sum)[4][2], int column, double* to) {
    double mine = 0.0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const double v = __shfl_sync(0xffffffffu, (column & 1) != 0 ? sum[t][1] : sum[t][0], 4 * (lane & 7) + (column >> 1));
      if ((lane >> 3) == t) mine = v;
    }
    finite = finite && (__double2hiint(mine) & 0x7ff00000) != 0x7ff00000;
    *to = mine;
  };
  const bool model = (which & 0xffu) != 0, tracker = which >> 8 != 0;
  unsigned left = which;
  for (int i = 0; i < (lane >> 2) && (left & (left - 1)) != 0; ++i) left &= left - 1;  // columns beyond the last repeat it
  const int mine = __ffs(left) - 1, array = mine >> 3;
  const float* const column = z + array * stride + (mine & 7) + (lane & 3) * kPS;
  double sum[4][2];
#pragma unroll
  for (int i = 0; i < 8; ++i) sum[i >> 1][i & 1] = 0.0;
  for (int b = 0; b < nb; ++b) {
    if ((reach >> b & 1) == 0) continue;  // a zero block of P
    const double* const pw = weights(b);
    const float* const zb = column + kPBlock * b * kPS;
#pragma unroll 1
    for (int h = 0; h < kPBlock; h += 16) {
#pragma unroll 2
      for (int s = 0; s < 4; ++s) {
        double w[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) w[t] = __ldg(pw + static_cast<size_t>(8 * t) * pitch + h + 4 * s);
        const double v = static_cast<double>(zb[(h + 4 * s) * kPS]);
#pragma unroll
        for (int t = 0; t < 4; ++t) dmma(sum[t], w[t], v);
      }
    }
  }
  left = which;
  for (int q = 0; left != 0; ++q, left &= left - 1) hand_over(sum, q, out + __ffs(left) - 1);
  if (__any_sync(0xffffffffu, !finite)) {
    // Infinities or NaN among the operands: a lane sums its own worker, without the zeros of P, which the products above turn
    // into NaN.
#pragma unroll 1
    for (int u = 0; u < 16; ++u) {
      if (!(u < 8 ? model : tracker)) continue;
      const int array = u >> 3;
      double own = 0.0;
      for (int b = 0; b < nb; ++b) {
        if ((reach >> b & 1) == 0) continue;
        const int pb = !circulant ? b : b >= c ? b - c : b - c + nb;
        const double* const pw = poly + static_cast<size_t>(lane) * pitch + kPBlock * pb;
        for (int w = 0; w < kPBlock; ++w)
          if (pw[w] != 0.0) own = fma(pw[w], static_cast<double>(z[array * stride + (kPBlock * b + w) * kPS + (u & 7)]), own);
      }
      out[u] = own;
    }
  }
}

template <bool kFold>
__device__ __noinline__ void exact_sums(const float* z, const double* poly, unsigned which, int circulant, int c, int nb, unsigned reach, double* out) {
  if (!kFold && __popc(which) <= 8) {
    exact_columns(z, poly, which, circulant, c, nb, reach, out);
    return;
  }
  const int lane = threadIdx.x & 31, pitch = nb * kPBlock;
  const int stride = nb * kPBlock * kPS;
  auto value = [&](int array, const float* at) {
    double v = static_cast<double>(at[0]);
    if (kFold && array != 0) v += static_cast<double>(at[stride]) - static_cast<double>(at[2 * stride]);
    return v;
  };
  auto weights = [&](int b) {  // this lane's entry of the first tile and k-step
    const int pb = !circulant ? b : b >= c ? b - c : b - c + nb;
    return poly + static_cast<size_t>(lane >> 2) * pitch + kPBlock * pb + (lane & 3);
  };
  bool finite = true;
  // lane l has tiles' rows l / 4, columns 2 (l % 4) + e; it wants row l, i.e. row l % 8 of tile l / 8
  auto hand_over = [&](const double (&sum)[4][2], int column, double* to) {
    double mine = 0.0;
#pragma unroll
    for (int t = 0; t < 4; ++t) {
      const double v = __shfl_sync(0xffffffffu, (column & 1) != 0 ? sum[t][1] : sum[t][0], 4 * (lane & 7) + (column >> 1));
      if ((lane >> 3) == t) mine = v;
    }
    finite = finite && (__double2hiint(mine) & 0x7ff00000) != 0x7ff00000;
    *to = mine;
  };
  const bool model = (which & 0xffu) != 0, tracker = which >> 8 != 0;
  double sum[2][4][2];
#pragma unroll
  for (int i = 0; i < 16; ++i) sum[i >> 3][i >> 1 & 3][i & 1] = 0.0;
  for (int b = 0; b < nb; ++b) {
    if ((reach >> b & 1) == 0) continue;
    const double* const pw = weights(b);
    const float* const zb = z + (kPBlock * b + (lane & 3)) * kPS + (lane >> 2);
#pragma unroll 1
    for (int h = 0; h < kPBlock; h += 16) {
#pragma unroll 2
      for (int s = 0; s < 4; ++s) {
        const float* const at = zb + (h + 4 * s) * kPS;
        double w[4];
#pragma unroll
        for (int t = 0; t < 4; ++t) w[t] = __ldg(pw + static_cast<size_t>(8 * t) * pitch + h + 4 * s);
        if (!kFold) {
          const double v = value(0, at), u = value(1, at + stride);
#pragma unroll
          for (int t = 0; t < 4; ++t) dmma(sum[0][t], w[t], v);
#pragma unroll
          for (int t = 0; t < 4; ++t) dmma(sum[1][t], w[t], u);
          continue;
        }
        if (model) {
          const double v = value(0, at);
#pragma unroll
          for (int t = 0; t < 4; ++t) dmma(sum[0][t], w[t], v);
        }
        if (tracker) {
          const double v = value(1, at + stride);
#pragma unroll
          for (int t = 0; t < 4; ++t) dmma(sum[1][t], w[t], v);
        }
      }
    }
  }
#pragma unroll
  for (int u = 0; u < 16; ++u) hand_over(sum[u >> 3], u & 7, out + u);
  if (__any_sync(0xffffffffu, !finite)) {
    // Infinities or NaN among the operands: a lane sums its own worker, without the zeros of P, which the products above turn
    // into NaN.
#pragma unroll 1
    for (int u = 0; u < 16; ++u) {
      if (!(u < 8 ? model : tracker)) continue;
      const int array = u >> 3;
      double own = 0.0;
      for (int b = 0; b < nb; ++b) {
        if ((reach >> b & 1) == 0) continue;
        const int pb = !circulant ? b : b >= c ? b - c : b - c + nb;
        const double* const pw = poly + static_cast<size_t>(lane) * pitch + kPBlock * pb;
        for (int w = 0; w < kPBlock; ++w)
          if (pw[w] != 0.0) own = fma(pw[w], value(array, z + array * stride + (kPBlock * b + w) * kPS + (u & 7)), own);
      }
      out[u] = own;
    }
  }
}

// kWide: the gradient in float64 (the precision of the rounds kernel, in whose place
// the call runs; beyond 128 workers, where it would run there, sigma xi in float64 too) instead of float32 at the rounded model (the other
// tensor-path kernels').  kRows: 64, 96, 128 or 256, n rounded up.
// kAtStart: the gradient at the model the step started from.
template <int kMode, bool kWide, int kRows, bool kAtStart>
__global__ void __launch_bounds__(kPThreads, 1)
step_rows_kernel(const StepParams p, const __grid_constant__ RowsMaps maps, const __grid_constant__ RowsTables tb,
                  const __grid_constant__ RowsPlan plan) {
  constexpr bool kTwo = kRows == 256;
  constexpr int H = kTwo ? 2 : 1, kCopies = kRows == 64 ? 2 : 1;
  // Up to 96 workers nothing is left to finish for a quarter of tensor memory's lanes, and so for the SM's fourth scheduler, whose
  // warps are the only ones to reach it: there they split.
  constexpr bool kFourth = kRows == 96;
  constexpr int kSplits = kFourth ? 6 : kPSplitWarps, kParts = kSplits / 2, kFinishers = kFourth ? 12 : kPFinishWarps;
  extern __shared__ unsigned char smem_unaligned[];
  unsigned char* const smem = smem_unaligned + ((1024u - (s_addr(smem_unaligned) & 1023u)) & 1023u);
  float* const e_mem = reinterpret_cast<float*>(smem);                        // [stage][g | a | c][rows][32], swizzled
  float* const raw_mem = reinterpret_cast<float*>(smem + plan.raw_at);        // [buffer][x | y][32 nb][32]
  unsigned char* const dig_mem = smem + plan.dig_at;                          // [buffer][block][digit][64 rows x 32 bytes]
  int* const magics = reinterpret_cast<int*>(smem + plan.scale_at);           // [slot][model | tracker coordinate]
  unsigned* const flags = reinterpret_cast<unsigned*>(magics + kPScaleSlots * kPColumns);  // [slot][array]: coordinates in float64
  int* const row_exp = reinterpret_cast<int*>(smem + plan.exp_at);
  float2* const maxima = reinterpret_cast<float2*>(smem + plan.max_at);       // [chunk parity][part][64 columns]
  uint8_t* const guard = smem + plan.guard_at;
  uint64_t* const raw_full = reinterpret_cast<uint64_t*>(smem + plan.ctrl_at);
  uint64_t* const raw_empty = raw_full + kPMaxBuffers;
  uint64_t* const dig_full = raw_empty + kPMaxBuffers;
  uint64_t* const dig_empty = dig_full + 2;
  uint64_t* const acc_full = dig_empty + 2;
  uint64_t* const acc_empty = acc_full + 2;
  uint64_t* const e_full = acc_empty + 2;
  uint64_t* const out_ready = e_full + kPMaxBuffers;
  uint64_t* const max_ready = out_ready + kPMaxBuffers;
  uint64_t* const drained = max_ready + 1;
  uint64_t* const ring_full = drained + 1;
  uint64_t* const ring_empty = ring_full + kPMaxRing;
  unsigned* const finished = reinterpret_cast<unsigned*>(ring_empty + kPMaxRing);  // [finishing warp]: units done
  uint32_t* const tmem_slot = finished + kPFinishWarps;
  static_assert((4 * kPMaxBuffers + 10 + 2 * kPMaxRing) * 8 + (kPFinishWarps + 1) * 4 <= kPCtrlBytes, "barrier area");

  const int tid = threadIdx.x, lane = tid & 31, warp = __shfl_sync(0xffffffffu, tid >> 5, 0);  // uniform for the compiler
  const int n = p.n, nb = tb.nb;
  const unsigned limit = p.spin_limit;
  for (int e = tid; e < 256; e += kPThreads) row_exp[e] = e < n ? tb.row_exp[e] : 0;
  for (int e = tid; e < tb.guard_groups * tb.guard_size; e += kPThreads) guard[e] = tb.guard[e];
  if (tid == 0) {
    for (int s = 0; s < kPMaxBuffers; ++s) {
      bar_init(&raw_full[s], 1);
      bar_init(&raw_empty[s], kSplits);
      bar_init(&e_full[s], 1);
      bar_init(&out_ready[s], kFinishers / kCopies);
    }
    for (int s = 0; s < 2; ++s) {
      bar_init(&dig_full[s], kSplits);
      bar_init(&dig_empty[s], 1);
    }
    for (int s = 0; s < kCopies; ++s) {
      bar_init(&acc_full[s], 1);
      bar_init(&acc_empty[s], kFinishers / kCopies);
    }
    bar_init(max_ready, kSplits);
    bar_init(drained, 1);
    for (int s = 0; s < kPMaxRing; ++s) {
      bar_init(&ring_full[s], 1);
      bar_init(&ring_empty[s], 1);
    }
    for (int w = 0; w < kPFinishWarps; ++w) finished[w] = 0;
    fence_barrier_init();
  }
  if (warp == kPMmaWarp) tmem_alloc(tmem_slot, kPTmemColumns);
  fence_async_shared();
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  constexpr uint32_t tmem = 0;  // all 512 columns are this CTA's: they start at address 0
  const bool ours = *tmem_slot == 0;
  if (tid == 0 && !ours) atomicExch(p.status, 2);
  // P into tensor memory, all of it or four tiles: thread = output worker = tensor memory lane
  if (ours && warp >= kPFinishWarp && warp < kPFinishWarp + 4) {
    const int row = (warp & 3) * 32 + lane, at = (row % (kRows == 64 ? 64 : kPRows) >> 3) * 256 + (row & 7) * 16;
    uint32_t to = tmem + kPPolyColumn + (static_cast<uint32_t>(warp & 3) << 21);
    for (int t = 0; t < (kTwo ? tb.use.residents : nb); ++t) {
      const int half = kTwo ? tb.use.resident[t] >> 4 : 0, plane = kTwo ? tb.plane_bytes[half] : kPPlaneBytes;
      const unsigned char* src = tb.tiles + half * tb.half_at + static_cast<size_t>(kTwo ? tb.use.resident[t] & 15 : t) * kPDigits * plane + at;
#pragma unroll
      for (int q = 0; q < kPDigits; ++q, src += plane, to += 8) {
        uint4 a = make_uint4(0, 0, 0, 0), b = a;  // a plane of the second half ends with its workers
        if (!kTwo || at < plane) {
          a = __ldg(reinterpret_cast<const uint4*>(src));
          b = __ldg(reinterpret_cast<const uint4*>(src + 128));
        }
        const uint32_t w[8] = {a.x, a.y, a.z, a.w, b.x, b.y, b.z, b.w};
        tmem_store8(to, w);
      }
    }
    tmem_wait_store();
  }
  tmem_fence_before();
  __syncthreads();
  tmem_fence_after();
  if (p.beside == 0) chain_wait();
  chain_next();

  // This CTA takes slabs blockIdx.x, blockIdx.x + gridDim.x, ... of 1 << chunk_shift chunks; unit v = chunk number * H + half
  const int shift = plan.chunk_shift;
  auto chunk_col = [&](int k) {  // below 2^31 + 64 in 32 bits
    return static_cast<long long>((((blockIdx.x + static_cast<unsigned>(k >> shift) * gridDim.x) << shift) + (k & ((1 << shift) - 1))) * kPS);
  };
  int chunks = ours && blockIdx.x < p.num_slabs ? static_cast<int>((p.num_slabs - blockIdx.x + gridDim.x - 1) / gridDim.x) << shift : 0;
  while (chunks > 0 && chunk_col(chunks - 1) >= p.d) --chunks;
  const int total = chunks * H;
  auto warp_wait = [&](uint64_t* bar, int phase) {  // every lane polls the same barrier: no broadcast of the verdict
    return __all_sync(0xffffffffu, bar_wait(bar, phase & 1, limit));
  };

  auto split = [&](int index) {
    // ---------------------------------------------------------------- splitting warps: thread = model or tracker of a coordinate
    const int array = index & 1, part = index >> 1;  // takes the half blocks part, part + kParts, ... of 16 workers
    const int column = array * kPS + lane, halves = 2 * nb;
    const bool idle = kMode == kModeDpsgd && array != 0;  // D-PSGD has no tracker: its rows of the digits are never used
    const int raw_floats = plan.ins * nb * kPBlock * kPS;
    const int array_floats = nb * kPBlock * kPS;
    const float* const first = raw_mem + array * array_floats + lane;
    const bool fold = kMode == kModeExternal && array != 0;  // Algorithm 2's tracker update, y + g_new - g
    unsigned char* const to = dig_mem + (2 * (lane >> 3) + array) * 256 + (lane & 7) * 16;
    bool ok = true;
    int raw = 0, raw_phase = 0, buf = 0, use = 0;
    const bool later = !kFourth && plan.raws > 1;
    bool held = false;  // the buffer of the chunk before this one has not been given back
    for (int k = 0; k < chunks && ok; ++k) {
      const int slot = k % kPScaleSlots;
      const float* const col = first + raw * raw_floats;
      ok = warp_wait(&raw_full[raw], raw_phase);
      if (!ok) break;
      if (kMode == kModeExternal && index == 0 && lane == 0) {  // g' = g_new: from the staged rows themselves
        const long long at = chunk_col(k);
        if (at < (p.d & ~3LL)) tile_store(&maps.gs, static_cast<int>(at), 0, raw_mem + raw * raw_floats + 2 * array_floats);
        store_commit();
      }
      auto value = [&](int w) {
        const float* const at = col + w * kPS;
        return fold ? at[0] + (at[array_floats] - at[2 * array_floats]) : at[0];
      };
      // largest magnitude, and the smallest of the largest magnitudes of the guard's groups
      float top_f = 0.f, low_f = __uint_as_float(0x7f800000u);
      if (!idle) {
        float change = 0.f;  // largest |g_new - g|
        auto largest = [&](auto four) {  // `four`: of four workers
#pragma unroll 1
          for (int h = part; h < halves; h += kParts) {
            float m[4];
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              float v[4];
              four(col + (16 * h + 4 * i) * kPS, v);
              m[i] = max_abs3(max_abs3(v[0], v[1], v[2]), v[3], 0.f);
            }
            top_f = max_abs3(max_abs3(m[0], m[1], m[2]), m[3], top_f);
          }
        };
        if (fold) {
          largest([&](const float* at, float (&v)[4]) {
            float t[4];
#pragma unroll
            for (int u = 0; u < 4; u += 2) {
              const float *const p0 = at + u * kPS, *const p1 = p0 + kPS;
              const F2 delta = sub2(pack2(p0[array_floats], p1[array_floats]), pack2(p0[2 * array_floats], p1[2 * array_floats]));
              unpack2(delta, t[u], t[u + 1]);
              unpack2(add2(pack2(p0[0], p1[0]), delta), v[u], v[u + 1]);
            }
            change = max_abs3(max_abs3(change, t[0], t[1]), t[2], t[3]);
          });
        } else {
          largest([&](const float* at, float (&v)[4]) {
#pragma unroll
            for (int u = 0; u < 4; ++u) v[u] = at[u * kPS];
          });
        }
        low_f = group_low<uchar4, uchar2>(value, guard, tb.guard_groups, tb.guard_size, part, kParts);
        // These sums lack what their two roundings leave out, 2^-24 of the difference and of themselves: below 2^-18 of the largest of
        // them while that is 2^-5 of the largest difference.  Else every warp looks anew, below.
        if (fold && change * 0x1p-5f > top_f) low_f = -1.f;
      }
      float2* const mx = maxima + (k & 1) * 4 * kPColumns + column;  // read again two chunks later, behind the next hand-over
      mx[part * kPColumns] = make_float2(top_f, low_f);
      __syncwarp();
      if (lane == 0) bar_arrive(max_ready);
      ok = warp_wait(max_ready, k);
      if (!ok) break;
#pragma unroll
      for (int i = 0; i < kParts; ++i) {
        const float2 other = mx[i * kPColumns];
        top_f = max_abs3(top_f, other.x, 0.f);
        low_f = fminf(low_f, other.y);
      }
      const bool cancels = fold && __any_sync(0xffffffffu, low_f < 0.f);  // the same in all warps of the array
      if (cancels) {
        auto sum = [&](int w) { return fold_value(col[w * kPS], col[w * kPS + array_floats], col[w * kPS + 2 * array_floats]); };
        top_f = 0.f;
#pragma unroll 2
        for (int w = 0; w < 16 * halves; w += 2) top_f = max_abs3(sum(w), sum(w + 1), top_f);
        low_f = group_low<uchar4, uchar2>(sum, guard, tb.guard_groups, tb.guard_size, 0, 1);
      }
      const unsigned top = __float_as_uint(top_f);
      // as float bits: not finite, too small for the scale; an output may read nothing near the largest operand
      const bool exact = top >= 0x7f800000u || (top != 0 && (top < kSmallest || low_f < tb.guard_tau * top_f));
      const int e = top == 0 || exact ? 30 : static_cast<int>((top + kRoundUp) >> 23) - 127;  // all |z| < 2^(e+1)
      const float scale = __uint_as_float(static_cast<unsigned>(157 - e) << 23);              // 2^(30 - e)
      const unsigned exact_lanes = __ballot_sync(0xffffffffu, exact);
      if (use > 0) ok = warp_wait(&dig_empty[buf], use - 1);
      if (!ok) break;
      // The slot was last read for chunk k - 4: the finishing warps read a unit's scales before they release the accumulators, and
      // the MMAs of chunk k - 2 at the latest (complete: dig_empty) came after that release for all units of k - 4.
      if (part == 0) {
        magics[slot * kPColumns + 16 * (lane >> 3) + 8 * array + (lane & 7)] = 0x43380000 + (exact ? 0 : e - 6) * (1 << 20);
        if (lane == 0) flags[slot * 2 + array] = exact_lanes;
      }
      if (!idle) {
        auto split_all = [&](auto four) {
#pragma unroll 1
          for (int h = part; h < halves; h += kParts) {
            uint32_t d[4][kPDigits];
#pragma unroll
            for (int u = 0; u < 4; ++u) four(col + (h * 16 + 4 * u) * kPS, d[u]);
            unsigned char* const at = to + (buf * nb + (h >> 1)) * kPBlockBytes + (h & 1) * 128;
#pragma unroll
            for (int q = 0; q < kPDigits; ++q) *reinterpret_cast<uint4*>(at + q * kPDigitBytes) = make_uint4(d[0][q], d[1][q], d[2][q], d[3][q]);
          }
        };
        if (cancels) {
          split_all([&](const float* src, uint32_t (&d)[kPDigits]) { four_fold_digits<true>(src, array_floats, kPS, scale, d); });
        } else if (fold) {
          split_all([&](const float* src, uint32_t (&d)[kPDigits]) { four_fold_digits<false>(src, array_floats, kPS, scale, d); });
        } else {
          split_all([&](const float* src, uint32_t (&d)[kPDigits]) { four_digits(src, kPS, scale, d); });
        }
      }
      fence_async_shared();  // the MMAs read the digits through the asynchronous proxy
      __syncwarp();
      if (lane == 0) bar_arrive(&dig_full[buf]);
      if (kMode == kModeExternal && index == 0 && lane == 0) store_wait_read();
      // The finishing warps read operands that were not split themselves: such a chunk's are kept until they are done (of two sets that
      // take turns the one whose chunk it is).  Behind the splitting of the next one, where there is another buffer: waiting before it
      // 100 workers, K = 2, d = 300 k, all in float64, took 1511 us instead of 1202, 60, d = 100 k 288 instead of 198.  (Not of 65 to 96:
      // one more value in the splitting warps that are compiled twice, and D-PSGD of 90, d = 100 k, alike, takes 82 us instead of 76.)
      if (__builtin_expect(held || (exact_lanes != 0 && !later), 0)) {
        const int of = held ? k - 1 : k;
        if (lane < kPFinishWarps && (kCopies == 1 || (lane >> 3) == (of & 1)) && !(kFourth && (lane & 3) == 3))
          ok = count_wait_relaxed(&finished[lane], static_cast<unsigned>((of + 1) * H), limit);
        ok = __all_sync(0xffffffffu, ok);
        asm volatile("fence.acq_rel.cta;" ::: "memory");
        if (lane == 0 && ok) bar_arrive(&raw_empty[!held ? raw : raw == 0 ? plan.raws - 1 : raw - 1]);
      }
      held = exact_lanes != 0 && later;
      if (exact_lanes == 0 && lane == 0 && ok) bar_arrive(&raw_empty[raw]);
      __syncwarp();
      if (++raw == plan.raws) {
        raw = 0;
        raw_phase ^= 1;
      }
      if (++buf == plan.digs) {
        buf = 0;
        ++use;
      }
    }
    if (kMode == kModeExternal && index == 0 && lane == 0) store_wait_all();
    if (!ok && lane == 0) atomicExch(p.status, 1);
  };
  // A branch per share of the registers: the compiler takes it from there.
  if (warp >= kPFinishWarp) {
    asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;" ::"n"(kPFinishRegisters));
    if (kFourth && (warp & 3) == 3) {
      split((warp >> 2) - 1);
    } else {
    // ---------------------------------------------------------------- finishing warps: thread = output worker
    // kCopies = 2: the upper half of the rows holds the same workers again; half of the groups take every other chunk, and of its
    // coordinates the upper rows the second eight of every sixteen.
    const int quarter = warp & 3, group = (warp - kPFinishWarp) >> 2, set = kCopies == 2 ? group >> 1 : 0;
    const int row = (kCopies == 2 ? quarter & 1 : quarter) * 32 + lane, part = kCopies == 2 ? 2 * (group & 1) + (quarter >> 1) : group;
    const uint32_t acc = tmem + (static_cast<uint32_t>(quarter) << 21) + 2 * kPGroup * part;
    const double alpha = p.alpha;
    constexpr bool kWideNoise = kWide && kTwo;
    const float sigma = static_cast<float>(p.sigma);
    const bool noisy = kMode != kModeExternal && p.sigma != 0.0;
    const int d = static_cast<int>(p.d), d_tma = d & ~3;  // columns below d_tma are written by the TMA stores
    const int stage_floats = plan.outs * plan.rows * kPS, raw_floats = plan.ins * nb * kPBlock * kPS;
    const int at0 = ((2 * part) ^ (row & 7)) << 2, at1 = at0 ^ 4;
    int st = set, st_phase = 0, raw = set, power = row_exp[row] << 20;
    if (kCopies == 2 && set >= plan.stages) st = 0, st_phase = 1;
    if (kCopies == 2 && set >= plan.raws) raw = 0;
    bool ok = true;
    for (int k = set, v = set; k < chunks && ok; k += kCopies) {
      const int slot = k % kPScaleSlots;
      const int j = static_cast<int>(chunk_col(k)) + kPGroup * part;
#pragma unroll 1
      for (int half = 0; half < H; ++half) {
        const int w = kPRows * half + row;
        const bool active = kPRows * half + (row & ~31) < n;  // of the whole warp
        ok = warp_wait(&acc_full[set], v / kCopies);
        if (!ok) break;
        tmem_fence_after();
        double sums[16];  // models, trackers
        double in_full[16];
        if (active) {
          // coordinates that were not split
          const unsigned exact = (flags[slot * 2] >> (kPGroup * part) & 0xffu) |
                                 (kMode != kModeDpsgd ? (flags[slot * 2 + 1] >> (kPGroup * part) & 0xffu) << 8 : 0u);
          if (__builtin_expect(exact != 0, 0)) {
            const int c = 4 * half + (row >> 5), pitch = nb * kPBlock;
            const double* const rows = tb.poly + (tb.circulant ? 0 : static_cast<size_t>(kPBlock * c) * pitch);
            exact_sums<kMode == kModeExternal>(raw_mem + raw * raw_floats + kPGroup * part, rows, exact, tb.circulant, c, nb, tb.reach[c], in_full);
          }
          const int* const magic = magics + slot * kPColumns + 2 * kPGroup * part;
          if (kTwo) power = row_exp[w] << 20;
          take_sums<kTwo>(acc, magic, power, sums);
          if (kMode != kModeDpsgd) take_sums<kTwo>(acc + kPGroup, magic + kPGroup, power, sums + 8);
          if (__builtin_expect(exact != 0, 0)) {
#pragma unroll
            for (int u = 0; u < 16; ++u)
              if (exact >> u & 1) sums[u] = in_full[u];
          }
        }
        tmem_fence_before();
        __syncwarp();
        if (lane == 0) bar_arrive(&acc_empty[set]);
        // ---- normals of this thread's worker: of the four lanes of a Philox call each draws two coordinates for all four
        float xi[8];
        if (noisy && active) {
          const unsigned long long jn = static_cast<unsigned long long>(p.coord_offset + j) + (lane & 3);
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            float t[4];
            normal_quad(p.round_key, jn + 4 * i, static_cast<uint32_t>(w >> 2), p.t_noise, kWideNoise ? 1.f : sigma, t);
            transpose_quad(t, lane & 3);
#pragma unroll
            for (int u = 0; u < 4; ++u) xi[4 * i + u] = t[u];
          }
        } else {
#pragma unroll
          for (int u = 0; u < 8; ++u) xi[u] = 0.f;
        }
        ok = warp_wait(&e_full[st], st_phase);
        if (!ok) break;
        if (active) {
          const bool mine = w < n;
          float* const sg = e_mem + st * stage_floats + row * kPS;  // caller-written gradients: x', y' only
          float* const sa = kMode == kModeExternal ? sg : sg + plan.rows * kPS;
          float* const sc = sa + plan.rows * kPS;
          auto take8 = [&](const float* src, float (&v)[8]) {
            const float4 a = *reinterpret_cast<const float4*>(src + at0), b = *reinterpret_cast<const float4*>(src + at1);
            v[0] = a.x, v[1] = a.y, v[2] = a.z, v[3] = a.w, v[4] = b.x, v[5] = b.y, v[6] = b.z, v[7] = b.w;
          };
          auto put8 = [&](float* to, const float (&v)[8]) {
            *reinterpret_cast<float4*>(to + at0) = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(to + at1) = make_float4(v[4], v[5], v[6], v[7]);
          };
          if (kMode != kModeDpsgd && p.y_obs != nullptr && mine) {  // optional observer: the gossiped tracker
#pragma unroll
            for (int u = 0; u < 8; ++u)
              if (j + u < d) p.y_obs[w * p.ld + j + u] = static_cast<float>(sums[8 + u]);
          }
          float gold[8], av[8], cv[8], from[8], xo[8], go[8], yo[8];
          if (kMode == kModeExternal) {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              xo[u] = static_cast<float>(fma(-alpha, sums[8 + u], sums[u]));
              yo[u] = static_cast<float>(sums[8 + u]);
            }
          } else {
            take8(sg, gold);
            // gradient point of Algorithm 2 as printed: the model the step started from, still in global memory - stored after this
            if (kAtStart) {
#pragma unroll
              for (int q = 0; q < 8; q += 4) {
                float4 s4 = make_float4(0.f, 0.f, 0.f, 0.f);
                if (mine && j + q < d) s4 = *reinterpret_cast<const float4*>(p.x + w * p.ld + j + q);
                from[q] = s4.x, from[q + 1] = s4.y, from[q + 2] = s4.z, from[q + 3] = s4.w;
              }
            }
            take8(sa, av);
            take8(sc, cv);
            // model update, y~ - g
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const double gd = static_cast<double>(gold[u]);
              sums[u] = fma(-alpha, kMode == kModeDpsgd ? gd : sums[8 + u], sums[u]);
              if (kMode != kModeDpsgd) sums[8 + u] -= gd;
              xo[u] = static_cast<float>(sums[u]);
              if (!kAtStart) from[u] = xo[u];
            }
            // gradient and fold
#pragma unroll
            for (int u = 0; u < 8; u += 2) {
              if (kWide) {
#pragma unroll
                for (int e = u; e < u + 2; ++e)
                  go[e] = static_cast<float>(fma(static_cast<double>(av[e]), (kAtStart ? static_cast<double>(from[e]) : sums[e]) - static_cast<double>(cv[e]),
                                                    kWideNoise ? static_cast<double>(sigma) * static_cast<double>(xi[e]) : static_cast<double>(xi[e])));
              } else {
                unpack2(fma2(pack2(av[u], av[u + 1]), sub2(pack2(from[u], from[u + 1]), pack2(cv[u], cv[u + 1])), pack2(xi[u], xi[u + 1])), go[u], go[u + 1]);
              }
            }
            if (kMode != kModeDpsgd) {
#pragma unroll
              for (int u = 0; u < 8; ++u) yo[u] = static_cast<float>(sums[8 + u] + static_cast<double>(go[u]));
            }
            put8(sg, go);
          }
          put8(sa, xo);
          if (kMode != kModeDpsgd) put8(sc, yo);
          if (j + kPGroup > d_tma && mine) {  // TMA clips a store at 16-byte granularity: the last d % 4 columns are written here
#pragma unroll 1
            for (int u = max(d_tma - j, 0); u < kPGroup && j + u < d; ++u) {
              const int at = (u < 4 ? at0 : at1) + (u & 3);
              p.g[w * p.ld + j + u] = kMode == kModeExternal ? p.g_ext[w * p.ld + j + u] : sg[at];
              p.x[w * p.ld + j + u] = sa[at];
              if (kMode != kModeDpsgd) p.y[w * p.ld + j + u] = sc[at];
            }
          }
        }
        fence_async_shared();  // results visible to the TMA stores
        __syncwarp();
        if (lane == 0) {
          bar_arrive(&out_ready[st]);
          // relaxed: what a reader of the count waits for, this unit's reads of x and y, went into the results above
          *const_cast<volatile unsigned*>(&finished[warp - kPFinishWarp]) = static_cast<unsigned>(v + 1);
        }
        v += kCopies;
        st += kCopies;
        if (st >= plan.stages) {
          st -= plan.stages;
          st_phase ^= 1;
        }
      }
      raw += kCopies;
      if (raw >= plan.raws) raw -= plan.raws;
    }
    if (!ok && lane == 0) atomicExch(p.status, 1);
    }
  } else if (warp < kPSplitWarps) {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPSplitRegisters));
    if (!kFourth) {
      split(warp);
    } else if ((warp & 3) == 3) {
      split(warp >> 2);
    }
  } else {
    asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;" ::"n"(kPIssueRegisters));
    if (warp == kPMmaWarp) {
    // ---------------------------------------------------------------- MMAs
    // The whole warp walks the loop, one lane issues: operands computed in uniform control flow stay in uniform registers.
    const uint64_t dig_base = mma_operand(s_addr(dig_mem), 256, 128), ring_base = mma_operand(s_addr(smem + plan.ring_at), 256, 128);
    const bool leader = lane == 0;
    constexpr uint64_t kDigit = kPDigitBytes / 16;
    // A tile in tensor memory: plane l of P with the digits 4 - l .. 4 of z -> weights 4 .. 4 + l
    auto six = [&](uint32_t a, uint64_t b, unsigned add) {
      mma_i8(tmem, a, b, mma_i8_desc(3 * kPColumns), add, leader);
      mma_i8(tmem + 3 * kPColumns, a, b + 3 * kDigit, mma_i8_desc(2 * kPColumns), add, leader);
      mma_i8(tmem, a + 8, b + kDigit, mma_i8_desc(4 * kPColumns), 1u, leader);
      mma_i8(tmem, a + 16, b + 2 * kDigit, mma_i8_desc(3 * kPColumns), 1u, leader);
      mma_i8(tmem, a + 24, b + 3 * kDigit, mma_i8_desc(2 * kPColumns), 1u, leader);
      mma_i8(tmem, a + 32, b + 4 * kDigit, mma_i8_desc(kPColumns), 1u, leader);
    };
    bool ok = true;
    int buf = 0, use = 0, slot = 0, round = 0;
    for (int k = 0, v = 0; k < chunks && ok; ++k) {
      ok = warp_wait(&dig_full[buf], use);
      for (int half = 0; half < H && ok; ++half, ++v) {
        if (v > 0) ok = warp_wait(&acc_empty[(v - 1) % kCopies], (v - 1) / kCopies);
        if (!ok) break;
        tmem_fence_after();
        unsigned add = 0;  // the first plane clears the accumulators
        uint64_t b = dig_base + buf * nb * (kPBlockBytes / 16);
        uint32_t a = tmem + kPPolyColumn;
        if (!kTwo) {
          for (int kb = 0; kb < nb; ++kb, b += kPBlockBytes / 16, a += kPDigits * 8) {
            six(a, b, add);
            add = 1;
          }
        } else {
          const int plane = tb.plane_bytes[half] / 16;
          uint32_t order = tb.use.order[half], place = tb.use.place[half];
          for (int t = 0; t < tb.use.count[half] && ok; ++t, order >>= 4, place >>= 4) {
            const uint64_t bt = b + (order & 15) * (kPBlockBytes / 16);
            if ((place & 15) != 15) {  // in tensor memory
              six(a + (place & 15) * (kPDigits * 8), bt, add);
              add = 1;
              continue;
            }
            uint64_t at = 0;
            int in_unit = 0;
#pragma unroll
            for (int l = 4; l >= 0; --l) {
              if (in_unit == 0) {
                ok = ok && warp_wait(&ring_full[slot], round);
                at = ring_base + slot * plan.unit * (kPPlaneBytes / 16);
              }
              if (!ok) break;
              if (l == 4) {
                mma_i8_shared(tmem, at, bt, mma_i8_desc(3 * kPColumns), add, leader);
                mma_i8_shared(tmem + 3 * kPColumns, at, bt + 3 * kDigit, mma_i8_desc(2 * kPColumns), add, leader);
              } else {
                mma_i8_shared(tmem, at, bt + (4 - l) * kDigit, mma_i8_desc((l + 1) * kPColumns), 1u, leader);
              }
              at += plane;
              if (++in_unit == plan.unit || l == 0) {
                mma_commit(&ring_empty[slot], leader);
                in_unit = 0;
                if (++slot == plan.ring) {
                  slot = 0;
                  ++round;
                }
              }
            }
            add = 1;
          }
        }
        if (ok) mma_commit(&acc_full[v % kCopies], leader);
      }
      if (ok) mma_commit(&dig_empty[buf], leader);
      if (++buf == plan.digs) {
        buf = 0;
        ++use;
      }
    }
    if (!ok) {  // nothing may be in flight when the tensor memory is given back
      if (leader) atomicExch(p.status, 1);
      mma_commit(drained, leader);
      warp_wait(drained, 0);
    }
  } else if (warp == kPLoadXYWarp) {
    if (lane == 0) {
      const unsigned bytes = (kMode == kModeDpsgd ? 1u : kMode == kModeExternal ? 4u : 2u) * nb * kPBlock * kPS * 4u;
      int k = 0, raw = 0, phase = 0;
      bool ok = true;
      for (; k < chunks; ++k) {
        if (p.stall_after >= 0 && static_cast<long long>(k) * H >= p.stall_after) break;  // self test: the loads stop
        if (phase > 0) ok = bar_wait(&raw_empty[raw], (phase - 1) & 1, limit);
        if (!ok) break;
        const int col = static_cast<int>(chunk_col(k));
        float* const dst = raw_mem + raw * plan.ins * nb * kPBlock * kPS;
        bar_expect_tx(&raw_full[raw], bytes);
        tile_load(dst, &maps.x, col, 0, &raw_full[raw]);
        if (kMode != kModeDpsgd) tile_load(dst + nb * kPBlock * kPS, &maps.y, col, 0, &raw_full[raw]);
        if (kMode == kModeExternal) {
          tile_load(dst + 2 * nb * kPBlock * kPS, &maps.a, col, 0, &raw_full[raw]);
          tile_load(dst + 3 * nb * kPBlock * kPS, &maps.g, col, 0, &raw_full[raw]);
        }
        if (++raw == plan.raws) {
          raw = 0;
          ++phase;
        }
      }
      if (!ok) atomicExch(p.status, 1);
      // nothing in flight when the CTA leaves (bounded)
      for (int back = 1; back <= plan.raws && back <= k; ++back) bar_wait(&raw_full[(k - back) % plan.raws], ((k - back) / plan.raws) & 1, limit);
    }
    __syncwarp();
  } else if (warp == kPTailWarp) {
    // ---------------------------------------------------------------- g, a, c in, g', x', y' out
    if (lane == 0) {
      const unsigned array = plan.rows * kPS;
      int asked = 0;
      auto load = [&](int v, int st) {
        if (p.stall_after >= 0 && v >= p.stall_after) return;
        asked = v + 1;
        if (kMode == kModeExternal) {  // nothing to load: the stage is free
          bar_arrive(&e_full[st]);
          return;
        }
        float* const dst = e_mem + st * 3 * array;
        const int col = static_cast<int>(chunk_col(v / H)), row = kPRows * (v % H);
        bar_expect_tx(&e_full[st], 3 * array * 4);
        tile_load(dst, &maps.g, col, row, &e_full[st]);
        tile_load(dst + array, &maps.a, col, row, &e_full[st]);
        tile_load(dst + 2 * array, &maps.c, col, row, &e_full[st]);
      };
      for (int v = 0; v < plan.stages && v < total; ++v) load(v, v);
      int st = 0, phase = 0;
      for (int v = 0; v < total; ++v) {
        if (!bar_wait(&out_ready[st], phase, limit)) {
          atomicExch(p.status, 1);
          break;
        }
        const float* const src = e_mem + st * plan.outs * array;  // now (g' |) x' | y'
        const long long col = chunk_col(v / H);
        const int row = kPRows * (v % H);
        if (col < (p.d & ~3LL)) {
          constexpr int kFirst = kMode == kModeExternal ? 0 : 1;
          if (kFirst != 0) tile_store(&maps.gs, static_cast<int>(col), row, src);
          tile_store(&maps.xs, static_cast<int>(col), row, src + kFirst * array);
          if (kMode != kModeDpsgd) tile_store(&maps.ys, static_cast<int>(col), row, src + (kFirst + 1) * array);
        }
        store_commit();
        store_wait_read();  // the stage may be refilled now
        if (v + plan.stages < total) load(v + plan.stages, st);
        if (++st == plan.stages) {
          st = 0;
          phase ^= 1;
        }
      }
      for (int back = 1; back <= plan.stages && back <= asked; ++back) bar_wait(&e_full[(asked - back) % plan.stages], ((asked - back) / plan.stages) & 1, limit);
      store_wait_all();
    }
    __syncwarp();
  } else if (kTwo) {
    // ---------------------------------------------------------------- planes of P from L2, plan.unit at a time
    if (lane == 0) {
      int slot = 0, round = 0, asked = 0;
      bool ok = true;
      for (int v = 0; v < total && ok; ++v) {
        const int half = v % H, plane = tb.plane_bytes[half];
        for (int t = 0; t < tb.use.count[half] && ok; ++t) {
          if ((tb.use.place[half] >> (4 * t) & 15) != 15) continue;
          const unsigned char* src = tb.tiles + half * tb.half_at + static_cast<size_t>(tb.use.order[half] >> (4 * t) & 15) * kPDigits * plane;
          for (int left = kPDigits; left > 0; left -= plan.unit, src += plan.unit * plane) {
            if (round > 0) ok = bar_wait(&ring_empty[slot], (round - 1) & 1, limit);
            if (!ok) break;
            const unsigned bytes = min(left, plan.unit) * plane;
            bar_expect_tx(&ring_full[slot], bytes);
            bytes_load(smem + plan.ring_at + slot * plan.unit * kPPlaneBytes, src, bytes, &ring_full[slot]);
            ++asked;
            if (++slot == plan.ring) {
              slot = 0;
              ++round;
            }
          }
        }
      }
      if (!ok) atomicExch(p.status, 1);
      for (int back = 1; back <= plan.ring && back <= asked; ++back) bar_wait(&ring_full[(asked - back) % plan.ring], ((asked - back) / plan.ring) & 1, limit);
    }
    __syncwarp();
  }
  }
  if (p.beside != 0) chain_wait();
  tmem_fence_before();
  __syncthreads();
  if (warp == kPMmaWarp) {
    tmem_fence_after();
    tmem_free(*tmem_slot, kPTmemColumns);
  }
}

typedef void (*RowsKernel)(const StepParams, const RowsMaps, const RowsTables, const RowsPlan);

template <int kRows, bool kAtStart>
RowsKernel pick_rows(const StepParams& p, bool wide) {
  if (p.mode == kModeDpsgd)
    return wide ? step_rows_kernel<kModeDpsgd, true, kRows, kAtStart> : step_rows_kernel<kModeDpsgd, false, kRows, kAtStart>;
  // up to 64 workers the DeTAG step never goes by the rounds' name (resolve_variant)
  return wide && kRows > 64 ? step_rows_kernel<kModeDetag, (kRows > 64), kRows, kAtStart> : step_rows_kernel<kModeDetag, false, kRows, kAtStart>;
}

template <int kRows>
RowsKernel pick_rows(const StepParams& p, bool wide) {
  if (p.mode == kModeExternal) return step_rows_kernel<kModeExternal, false, kRows, false>;
  return p.grad_at_start != 0 ? pick_rows<kRows, true>(p, wide) : pick_rows<kRows, false>(p, wide);
}

// [n rows][d columns] float32 with row pitch ld, tiles of box_rows x 32 columns in the 128-byte swizzle, zero fill outside.
bool make_swizzled_map(CUtensorMap* m, const float* base, int n, long long d, long long ld, int box_rows) {
  EncodeTiledFn fn = encode_tiled_fn();
  if (!fn) return false;
  const cuuint64_t dims[2] = {static_cast<cuuint64_t>(d), static_cast<cuuint64_t>(n)};
  const cuuint64_t strides[1] = {static_cast<cuuint64_t>(ld) * sizeof(float)};
  const cuuint32_t box[2] = {kPS, static_cast<cuuint32_t>(box_rows)};
  const cuuint32_t elem[2] = {1, 1};
  return fn(m, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 2, const_cast<float*>(base), dims, strides, box, elem, CU_TENSOR_MAP_INTERLEAVE_NONE,
            CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

}  // namespace

namespace {

// Which tiles the MMAs of a half take: those with a digit, the ones that stay in tensor memory (four, first those that both halves
// use, as in a block-circulant matrix) between those that travel, which thus have the time of two.
void place_tiles(int n, int nb, const unsigned (&used)[2], SplitPoly& made) {
  constexpr int kResidents = 4, kTravels = 15;
  auto tile = [&](int half, int b) {
    return &made.weights[static_cast<size_t>(half) * nb * kPDigits * kPPlaneBytes + static_cast<size_t>(b) * kPDigits * plane_bytes(n, half)];
  };
  int twin[8], place[2][8];
  for (int b = 0; b < nb; ++b) {
    twin[b] = -1;
    place[0][b] = place[1][b] = kTravels;
    for (int c = 0; c < nb && plane_bytes(n, 0) == plane_bytes(n, 1) && (used[0] >> b & 1); ++c)
      if (std::memcmp(tile(0, b), tile(1, c), kPDigits * kPPlaneBytes) == 0) twin[b] = c;
  }
  RowsTiles& t = made.use;
  auto keep = [&](int half, int b) {
    if (t.residents == kResidents || !(used[half] >> b & 1) || place[half][b] != kTravels) return;
    place[half][b] = t.residents;
    if (half == 0 && twin[b] >= 0) place[1][twin[b]] = t.residents;
    t.resident[t.residents++] = static_cast<unsigned char>(half << 4 | b);
  };
  for (int b = 0; b < nb; ++b)
    if (twin[b] >= 0) keep(0, b);
  for (int b = 0; b < nb; ++b)
    for (int half = 0; half < 2; ++half) keep(half, b);
  for (int half = 0; half < 2; ++half) {
    int left[2] = {0, 0}, next[2] = {0, 0};  // travelling, staying
    for (int b = 0; b < nb; ++b)
      if (used[half] >> b & 1) ++left[place[half][b] == kTravels ? 0 : 1];
    for (int turn = 0; left[0] + left[1] > 0; ++turn) {
      const int kind = left[0] == 0 ? 1 : left[1] == 0 ? 0 : turn & 1;
      int& b = next[kind];
      while (!(used[half] >> b & 1) || (place[half][b] == kTravels ? 0 : 1) != kind) ++b;
      t.order[half] |= static_cast<uint32_t>(b) << (4 * t.count[half]);
      t.place[half] |= static_cast<uint32_t>(place[half][b]) << (4 * t.count[half]++);
      ++b;
      --left[kind];
    }
  }
}

}  // namespace

// Digits of P, the rows' exponents, which of its parts are zero.  `poly`: the n x n matrix, or (circulant: the
// blocks depend on their distance only) its first 32 rows.  Leaves `out` empty when the kernel does not take the matrix:
// n outside 33 .. 256, an entry or a row that cannot be scaled.
void rows_polynomial(int n, const std::vector<double>& poly, bool circulant, const SplitPoly& other, SplitPoly& out) {
  out = SplitPoly{};
  if (n <= 32 || n > 256 || encode_tiled_fn() == nullptr) return;
  const int nb = (n + kPBlock - 1) / kPBlock, rows = circulant ? kPBlock : n, wide = nb * kPBlock, halves = n > kPRows ? 2 : 1;
  std::vector<int64_t> digits;
  SplitPoly made{};
  if (!split_digits(n, poly, rows, wide, digits, made.row_exp)) return;
  if (other.guard.empty()) {
    split_guard(n, poly, rows, made);
  } else {  // the other kernel's tables have been made
    made.guard = other.guard;
    made.guard_size = other.guard_size;
    made.guard_tau = other.guard_tau;
    made.unequal = other.unequal;
  }
  if (rows_plan(n, kModeDetag, static_cast<int>(made.guard.size())).bytes == 0) return;
  unsigned used[2] = {0, 0};
  made.weights.assign(static_cast<size_t>(halves) * nb * kPDigits * kPPlaneBytes, 0);
  for (int i = 0; i < n; ++i) {
    const int half = i / kPRows, r = i % kPRows, shift = circulant ? i / kPBlock : 0;  // block row c: block row 0, c blocks further
    const double* row = &poly[static_cast<size_t>(i % rows) * n];
    const int64_t* src = &digits[static_cast<size_t>(i % rows) * wide];
    for (int b = 0; b < nb; ++b) {
      const int from = (b - shift + nb) % nb * kPBlock;
      // planes of core matrices of 8 rows x 16 bytes, the two of a row group side by side
      const int plane = plane_bytes(n, half);
      unsigned char* at = &made.weights[static_cast<size_t>(half) * nb * kPDigits * kPPlaneBytes + static_cast<size_t>(b) * kPDigits * plane + (r / 8) * 256 + (r % 8) * 16];
      int64_t any = 0;
      for (int w = 0; w < kPBlock; ++w) {
        const int64_t v = src[from + w];
        any |= v;
        if (from + w < n && row[from + w] != 0.0) made.reach[i / kPBlock] |= static_cast<unsigned char>(1u << b);
        if (v != 0)
          for (int l = 0; l < kPDigits; ++l) at[(kPDigits - 1 - l) * plane + (w / 16) * 128 + w % 16] = static_cast<unsigned char>(v >> (8 * l));
      }
      if (any != 0) used[half] |= 1u << b;
    }
  }
  if (halves == 2) place_tiles(n, nb, used, made);
  const int padded = circulant ? kPBlock : wide;
  made.poly.assign(static_cast<size_t>(padded) * wide, 0.0);
  for (int i = 0; i < rows; ++i) std::copy(&poly[static_cast<size_t>(i) * n], &poly[static_cast<size_t>(i) * n] + n, &made.poly[static_cast<size_t>(i) * wide]);
  made.circulant = circulant;
  out = std::move(made);
}

// Four arrays are staged for caller-written gradients: up to 192 workers.
bool rows_take_external(const SplitPoly& poly) {
  return !poly.weights.empty() && rows_plan(static_cast<int>(poly.row_exp.size()), kModeExternal, static_cast<int>(poly.guard.size())).bytes != 0;
}

bool build_maps_rows(const StepParams& p, TensorMapSet* out) {
  RowsMaps& m = *reinterpret_cast<RowsMaps*>(out->bytes);
  const float* y = p.mode == kModeDpsgd ? p.x : p.y;  // D-PSGD has no tracker: those maps are never used
  const int all = (p.n + kPBlock - 1) / kPBlock * kPBlock, rows = stage_rows(p.n);
  const long long d_tma = p.d & ~3LL;  // the stores' tensor ends on a 16-byte boundary
  if (!make_map(&m.x, p.x, p.n, p.d, p.ld, all, kPS) || !make_map(&m.y, y, p.n, p.d, p.ld, all, kPS)) return false;
  if (p.mode == kModeExternal) {  // both gradients are staged like x and y, and the newest is stored from there
    if (!make_map(&m.g, p.g, p.n, p.d, p.ld, all, kPS) || !make_map(&m.a, p.g_ext, p.n, p.d, p.ld, all, kPS)) return false;
    if (d_tma > 0 && !make_map(&m.gs, p.g, p.n, d_tma, p.ld, all, kPS)) return false;
    m.c = m.a;  // never used
  } else {
    if (!make_swizzled_map(&m.g, p.g, p.n, p.d, p.ld, rows) || !make_swizzled_map(&m.a, p.a, p.n, p.d, p.ld, rows) ||
        !make_swizzled_map(&m.c, p.c, p.n, p.d, p.ld, rows))
      return false;
    if (d_tma > 0 && !make_swizzled_map(&m.gs, p.g, p.n, d_tma, p.ld, rows)) return false;
  }
  if (d_tma > 0 && (!make_swizzled_map(&m.xs, p.x, p.n, d_tma, p.ld, rows) || !make_swizzled_map(&m.ys, y, p.n, d_tma, p.ld, rows))) return false;
  if (d_tma == 0) m.xs = m.ys = m.gs = m.x;  // never used
  return true;
}

int launch_step_rows(StepParams p, const TensorMapSet& maps, const SplitPoly& poly, const SplitDevice& dev, bool wide,
                      int sm_count, cudaStream_t stream) {
  if (poly.weights.empty()) return static_cast<int>(cudaErrorInvalidValue);
  RowsTables tb{};
  tb.tiles = static_cast<const unsigned char*>(dev.weights);
  tb.row_exp = dev.row_exp;
  tb.poly = dev.poly;
  tb.guard = dev.guard;
  tb.guard_size = poly.guard_size;
  tb.guard_groups = static_cast<int>(poly.guard.size()) / poly.guard_size;
  tb.guard_tau = poly.guard_tau;
  tb.circulant = poly.circulant ? 1 : 0;
  tb.nb = (p.n + kPBlock - 1) / kPBlock;
  tb.half_at = tb.nb * kPDigits * kPPlaneBytes;
  for (int half = 0; half < 2; ++half) tb.plane_bytes[half] = plane_bytes(p.n, half);
  tb.use = poly.use;
  std::memcpy(tb.reach, poly.reach, sizeof tb.reach);
  RowsPlan plan = rows_plan(p.n, p.mode, static_cast<int>(poly.guard.size()));
  if (plan.bytes == 0) return static_cast<int>(cudaErrorInvalidValue);
  const long long chunks = (p.d + kPS - 1) / kPS;
  plan.chunk_shift = chunks > 16LL * sm_count ? 1 : 0;
  p.S = kPS << plan.chunk_shift;
  p.num_slabs = (p.d + p.S - 1) / p.S;
  const RowsKernel kernel = p.n > kPRows ? pick_rows<256>(p, wide) : p.n > 96 ? pick_rows<128>(p, wide) : p.n > 64 ? pick_rows<96>(p, wide) : pick_rows<64>(p, wide);
  const int e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), plan.bytes);
  if (e != 0) return e;
  const long long grid = p.num_slabs < sm_count ? p.num_slabs : sm_count;
  if (grid <= 0) return 0;
  return launch_chained(kernel, static_cast<unsigned>(grid), kPThreads, plan.bytes, stream, p, *reinterpret_cast<const RowsMaps*>(maps.bytes), tb, plan);
}

}  // namespace detag
