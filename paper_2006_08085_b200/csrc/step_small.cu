// DeTAG step for at most 16 workers, held in registers from the loads to the stores.
//
// AG_K(z) = P z with P = P_K(M) from the host, on the float64 tensor path (mma m8n8k4) with the operands' roles chosen so that
// nothing has to move between lanes: eight coordinates are the M index, the input workers the contraction index and the
// output workers the N index, permuted so that column 2 q + e of the output block b stands for worker q + 4 (2 b + e).  A
// lane (c = lane / 4, q = lane % 4) then supplies workers q, q + 4, ... of coordinate c and receives the same workers of the
// same coordinate: it loads its elements from global memory, takes them through all of the step and writes them back.  No
// shared memory, no barriers; the next step of several in one launch finds its operands in place.
//
// A warp takes 8 V coordinates; lane c owns the V neighbouring ones from V c on, so that a row is read as V-word vectors, and
// its tile t consists of the t-th of every lane.  The four workers of a Philox call are the four lanes of a coordinate at the
// same place: each lane draws whole calls, as many as there are for four lanes, and a 4 x 4 transpose hands them out.
//
// Bound: HBM for single steps (n = 8, d = 8 M 327 us, 0.96 of the copy rate; n = 16, d = 4 M 378 us, 0.83), at d = 270 k the launch
// and the loads' latency (n = 16 29 us for 21 of HBM time); for many steps the special-function pipe, five conversions per
// worker-coordinate and step beside the normals (n = 8, d = 62 k, twenty steps: 28 us).  One thread per coordinate, its column in
// shared memory and the sums on the scalar float64 pipe, took 133 instructions per worker-coordinate at n = 16 and 399, 499, 41
// and 45 us; caller-written gradients of 16 workers, d = 270 k, went from 35 us on the staged kernel to 25.
//
// Measured on the way: loads behind a branch (rows beyond n) 599 us at n = 13, d = 4 M, clamped and selected 350; V = 2 for
// single steps 514 us at n = 8, d = 8 M (64-byte row pieces), within 2 % at n = 16, d = 270 k; 128 registers instead of 168 at
// n = 16 421 us for d = 4 M; blocks of 64 threads the same.
#include <cuda_runtime.h>

#include "chain.cuh"
#include "detag_internal.h"
#include "noise.cuh"
#include "pipeline.cuh"

namespace detag {

namespace {

constexpr int kSmallThreads = 128;

template <int V>
struct Vec;
template <>
struct Vec<2> {
  typedef float2 Type;
};
template <>
struct Vec<4> {
  typedef float4 Type;
};

// Blocks per SM the registers are planned for: what the five arrays' vectors and the sums need, but for 4 to 40 bytes that the
// printed timing of 12 to 16 workers and the default step of 13 to 15 spill.  More blocks
// at fewer registers lose (n = 16: above), fewer do not gain; many steps at n = 16 in 6 blocks 76 us for 68.
constexpr int small_blocks(int R, int V, bool many) { return many ? 4 : R * V <= 8 ? 5 : R * V <= 12 ? 4 : 3; }

// R: workers per lane, n rounded up to 4 R; kFull: n == 4 R.  V: coordinates per lane.  kMany: p.steps iterations (DeTAG with
// the synthetic gradient only).
template <int R, bool kFull, int V, int kMode, bool kAtStart, bool kMany>
__global__ void __launch_bounds__(kSmallThreads, small_blocks(R, V, kMany)) step_small_kernel(const StepParams p) {
  typedef typename Vec<V>::Type VecT;
  constexpr int kBlocks = (R + 1) / 2;        // output blocks of eight workers
  constexpr int kDraws = (R * V + 3) / 4;     // Philox calls of a lane
  const int lane = threadIdx.x & 31, q = lane & 3, c = lane >> 2;
  const long long warp = (blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x) >> 5;
  const long long first = warp * (8 * V);     // the warp's first coordinate
  if (first >= p.d) return;                   // whole warps
  const long long j = first + V * c;          // this lane's first coordinate; rows are padded to a multiple of four
  const bool inside = j < p.d;
  const int n = kFull ? 4 * R : p.n;
  const double alpha = p.alpha;
  const float sigma = static_cast<float>(p.sigma);
  const bool noisy = kMode != kModeExternal && p.sigma != 0.0;
  const float* const pa = kMode == kModeExternal ? p.g_ext : p.a;

  // ---- everything is asked for before anything is used.  Workers beyond n count as zero; they read a row that is there, so
  // that no branch keeps the loads apart.  Coordinates beyond d take what the rows' padding or the warp's first column holds:
  // they keep to themselves and are not stored.
  const long long at = inside ? j : first;
  auto load = [&](const float* base, float (&v)[R][V]) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      const int row = q + 4 * i;
      const VecT w = *reinterpret_cast<const VecT*>(base + (kFull || row < n ? row : n - 1) * p.ld + at);
      const float* const e = reinterpret_cast<const float*>(&w);
#pragma unroll
      for (int t = 0; t < V; ++t) v[i][t] = kFull || row < n ? e[t] : 0.f;
    }
  };
  chain_wait();
  chain_next();
  float x[R][V], y[R][V], g[R][V], a[R][V], cc[R][V];
  load(p.x, x);
  if (kMode != kModeDpsgd) load(p.y, y);
  load(p.g, g);
  load(pa, a);
  if (kMode != kModeExternal) load(p.c, cc);
  double frag[R][kBlocks];  // [input step][output block]: P[worker of column c][worker q of the step]
#pragma unroll
  for (int k = 0; k < R; ++k)
#pragma unroll
    for (int b = 0; b < kBlocks; ++b) {
      const int out = (c >> 1) + 4 * (2 * b + (c & 1)), in = 4 * k + q;
      frag[k][b] = out < n && in < n ? p.poly[out * n + in] : 0.0;
    }

  double gd[R][V];  // the old gradient widened; the next of several steps starts from what this one folded
#pragma unroll
  for (int i = 0; i < R; ++i)
#pragma unroll
    for (int t = 0; t < V; ++t) gd[i][t] = static_cast<double>(g[i][t]);

  auto step = [&](uint32_t t_noise) {
    float xi[R][V];
#pragma unroll
    for (int i = 0; i < R; ++i)
#pragma unroll
      for (int t = 0; t < V; ++t) xi[i][t] = 0.f;
    if (noisy) {
#pragma unroll
      for (int h = 0; h < kDraws; ++h) {
        // call 4 h + lane's place: coordinate (its number) % V, quad (its number) / V
        const int mine_t = V == 4 ? q : q % V, mine_i = V == 4 ? h : (4 / V) * h + q / V;
        float v[4];
        normal_quad(p.round_key, static_cast<unsigned long long>(p.coord_offset + j + mine_t), static_cast<uint32_t>(mine_i), t_noise, sigma, v);
        transpose_quad(v, q);
#pragma unroll
        for (int s = 0; s < 4; ++s) {
          const int number = 4 * h + s;
          if (number / V < R) xi[number / V][number % V] = v[s];
        }
      }
    }
#pragma unroll
    for (int t = 0; t < V; ++t) {
      // cx ends as x' = P (x - alpha y), by linearity; cy starts at -g and ends as y~ - g, so that the fold is cy + g'.
      // Caller-written gradients: the operand is the tracker folded with them, cy starts at zero.  D-PSGD: cx starts at
      // -alpha g and sums P x.
      double cx[kBlocks][2], cy[kBlocks][2];
#pragma unroll
      for (int i = 0; i < 2 * kBlocks; ++i) {
        const double old = i < R && kMode != kModeExternal ? -gd[i < R ? i : 0][t] : 0.0;
        cx[i >> 1][i & 1] = kMode == kModeDpsgd ? alpha * old : 0.0;
        cy[i >> 1][i & 1] = kMode == kModeDetag ? old : 0.0;
      }
#pragma unroll
      for (int k = 0; k < R; ++k) {
        double u = static_cast<double>(x[k][t]), yd = 0.0;
        if (kMode != kModeDpsgd) {
          yd = static_cast<double>(y[k][t]);
          if (kMode == kModeExternal) yd += static_cast<double>(a[k][t]) - gd[k][t];  // Algorithm 2's tracker update
          u = fma(-alpha, yd, u);
        }
#pragma unroll
        for (int b = 0; b < kBlocks; ++b) {
          if (kMode != kModeDpsgd) dmma(cy[b], yd, frag[k][b]);
          dmma(cx[b], u, frag[k][b]);
        }
      }
#pragma unroll
      for (int i = 0; i < R; ++i) {
        const double sy = cy[i >> 1][i & 1];
        const float xn = static_cast<float>(cx[i >> 1][i & 1]);  // x' (float64 sum, rounded once)
        if (!kMany && kMode != kModeDpsgd && p.y_obs != nullptr && (kFull || q + 4 * i < n) && j + t < p.d)  // optional observer: the gossiped tracker
          p.y_obs[(q + 4 * i) * p.ld + j + t] = static_cast<float>(kMode == kModeDetag ? sy + gd[i][t] : sy);
        if (kMode == kModeExternal) {
          g[i][t] = a[i][t];                    // the gradient just folded becomes g_old
          y[i][t] = static_cast<float>(sy);     // the gossiped tracker
        } else {
          const float gn = fmaf(a[i][t], (kAtStart ? x[i][t] : xn) - cc[i][t], xi[i][t]);  // stochastic gradient
          gd[i][t] = static_cast<double>(gn);
          if (kMode == kModeDetag) y[i][t] = static_cast<float>(sy + gd[i][t]);  // fold: (y~ - g) + g', g' as stored
          g[i][t] = gn;
        }
        x[i][t] = xn;
      }
    }
  };
  if (kMany) {
#pragma unroll 1
    for (int s = 0; s < p.steps; ++s) step(p.t_noise + static_cast<uint32_t>(s));
  } else {
    step(p.t_noise);
  }

  if (!inside) return;
  auto store = [&](float* base, const float (&v)[R][V]) {
#pragma unroll
    for (int i = 0; i < R; ++i) {
      if (!kFull && q + 4 * i >= n) continue;
      float* const to = base + (q + 4 * i) * p.ld + j;
      if (j + V <= p.d) {
        VecT w;
        float* const e = reinterpret_cast<float*>(&w);
#pragma unroll
        for (int t = 0; t < V; ++t) e[t] = v[i][t];
        *reinterpret_cast<VecT*>(to) = w;
      } else {  // nothing beyond column d is written
#pragma unroll
        for (int t = 0; t < V; ++t)
          if (j + t < p.d) to[t] = v[i][t];
      }
    }
  };
  store(p.x, x);
  if (kMode != kModeDpsgd) store(p.y, y);
  store(p.g, g);
}

typedef void (*SmallKernel)(const StepParams);

template <int R, bool kFull>
SmallKernel pick_small(const StepParams& p) {
  if (p.mode == kModeExternal) return step_small_kernel<R, kFull, 4, kModeExternal, false, false>;
  if (p.mode == kModeDpsgd) return p.grad_at_start ? step_small_kernel<R, kFull, 4, kModeDpsgd, true, false> : step_small_kernel<R, kFull, 4, kModeDpsgd, false, false>;
  return p.grad_at_start ? step_small_kernel<R, kFull, 4, kModeDetag, true, false> : step_small_kernel<R, kFull, 4, kModeDetag, false, false>;
}

template <int R, bool kFull>
SmallKernel pick_many(const StepParams& p, bool wide) {
  if (R == 1 && wide) return p.grad_at_start ? step_small_kernel<1, kFull, 4, kModeDetag, true, true> : step_small_kernel<1, kFull, 4, kModeDetag, false, true>;
  return p.grad_at_start ? step_small_kernel<R, kFull, 2, kModeDetag, true, true> : step_small_kernel<R, kFull, 2, kModeDetag, false, true>;
}

template <int R>
int launch_small(const StepParams& p, int sm_count, cudaStream_t stream) {
  const bool many = p.steps > 1, full = p.n == 4 * R;
  // Many steps: half as many coordinates to a warp, twice the warps to hide the chain of a step behind.  But with up to 4 workers a
  // lane throws half of its Philox call away then: once every scheduler has a warp, four coordinates per lane (3 workers, twenty
  // steps, two -> four: d = 4096 9.2 -> 10.2 us, 14 k 10.2 both, 32 k 14.3 -> 12.3, 150 k 40 -> 30, 1 M 233 -> 166).
  const bool wide = !many || (R == 1 && p.d > 64LL * sm_count);
  const SmallKernel kernel = many ? (full ? pick_many<R, true>(p, wide) : pick_many<R, false>(p, wide))
                                  : (full ? pick_small<R, true>(p) : pick_small<R, false>(p));
  // Short vectors: smaller blocks, so that every SM gets a share.
  const int width = wide ? 32 : 16;
  const long long warps = (p.d + width - 1) / width;
  const int per_block = warps >= 4LL * sm_count ? 4 : warps >= 2LL * sm_count ? 2 : 1;
  const unsigned grid = static_cast<unsigned>((warps + per_block - 1) / per_block);
  if (!many) return launch_chained(kernel, grid, 32 * per_block, 0, stream, p);
  // All blocks of many steps are on the SMs at once, and blocks of the next launch that wait in the places left over would
  // spread them unevenly (8 workers, d = 62 k, twenty steps: 27.5 us for 26.6).
  kernel<<<grid, 32 * per_block, 0, stream>>>(p);
  return static_cast<int>(cudaGetLastError());
}

}  // namespace

// p.steps > 1: that many iterations.
int launch_step_small(const StepParams& p, int sm_count, cudaStream_t stream) {
  if (p.n > kMaxSmallWorkers || p.d <= 0 || (p.steps > 1 && p.mode != kModeDetag)) return static_cast<int>(cudaErrorInvalidValue);
  if (p.n <= 4) return launch_small<1>(p, sm_count, stream);
  if (p.n <= 8) return launch_small<2>(p, sm_count, stream);
  if (p.n <= 12) return launch_small<3>(p, sm_count, stream);
  return launch_small<4>(p, sm_count, stream);
}

}  // namespace detag
