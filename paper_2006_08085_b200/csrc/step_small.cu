// DeTAG step for at most 16 workers: a thread takes the whole column of workers of a coordinate.
//
// AG_K(z) = P z with P = P_K(M) from the host.  A column of n <= 16 workers is 2 n^2 float64 multiply-adds for the two
// contractions, at most 32 per worker-coordinate: half a clock per worker-coordinate and SM on the scalar float64 pipe
// against 1.3 clocks of HBM traffic, so the tensor path has nothing to win here - it works on 32 padded rows, which for
// eight workers is three quarters of its noise, gradient and shared-memory work for nothing.  P sits in shared memory, four
// output workers of one input worker side by side (two 16-byte broadcasts for eight multiply-adds).  Rows are read and written as neighbouring
// lanes' neighbouring words; nothing is staged, no thread waits for another, and the remainder of d needs no path of its
// own.  Several steps per launch keep the column in registers from one to the next.
//
// Bound: HBM up to 12 workers (8 workers, d = 8 M: 362 us, 0.86 of the copy rate; the tensor-path kernel took 1005 us), at
// 16 the issue slots, 133 instructions per worker-coordinate (d = 4 M: 474 us, before 568; address arithmetic with one
// byte offset per row for all arrays instead of one per access took it from 178 instructions and 537 us; two coordinates
// per thread cost 962 us for want of warps).  Twenty steps in one launch, 8 workers, d = 62 k: 45 us, before 127.
#include <cuda_runtime.h>

#include "detag_internal.h"
#include "noise.cuh"

namespace detag {

namespace {

constexpr int kSmallThreads = 128;

// Blocks per SM the registers are planned for.
constexpr int small_blocks(int N, bool many) { return many ? (N <= 8 ? 3 : 2) : 6; }

// N: n rounded up to a multiple of four, kFull: n == N.  kMany: p.steps iterations (DeTAG with the synthetic gradient only).
template <int N, bool kFull, int kMode, bool kAtStart, bool kMany>
__global__ void __launch_bounds__(kSmallThreads, small_blocks(N, kMany)) step_small_kernel(const StepParams p) {
  __shared__ __align__(16) double poly[N / 4][N][4];  // [output quad][input worker][output], zero beyond n
  // The column's operands of the contractions, u = x - alpha y (D-PSGD: x) and the tracker, widened once; every thread its
  // own entries.  In registers they would leave room for half the warps.
  __shared__ double operands[(kMode == kModeDpsgd ? 1 : 2) * N * kSmallThreads];
  double* const op_u = operands + threadIdx.x;
  double* const op_y = op_u + N * kSmallThreads;
  for (int e = threadIdx.x; e < N * N; e += blockDim.x) {
    const int i = e / N, k = e % N;
    poly[i >> 2][k][i & 3] = i < p.n && k < p.n ? p.poly[i * p.n + k] : 0.0;
  }
  __syncthreads();
  const long long j = blockIdx.x * static_cast<long long>(blockDim.x) + threadIdx.x;
  if (j >= p.d) return;
  const int n = kFull ? N : p.n;
  const double alpha = p.alpha;
  const float sigma = static_cast<float>(p.sigma);
  const bool noisy = p.sigma != 0.0;
  const unsigned long long jn = static_cast<unsigned long long>(p.coord_offset + j);
  // One byte offset per row serves all arrays.
  const long long pitch = p.ld * 4, start = j * 4;
  auto at = [](const float* base, long long off) { return reinterpret_cast<const float*>(reinterpret_cast<const char*>(base) + off); };
  // Rows beyond n read row n - 1 and count as zero: no branch around a read.
  auto rows4 = [&](const float* base, int q, const long long (&off)[4], float (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float t = *at(base, off[i]);
      v[i] = kFull || q + i < n ? t : 0.f;
    }
  };
  auto offsets = [&](int q, long long (&off)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i) off[i] = start + (kFull || q + i < n ? q + i : n - 1) * pitch;
  };
  const float* const pa = kMode == kModeExternal ? p.g_ext : p.a;

  float xs[kMany ? N / 4 : 1][4], ys[kMany ? N / 4 : 1][4], gs[kMany ? N / 4 : 1][4], as[kMany ? N / 4 : 1][4],
      cs[kMany ? N / 4 : 1][4];
  // all rows are asked for before the first is used
  constexpr int kQuads = N / 4;
#pragma unroll
  for (int f = 0; f < N / 4; f += kQuads) {
    float xv[kQuads][4], yv[kQuads][4], gv[kQuads][4], gn[kQuads][4];
#pragma unroll
    for (int q = 0; q < kQuads; ++q) {
      long long off[4];
      offsets(4 * (f + q), off);
      rows4(p.x, 4 * (f + q), off, xv[q]);
      if (kMode != kModeDpsgd) rows4(p.y, 4 * (f + q), off, yv[q]);
      if (kMode == kModeExternal) {
        rows4(pa, 4 * (f + q), off, gn[q]);
        rows4(p.g, 4 * (f + q), off, gv[q]);
      }
    }
#pragma unroll
    for (int q = 0; q < kQuads; ++q)
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const int k = 4 * (f + q) + i;
        double y = kMode == kModeDpsgd ? 0.0 : static_cast<double>(yv[q][i]);
        // Algorithm 2's tracker update with the caller's newest gradient
        if (kMode == kModeExternal) y += static_cast<double>(gn[q][i]) - static_cast<double>(gv[q][i]);
        op_u[k * kSmallThreads] = kMode == kModeDpsgd ? static_cast<double>(xv[q][i]) : fma(-alpha, y, static_cast<double>(xv[q][i]));
        if (kMode != kModeDpsgd) op_y[k * kSmallThreads] = y;
        if (kMany) xs[f + q][i] = xv[q][i];
      }
  }

  // Four output workers: contractions, noise, gradient, fold.  x_at: the model the step started from (kAtStart).
  auto quad = [&](int q, uint32_t t, const float (&gv)[4], const float (&av)[4], const float (&cv)[4], const float (&x_at)[4],
                  float (&xo)[4], float (&yo)[4], float (&go)[4], double (&cy)[4]) {
    double cx[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      cx[i] = kMode == kModeDpsgd ? -alpha * static_cast<double>(gv[i]) : 0.0;
      cy[i] = kMode == kModeDetag ? static_cast<double>(-gv[i]) : 0.0;  // ends as y~ - g
    }
#pragma unroll
    for (int k = 0; k < N; ++k) {
      // a few shared-memory reads in flight at a time: all of a quad's, moved to its front, would not fit in registers
      if (k % 4 == 0) asm volatile("" ::: "memory");
      const double2 p01 = *reinterpret_cast<const double2*>(&poly[q >> 2][k][0]);
      const double2 p23 = *reinterpret_cast<const double2*>(&poly[q >> 2][k][2]);
      const double pk[4] = {p01.x, p01.y, p23.x, p23.y};
      const double u = op_u[k * kSmallThreads], y = kMode == kModeDpsgd ? 0.0 : op_y[k * kSmallThreads];
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        cx[i] = fma(pk[i], u, cx[i]);
        if (kMode != kModeDpsgd) cy[i] = fma(pk[i], y, cy[i]);
      }
    }
    float xi[4] = {0.f, 0.f, 0.f, 0.f};
    if (kMode != kModeExternal && noisy) normal_quad(p.round_key, jn, static_cast<uint32_t>(q >> 2), t, xi);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      xo[i] = static_cast<float>(cx[i]);  // x' (float64 sum, rounded once)
      if (kMode == kModeExternal) {
        go[i] = av[i];                      // the gradient just folded becomes g_old
        yo[i] = static_cast<float>(cy[i]);  // the gossiped tracker
      } else {
        go[i] = fmaf(av[i], (kAtStart ? x_at[i] : xo[i]) - cv[i], sigma * xi[i]);  // stochastic gradient
        yo[i] = static_cast<float>(cy[i] + static_cast<double>(go[i]));            // fold: (y~ - g) + g', g' as stored
      }
    }
  };
  auto store4 = [&](float* base, int q, const long long (&off)[4], const float (&v)[4]) {
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (kFull || q + i < n) *const_cast<float*>(at(base, off[i])) = v[i];
  };

  if (kMany) {
#pragma unroll
    for (int q = 0; q < N / 4; ++q) {
      long long off[4];
      offsets(4 * q, off);
      rows4(p.g, 4 * q, off, gs[q]);
      rows4(pa, 4 * q, off, as[q]);
      rows4(p.c, 4 * q, off, cs[q]);
    }
#pragma unroll 1
    for (int step = 0; step < p.steps; ++step) {
#pragma unroll
      for (int q = 0; q < N / 4; ++q) {
        double cy[4];
        float g4[4], x4[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          g4[i] = gs[q][i];
          x4[i] = xs[q][i];
        }
        quad(4 * q, p.t_noise + static_cast<uint32_t>(step), g4, as[q], cs[q], x4, xs[q], ys[q], gs[q], cy);
      }
      if (step + 1 < p.steps) {
#pragma unroll
        for (int q = 0; q < N / 4; ++q)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const double y = static_cast<double>(ys[q][i]);
            op_u[(4 * q + i) * kSmallThreads] = fma(-alpha, y, static_cast<double>(xs[q][i]));
            op_y[(4 * q + i) * kSmallThreads] = y;
          }
      }
    }
#pragma unroll
    for (int q = 0; q < N / 4; ++q) {
      long long off[4];
      offsets(4 * q, off);
      store4(p.x, 4 * q, off, xs[q]);
      store4(p.y, 4 * q, off, ys[q]);
      store4(p.g, 4 * q, off, gs[q]);
    }
    return;
  }
  float gn[4], an[4], cn[4], xn[4];  // the next quad's rows are on their way while one is worked on
  long long next[4];
  auto fetch = [&](int q) {
    if (kMode != kModeExternal) {
      rows4(p.g, q, next, gn);
      rows4(p.c, q, next, cn);
    }
    rows4(pa, q, next, an);
    if (kAtStart) rows4(p.x, q, next, xn);  // still the old model: this thread overwrites it below
  };
  offsets(0, next);
  fetch(0);
#pragma unroll 1
  for (int q = 0; q < N; q += 4) {
    float gv[4], av[4], cv[4], xv[4], xo[4], yo[4], go[4];
    double cy[4];
    long long off[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      gv[i] = gn[i];
      av[i] = an[i];
      cv[i] = cn[i];
      xv[i] = xn[i];
      off[i] = next[i];
      if (kFull) next[i] += 4 * pitch;
    }
    if (!kFull) offsets(q + 4, next);
    if (q + 4 < N) fetch(q + 4);
    quad(q, p.t_noise, gv, av, cv, xv, xo, yo, go, cy);
    store4(p.x, q, off, xo);
    if (kMode != kModeDpsgd) store4(p.y, q, off, yo);
    store4(p.g, q, off, go);
    if (kMode != kModeDpsgd && p.y_obs != nullptr) {  // optional observer: the gossiped tracker
      float yg[4];
#pragma unroll
      for (int i = 0; i < 4; ++i)
        yg[i] = kMode == kModeDetag ? static_cast<float>(cy[i] + static_cast<double>(gv[i])) : yo[i];
      store4(p.y_obs, q, off, yg);
    }
  }
}

typedef void (*SmallKernel)(const StepParams);

template <int N, bool kFull>
SmallKernel pick_small(const StepParams& p) {
  if (p.steps > 1)
    return p.grad_at_start ? step_small_kernel<N, kFull, kModeDetag, true, true> : step_small_kernel<N, kFull, kModeDetag, false, true>;
  if (p.mode == kModeExternal) return step_small_kernel<(N <= 8 ? N : 8), kFull, kModeExternal, false, false>;  // n <= 8
  if (p.mode == kModeDpsgd) return step_small_kernel<N, kFull, kModeDpsgd, false, false>;
  return p.grad_at_start ? step_small_kernel<N, kFull, kModeDetag, true, false> : step_small_kernel<N, kFull, kModeDetag, false, false>;
}

template <int N>
int launch_small(const StepParams& p, int sm_count, cudaStream_t stream) {
  const SmallKernel kernel = p.n == N ? pick_small<N, true>(p) : pick_small<N, false>(p);
  // short vectors: smaller blocks, so that every SM gets a share
  const int threads = p.d >= kSmallThreads * static_cast<long long>(sm_count) ? kSmallThreads : p.d >= 64LL * sm_count ? 64 : 32;
  const long long grid = (p.d + threads - 1) / threads;
  kernel<<<static_cast<unsigned>(grid), threads, 0, stream>>>(p);
  return static_cast<int>(cudaGetLastError());
}

}  // namespace

// p.steps > 1: that many iterations.
int launch_step_small(const StepParams& p, int sm_count, cudaStream_t stream) {
  if (p.n > kMaxSmallWorkers || p.d <= 0 || (p.mode == kModeExternal && p.n > 8) || (p.steps > 1 && p.mode != kModeDetag)) return static_cast<int>(cudaErrorInvalidValue);
  if (p.n <= 4) return launch_small<4>(p, sm_count, stream);
  if (p.n <= 8) return launch_small<8>(p, sm_count, stream);
  if (p.n <= 12) return launch_small<12>(p, sm_count, stream);
  return launch_small<16>(p, sm_count, stream);
}

}  // namespace detag
