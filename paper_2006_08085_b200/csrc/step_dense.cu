// DeTAG step with the dense polynomial for 17 to 48 workers on the float64 tensor path, the lanes' roles as in step_small.cu.
//
// AG_K(z) = P z with P = P_K(M) from the host, as float64 MMAs (m8n8k4): eight coordinates are the M index, the input workers
// the contraction index, the output workers the N index, permuted so that column 2 q + e of the output block b stands for
// worker q + 4 (2 b + e).  A lane (c = lane / 4, q = lane % 4) supplies workers q, q + 4, ... of its coordinates and receives
// the same ones: operands, sums and the element-wise tail of a coordinate never leave the lane.
//
// Four warps (a group) take a slab of 64 coordinates, sixteen each, a lane two neighbours (both share a fragment of P, which
// comes from shared memory); beyond 32 workers eight warps with a coordinate per lane, for the sums of two would leave room for
// half the warps.  Slabs of 64 because rows have to travel in pieces of 256 bytes: warps on their own with 64-byte
// pieces reached 0.38 of the copy rate, by TMA and by cp.async alike.  A group has one buffer for the operands of the products
// (x, y; up to 32 workers g) and one for the rest, over which the results are written.  There is no loading and no storing
// thread: the warp that is the last of its group to be done with the operands asks for the next slab's, which travel while the
// tail is worked on; the last to have written its results sends them out and asks for the next slab's inputs of the tail
// when the store has been read, at the start of its next products.  Every wait is bounded.
//
// A tile is one three-dimensional box {32 coordinates, 2 halves, rows} in the 128-byte swizzle: whole 256-byte row pieces, and
// every access of a half warp falls into different banks.  The last d % 64 coordinates are read and written by their lanes.
//
// Bound: HBM and the power cap up to 32 workers (d = 25.6 M, six rounds 4.8 ms in short runs, 0.83 of the copy rate; the kernel
// with padded tiles, a loading and a storing thread 5.17; D-PSGD, d = 3 M 417 us, 0.84), beyond them the FP64 pipe: 12 MMAs of
// 16.3 cycles and three scalar operations per 32 worker-coordinates and scheduler at 48 workers, 200 cycles for 176 of HBM, of which
// six warps per scheduler keep 0.7 busy (d = 1 M 372 us; the integer tensor path 428).  Up to 24 workers padding was what it
// saves: 24, d = 3 M 569 -> 400 us, 17 582 -> 340.
//
// Measured on the way (us): the normals drawn in the tail instead of before the wait for its inputs, 32 workers d = 25.6 M 4900
// for 4805; products in a loop unrolled twice 5190 at 32 workers, at 48 390 where the straight line of MMAs takes 410; loads of a
// ragged slab one after the other 17 instead of 12 at d = 9000.  Two coordinates per lane and three groups of four warps beyond 32
// workers: 48 382 for 372, printed timing 411 for 395, 33 276 for 258, 33 with d = 100 k 37.2 for 33.9, but caller-written gradients of
// 48 391 for 397; two groups of eight 380.  One coordinate per lane up to 32: 24 456 for 408, 32 with d = 30 k 14.5 for 12.4.
#include <cuda.h>
#include <cuda_runtime.h>

#include "chain.cuh"
#include "detag_internal.h"
#include "noise.cuh"
#include "packed.cuh"
#include "pipeline.cuh"
#include "tma.cuh"

namespace detag {

namespace {

constexpr int kDS = 64;  // coordinates per slab
// Coordinates per lane, warps per group, threads per CTA.
__host__ __device__ constexpr int dense_coords(int R) { return R <= 8 ? 2 : 1; }
__host__ __device__ constexpr int dense_warps(int R) { return 8 / dense_coords(R); }
__host__ __device__ constexpr int dense_groups(int R) { return R <= 8 ? 4 : 3; }
__host__ __device__ constexpr int dense_threads(int R) { return dense_groups(R) * dense_warps(R) * 32; }
__host__ __device__ constexpr int dense_blocks(int R) { return (R + 1) / 2; }
__host__ __device__ constexpr int dense_frag_bytes(int R) { return R * dense_blocks(R) * 32 * 8; }
__host__ __device__ constexpr int dense_group_bytes(int R) { return (R <= 8 ? 6 : 5) * R * 1024; }
// barriers and counters, and slack to align the tiles to 1 KiB, at the end
__host__ __device__ constexpr int dense_smem_bytes(int R) { return dense_groups(R) * dense_group_bytes(R) + dense_frag_bytes(R) + 128 + 1024; }
static_assert(4 * (2 * 8 + 4 * 4) <= 128, "barrier area");
static_assert(dense_smem_bytes(12) <= 232448 && dense_smem_bytes(8) <= 232448, "shared memory plan");

struct DenseMaps {
  CUtensorMap x, y, g, a, c;  // boxes {32, 2, 4 R rows}: loads and (x, y, g) stores
};
static_assert(sizeof(DenseMaps) <= sizeof(TensorMapSet), "tensor map storage");

// One more arrival at a counter of the CTA; true for every `of`-th.  Orders what the warp did before (after __syncwarp) before
// what the last one does next.
__device__ __forceinline__ bool last_of(unsigned* counter, unsigned of) {
  unsigned before;
  asm volatile("atom.acq_rel.cta.shared::cta.add.u32 %0, [%1], 1;" : "=r"(before) : "r"(s_addr(counter)) : "memory");
  return before % of == of - 1;
}

// The first `bytes` of kBytes (4 or 8) bytes, then zeros; asynchronous.
template <int kBytes>
__device__ __forceinline__ void copy_bytes(float* to, const float* from, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], %2, %3;" ::"r"(s_addr(to)), "l"(from), "n"(kBytes), "r"(bytes) : "memory");
}

// R: workers per lane, n rounded up to 4 R.  kWide: the gradient in float64 instead of float32 at the rounded model.
// kMany: p.steps iterations (DeTAG with the synthetic gradient, up to 32 workers): every lane's results take the places of its
// own operands.
template <int R, int kMode, bool kAtStart, bool kWide, bool kMany = false>
__global__ void __launch_bounds__(dense_threads(R), 1) step_dense_kernel(const StepParams p, const __grid_constant__ DenseMaps maps) {
  constexpr int kBlocks = dense_blocks(R), kGroups = dense_groups(R), kTile = R * 256;  // floats of an array's tile
  constexpr int V = dense_coords(R), kWarps = dense_warps(R);
  // Where g is: with the operands (up to 32 workers, so that y~ - g is what the products sum up to, as in the kernel of
  // several steps), or with the tail's inputs.
  constexpr bool kEarly = R <= 8;
  constexpr unsigned kTileBytes = kTile * 4;
  extern __shared__ unsigned char smem_unaligned[];
  unsigned char* const smem = smem_unaligned + ((1024u - (s_addr(smem_unaligned) & 1023u)) & 1023u);
  const int lane = threadIdx.x & 31, warp = __shfl_sync(0xffffffffu, threadIdx.x >> 5, 0), q = lane & 3, c = lane >> 2;
  const int group = warp / kWarps, part = warp % kWarps;
  float* const tiles = reinterpret_cast<float*>(smem + group * dense_group_bytes(R));
  double* const frag = reinterpret_cast<double*>(smem + kGroups * dense_group_bytes(R));  // [input step][output block][lane]
  uint64_t* const bars = reinterpret_cast<uint64_t*>(smem + kGroups * dense_group_bytes(R) + dense_frag_bytes(R));
  uint64_t *const in_full = bars + 2 * group, *const tail_full = in_full + 1;
  unsigned* const in_done = reinterpret_cast<unsigned*>(bars + 2 * kGroups) + 4 * group;  // warps done, slabs asked for
  unsigned *const tail_done = in_done + 1, *const in_asked = in_done + 2, *const tail_asked = in_done + 3;
  const int n = p.n;
  // operands x | y | (g), then what the results replace: (g -> g') | a -> x' | c -> y'; up to 32 workers g' has a place of its own
  float* const tx = tiles;
  float* const ty = tx + kTile;
  float* const tg = ty + kTile;
  float* const t_gout = kEarly ? tg + kTile : tg;
  float* const ta = t_gout + kTile;
  float* const tc = ta + kTile;
  // this lane's coordinates of row q; rows q + 4 i are 256 floats apart and have the same place in the swizzle
  const int within = 8 * V * part + V * c, half = within >> 5, chunk = (within & 31) >> 2;
  auto place = [&](int row) { return row * kDS + half * 32 + ((chunk ^ ((2 * row + half) & 7)) << 2) + (within & 3); };
  const int off = place(q);
  // Two elements at a time: of row i its two coordinates, or of rows i and i + 1 the one.
  auto row_of = [](int i, int m) { return V == 2 ? i : i + m; };
  auto coord_of = [](int m) { return V == 2 ? m : 0; };
  auto get = [&](const float* tile, int i) {
    if (V == 2) return *reinterpret_cast<const float2*>(tile + off + i * 256);
    return make_float2(tile[off + i * 256], i + 1 < R ? tile[off + (i + 1) * 256] : 0.f);
  };
  auto put = [&](float* tile, int i, float2 v) {
    if (V == 2) {
      *reinterpret_cast<float2*>(tile + off + i * 256) = v;
    } else {
      tile[off + i * 256] = v.x;
      if (i + 1 < R) tile[off + (i + 1) * 256] = v.y;
    }
  };
  auto one = [&](const float* tile, int i, int t) { return tile[off + i * 256 + t]; };

  const double alpha = p.alpha;
  const float sigma = static_cast<float>(p.sigma);
  const bool noisy = kMode != kModeExternal && p.sigma != 0.0;
  const unsigned limit = p.spin_limit;
  const int whole = static_cast<int>(p.d / kDS), slabs = static_cast<int>((p.d + kDS - 1) / kDS), stride = gridDim.x * kGroups;
  int slab = blockIdx.x + gridDim.x * group;

  auto load_operands = [&](int s, int k) {  // one thread, for the group's k-th slab
    *in_asked = k + 1;
    bar_expect_tx(in_full, (1u + (kMode != kModeDpsgd) + kEarly) * kTileBytes);
    rows_load(tx, &maps.x, 2 * s, 0, in_full);
    if (kMode != kModeDpsgd) rows_load(ty, &maps.y, 2 * s, 0, in_full);
    if (kEarly) rows_load(tg, &maps.g, 2 * s, 0, in_full);
  };
  auto load_tail = [&](int s, int k) {
    *tail_asked = k + 1;
    bar_expect_tx(tail_full, (1u + (kMode != kModeExternal) + !kEarly) * kTileBytes);
    if (!kEarly) rows_load(tg, &maps.g, 2 * s, 0, tail_full);
    rows_load(ta, &maps.a, 2 * s, 0, tail_full);
    if (kMode != kModeExternal) rows_load(tc, &maps.c, 2 * s, 0, tail_full);
  };
  if (part == 0 && lane == 0) {
    bar_init(in_full, 1);
    bar_init(tail_full, 1);
    *in_done = *tail_done = *in_asked = *tail_asked = 0;
    fence_barrier_init();
    fence_async_shared();
    chain_wait();
    if (slab < p.operands_end) load_operands(slab, 0);
    if (slab < p.tails_end) load_tail(slab, 0);
  }
#pragma unroll
  for (int e = threadIdx.x; e < R * kBlocks * 32; e += dense_threads(R)) {  // while the first loads are on their way
    const int l = e & 31, b = (e >> 5) % kBlocks, k = (e >> 5) / kBlocks;
    const int out = (l >> 3) + 4 * (2 * b + ((l >> 2) & 1)), in = 4 * k + (l & 3);
    frag[e] = out < n && in < n ? p.poly[out * n + in] : 0.0;
  }
  __syncthreads();
  chain_wait();
  chain_next();
  bool owes = false;  // this thread sent the last results out and has not yet asked for the next inputs
  bool ok = true;
  int use = 0;
  for (; slab < slabs; slab += stride, ++use) {
    const bool ragged = slab >= whole;
    const long long j = static_cast<long long>(slab) * kDS + within;  // this lane's first coordinate
    if (!ragged) ok = bar_wait(in_full, use & 1, limit);
    if (owes) {
      store_wait_read();
      if (slab < p.tails_end) {
        load_tail(slab, use);
      } else if (ragged) {
        bar_arrive(tail_full);
      }
      owes = false;
    }
    // what comes with the tail's inputs is needed in the products (caller-written gradients), or they are a ragged slab's:
    // its lanes' elements are read here, over tiles whose store has been read
    if (kMode == kModeExternal || ragged) {
      if (!ragged || use > 0) ok = bar_wait(tail_full, use & 1, limit) && ok;
    }
    ok = __all_sync(0xffffffffu, ok) != 0;
    if (!ok) break;
    if (ragged) {
      const int bytes = j + V <= p.d ? 4 * V : j < p.d ? 4 : 0;  // the others become zeros
      auto take = [&](float* tile, const float* base) {
#pragma unroll 1
        for (int i = 0; i < R; ++i) {
          const bool there = bytes != 0 && q + 4 * i < n;
          copy_bytes<4 * V>(tile + off + i * 256, there ? base + (q + 4 * i) * p.ld + j : base, there ? bytes : 0);
        }
      };
      take(tx, p.x);
      if (kMode != kModeDpsgd) take(ty, p.y);
      take(tg, p.g);
      take(ta, kMode == kModeExternal ? p.g_ext : p.a);
      if (kMode != kModeExternal) take(tc, p.c);
      asm volatile("cp.async.wait_all;" ::: "memory");  // every lane reads its own,
      if (R > 8) __syncwarp();                          // and the other lanes' where a sum is not finite
    }
#pragma unroll 1
    for (int step = 0; step < (kMany ? p.steps : 1); ++step) {
      const bool final_step = !kMany || step + 1 == p.steps;
      const uint32_t t_noise = p.t_noise + (kMany ? static_cast<uint32_t>(step) : 0u);
      // cx ends as x' = P (x - alpha y), by linearity; cy starts at -g and ends as y~ - g, or ends as y~.  Caller-written gradients:
      // the operand is the tracker folded with them.  D-PSGD: cx starts at -alpha g, or ends without it, and sums P x.
      double cx[kBlocks][V][2], cy[kBlocks][V][2];  // [block][coordinate][worker of the lane's two]
#pragma unroll
      for (int i = 0; i < 2 * kBlocks; ++i)
#pragma unroll
        for (int t = 0; t < V; ++t) {
          const float g = kEarly && kMode != kModeExternal && i < R ? one(tg, i, t) : 0.f;
          cx[i >> 1][t][i & 1] = kMode == kModeDpsgd && kEarly ? -alpha * static_cast<double>(g) : 0.0;
          cy[i >> 1][t][i & 1] = kMode == kModeDetag && kEarly ? static_cast<double>(-g) : 0.0;
        }
      float x_old[kAtStart ? R : 1][V];
      constexpr int kUnroll = kAtStart || R <= 10 ? R : 2;  // the printed timing keeps the old model in registers
#pragma unroll kUnroll
      for (int k = 0; k < R; ++k) {
        double u[V], y[V];
#pragma unroll
        for (int t = 0; t < V; ++t) {
          const float x = one(tx, k, t);
          if (kAtStart) x_old[kAtStart ? k : 0][t] = x;
          u[t] = static_cast<double>(x);
          y[t] = 0.0;
          if (kMode != kModeDpsgd) {
            y[t] = static_cast<double>(one(ty, k, t));
            if (kMode == kModeExternal) y[t] += static_cast<double>(one(ta, k, t)) - static_cast<double>(one(tg, k, t));  // Algorithm 2's tracker update
            u[t] = fma(-alpha, y[t], u[t]);
          }
        }
#pragma unroll
        for (int b = 0; b < kBlocks; ++b) {
          const double f = frag[(k * kBlocks + b) * 32 + lane];
#pragma unroll
          for (int t = 0; t < V; ++t) {
            if (kMode != kModeDpsgd) dmma(cy[b][t], y[t], f);
            dmma(cx[b][t], u[t], f);
          }
        }
      }
      if (R > 8) {
        // Infinities or NaN among the operands: zeros of P have carried them to workers that do not hear of them.  Each lane
        // then sums its own workers anew, without those.  (As float bits the upper half of a double that is not finite is a NaN.)
        float seen = 0.f;
#pragma unroll
        for (int b = 0; b < kBlocks; ++b)
#pragma unroll
          for (int t = 0; t < V; ++t) {
            seen = max_abs3(seen, __int_as_float(__double2hiint(cx[b][t][0])), __int_as_float(__double2hiint(cx[b][t][1])));
            if (kMode != kModeDpsgd) seen = max_abs3(seen, __int_as_float(__double2hiint(cy[b][t][0])), __int_as_float(__double2hiint(cy[b][t][1])));
          }
        if (__any_sync(0xffffffffu, seen != seen)) {
#pragma unroll
          for (int b = 0; b < kBlocks; ++b)
#pragma unroll
            for (int t = 0; t < V; ++t)
#pragma unroll
              for (int e = 0; e < 2; ++e) {
                double sx = 0.0, sy = 0.0;
#pragma unroll 1
                for (int in = 0; in < n; ++in) {
                  const double w = frag[((in >> 2) * kBlocks + b) * 32 + q * 8 + e * 4 + (in & 3)];
                  if (w == 0.0) continue;
                  const int at = (in >> 2) * 256 + place(in & 3) + t;
                  double u = static_cast<double>(tx[at]), y = 0.0;
                  if (kMode != kModeDpsgd) {
                    y = static_cast<double>(ty[at]);
                    if (kMode == kModeExternal) y += static_cast<double>(ta[at]) - static_cast<double>(tg[at]);
                    u = fma(-alpha, y, u);
                  }
                  sx = fma(w, u, sx);
                  sy = fma(w, y, sy);
                }
                cx[b][t][e] = sx;
                cy[b][t][e] = sy;
              }
        }
      }
      if (!kMany) {  // several steps write their results over the operands
        __syncwarp();
        if (lane == 0 && last_of(in_done, kWarps) && slab + stride < p.operands_end) load_operands(slab + stride, use + 1);
      }
      // Normals, all before the wait where their registers allow it.  Two coordinates: lane q draws coordinate q % 2, quad
      // 2 h + q / 2, and entry s of what it gets in return is coordinate s % 2, quad 2 h + s / 2.  One: lane q draws quad 4 h + q.
      constexpr int kDraws = V == 2 ? kBlocks : (R + 3) / 4;
      float v[kDraws][4];
      auto draw = [&](int h) {
        v[h][0] = v[h][1] = v[h][2] = v[h][3] = 0.f;
        if (noisy) {
          normal_quad(p.round_key, static_cast<unsigned long long>(p.coord_offset + j + (V == 2 ? q & 1 : 0)),
                      static_cast<uint32_t>(V == 2 ? 2 * h + (q >> 1) : 4 * h + q), t_noise, sigma, v[h]);
          transpose_quad(v[h], q);
        }
      };
      auto normal = [&](int i, int t) { return V == 2 ? v[i >> 1][2 * (i & 1) + t] : v[i >> 2][i & 3]; };
      constexpr bool kDrawFirst = R <= 10 || V == 1;
      if (kDrawFirst) {
#pragma unroll
        for (int h = 0; h < kDraws; ++h) draw(h);
      }
      if (kMode != kModeExternal && !ragged && step == 0) ok = bar_wait(tail_full, use & 1, limit);
      ok = __all_sync(0xffffffffu, ok) != 0;
      if (!ok) break;
      // ---- element-wise tail, two elements at a time
#pragma unroll
      for (int i = 0; i < R; i += 3 - V) {
        if (!kDrawFirst && (i & 1) == 0) draw(i >> 1);
        double sx[2], sy[2];
        float nv[2] = {0.f, 0.f}, old[2] = {0.f, 0.f};
#pragma unroll
        for (int m = 0; m < 2; ++m) {
          const int r = row_of(i, m), t = coord_of(m);
          sx[m] = r < R ? cx[r >> 1][t][r & 1] : 0.0;
          sy[m] = r < R ? cy[r >> 1][t][r & 1] : 0.0;
          if (r < R) nv[m] = normal(r, t);
          if (kAtStart && r < R) old[m] = x_old[kAtStart ? r : 0][t];
        }
        float2 go, g = make_float2(0.f, 0.f);
        if (!kEarly && kMode != kModeExternal) {
          g = get(tg, i);
          if (kMode == kModeDpsgd) {
            sx[0] = fma(-alpha, static_cast<double>(g.x), sx[0]);
            sx[1] = fma(-alpha, static_cast<double>(g.y), sx[1]);
          } else {
            sy[0] -= static_cast<double>(g.x);
            sy[1] -= static_cast<double>(g.y);
          }
        }
        const float2 xo = make_float2(static_cast<float>(sx[0]), static_cast<float>(sx[1]));  // x' (float64 sum, rounded once)
        float2 yo = xo;
        if (kMode == kModeExternal) {
          go = get(ta, i);  // the gradient just folded becomes g_old
          yo = make_float2(static_cast<float>(sy[0]), static_cast<float>(sy[1]));  // the gossiped tracker
        } else {
          const float2 a = get(ta, i), cc = get(tc, i);
          if (kWide) {
            go.x = static_cast<float>(fma(static_cast<double>(a.x), (kAtStart ? static_cast<double>(old[0]) : sx[0]) - static_cast<double>(cc.x), static_cast<double>(nv[0])));
            go.y = static_cast<float>(fma(static_cast<double>(a.y), (kAtStart ? static_cast<double>(old[1]) : sx[1]) - static_cast<double>(cc.y), static_cast<double>(nv[1])));
          } else {
            const F2 at = kAtStart ? pack2(old[0], old[1]) : pack2(xo.x, xo.y);  // stochastic gradient
            unpack2(fma2(pack2(a.x, a.y), sub2(at, pack2(cc.x, cc.y)), pack2(nv[0], nv[1])), go.x, go.y);
          }
          if (kMode == kModeDetag)  // fold: (y~ - g) + g', g' as stored
            yo = make_float2(static_cast<float>(sy[0] + static_cast<double>(go.x)), static_cast<float>(sy[1] + static_cast<double>(go.y)));
        }
        if (!kMany && kMode != kModeDpsgd && p.y_obs != nullptr) {  // optional observer: the gossiped tracker
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const int row = q + 4 * row_of(i, m);
            const long long at = row * p.ld + j + coord_of(m);
            if (row_of(i, m) >= R || row >= n || j + coord_of(m) >= p.d) continue;
            // g: where the products have taken it in already it is still in global memory, not yet stored over
            const float old_g = kMode == kModeDetag && kEarly ? p.g[at] : m == 0 ? g.x : g.y;
            p.y_obs[at] = static_cast<float>(sy[m] + static_cast<double>(old_g));
          }
        }
        if (!final_step) {
          put(tg, i, go);
          put(tx, i, xo);
          put(ty, i, yo);
        } else if (!ragged) {
          put(t_gout, i, go);
          put(ta, i, xo);
          if (kMode != kModeDpsgd) put(tc, i, yo);
        } else {
#pragma unroll
          for (int m = 0; m < 2; ++m) {
            const int row = q + 4 * row_of(i, m);
            const long long at = row * p.ld + j + coord_of(m);
            if (row_of(i, m) >= R || row >= n || j + coord_of(m) >= p.d) continue;
            p.g[at] = m == 0 ? go.x : go.y;
            p.x[at] = m == 0 ? xo.x : xo.y;
            if (kMode != kModeDpsgd) p.y[at] = m == 0 ? yo.x : yo.y;
          }
        }
      }
    }
    if (!ok) break;
    // What was written here comes before what the TMA does next: the results before their stores and, of several steps, the
    // intermediate ones before the next operands that are loaded over them.
    fence_async_shared();
    __syncwarp();
    if (kMany && lane == 0 && last_of(in_done, kWarps) && slab + stride < p.operands_end) load_operands(slab + stride, use + 1);
    if (!ragged) {
      if (lane == 0 && last_of(tail_done, kWarps)) {
        rows_store(&maps.g, 2 * slab, 0, t_gout);
        rows_store(&maps.x, 2 * slab, 0, ta);
        if (kMode != kModeDpsgd) rows_store(&maps.y, 2 * slab, 0, tc);
        store_commit();
        owes = slab + stride < slabs;
      }
    }
  }
  if (!ok) {
    // Copies still in flight land in this CTA's shared memory: wait for the last that were asked for (bounded) before leaving.
    // A warp that asks for more after this is still in its loop: it sees them land, or gets here itself.
    if (lane == 0) atomicExch(p.status, 1);
    const unsigned in = *const_cast<volatile unsigned*>(in_asked), tail = *const_cast<volatile unsigned*>(tail_asked);
    if (in != 0) bar_wait(in_full, (in - 1) & 1, limit);
    if (tail != 0) bar_wait(tail_full, (tail - 1) & 1, limit);
  }
  if (lane == 0) store_wait_all();
}

typedef void (*DenseKernel)(const StepParams, const DenseMaps);

template <int R>
int launch_kernel(DenseKernel kernel, StepParams p, const TensorMapSet& maps, int sm_count, cudaStream_t stream) {
  const int e = ensure_dynamic_smem(reinterpret_cast<const void*>(kernel), dense_smem_bytes(R));
  if (e != 0) return e;
  const long long slabs = (p.d + kDS - 1) / kDS, grid = slabs < sm_count ? slabs : sm_count;
  p.operands_end = p.tails_end = static_cast<int>(p.d / kDS);
  // Self test of failure detection: a block's first stall_after slabs are loaded, of the others nothing or, if the number is odd,
  // all but the tail's inputs - both waits can run out, the second with the next operands on their way.  The limits come from
  // here because a test in the kernel, run once a slab by one thread, took 48 workers from 388 to 402 us (d = 1 M).
  if (p.stall_after >= 0 && p.stall_after <= p.tails_end / grid) {
    p.tails_end = static_cast<int>(p.stall_after * grid);
    if (p.stall_after % 2 == 0) p.operands_end = p.tails_end;
  }
  return launch_chained(kernel, static_cast<unsigned>(grid), dense_threads(R), dense_smem_bytes(R), stream, p, *reinterpret_cast<const DenseMaps*>(maps.bytes));
}

template <int R>
int launch_dense(const StepParams& p, const TensorMapSet& maps, int sm_count, cudaStream_t stream) {
  DenseKernel kernel = step_dense_kernel<R, kModeExternal, false, false>;
  if (p.mode == kModeDpsgd) {  // beyond 32 workers it goes by the rounds' name and has their gradient in float64
    kernel = p.grad_at_start ? step_dense_kernel<R, kModeDpsgd, true, (R > 8)> : step_dense_kernel<R, kModeDpsgd, false, (R > 8)>;
  } else if (p.mode == kModeDetag) {
    kernel = p.grad_at_start ? step_dense_kernel<R, kModeDetag, true, false> : step_dense_kernel<R, kModeDetag, false, false>;
  }
  return launch_kernel<R>(kernel, p, maps, sm_count, stream);
}

template <int R>
int launch_many(const StepParams& p, const TensorMapSet& maps, int sm_count, cudaStream_t stream) {
  return launch_kernel<R>(p.grad_at_start ? step_dense_kernel<R, kModeDetag, true, false, true> : step_dense_kernel<R, kModeDetag, false, false, true>, p, maps, sm_count, stream);
}

}  // namespace

bool build_maps_dense(const StepParams& p, TensorMapSet* out) {
  DenseMaps& m = *reinterpret_cast<DenseMaps*>(out->bytes);
  const int rows = (p.n + 3) / 4 * 4;
  const float* y = p.mode == kModeDpsgd ? p.x : p.y;  // D-PSGD has no tracker, caller-written gradients no objective: never used
  const float* a = p.mode == kModeExternal ? p.g_ext : p.a;
  const float* c = p.mode == kModeExternal ? p.g_ext : p.c;
  return make_half_map(&m.x, p.x, p.n, p.d, p.ld, rows) && make_half_map(&m.y, y, p.n, p.d, p.ld, rows) &&
         make_half_map(&m.g, p.g, p.n, p.d, p.ld, rows) && make_half_map(&m.a, a, p.n, p.d, p.ld, rows) &&
         make_half_map(&m.c, c, p.n, p.d, p.ld, rows);
}

// p.steps iterations, up to 32 workers.
int launch_step_dense_many(const StepParams& p, const TensorMapSet& maps, int sm_count, cudaStream_t stream) {
  if (p.n <= kMaxSmallWorkers || p.n > 32 || p.d <= 0 || p.d > 0x7fffffffLL || p.mode != kModeDetag) return static_cast<int>(cudaErrorInvalidValue);
  switch ((p.n + 3) / 4) {
    case 5: return launch_many<5>(p, maps, sm_count, stream);
    case 6: return launch_many<6>(p, maps, sm_count, stream);
    case 7: return launch_many<7>(p, maps, sm_count, stream);
    default: return launch_many<8>(p, maps, sm_count, stream);
  }
}

int launch_step_dense(const StepParams& p, const TensorMapSet& maps, int sm_count, cudaStream_t stream) {
  if (p.n <= kMaxSmallWorkers || p.n > kMaxDenseStepWorkers || p.d <= 0 || p.d > 0x7fffffffLL) return static_cast<int>(cudaErrorInvalidValue);
  switch ((p.n + 3) / 4) {
    case 5: return launch_dense<5>(p, maps, sm_count, stream);
    case 6: return launch_dense<6>(p, maps, sm_count, stream);
    case 7: return launch_dense<7>(p, maps, sm_count, stream);
    case 8: return launch_dense<8>(p, maps, sm_count, stream);
    case 9: return launch_dense<9>(p, maps, sm_count, stream);
    case 10: return launch_dense<10>(p, maps, sm_count, stream);
    case 11: return launch_dense<11>(p, maps, sm_count, stream);
    default: return launch_dense<12>(p, maps, sm_count, stream);
  }
}

}  // namespace detag
