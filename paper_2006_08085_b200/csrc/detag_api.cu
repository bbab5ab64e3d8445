// Host side of the C ABI declared in include/detag.h: argument checking, the host-side numerics
// (momentum, polynomial of the gossip matrix), workspace layout and kernel launches.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <new>
#include <utility>

#include "detag_internal.h"
#include "torus_basis.h"

using detag::StepParams;

namespace {

size_t align_up(size_t v) { return (v + detag::kWsAlign - 1) / detag::kWsAlign * detag::kWsAlign; }

struct WsLayout {
  size_t status, result, row_ptr, col_idx, vals, poly, torus, partials, total;
  struct { size_t weights, row_exp, guard, poly; } split, rows;
};

WsLayout ws_layout(const detag_state* s) {
  WsLayout l{};
  size_t off = 0;
  l.status = off;
  l.result = off + 64;
  off += detag::kWsAlign;
  l.row_ptr = off;
  off += align_up((s->n + 1) * sizeof(int32_t));
  l.col_idx = off;
  off += align_up(s->col_idx.size() * sizeof(int32_t));
  l.vals = off;
  off += align_up(s->vals.size() * sizeof(double));
  l.poly = off;
  off += align_up(s->poly.size() * sizeof(double));
  l.torus = off;
  off += align_up(s->torus_frag.size() * sizeof(double));
  const std::pair<const detag::SplitPoly*, decltype(l.split)*> tables[2] = {{&s->split, &l.split}, {&s->rows, &l.rows}};
  for (const auto& t : tables) {
    t.second->weights = off;
    off += align_up(t.first->weights.size());
    t.second->row_exp = off;
    off += align_up(t.first->row_exp.size() * sizeof(int32_t));
    t.second->guard = off;
    off += align_up(t.first->guard.size());
    t.second->poly = off;
    off += align_up(t.first->poly.size() * sizeof(double));
  }
  l.partials = off;
  off += align_up(detag::kMaxPartials * sizeof(double));
  l.total = off;
  return l;
}

int fail(detag_state* s, int code, const char* what) {
  if (s) s->err = what;
  return code;
}

int fail_cuda(detag_state* s, int cuda_code, const char* where) {
  if (s) {
    char buf[256];
    std::snprintf(buf, sizeof buf, "%s: %s", where, cudaGetErrorString(static_cast<cudaError_t>(cuda_code)));
    s->err = buf;
  }
  return DETAG_ERR_CUDA;
}

// P_K(M) by the matrix form of Algorithm 3: P_{-1} = P_0 = I, P_{r+1} = (1+eta) M P_r - eta P_{r-1}.
void gossip_polynomial(const detag_state* s, std::vector<double>& out) {
  const int n = s->n;
  std::vector<double> prev(static_cast<size_t>(n) * n, 0.0), cur, next(static_cast<size_t>(n) * n), acc(n);
  for (int i = 0; i < n; ++i) prev[static_cast<size_t>(i) * n + i] = 1.0;
  cur = prev;
  for (int r = 0; r < s->K; ++r) {
    for (int i = 0; i < n; ++i) {
      std::fill(acc.begin(), acc.end(), 0.0);
      for (int k = s->row_ptr[i]; k < s->row_ptr[i + 1]; ++k) {
        const double w = s->vals[k];
        const double* row = &cur[static_cast<size_t>(s->col_idx[k]) * n];
        for (int j = 0; j < n; ++j) acc[j] += w * row[j];
      }
      const double* old = &prev[static_cast<size_t>(i) * n];
      double* out_row = &next[static_cast<size_t>(i) * n];
      for (int j = 0; j < n; ++j) out_row[j] = (1.0 + s->eta) * acc[j] - s->eta * old[j];
    }
    prev.swap(cur);
    cur.swap(next);
  }
  out = cur;
}

// Rows 32 further are the same entries 32 columns further: then so is every polynomial of M, and its 32 x 32 blocks
// depend on their distance only.
bool block_circulant(const detag_state* s) {
  constexpr int kBlock = 32;
  const int n = s->n;
  if (n % kBlock != 0) return false;
  std::vector<double> row(n, 0.0);
  for (int i = 0; i < n; ++i) {
    const int next = (i + kBlock) % n;
    if (s->row_ptr[i + 1] - s->row_ptr[i] != s->row_ptr[next + 1] - s->row_ptr[next]) return false;
    for (int k = s->row_ptr[i]; k < s->row_ptr[i + 1]; ++k) row[s->col_idx[k]] = s->vals[k];
    bool same = true;
    for (int k = s->row_ptr[next]; k < s->row_ptr[next + 1]; ++k)
      same = same && row[(s->col_idx[k] - kBlock + n) % n] == s->vals[k];
    for (int k = s->row_ptr[i]; k < s->row_ptr[i + 1]; ++k) row[s->col_idx[k]] = 0.0;
    if (!same) return false;
  }
  return true;
}

// Rows 0 .. 31 of P_K(M), for a matrix whose 32 x 32 blocks depend on their distance only: the recursion of Algorithm 3
// on those rows alone, P_{r+1} = (1+eta) P_r M - eta P_{r-1} (P_r is a polynomial of M and commutes with it).
void first_block_row(const detag_state* s, std::vector<double>& out) {
  constexpr int kRows = 32;
  const int n = s->n;
  out.assign(static_cast<size_t>(kRows) * n, 0.0);
  if (!s->circ_row.empty()) {  // circulant: shifts of the first row, which is known
    for (int i = 0; i < kRows; ++i)
      for (int j = 0; j < n; ++j) out[static_cast<size_t>(i) * n + j] = s->circ_row[j >= i ? j - i : j - i + n];
    return;
  }
  std::vector<double> prev(n), cur(n), next(n);
  for (int i = 0; i < kRows; ++i) {
    std::fill(prev.begin(), prev.end(), 0.0);
    prev[i] = 1.0;
    cur = prev;
    for (int r = 0; r < s->K; ++r) {
      std::fill(next.begin(), next.end(), 0.0);
      for (int k = 0; k < n; ++k)
        if (cur[k] != 0.0)
          for (int e = s->row_ptr[k]; e < s->row_ptr[k + 1]; ++e) next[s->col_idx[e]] += cur[k] * s->vals[e];
      for (int j = 0; j < n; ++j) next[j] = (1.0 + s->eta) * next[j] - s->eta * prev[j];
      prev.swap(cur);
      cur.swap(next);
    }
    std::copy(cur.begin(), cur.end(), out.begin() + static_cast<size_t>(i) * n);
  }
}

// Of the 32 x 32 blocks of P_K(M), those per 32 rows whose workers hear from one another in K rounds (n <= 256).
double reached_blocks(const detag_state* s) {
  const int n = s->n, nb = (n + 31) / 32;
  std::vector<uint32_t> from(static_cast<size_t>(n) * nb, 0), next;
  for (int i = 0; i < n; ++i) from[static_cast<size_t>(i) * nb + i / 32] = 1u << (i % 32);
  for (int r = 0; r < s->K; ++r) {
    next = from;
    for (int i = 0; i < n; ++i)
      for (int k = s->row_ptr[i]; k < s->row_ptr[i + 1]; ++k)
        for (int b = 0; b < nb; ++b) next[static_cast<size_t>(i) * nb + b] |= from[static_cast<size_t>(s->col_idx[k]) * nb + b];
    if (next == from) break;
    from.swap(next);
  }
  int count = 0;
  for (int c = 0; c < nb; ++c)
    for (int b = 0; b < nb; ++b) {
      uint32_t any = 0;
      for (int i = 32 * c; i < n && i < 32 * c + 32; ++i) any |= from[static_cast<size_t>(i) * nb + b];
      count += any != 0 ? 1 : 0;
    }
  return static_cast<double>(count) / nb;
}

// Circulant M (row i = row 0 shifted by i): then P_K(M) is circulant too; its row 0 is computed with the
// recursion of Algorithm 3 on a single row and stored as a band around the diagonal.
void analyse_circulant(detag_state* s) {
  const int n = s->n;
  std::vector<double> row0(n, 0.0);
  for (int k = s->row_ptr[0]; k < s->row_ptr[1]; ++k) row0[s->col_idx[k]] = s->vals[k];
  for (int i = 1; i < n; ++i) {
    if (s->row_ptr[i + 1] - s->row_ptr[i] != s->row_ptr[1] - s->row_ptr[0]) return;
    for (int k = s->row_ptr[i]; k < s->row_ptr[i + 1]; ++k)
      if (s->vals[k] != row0[((s->col_idx[k] - i) % n + n) % n]) return;
  }
  s->circulant = true;
  // row 0 of P_r: q_{r+1}[j] = (1+eta) sum_k M[0][k] q_r[(j - k) mod n] - eta q_{r-1}[j]   (circulant product)
  std::vector<double> prev(n, 0.0), cur, next(n);
  prev[0] = 1.0;
  cur = prev;
  for (int r = 0; r < s->K; ++r) {
    std::fill(next.begin(), next.end(), 0.0);
    for (int k = s->row_ptr[0]; k < s->row_ptr[1]; ++k) {
      const double w = s->vals[k];
      const int shift = s->col_idx[k];  // next[j] += w cur[(j - shift) mod n]
      for (int j = 0; j < shift; ++j) next[j] += w * cur[j - shift + n];
      for (int j = shift; j < n; ++j) next[j] += w * cur[j - shift];
    }
    for (int j = 0; j < n; ++j) next[j] = (1.0 + s->eta) * next[j] - s->eta * prev[j];
    prev.swap(cur);
    cur.swap(next);
  }
  int hb = 0;
  for (int j = 0; j < n; ++j)
    if (cur[j] != 0.0) {
      const int delta = j <= n / 2 ? j : n - j;
      if (delta > hb) hb = delta;
    }
  s->half_band = hb;
  if (n <= detag::kMaxSplitWorkers) s->circ_row = cur;
  if (hb <= 16 && n >= 2 * hb + 1)
    for (int delta = -16; delta <= 16; ++delta)
      s->band[delta + 16] = (delta >= -hb && delta <= hb) ? cur[((delta % n) + n) % n] : 0.0;
}

// Block-circulant M with 8-worker blocks whose block (r, r') depends on the distance (r' - r) mod R only, equal for
// +k and -k (tori): the real Fourier basis Q of the R-cycle block-diagonalises every polynomial of M,
//     P_K(M) = sum_p (q_p q_p^T) (x) P_K(Mhat_p) ,   Mhat_p = sum_k cos(2 pi f_p k / R) G_k .
// The 8 x 8 blocks P_K(Mhat_p) come from the recursion of Algorithm 3 on Mhat_p; the result is accepted only if it
// reproduces the dense polynomial.
void analyse_torus(detag_state* s) {
  const int n = s->n, C = 8;
  if (s->poly.empty() || n % C != 0 || !detag::torus_variant_available(n)) return;
  const int R = n / C;
  std::vector<double> m;
  detag::csr_to_dense(n, s->row_ptr.data(), s->col_idx.data(), s->vals.data(), m);
  auto M = [&](int r, int c, int r2, int c2) { return m[static_cast<size_t>(r * C + c) * n + (r2 * C + c2)]; };
  for (int r = 0; r < R; ++r)
    for (int k = 0; k < R; ++k)
      for (int c = 0; c < C; ++c)
        for (int c2 = 0; c2 < C; ++c2) {
          if (M(r, c, (r + k) % R, c2) != M(0, c, k, c2)) return;        // block circulant
          if (M(0, c, k, c2) != M(0, c, (R - k) % R, c2)) return;        // the same block at distance +k and -k
        }
  const double kPi = 3.14159265358979323846;
  std::vector<double> q(static_cast<size_t>(R) * R);  // the kernel's basis, row p = basis vector p
  std::vector<int> freq(R);
  for (int p = 0; p < R; ++p) {
    freq[p] = detag::torus_frequency(R, p);
    for (int r = 0; r < R; ++r) q[p * R + r] = detag::torus_q(R, p, r);
  }
  std::vector<double> phat(static_cast<size_t>(R) * C * C);
  for (int p = 0; p < R; ++p) {
    double mh[8][8], prev[8][8], cur[8][8], next[8][8];
    for (int c = 0; c < C; ++c)
      for (int c2 = 0; c2 < C; ++c2) {
        double acc = 0.0;
        for (int k = 0; k < R; ++k) acc += std::cos(2.0 * kPi * freq[p] * k / R) * M(0, c, k, c2);
        mh[c][c2] = acc;
        prev[c][c2] = cur[c][c2] = c == c2 ? 1.0 : 0.0;
      }
    for (int round = 0; round < s->K; ++round) {  // P_{r+1} = (1+eta) Mhat P_r - eta P_{r-1}
      for (int c = 0; c < C; ++c)
        for (int c2 = 0; c2 < C; ++c2) {
          double acc = 0.0;
          for (int k = 0; k < C; ++k) acc += mh[c][k] * cur[k][c2];
          next[c][c2] = (1.0 + s->eta) * acc - s->eta * prev[c][c2];
        }
      std::memcpy(prev, cur, sizeof cur);
      std::memcpy(cur, next, sizeof cur);
    }
    for (int c = 0; c < C; ++c)
      for (int c2 = 0; c2 < C; ++c2) phat[(static_cast<size_t>(p) * C + c) * C + c2] = cur[c][c2];
  }
  // the decomposition must give back the dense polynomial
  double worst = 0.0, scale = 0.0;
  for (int r = 0; r < R; ++r)
    for (int r2 = 0; r2 < R; ++r2)
      for (int c = 0; c < C; ++c)
        for (int c2 = 0; c2 < C; ++c2) {
          double acc = 0.0;
          for (int p = 0; p < R; ++p) acc += q[p * R + r] * q[p * R + r2] * phat[(static_cast<size_t>(p) * C + c) * C + c2];
          const double want = s->poly[static_cast<size_t>(r * C + c) * n + (r2 * C + c2)];
          worst = std::fmax(worst, std::fabs(acc - want));
          scale = std::fmax(scale, std::fabs(want));
        }
  if (!(worst <= 1e-13 * std::fmax(1.0, scale))) return;
  s->torus = true;
  // fragment order of the kernel: entry (p, k-step s, lane) is Phat_p[c'][c] with the contraction index
  // c = lane % 4 + 4 s and the output position c' = pi(lane / 4), pi(2 q + e) = q + 4 e (see step_torus.cu)
  s->torus_frag.resize(static_cast<size_t>(R) * 2 * 32);
  // For R = 8 the kernel's butterflies leave out the basis' normalisation (1/sqrt(8) for the constant and the
  // alternating vector, 1/2 for the others) on the way in and on the way out: both factors go into the block.
  for (int p = 0; p < R; ++p) {
    const double scale = R == 8 ? ((p == 0 || p == R - 1) ? 0.125 : 0.25) : 1.0;
    for (int st = 0; st < 2; ++st)
      for (int lane = 0; lane < 32; ++lane)
        s->torus_frag[(static_cast<size_t>(p) * 2 + st) * 32 + lane] =
            scale * phat[(static_cast<size_t>(p) * C + ((lane / 4) >> 1) + 4 * ((lane / 4) & 1)) * C + (lane % 4) + 4 * st];
  }
}

bool torus_ok(const detag_state* s) { return s->torus && s->d <= 0x7fffffffLL; }

// The circulant kernel takes polynomials whose half-band is at most 16; the integer tensor path the others up to 256 workers.
bool ring_band(const detag_state* s) { return detag::ring_variant_available(s->n, s->half_band); }

bool band_ok(const detag_state* s) {
  return s->circulant && s->d <= 0x7fffffffLL && (ring_band(s) || (detag::ring_variant_available(s->n, 0) && s->n <= detag::kMaxSplitWorkers));
}

int step_mode(const detag_state* s) {
  if (s->algorithm == DETAG_ALGORITHM_DPSGD) return detag::kModeDpsgd;
  return s->gradient_source == DETAG_GRADIENT_EXTERNAL ? detag::kModeExternal : detag::kModeDetag;
}

StepParams make_params(const detag_state* s) {
  StepParams p{};
  p.n = s->n;
  p.nnz = static_cast<int>(s->col_idx.size());
  p.K = s->K;
  p.d = s->d;
  p.ld = s->ld;
  p.coord_offset = s->coord_offset;
  p.x = s->x;
  p.y = s->y;
  p.g = s->g;
  p.a = s->a;
  p.c = s->c;
  p.y_obs = s->y_obs;
  p.row_ptr = s->d_row_ptr;
  p.col_idx = s->d_col_idx;
  p.vals = s->d_vals;
  p.poly = s->d_poly;
  p.torus = s->d_torus;
  p.tables = s->d_tables;
  p.eta = s->eta;
  p.alpha = s->alpha;
  p.sigma = s->sigma;
  for (uint32_t round = 0; round < 10; ++round) {
    p.round_key[2 * round] = static_cast<uint32_t>(s->seed & 0xffffffffu) + round * 0x9E3779B9u;
    p.round_key[2 * round + 1] = static_cast<uint32_t>(s->seed >> 32) + round * 0xBB67AE85u;
  }
  p.status = s->d_status;
  p.grad_at_start = s->gradient_point == DETAG_GRADIENT_AT_PHASE_START ? 1 : 0;
  p.mode = step_mode(s);
  p.g_ext = s->g_ext;
  p.spin_limit = s->spin_limit;
  p.stall_after = s->stall_after;
  return p;
}

bool dense_ok(const detag_state* s) {
  if (s->d > 0x7fffffffLL) return false;
  return detag::dense_variant_available(s->n);
}

// Host cost model.  The product with the polynomial beats the sparse rounds wherever a kernel takes it: K rounds cost
// K * (nnz per row) shared-memory gathers of 16 bytes per element and array and two barriers each.  Tori of 8-worker blocks
// take the transform kernel (24 multiply-adds per element and array).  Caller-written gradients run on the dense kernels
// for n <= 48 (under the rounds' name beyond 32), beyond on step_rows.cu (to 192) or as rounds (rows_beat_rounds).
bool variant_runs_mode(const detag_state* s, int variant) {
  if (step_mode(s) == detag::kModeDetag) return true;
  if (variant == DETAG_VARIANT_RING) return step_mode(s) == detag::kModeDpsgd;
  return variant == DETAG_VARIANT_CSR || (variant == DETAG_VARIANT_DENSE && s->n <= 32);  // n > 32: DeTAG step only
}

int resolve_variant(const detag_state* s) {
  if (s->variant_forced != DETAG_VARIANT_AUTO) return s->variant_forced;
  // a ring whose band fits takes the circulant kernel from n = 64 on; rings with a dense polynomial go by that name too,
  // beyond 64 workers
  const bool ring = band_ok(s) && (ring_band(s) || s->n > 64);
  if (step_mode(s) == detag::kModeDpsgd && s->n > 32 && ring) return DETAG_VARIANT_RING;
  if (step_mode(s) != detag::kModeDetag) return (s->n <= 32 && dense_ok(s)) ? DETAG_VARIANT_DENSE : DETAG_VARIANT_CSR;
  if (s->n > 32 && ring) return DETAG_VARIANT_RING;
  if (s->n > 32 && torus_ok(s)) return DETAG_VARIANT_TORUS;
  if (dense_ok(s)) {
    if (s->n > 64) {
      // Where no structure decides, the rounds if a float64 product on the tensor path (blocks of eight workers on four
      // schedulers) would take longer, in ms at d = 2 M: one or two rounds on graphs of degree four.  Both run on the
      // integer tensor path now where that takes the matrix (split_ok; 100 workers, d = 2 M: 2.0 ms for two rounds, 3.9 as
      // rounds); what the choice still decides is the name the call goes by and with it the precision of the gradient, which
      // the rounds evaluate in float64 and the products in float32 at the stored model.
      const int blocks = (s->n + 7) / 8, blocks_eff = blocks % 4 == 3 ? blocks + 1 : blocks;
      const double dense_ms = 0.0412 * blocks_eff * blocks / 2.0;
      const double rounds_ms = 0.024 * s->n + 0.00155 * s->K * static_cast<double>(s->col_idx.size());
      if (rounds_ms < dense_ms) return DETAG_VARIANT_CSR;
    }
    return DETAG_VARIANT_DENSE;
  }
  return DETAG_VARIANT_CSR;
}

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

int query_device(detag_state* s) {
  cudaError_t e = cudaGetDevice(&s->device);
  if (e != cudaSuccess) return fail_cuda(s, e, "cudaGetDevice");
  e = cudaDeviceGetAttribute(&s->sm_count, cudaDevAttrMultiProcessorCount, s->device);
  if (e != cudaSuccess) return fail_cuda(s, e, "cudaDeviceGetAttribute(sm count)");
  e = cudaDeviceGetAttribute(&s->smem_optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, s->device);
  if (e != cudaSuccess) return fail_cuda(s, e, "cudaDeviceGetAttribute(shared memory)");
  return DETAG_OK;
}

// Kernel families that take tensor maps.
enum { kFamilyMma = 1, kFamilyTorus = 2, kFamilyRing = 3, kFamilySplit = 4, kFamilyDense = 5, kFamilyRows = 6 };

// Tensor maps for the buffers in `p`: built on first use, then found again by buffer addresses and sizes
// (detag_step always hits; detag_step_host cycles through its two chunk slots and the ragged last chunk).
const detag::TensorMapSet* maps_for(detag_state* s, int family, const StepParams& p) {
  const void* slot_a = p.mode == detag::kModeExternal ? static_cast<const void*>(p.g_ext) : p.a;
  const void* key[5] = {p.x, p.mode == detag::kModeDpsgd ? nullptr : p.y, p.g, slot_a,
                        p.mode == detag::kModeExternal ? nullptr : p.c};
  for (auto& en : s->map_cache) {
    if (en.family == family && en.d == p.d && en.ld == p.ld && std::memcmp(en.ptr, key, sizeof key) == 0)
      return &en.maps;
  }
  constexpr size_t kEntries = 6;
  detag_state::MapEntry* slot;
  if (s->map_cache.size() < kEntries) {
    s->map_cache.emplace_back();
    slot = &s->map_cache.back();
  } else {
    slot = &s->map_cache[s->map_next];
    s->map_next = (s->map_next + 1) % kEntries;
  }
  detag_state::MapEntry& en = *slot;
  en.family = 0;  // invalid until built
  const bool ok = family == kFamilyMma    ? detag::build_maps_mma(p, &en.maps)
                  : family == kFamilyRing ? detag::build_maps_ring(p, &en.maps)
                  : family == kFamilySplit ? detag::build_maps_split(p, &en.maps)
                  : family == kFamilyDense ? detag::build_maps_dense(p, &en.maps)
                  : family == kFamilyRows  ? detag::build_maps_rows(p, &en.maps)
                                          : detag::build_maps_torus(p, &en.maps);
  if (!ok) return nullptr;
  en.family = family;
  en.d = p.d;
  en.ld = p.ld;
  std::memcpy(en.ptr, key, sizeof key);
  return &en.maps;
}

// The integer tensor path: lanes as coordinates, or (rows) as output workers.
int launch_split(detag_state* s, const StepParams& p, bool rows, bool wide, cudaStream_t stream) {
  const detag::TensorMapSet* maps = maps_for(s, rows ? kFamilyRows : kFamilySplit, p);
  if (!maps) return fail(s, DETAG_ERR_CUDA, "tensor map encoding failed");
  const WsLayout l = ws_layout(s);
  const auto& at = rows ? l.rows : l.split;
  const unsigned char* base = p.tables;
  const detag::SplitDevice tables{base + at.weights, reinterpret_cast<const int32_t*>(base + at.row_exp), base + at.guard,
                                  reinterpret_cast<const double*>(base + at.poly)};
  s->launched[p.beside] = rows ? "step_rows" : "step_split";
  const int e = rows ? detag::launch_step_rows(p, *maps, s->rows, tables, wide, s->sm_count, stream)
                     : detag::launch_step_split(p, *maps, s->split, tables, wide, s->sm_count, stream);
  return e != 0 ? fail_cuda(s, e, "step kernel launch") : DETAG_OK;
}

// The columns from `first` on, which the circulant kernel leaves (it takes whole 64-coordinate slabs), in the same call, beside
// it (64-ring, K = 4, d = 14001 21.3 -> 14.6 us in one launch, 256, d = 60001 188 -> 143 in two): through the integer tensor path up to
// 128 workers (one chunk or two 8 .. 11 us), beyond as rounds, whose latency is the smaller one (256 workers 6 us and 1.7 a round,
// step_split.cu's slab 38), and so where the caller asked for the circulant kernel, which runs in float64 throughout.
int launch_tail_columns(detag_state* s, const StepParams& p, long long first, cudaStream_t stream) {
  StepParams pt = p;
  pt.d = p.d - first;
  pt.coord_offset = p.coord_offset + first;
  pt.x = p.x + first;
  pt.y = p.y + first;
  pt.g = p.g + first;
  pt.a = p.a + first;
  pt.c = p.c + first;
  if (p.y_obs) pt.y_obs = p.y_obs + first;
  pt.beside = first > 0 ? 1 : 0;
  if (p.n <= 128 && !s->rows.weights.empty() && s->variant_forced == DETAG_VARIANT_AUTO) return launch_split(s, pt, true, false, stream);
  s->launched[pt.beside] = "step_csr";
  const int rc = detag::plan_step_csr(pt, s->smem_optin);
  if (rc != DETAG_OK) return fail(s, rc, "graph too large for the shared-memory plan");
  const int e = detag::launch_step_csr(pt, s->sm_count, stream);
  return e != 0 ? fail_cuda(s, e, "step kernel launch") : DETAG_OK;
}

// The integer tensor path takes the dense and circulant products with 48 < n <= 256, and, where the choice is the
// library's, the rounds of such matrices too.  Circulant bands stay on their float64 kernel, which needs no test of the
// operands; us per step, integer path -> that one: 64 workers, d = 2 M, K = 1 1099 -> 1035, K = 16 1020 -> 1035; 128, d = 1 M,
// K = 1 1260 -> 1031, K = 16 1103 -> 1031; 224, d = 500 k, K = 16 1198 -> 927; 256, d = 1 M, K = 1 3157 -> 2032, K = 16
// 2620 -> 2032; 256, d = 4096 82 -> 30.  (Bands of half-width 12 to 16 of up to 128 workers gain on the integer path with operands alike -
// 64, K = 12, d = 60 k 47 -> 45, 128, K = 16 105 -> 73 - and lose with operands spread over four decades: 47 -> 163, 119 -> 272.)
// Unless the choice is the library's and d is ragged, up to 128 workers, and so short that one launch takes less than two side by
// side: 64 workers, K = 4, d = 3001 13.8 -> 9.6; 128, 3001 15.3 -> 12.4, but 9001 15.9 -> 18.7; 256, 3001
// 42.8 -> 67.  Longer ones of 64 would gain too, with operands alike (d = 60001 50.4 -> 40.5; spread 69 -> 172).
bool split_ok(const detag_state* s, const StepParams& p, int variant) {
  if ((s->split.weights.empty() && s->rows.weights.empty()) || p.d > 0x7fffffffLL) return false;
  if (variant == DETAG_VARIANT_CSR) return s->variant_forced == DETAG_VARIANT_AUTO;
  if (variant == DETAG_VARIANT_DENSE) return true;
  if (variant != DETAG_VARIANT_RING) return false;
  if (!ring_band(s)) return true;
  if (s->variant_forced != DETAG_VARIANT_AUTO) return false;
  // by the length of the state, not of a staged chunk: host-resident stepping gives the same bits
  return s->d % 64 != 0 && s->d <= (s->n <= 64 ? 4LL : s->n <= 128 ? 1LL : 0LL) * 32 * s->sm_count;
}

// Whether step_rows.cu takes less than the rounds: caller-written gradients up to 192 workers, beyond 128 matrices without block
// structure.  Estimates of both in us (`sms`: as if on that many SMs).  Rounds -> there, operands alike: caller-written,
// 100 workers, K = 6, d = 1 M 3177 -> 862, 20 k 76 -> 27, ring of 54, K = 1, d = 27 k 13.9 against 24.1; 144, K = 6, d = 500 k 3396 -> 984,
// 256, K = 12, d = 200 k 3830 -> 750, ring of 144, K = 4, d = 8931 35.6 against 48.1.  On short vectors rounds take their latency, one after the other:
// caller-written, 124 workers, K = 12, d = 785 31.7 us; 226, K = 16, d = 246 32.5.
// The rounds do not care how operands differ, and there what cannot share a scale is summed in float64 at up to five times the time (14 us more
// per turn of the SMs at 100 workers, 55 at 250).  So the estimate is for operands spread over four decades: few rounds on sparse graphs
// then stay rounds, which alike would gain.  Of passes of eight coordinates the share that is held up goes with the fourth root of the coordinates'
// (0.2 at 0.003, 0.36 at 0.015, 0.6 at 0.12, 0.8 at 0.45, measured).  A limit of 1.1 for caller-written gradients, 1.35 for the others, for which the
// estimate is the more careful one: where it says 0.74 of the rounds' speed or more 0.8 is the least that was measured.  Rounds' time / time there, operands alike, spread over two, over four
// decades, d = 150 k: caller-written, 100 workers, K = 3 1.7, 1.3, 0.59, K = 5 2.5, 2.1, 1.8; 128, K = 4 2.4, 1.9, 0.98; 160, K = 5 2.9, 0.98, 0.63; 192, K = 5 2.4, 1.7, 0.68; DeTAG, 140, K = 3 1.9, 1.2, 0.53,
// K = 4 2.3, 1.7, 0.75, K = 6 3.1, 2.9, 1.7; 215, K = 5 3.1, 1.6, 0.78, K = 6 3.6, 1.2, 0.91; 250, K = 4 2.1, 0.94, 0.52; D-PSGD, 180, K = 5 2.3, 0.75, 0.57; 155-ring, K = 6 2.4, 2.1, 0.77, K = 10 3.3,
// 2.8, 1.2; 14 x 13 torus, K = 3 1.9, 1.7, 0.50, K = 6 2.7, 2.5, 0.87.
bool rows_beat_rounds(const detag_state* s, int mode, int sms) {
  const detag::SplitPoly& t = s->rows;
  const double n = s->n, d = static_cast<double>(s->d), turns = std::ceil(d / (32.0 * sms)), nb = std::ceil(n / 32.0);
  const double products = s->K * static_cast<double>(s->col_idx.size());
  const bool sparse = t.guard.size() > static_cast<size_t>(s->n);
  // The 32 x 32 blocks that the float64 sums go through per 32 outputs.  Before the tables are made the share is the least that was found
  // for graphs with fewer than 2.5 walks of K steps, degree - 1 onwards at each, per worker, and none beyond.
  double share = t.unequal, blocks = s->reach;
  if (t.guard.empty()) {
    share = std::pow(std::fmax(products / s->K / n - 2.0, 0.0), s->K) < 2.5 * n ? 0.15 : 0.0;
  } else {
    int reach = 0;
    for (unsigned char r : t.reach) reach += __builtin_popcount(r);
    blocks = reach / nb;
  }
  double here, unequal, rounds, latency, limit = 1.35;
  if (mode == detag::kModeExternal) {
    limit = 1.1;
    if (n > 128) {
      here = 10.0 + 0.065 * n * turns * (sparse ? 1.05 : 1.0);
      unequal = 2.0 + 8.0 * blocks;
      rounds = 6.0 + (1.2 + 0.003 * n + 0.00105 * products) * d / 1000.0;
    } else {  // of 65 to 96 workers six warps for the test of the operands
      here = 8.0 + turns * (n <= 64 ? 0.6 + 0.036 * n : n <= 96 ? 0.063 * n * (sparse ? 1.3 : 1.0) : (3.4 + 0.009 * n) * (sparse ? 1.2 : 1.0));
      unequal = (n <= 64 ? 2.5 : n <= 96 ? 5.5 : 3.5) * blocks;
      rounds = 6.0 + (0.0085 * n + 0.00078 * products) * (n <= 64 ? 0.86 : 1.0) * d / 1000.0;
    }
    latency = 6.0 + 0.0155 * n * s->K;
  } else {
    here = 10.0 + 0.065 * n * turns * (sparse ? 1.07 : 1.0);
    unequal = 3.0 + 1.2 * nb + 5.0 * blocks;
    rounds = (1.35 + 0.004 * n + 0.0011 * products) * d / 1000.0;
    latency = 6.0 + 0.0068 * n * s->K;
    if (mode == detag::kModeDpsgd) {  // one array
      here *= 0.88;
      unequal *= 0.85;
      rounds *= 0.68;
    }
  }
  rounds = std::fmax(std::fmax(rounds, latency), 8.0);
  return here < rounds && here + std::sqrt(std::sqrt(share)) * unequal * d / (32.0 * sms) < limit * rounds;
}

// Of 97 to 128 workers, calls in which reading the model a second time, in pieces of 32 bytes, costs the printed timing more than
// step_rows.cu gains: step_split.cu -> there, n = 98, d = 1 M 1021 -> 990, 2 M 2040 -> 2082; 112, 600 k 647 -> 614, 1 M 1077 -> 1087, 2 M 2143 -> 2333; 128, 600 k
// 703 -> 662, 1 M 1167 -> 1218, 2 M 2318 -> 2616.
bool long_calls(const detag_state* s, int sms) { return s->n * std::ceil(static_cast<double>(s->d) / (32.0 * sms)) > 24000.0; }

// Which of its two kernels.  us per step, lanes as coordinates -> as output workers: 100 workers, d = 2 k 13.0 -> 9.4, 20 k 31.8 -> 26.0,
// 1 M 938 -> 859; 128, 40 k 53.2 -> 42.7; D-PSGD of 96, 10 k 17.5 -> 14.5, 1 M 707 -> 639 (but, where operands spread over four decades go to
// float64, 90, K = 2, d = 100 k 273 -> 420), but the DeTAG step of 80, 20 k 23.1 -> 24.0, of 96,
// 8 k 12.4 -> 14.4, 300 k 224 -> 234, only the shortest of these better (96, 3000 11.7 -> 10.9, K = 1, 700 12.8 -> 11.4); 64, 10 k 12.9 -> 11.0,
// 100 k 55.4 -> 54.4, but 300 k 150 -> 160 (rows in pieces of 128 bytes): up to 64 workers therefore calls whose blocks have at most 32 chunks of
// 32 coordinates to do.  What would run as rounds otherwise runs here if rows_beat_rounds says so.  Block-circulant
// matrices beyond 160 workers come here while P is dense and calls are not long (lanes as coordinates -> here: 256-ring, K = 40, d = 4 k
// 34.6 -> 21.9, 60 k 263 -> 233, 16 x 16 torus, K = 9, 10 k 65 -> 49, 60 k 197 -> 186, but 100 k 303 -> 310, 189 k 554 -> 600; 224, 60 k 171 -> 166, but 75 k 195 -> 205;
// 192, 19 k 62 -> 58, but 60 k 134 -> 145; D-PSGD, 14 k 56 -> 46, but 18 k 57 -> 58), all with a chunk per block at most.
bool rows_ok(const detag_state* s, const StepParams& p) {
  if (s->rows.weights.empty()) return false;
  if (p.mode == detag::kModeExternal) return detag::rows_take_external(s->rows) && rows_beat_rounds(s, p.mode, s->sm_count);
  const double turns = std::ceil(static_cast<double>(s->d) / (32.0 * s->sm_count));
  if (p.n <= 64) return turns <= 32.0 || s->split.weights.empty();
  if (p.n > 96 && p.n <= 128) return !(p.mode == detag::kModeDetag && p.grad_at_start != 0 && long_calls(s, s->sm_count) && !s->split.weights.empty());
  if (p.n <= 128) return p.mode == detag::kModeDpsgd ? turns <= 1.0 || s->rows.unequal < 0.04f : s->d <= 24LL * s->sm_count;
  if (s->split.weights.empty()) return rows_beat_rounds(s, p.mode, s->sm_count);
  const bool dense = s->rows.use.count[0] + s->rows.use.count[1] == 2 * ((p.n + 31) / 32);
  // two chunks a block are one slab of 64 coordinates there (12 x 16 torus, d = 4863 24.0 against 27.5, but 256-ring, K = 40, d = 9 k 85 -> 38)
  if (p.n <= 192 && turns > 1.0 && turns <= 2.0) return false;
  return turns <= (p.n <= 160 || !dense ? 1.0 : p.mode == detag::kModeDpsgd ? 3.0 : p.n <= 192 ? 6.0 : 13.0);
}

// Up to 16 workers the step runs in registers, without staging.  us per step, tensor-path kernel with its stages and barriers
// -> that one: 8 workers, d = 8 M 1005 -> 327; 12, d = 4 M 565 -> 273; 13, d = 4 M 565 -> 350; 16, d = 4 M 568 -> 378, d = 270 k
// 47 -> 29; caller-written gradients, 16, d = 4 M 415 -> 321, d = 270 k 34.9 -> 24.9.  The failure-detection self test wants
// bounded waits, of which that kernel has none: it runs the tensor-path kernel.
bool small_ok(const StepParams& p) {
  return p.n <= detag::kMaxSmallWorkers && p.stall_after < 0;
}

// Groups of warps with a slab each take the dense product of 17 to 48 workers, in all modes, and where the choice is the
// library's what the rounds would run there (caller-written gradients and D-PSGD beyond 32).  us per step, the kernel with
// padded tiles (up to 32) or the integer tensor path -> that one: 17 workers, d = 3 M 582 -> 340; 24 569 -> 414; 28 572 -> 531; 32
// 600 -> 580, d = 25.6 M 5030 -> 4805, printed timing, d = 3 M 790 -> 578; 33, d = 1 M 411 -> 272; 40 427 -> 292; 48 430 -> 393; D-PSGD
// of 32, d = 3 M 415 -> 405, of 48, d = 1 M 444 -> 265; caller-written gradients of 24, d = 3 M 448 -> 410, of 48, d = 1 M 664 (rounds)
// -> 391.  But caller-written gradients of 28 470 -> 496, of 32 498 -> 535.  At every length: with one slab per SM the integer path is
// up to 0.25 us ahead (48, d = 9400 9.50 -> 9.67, D-PSGD 9.17 -> 7.69), but its sums are not the same bits, and a shard of the
// coordinates gives what the whole gives.
bool dense_step_ok(const detag_state* s, const StepParams& p, int variant) {
  if (p.n <= detag::kMaxSmallWorkers || p.n > detag::kMaxDenseStepWorkers || p.poly == nullptr || p.d > 0x7fffffffLL) return false;
  if (p.mode == detag::kModeExternal && p.n > 24 && p.n <= 32) return false;
  return variant == DETAG_VARIANT_DENSE || (variant == DETAG_VARIANT_CSR && s->variant_forced == DETAG_VARIANT_AUTO);
}

// Picks the kernel variant, plans it for the sizes in `p` and launches it.
int launch_step(detag_state* s, StepParams& p, cudaStream_t stream) {
  int e = 0;
  s->launched[0] = s->launched[1] = "";
  const int variant = resolve_variant(s);
  if (!variant_runs_mode(s, variant))
    return fail(s, DETAG_ERR_UNSUPPORTED,
                "this kernel variant runs the DeTAG step with the synthetic gradient only; use AUTO or CSR");
  if (p.mode != detag::kModeExternal && (!p.a || !p.c))
    return fail(s, DETAG_ERR_UNBOUND, "the synthetic gradient needs the objective arrays a and c");
  if (p.mode == detag::kModeExternal && !p.g_ext)
    return fail(s, DETAG_ERR_UNBOUND, "caller-written gradients selected but no gradient array given");
  if (dense_step_ok(s, p, variant)) {
    const detag::TensorMapSet* maps = maps_for(s, kFamilyDense, p);
    if (!maps) return fail(s, DETAG_ERR_CUDA, "tensor map encoding failed");
    s->launched[0] = "step_dense";
    e = detag::launch_step_dense(p, *maps, s->sm_count, stream);
    return e != 0 ? fail_cuda(s, e, "step kernel launch") : DETAG_OK;
  }
  if (split_ok(s, p, variant)) {
    const bool rows = rows_ok(s, p);
    if (rows || (!s->split.weights.empty() && p.mode != detag::kModeExternal))
      return launch_split(s, p, rows, variant == DETAG_VARIANT_CSR, stream);
  }
  // what the integer tensor path does not take although its variant promises it (a polynomial whose entries cannot be
  // scaled, e.g. under an absurd momentum) runs as rounds
  const bool as_rounds = (variant == DETAG_VARIANT_DENSE && p.n > 32) || (variant == DETAG_VARIANT_RING && !ring_band(s));
  switch (as_rounds ? DETAG_VARIANT_CSR : variant) {
    case DETAG_VARIANT_DENSE: {
      if (small_ok(p)) {
        s->launched[0] = "step_small";
        e = detag::launch_step_small(p, s->sm_count, stream);
        break;
      }
      const detag::TensorMapSet* maps = maps_for(s, kFamilyMma, p);
      if (!maps) return fail(s, DETAG_ERR_CUDA, "tensor map encoding failed");
      s->launched[0] = "step_mma";
      e = detag::launch_step_mma(p, *maps, s->sm_count, stream);
      break;
    }
    case DETAG_VARIANT_RING: {
      const long long d_main = p.d & ~63LL;
      if (d_main > 0) {
        StepParams pm = p;
        pm.d = d_main;
        const detag::TensorMapSet* maps = maps_for(s, kFamilyRing, pm);
        if (!maps) return fail(s, DETAG_ERR_CUDA, "tensor map encoding failed");
        s->launched[0] = "step_ring";
        e = detag::launch_step_ring(pm, *maps, s->band, s->sm_count, stream);
        if (e != 0) return fail_cuda(s, e, "step kernel launch");
      }
      if (d_main < p.d) {
        const int rc = launch_tail_columns(s, p, d_main, stream);
        if (rc != DETAG_OK) return rc;
      }
      break;
    }
    case DETAG_VARIANT_TORUS: {
      const detag::TensorMapSet* maps = maps_for(s, kFamilyTorus, p);
      if (!maps) return fail(s, DETAG_ERR_CUDA, "tensor map encoding failed");
      s->launched[0] = "step_torus";
      e = detag::launch_step_torus(p, *maps, p.torus, s->sm_count, stream);
      break;
    }
    case DETAG_VARIANT_CSR:
    default: {
      s->launched[0] = "step_csr";
      const int rc = detag::plan_step_csr(p, s->smem_optin);
      if (rc != DETAG_OK) return fail(s, rc, "graph too large for the shared-memory plan");
      e = detag::launch_step_csr(p, s->sm_count, stream);
    }
  }
  if (e != 0) return fail_cuda(s, e, "step kernel launch");
  return DETAG_OK;
}

}  // namespace

extern "C" {

int detag_create(detag_state** out, int n, int64_t d, const int32_t* row_ptr, const int32_t* col_idx,
                 const double* vals, int K, double eta, double alpha) {
  if (!out) return DETAG_ERR_ARG;
  *out = nullptr;
  if (n <= 0 || d <= 0 || K < 1 || !std::isfinite(alpha)) return DETAG_ERR_ARG;
  int rc = detag::validate_csr(n, row_ptr, col_idx, vals);
  if (rc != DETAG_OK) return rc;
  if (n > detag::kMaxWorkers) return DETAG_ERR_UNSUPPORTED;
  const int nnz = row_ptr[n];
  // doubly stochastic: every row and column sums to one
  std::vector<double> col_sum(n, 0.0);
  for (int i = 0; i < n; ++i) {
    double row_sum = 0.0;
    for (int k = row_ptr[i]; k < row_ptr[i + 1]; ++k) {
      row_sum += vals[k];
      col_sum[col_idx[k]] += vals[k];
    }
    if (std::fabs(row_sum - 1.0) > 1e-9) return DETAG_ERR_NOT_STOCHASTIC;
  }
  for (int j = 0; j < n; ++j)
    if (std::fabs(col_sum[j] - 1.0) > 1e-9) return DETAG_ERR_NOT_STOCHASTIC;

  if (std::isnan(eta)) {
    double lam = 0.0;
    rc = detag_spectral(n, row_ptr, col_idx, vals, nullptr, nullptr, &lam, &eta);
    if (rc != DETAG_OK) return rc;
  } else if (!std::isfinite(eta)) {
    return DETAG_ERR_ARG;
  }

  detag_state* s = new (std::nothrow) detag_state();
  if (!s) return DETAG_ERR_ARG;
  s->n = n;
  s->d = d;
  s->K = K;
  s->eta = eta;
  s->alpha = alpha;
  s->row_ptr.assign(row_ptr, row_ptr + n + 1);
  s->col_idx.assign(col_idx, col_idx + nnz);
  s->vals.assign(vals, vals + nnz);
  std::vector<double> poly;
  if (n <= 128) gossip_polynomial(s, poly);
  if (n <= 64) s->poly = poly;  // what the small kernels and the torus analysis use
  analyse_circulant(s);
  analyse_torus(s);
  if (n > detag::kMaxDenseStepWorkers && n <= detag::kMaxSplitWorkers) {
    // tables for whichever of the two kernels may be asked (rows_ok); those of step_rows.cu take 1 .. 3 ms to make beyond 128 workers
    // and are left out where no call would use them on a device of up to 160 SMs (256 workers, K = 4, d = 200 k 3.5 ms -> 0.05 and 0.85 MB less of
    // workspace)
    auto used = [&]() {
      return rows_beat_rounds(s, detag::kModeDetag, 160) || rows_beat_rounds(s, detag::kModeDpsgd, 160) ||
             (n <= 192 && rows_beat_rounds(s, detag::kModeExternal, 160));
    };
    const bool blocks = block_circulant(s);
    if (n > 128 && !blocks) s->reach = reached_blocks(s);
    const bool rows = n <= 128 || (blocks ? n <= 192 || d <= 13LL * 32 * 160 : used());
    if (blocks) {
      first_block_row(s, poly);
    } else if (n > 128 && rows) {
      gossip_polynomial(s, poly);
    }
    if (n <= 64 ? d > 32LL * 32 * 100 : n <= 96 || (n <= 128 ? long_calls(s, 100) : blocks)) detag::split_polynomial(n, poly, blocks, s->split);
    if (rows) detag::rows_polynomial(n, poly, blocks, s->split, s->rows);
    if (n > 128 && !blocks && !used()) s->rows = detag::SplitPoly{};
  }
  s->map_cache.reserve(8);
  // the workspace's tables as they are uploaded, the cleared status block in front
  const WsLayout l = ws_layout(s);
  s->image.assign(l.partials, 0);
  auto put = [&](size_t at, const void* src, size_t bytes) {
    if (bytes != 0) std::memcpy(&s->image[at], src, bytes);
  };
  put(l.row_ptr, s->row_ptr.data(), s->row_ptr.size() * sizeof(int32_t));
  put(l.col_idx, s->col_idx.data(), s->col_idx.size() * sizeof(int32_t));
  put(l.vals, s->vals.data(), s->vals.size() * sizeof(double));
  put(l.poly, s->poly.data(), s->poly.size() * sizeof(double));
  put(l.torus, s->torus_frag.data(), s->torus_frag.size() * sizeof(double));
  auto put_split = [&](const auto& at, const detag::SplitPoly& t) {
    put(at.weights, t.weights.data(), t.weights.size());
    put(at.row_exp, t.row_exp.data(), t.row_exp.size() * sizeof(int32_t));
    put(at.guard, t.guard.data(), t.guard.size());
    put(at.poly, t.poly.data(), t.poly.size() * sizeof(double));
  };
  put_split(l.split, s->split);
  put_split(l.rows, s->rows);
  *out = s;
  return DETAG_OK;
}

int detag_workspace_bytes(const detag_state* s, size_t* bytes) {
  if (!s || !bytes) return DETAG_ERR_ARG;
  *bytes = ws_layout(s).total;
  return DETAG_OK;
}

int detag_bind(detag_state* s, int64_t ld, float* x, float* y, float* g, const float* a, const float* c,
               void* workspace, size_t workspace_bytes) {
  if (!s) return DETAG_ERR_ARG;
  if (!x || !y || !g || !workspace) return fail(s, DETAG_ERR_ARG, "detag_bind: null buffer");
  if (ld < s->d || (ld & 3) != 0) return fail(s, DETAG_ERR_ARG, "detag_bind: ld must be >= d and a multiple of 4");
  if (!aligned16(x) || !aligned16(y) || !aligned16(g) || !aligned16(a) || !aligned16(c))  // NULL counts as aligned
    return fail(s, DETAG_ERR_ARG, "detag_bind: state arrays must be 16-byte aligned");
  if ((reinterpret_cast<uintptr_t>(workspace) % detag::kWsAlign) != 0)
    return fail(s, DETAG_ERR_ARG, "detag_bind: workspace must be 256-byte aligned");
  const WsLayout l = ws_layout(s);
  if (workspace_bytes < l.total) return fail(s, DETAG_ERR_ARG, "detag_bind: workspace too small");

  const int qrc = query_device(s);
  if (qrc != DETAG_OK) return qrc;
  cudaError_t e = cudaSuccess;

  unsigned char* base = static_cast<unsigned char*>(workspace);
  s->d_status = reinterpret_cast<int*>(base + l.status);
  s->d_result = reinterpret_cast<double*>(base + l.result);
  s->d_row_ptr = reinterpret_cast<int32_t*>(base + l.row_ptr);
  s->d_col_idx = reinterpret_cast<int32_t*>(base + l.col_idx);
  s->d_vals = reinterpret_cast<double*>(base + l.vals);
  s->d_poly = s->poly.empty() ? nullptr : reinterpret_cast<double*>(base + l.poly);
  s->d_torus = s->torus_frag.empty() ? nullptr : reinterpret_cast<double*>(base + l.torus);
  s->d_tables = base;
  s->d_partials = reinterpret_cast<double*>(base + l.partials);

  e = cudaMemcpy(base, s->image.data(), s->image.size(), cudaMemcpyHostToDevice);  // status word and result cleared
  if (e != cudaSuccess) return fail_cuda(s, e, "detag_bind: workspace upload");

  s->ld = ld;
  s->x = x;
  s->y = y;
  s->g = g;
  s->a = a;
  s->c = c;
  s->ws = workspace;
  s->ws_bytes = workspace_bytes;
  s->bound = true;
  return DETAG_OK;
}

int detag_observe_gossiped_tracker(detag_state* s, float* y_gossip) {
  if (!s) return DETAG_ERR_ARG;
  if (y_gossip && !aligned16(y_gossip)) return fail(s, DETAG_ERR_ARG, "observer buffer must be 16-byte aligned");
  s->y_obs = y_gossip;
  return DETAG_OK;
}

int detag_set_noise(detag_state* s, double sigma, uint64_t seed, int64_t coord_offset) {
  if (!s) return DETAG_ERR_ARG;
  if (!std::isfinite(sigma) || sigma < 0.0 || coord_offset < 0)
    return fail(s, DETAG_ERR_ARG, "detag_set_noise: bad value");
  s->sigma = sigma;
  s->seed = seed;
  s->coord_offset = coord_offset;
  return DETAG_OK;
}

int detag_set_variant(detag_state* s, int variant) {
  if (!s) return DETAG_ERR_ARG;
  switch (variant) {
    case DETAG_VARIANT_AUTO:
    case DETAG_VARIANT_CSR:
      break;
    case DETAG_VARIANT_DENSE:
      if (!dense_ok(s)) return fail(s, DETAG_ERR_UNSUPPORTED, "detag_set_variant: dense variant needs n <= 128");
      break;
    case DETAG_VARIANT_TORUS:
      if (!torus_ok(s))
        return fail(s, DETAG_ERR_UNSUPPORTED,
                    "detag_set_variant: torus variant needs n = 32 or 64 and a matrix that is block circulant in "
                    "8-worker blocks, symmetric in the block distance");
      break;
    case DETAG_VARIANT_RING:
      if (!band_ok(s))
        return fail(s, DETAG_ERR_UNSUPPORTED,
                    "detag_set_variant: ring variant needs a circulant matrix, n a multiple of 32, n >= 64, and K*bandwidth <= 16 or n <= 256");
      break;
    default:
      return fail(s, DETAG_ERR_ARG, "detag_set_variant: unknown variant");
  }
  s->variant_forced = variant;
  return DETAG_OK;
}

int detag_get_variant(const detag_state* s, int* variant) {
  if (!s || !variant) return DETAG_ERR_ARG;
  *variant = resolve_variant(s);
  return DETAG_OK;
}

int detag_set_gradient_point(detag_state* s, int where) {
  if (!s) return DETAG_ERR_ARG;
  if (where != DETAG_GRADIENT_AT_NEW_MODEL && where != DETAG_GRADIENT_AT_PHASE_START)
    return fail(s, DETAG_ERR_ARG, "detag_set_gradient_point: unknown value");
  s->gradient_point = where;
  return DETAG_OK;
}

int detag_get_gradient_point(const detag_state* s, int* where) {
  if (!s || !where) return DETAG_ERR_ARG;
  *where = s->gradient_point;
  return DETAG_OK;
}

int detag_set_algorithm(detag_state* s, int algorithm) {
  if (!s) return DETAG_ERR_ARG;
  if (algorithm != DETAG_ALGORITHM_DETAG && algorithm != DETAG_ALGORITHM_DPSGD)
    return fail(s, DETAG_ERR_ARG, "detag_set_algorithm: unknown value");
  if (algorithm == DETAG_ALGORITHM_DPSGD && s->gradient_source == DETAG_GRADIENT_EXTERNAL)
    return fail(s, DETAG_ERR_UNSUPPORTED, "detag_set_algorithm: D-PSGD runs with the synthetic gradient only");
  s->algorithm = algorithm;
  return DETAG_OK;
}

int detag_get_algorithm(const detag_state* s, int* algorithm) {
  if (!s || !algorithm) return DETAG_ERR_ARG;
  *algorithm = s->algorithm;
  return DETAG_OK;
}

int detag_set_gradient_source(detag_state* s, int source, const float* g_new) {
  if (!s) return DETAG_ERR_ARG;
  if (source == DETAG_GRADIENT_SYNTHETIC) {
    s->gradient_source = source;
    s->g_ext = nullptr;
    return DETAG_OK;
  }
  if (source != DETAG_GRADIENT_EXTERNAL) return fail(s, DETAG_ERR_ARG, "detag_set_gradient_source: unknown value");
  if (!g_new || !aligned16(g_new))
    return fail(s, DETAG_ERR_ARG, "detag_set_gradient_source: the gradient array must be non-null and 16-byte aligned");
  if (s->algorithm == DETAG_ALGORITHM_DPSGD)
    return fail(s, DETAG_ERR_UNSUPPORTED, "detag_set_gradient_source: D-PSGD runs with the synthetic gradient only");
  s->gradient_source = source;
  s->g_ext = g_new;
  return DETAG_OK;
}

int detag_debug_inject_stall(detag_state* s, int64_t after_tiles, uint32_t poll_limit) {
  if (!s) return DETAG_ERR_ARG;
  if (after_tiles < 0) {  // back to normal
    s->stall_after = -1;
    s->spin_limit = 1u << 20;
    return DETAG_OK;
  }
  if (poll_limit < 16 || poll_limit > (1u << 20))
    return fail(s, DETAG_ERR_ARG, "detag_debug_inject_stall: poll limit outside [16, 2^20]");
  s->stall_after = after_tiles;
  s->spin_limit = poll_limit;
  return DETAG_OK;
}

int detag_debug_expire_wait(detag_state* s, uint32_t polls, void* stream) {
  if (!s) return DETAG_ERR_ARG;
  if (!s->bound) return fail(s, DETAG_ERR_UNBOUND, "detag_debug_expire_wait before detag_bind");
  if (polls < 1 || polls > (1u << 20)) return fail(s, DETAG_ERR_ARG, "detag_debug_expire_wait: polls outside [1, 2^20]");
  const int e = detag::launch_expire_wait(s->d_status, polls, static_cast<cudaStream_t>(stream));
  if (e != 0) return fail_cuda(s, e, "detag_debug_expire_wait launch");
  return DETAG_OK;
}

int detag_phase_length(int n, double lambda, double varsigma0_sq, double T, double delta_L, int* R) {
  if (!R || n < 1 || !(lambda >= 0.0) || !(lambda < 1.0)) return DETAG_ERR_ARG;
  double num = 0.5 * std::log(static_cast<double>(n));
  if (varsigma0_sq > 0.0 && T > 0.0 && delta_L > 0.0) {
    const double second = 0.5 * std::log(varsigma0_sq * T / delta_L);
    if (second > num) num = second;
  }
  const double r = std::ceil(num / std::sqrt(1.0 - lambda));
  *R = r < 1.0 ? 1 : (r > 2147483647.0 ? 2147483647 : static_cast<int>(r));
  return DETAG_OK;
}

int detag_init(detag_state* s, void* stream) {
  if (!s) return DETAG_ERR_ARG;
  if (!s->bound) return fail(s, DETAG_ERR_UNBOUND, "detag_init before detag_bind");
  StepParams p = make_params(s);
  p.t_noise = 0;
  int e;
  if (p.mode == detag::kModeExternal) {
    if (!p.g_ext) return fail(s, DETAG_ERR_UNBOUND, "caller-written gradients selected but no gradient array given");
    e = detag::launch_init_external(p, s->sm_count, static_cast<cudaStream_t>(stream));
  } else {
    if (!p.a || !p.c) return fail(s, DETAG_ERR_UNBOUND, "the synthetic gradient needs the objective arrays a and c");
    e = detag::launch_init_gradient(p, s->sm_count, static_cast<cudaStream_t>(stream));
  }
  if (e != 0) return fail_cuda(s, e, "detag_init launch");
  s->t = 0;
  return DETAG_OK;
}

int detag_step(detag_state* s, void* stream) {
  if (!s) return DETAG_ERR_ARG;
  if (!s->bound) return fail(s, DETAG_ERR_UNBOUND, "detag_step before detag_bind");
  StepParams p = make_params(s);
  p.t_noise = static_cast<uint32_t>(s->t + 1);
  const int rc = launch_step(s, p, static_cast<cudaStream_t>(stream));
  if (rc != DETAG_OK) return rc;
  s->t += 1;
  return DETAG_OK;
}

int detag_step_many(detag_state* s, int count, void* stream) {
  if (!s) return DETAG_ERR_ARG;
  if (count < 1) return fail(s, DETAG_ERR_ARG, "detag_step_many: count must be at least 1");
  if (!s->bound) return fail(s, DETAG_ERR_UNBOUND, "detag_step_many before detag_bind");
  if (count >= 2 && step_mode(s) == detag::kModeExternal)
    return fail(s, DETAG_ERR_ARG, "detag_step_many: caller-written gradients need one call per step");
  // the fused kernels exist for the dense polynomial with n <= 32; the observer wants every step's tracker
  if (count >= 2 && resolve_variant(s) == DETAG_VARIANT_DENSE && s->n <= 32 && s->y_obs == nullptr &&
      step_mode(s) == detag::kModeDetag) {
    // A launch is cut off at kMaxFusedSteps so that no thread of the kernel waits on a peer for longer than its
    // bounded waits allow (a tile of 1024 steps takes some tens of milliseconds; the waits give up after seconds).
    constexpr int kMaxFusedSteps = 1024;
    for (int done = 0; done < count;) {
      const int now = count - done < kMaxFusedSteps ? count - done : kMaxFusedSteps;
      StepParams p = make_params(s);
      p.t_noise = static_cast<uint32_t>(s->t + 1);
      p.steps = now;
      if (!p.a || !p.c) return fail(s, DETAG_ERR_UNBOUND, "the synthetic gradient needs the objective arrays a and c");
      int e;
      s->launched[1] = "";
      if (small_ok(p)) {
        s->launched[0] = "step_small";
        e = detag::launch_step_small(p, s->sm_count, static_cast<cudaStream_t>(stream));
      } else {
        // Groups of four warps take a slab's steps in turn; the kernel with padded tiles puts eight warps on one, which is ahead
        // while there are at most two slabs per SM, and where nothing is padded beyond three, which the groups take side by side and
        // its two in two turns.  us, padded -> groups, for ten steps: 17 workers, d = 9000 26.6 -> 22.5, d = 72 k 127 -> 71; 24, d = 9000
        // 26.6 -> 23.9; 28, d = 18 k 39.0 -> 41.0, d = 36 k 68 -> 59; for twenty: 28, d = 1 M 3044 -> 2790; 32, d = 25 k 103 -> 97,
        // d = 30 k 122 -> 124, d = 45 k 162 -> 179, d = 60 k 220 -> 217, d = 150 k 473 -> 486, d = 1 M 3077 -> 3171; printed timing,
        // d = 150 k 482 -> 491.
        // (At most 16 get here for the self test of failure detection.)
        const bool padded = p.n <= detag::kMaxSmallWorkers || (p.n > 24 && p.d <= 128LL * s->sm_count) || (p.n > 28 && p.d > 192LL * s->sm_count);
        const detag::TensorMapSet* maps = maps_for(s, padded ? kFamilyMma : kFamilyDense, p);
        if (!maps) return fail(s, DETAG_ERR_CUDA, "tensor map encoding failed");
        s->launched[0] = padded ? "step_mma_many" : "step_dense";
        e = padded ? detag::launch_step_mma_many(p, *maps, s->sm_count, static_cast<cudaStream_t>(stream))
                   : detag::launch_step_dense_many(p, *maps, s->sm_count, static_cast<cudaStream_t>(stream));
      }
      if (e != 0) return fail_cuda(s, e, "detag_step_many launch");
      s->t += now;
      done += now;
    }
    return DETAG_OK;
  }
  for (int i = 0; i < count; ++i) {
    const int rc = detag_step(s, stream);
    if (rc != DETAG_OK) return rc;
  }
  return DETAG_OK;
}

int detag_host_staging_bytes(const detag_state* s, int64_t chunk_coords, size_t* bytes) {
  if (!s || !bytes || chunk_coords < 128 || (chunk_coords % 128) != 0) return DETAG_ERR_ARG;
  *bytes = ws_layout(s).total + static_cast<size_t>(2) * 5 * s->n * static_cast<size_t>(chunk_coords) * sizeof(float);
  return DETAG_OK;
}

int detag_step_host(detag_state* s, int64_t ld_host, float* x, float* y, float* g, const float* a, const float* c,
                    void* staging, size_t staging_bytes, void* stream) {
  if (!s) return DETAG_ERR_ARG;
  if (!x || !y || !g || !a || !c || !staging) return fail(s, DETAG_ERR_ARG, "detag_step_host: null buffer");
  if (step_mode(s) == detag::kModeExternal)
    return fail(s, DETAG_ERR_UNSUPPORTED, "detag_step_host: caller-written gradients are not offered on host-resident state");
  if (ld_host < s->d) return fail(s, DETAG_ERR_ARG, "detag_step_host: ld_host < d");
  if ((reinterpret_cast<uintptr_t>(staging) % detag::kWsAlign) != 0)
    return fail(s, DETAG_ERR_ARG, "detag_step_host: staging must be 256-byte aligned");
  const WsLayout l = ws_layout(s);
  const size_t per_coord = static_cast<size_t>(2) * 5 * s->n * sizeof(float);
  if (staging_bytes < l.total + per_coord * 128)
    return fail(s, DETAG_ERR_ARG, "detag_step_host: staging too small for a 128-coordinate chunk");
  long long chunk = static_cast<long long>((staging_bytes - l.total) / per_coord) / 128 * 128;
  const long long d_up = (s->d + 127) / 128 * 128;
  if (chunk > d_up) chunk = d_up;

  int rc = query_device(s);
  if (rc != DETAG_OK) return rc;
  cudaError_t e = cudaSuccess;
  for (int k = 0; k < 2 && e == cudaSuccess; ++k)
    if (!s->host_stream[k]) e = cudaStreamCreateWithFlags(&s->host_stream[k], cudaStreamNonBlocking);
  for (int k = 0; k < 3 && e == cudaSuccess; ++k)
    if (!s->host_event[k]) e = cudaEventCreateWithFlags(&s->host_event[k], cudaEventDisableTiming);
  if (e != cudaSuccess) return fail_cuda(s, e, "detag_step_host: stream/event creation");

  cudaStream_t user = static_cast<cudaStream_t>(stream);
  unsigned char* base = static_cast<unsigned char*>(staging);
  // Graph tables at the head of the staging area, ordered on the caller's stream.  The status word there is
  // cleared when a staging area is first used, not on every call: a time-out stays visible to detag_status.
  int* status_word = reinterpret_cast<int*>(base + l.status);
  const size_t skip = s->d_status_host != status_word ? 0 : l.row_ptr;
  s->d_status_host = status_word;
  e = cudaMemcpyAsync(base + skip, s->image.data() + skip, s->image.size() - skip, cudaMemcpyHostToDevice, user);
  if (e == cudaSuccess) e = cudaEventRecord(s->host_event[2], user);
  for (int k = 0; k < 2 && e == cudaSuccess; ++k) e = cudaStreamWaitEvent(s->host_stream[k], s->host_event[2], 0);
  if (e != cudaSuccess) return fail_cuda(s, e, "detag_step_host: table upload");

  StepParams p = make_params(s);
  p.row_ptr = reinterpret_cast<int32_t*>(base + l.row_ptr);
  p.col_idx = reinterpret_cast<int32_t*>(base + l.col_idx);
  p.vals = reinterpret_cast<double*>(base + l.vals);
  p.poly = s->poly.empty() ? nullptr : reinterpret_cast<double*>(base + l.poly);
  p.torus = s->torus_frag.empty() ? nullptr : reinterpret_cast<double*>(base + l.torus);
  p.tables = base;
  p.status = status_word;
  p.y_obs = nullptr;
  p.t_noise = static_cast<uint32_t>(s->t + 1);
  p.ld = chunk;
  float* slots = reinterpret_cast<float*>(base + l.total);
  const size_t arr = static_cast<size_t>(s->n) * chunk;  // elements of one staged array
  const size_t hp = static_cast<size_t>(ld_host) * sizeof(float), dp = static_cast<size_t>(chunk) * sizeof(float);

  long long k = 0;
  for (long long j0 = 0; j0 < s->d; j0 += chunk, ++k) {
    const long long w = (s->d - j0 < chunk) ? s->d - j0 : chunk;
    cudaStream_t st = s->host_stream[k & 1];
    float* sx = slots + (k & 1) * 5 * arr;
    float *sy = sx + arr, *sg = sy + arr, *sa = sg + arr, *sc = sa + arr;
    const size_t wb = static_cast<size_t>(w) * sizeof(float);
    e = cudaMemcpy2DAsync(sx, dp, x + j0, hp, wb, s->n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpy2DAsync(sy, dp, y + j0, hp, wb, s->n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpy2DAsync(sg, dp, g + j0, hp, wb, s->n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpy2DAsync(sa, dp, a + j0, hp, wb, s->n, cudaMemcpyHostToDevice, st);
    if (e == cudaSuccess) e = cudaMemcpy2DAsync(sc, dp, c + j0, hp, wb, s->n, cudaMemcpyHostToDevice, st);
    if (e != cudaSuccess) return fail_cuda(s, e, "detag_step_host: host-to-device copy");
    p.x = sx; p.y = sy; p.g = sg; p.a = sa; p.c = sc;
    p.d = w;
    p.coord_offset = s->coord_offset + j0;
    rc = launch_step(s, p, st);
    if (rc != DETAG_OK) return rc;
    e = cudaMemcpy2DAsync(x + j0, hp, sx, dp, wb, s->n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpy2DAsync(y + j0, hp, sy, dp, wb, s->n, cudaMemcpyDeviceToHost, st);
    if (e == cudaSuccess) e = cudaMemcpy2DAsync(g + j0, hp, sg, dp, wb, s->n, cudaMemcpyDeviceToHost, st);
    if (e != cudaSuccess) return fail_cuda(s, e, "detag_step_host: device-to-host copy");
  }
  for (int q = 0; q < 2 && e == cudaSuccess; ++q) {
    e = cudaEventRecord(s->host_event[q], s->host_stream[q]);
    if (e == cudaSuccess) e = cudaStreamWaitEvent(user, s->host_event[q], 0);
  }
  if (e != cudaSuccess) return fail_cuda(s, e, "detag_step_host: join");
  s->t += 1;
  return DETAG_OK;
}

int detag_consensus_error(detag_state* s, void* stream, double* host_out) {
  if (!s || !host_out) return DETAG_ERR_ARG;
  if (!s->bound) return fail(s, DETAG_ERR_UNBOUND, "detag_consensus_error before detag_bind");
  const StepParams p = make_params(s);
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  const int e = detag::launch_consensus_error(p, s->d_partials, s->d_result, s->sm_count, st);
  if (e != 0) return fail_cuda(s, e, "detag_consensus_error launch");
  cudaError_t ce = cudaMemcpyAsync(host_out, s->d_result, sizeof(double), cudaMemcpyDeviceToHost, st);
  if (ce == cudaSuccess) ce = cudaStreamSynchronize(st);
  if (ce != cudaSuccess) return fail_cuda(s, ce, "detag_consensus_error copy");
  return DETAG_OK;
}

int detag_get_step(const detag_state* s, int64_t* t) {
  if (!s || !t) return DETAG_ERR_ARG;
  *t = s->t;
  return DETAG_OK;
}

int detag_set_step(detag_state* s, int64_t t) {
  if (!s || t < 0) return DETAG_ERR_ARG;
  s->t = t;
  return DETAG_OK;
}

int detag_status(detag_state* s, void* stream) {
  if (!s) return DETAG_ERR_ARG;
  if (!s->bound && !s->d_status_host) return fail(s, DETAG_ERR_UNBOUND, "detag_status before detag_bind or detag_step_host");
  int word[2] = {0, 0};
  cudaStream_t st = static_cast<cudaStream_t>(stream);
  cudaError_t e = cudaSuccess;
  if (s->bound) e = cudaMemcpyAsync(&word[0], s->d_status, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess && s->d_status_host)
    e = cudaMemcpyAsync(&word[1], s->d_status_host, sizeof(int), cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return fail_cuda(s, e, "detag_status");
  if (word[0] == 2 || word[1] == 2) return fail(s, DETAG_ERR_CUDA, "a kernel found its shared or tensor memory misplaced");
  if (word[0] != 0 || word[1] != 0) return fail(s, DETAG_ERR_TIMEOUT, "a device-side wait gave up");
  s->d_status_host = nullptr;  // read and clean: the staging area is not referred to again until the next host step
  return DETAG_OK;
}

const char* detag_debug_kernel(const detag_state* s, int part) { return s && (part == 0 || part == 1) ? s->launched[part] : ""; }

const char* detag_last_error(const detag_state* s) { return s ? s->err.c_str() : ""; }

int detag_destroy(detag_state* s) {
  if (!s) return DETAG_ERR_ARG;
  for (int k = 0; k < 2; ++k)
    if (s->host_stream[k]) {
      cudaStreamSynchronize(s->host_stream[k]);
      cudaStreamDestroy(s->host_stream[k]);
    }
  for (int k = 0; k < 3; ++k)
    if (s->host_event[k]) cudaEventDestroy(s->host_event[k]);
  delete s;
  return DETAG_OK;
}

}  // extern "C"
