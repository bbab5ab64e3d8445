// Internal declarations shared by the host API and the kernel launchers of libdetag.
#ifndef DETAG_INTERNAL_H
#define DETAG_INTERNAL_H

#include <cstddef>
#include <cstdint>
#include <string>
#include <vector>

#include "detag.h"

typedef struct CUstream_st* cudaStream_t;

namespace detag {

constexpr int kMaxWorkers = 1024;       // detag_create limit on n
constexpr int kMaxDenseWorkers = 128;   // dense variant: limit on n
constexpr int kMaxSmallWorkers = 16;    // step in registers: limit on n
constexpr int kMaxDenseStepWorkers = 48;  // dense product, groups of warps: limit on n
constexpr int kMaxSplitWorkers = 256;   // integer tensor path: limit on n
constexpr int kMaxPartials = 2048;      // per-CTA partial sums of the consensus-error reduction
constexpr size_t kWsAlign = 256;

// Everything a step / init / reduction kernel needs, passed by value.
struct StepParams {
  int n;
  int nnz;
  int K;
  int S;           // slab width in coordinates (power of two)
  int log2S;
  int csr_sub;     // generic rounds kernel: independent pieces the slab is cut into
  int csr_threads; // generic rounds kernel: threads per block (1024, or 512 with two blocks per SM)
  long long d;
  long long ld;
  long long num_slabs;
  long long coord_offset;  // global index of column 0 (noise counter)
  float* x;
  float* y;
  float* g;
  const float* a;
  const float* c;
  float* y_obs;  // optional gossiped-tracker output, may be null
  const int32_t* row_ptr;
  const int32_t* col_idx;
  const double* vals;
  const double* poly;  // dense P_K(M), row-major n x n (null when n > 64)
  const unsigned char* tables;  // the workspace, for the integer tensor path's tables
  const double* torus; // block-circulant kernel: per-frequency 8 x 8 polynomial blocks in fragment order (or null)
  double eta;
  double alpha;
  double sigma;
  uint32_t round_key[20];  // Philox round keys of the noise seed (noise.cuh)
  uint32_t t_noise;  // step index that enters the noise counter
  int grad_at_start;  // nonzero: the gradient is taken at the model the step started from (Algorithm 2 as printed)
  int steps;          // consecutive steps in one launch (multi-step kernel only)
  int mode;           // kModeDetag, kModeExternal or kModeDpsgd
  const float* g_ext; // kModeExternal: the caller's newest stochastic gradient, [n][ld]
  unsigned spin_limit;    // polls after which a device-side wait gives up
  int operands_end, tails_end;  // step_dense.cu: slabs from here on are not asked for
  // This launch's columns are not the ones of the launch before it (the last columns of a band): it runs beside that one.  The launches
  // before that are complete when it starts, for that one has waited for them before it let this one begin (chain.cuh); it waits at
  // its end instead, so that whoever waits for it has waited for both.
  int beside;
  long long stall_after;  // failure-detection self test: a CTA's producer stops loading after this many tiles (< 0: off)
  int* status;
};

// What a step computes (the `mode` of StepParams)
constexpr int kModeDetag = 0;     // DeTAG with the library's own synthetic gradient (y holds the folded tracker)
constexpr int kModeExternal = 1;  // DeTAG with caller-written gradients: fold, gossip, model update; no gradient evaluation
constexpr int kModeDpsgd = 2;     // D-PSGD: x' = AG_K(x) - alpha g, g' = synthetic gradient at x'; no tracker

// Room for the tensor maps of one launch (eight 128-byte CUtensorMap objects), built once per set of bound
// buffers and kept in the state.
struct alignas(64) TensorMapSet {
  unsigned char bytes[8 * 128];
};

// Tiles (128 outputs x 32 inputs) of the polynomial that the MMAs take for either half of the outputs.
struct RowsTiles {
  uint32_t order[2], place[2];  // four bits each: input block; where it stays in tensor memory, 15: it travels
  int count[2], residents;
  unsigned char resident[4];    // half << 4 | input block
};

// P_K(M) as a kernel of the integer tensor path takes it: its base-256 digits, the exponent of every row's scale, the groups of
// inputs that tell when a coordinate's operands may share one scale, and P itself.  Empty when neither kernel takes the matrix.
struct SplitPoly {
  std::vector<unsigned char> weights;  // digits: tiles of 128 outputs x 32 inputs, or the distinct 32 x 32 blocks
  std::vector<int32_t> row_exp;
  std::vector<double> poly;  // in float64, padded; step_split.cu: transposed
  std::vector<uint8_t> guard;  // groups of guard_size inputs
  int guard_size;
  float unequal;           // share of coordinates (a bound) that stay in float64 when operands are spread over four decades
  float guard_tau;         // each group's largest operand must be at least this share of the coordinate's largest
  bool circulant;          // the 32 x 32 blocks depend on their distance only: `poly` holds output workers 0 .. 31
  unsigned char id[64];    // step_split.cu: [output block][input block] -> distinct block, 255: no digit of it is set
  RowsTiles use;           // step_rows.cu beyond 128 workers
  unsigned char reach[8];  // [32 outputs], a bit per input block: some entry of P is not zero
};

// host helpers (spectral.cpp)
int validate_csr(int n, const int32_t* row_ptr, const int32_t* col_idx, const double* vals);
void csr_to_dense(int n, const int32_t* row_ptr, const int32_t* col_idx, const double* vals, std::vector<double>& m);
bool is_symmetric(int n, const std::vector<double>& m, double tol);
void jacobi_eigenvalues(int n, std::vector<double>& a, std::vector<double>& ev);
double eta_from_lambda(double lam);

// kernel launchers; each returns a cudaError_t value as int (0 = success)
int launch_init_gradient(const StepParams& p, int sm_count, cudaStream_t stream);
int plan_step_csr(StepParams& p, int smem_optin_bytes);  // chooses S; DETAG_ERR_UNSUPPORTED if nothing fits
int launch_step_csr(const StepParams& p, int sm_count, cudaStream_t stream);
bool dense_variant_available(int n);  // n <= kMaxDenseWorkers and the driver offers tensor-map encoding
// Tensor-path kernels: build_* fills the tensor maps for the buffers in `p` (false: the driver refused one);
// launch_* takes the maps built for exactly those buffers.
bool build_maps_mma(const StepParams& p, TensorMapSet* maps);
int launch_step_mma(StepParams p, const TensorMapSet& maps, int sm_count, cudaStream_t stream);       // n <= 32
int launch_step_mma_many(StepParams p, const TensorMapSet& maps, int sm_count, cudaStream_t stream);  // p.steps steps
// circulant kernel (step_ring.cu): n % 32 == 0, 64 <= n <= 1024, half-band <= 16
bool ring_variant_available(int n, int half_band);
bool build_maps_ring(const StepParams& p, TensorMapSet* maps);  // p.d a multiple of 64
int launch_step_ring(StepParams p, const TensorMapSet& maps, const double* band, int sm_count, cudaStream_t stream);
bool torus_variant_available(int n);               // block-circulant kernel: n = 32 or 64 (4 or 8 blocks of 8)
bool build_maps_torus(const StepParams& p, TensorMapSet* maps);
int launch_step_torus(StepParams p, const TensorMapSet& maps, const double* phat_frag /* device */, int sm_count,
                      cudaStream_t stream);
// the step in registers (step_small.cu): n <= 16, all modes; p.steps iterations
int launch_step_small(const StepParams& p, int sm_count, cudaStream_t stream);
// dense product, groups of warps with a slab each (step_dense.cu): 16 < n <= 48, all modes
bool build_maps_dense(const StepParams& p, TensorMapSet* maps);
int launch_step_dense(const StepParams& p, const TensorMapSet& maps, int sm_count, cudaStream_t stream);
int launch_step_dense_many(const StepParams& p, const TensorMapSet& maps, int sm_count, cudaStream_t stream);  // n <= 32, p.steps steps
// polynomial on the integer tensor path, 48 < n <= 256
void split_guard(int n, const std::vector<double>& poly, int rows, SplitPoly& out);
bool split_digits(int n, const std::vector<double>& poly, int rows, int wide, std::vector<int64_t>& digits, std::vector<int32_t>& row_exp);
struct SplitDevice {  // the tables of a SplitPoly in the workspace
  const void* weights;
  const int32_t* row_exp;
  const uint8_t* guard;
  const double* poly;
};
// step_split.cu: lanes are coordinates; the distinct blocks have to fit in shared memory
void split_polynomial(int n, const std::vector<double>& poly, bool circulant, SplitPoly& out);
bool build_maps_split(const StepParams& p, TensorMapSet* maps);
int launch_step_split(StepParams p, const TensorMapSet& maps, const SplitPoly& poly, const SplitDevice& tables,
                      bool wide_gradient, int sm_count, cudaStream_t stream);
// step_rows.cu: lanes are output workers; any matrix
void rows_polynomial(int n, const std::vector<double>& poly, bool circulant, const SplitPoly& other, SplitPoly& out);
bool rows_take_external(const SplitPoly& poly);
bool build_maps_rows(const StepParams& p, TensorMapSet* maps);
int launch_step_rows(StepParams p, const TensorMapSet& maps, const SplitPoly& poly, const SplitDevice& tables,
                     bool wide_gradient, int sm_count, cudaStream_t stream);
int launch_consensus_error(const StepParams& p, double* partials, double* result, int sm_count, cudaStream_t stream);
int launch_init_external(const StepParams& p, int sm_count, cudaStream_t stream);  // y = g = g_ext
int launch_expire_wait(int* status, unsigned polls, cudaStream_t stream);          // a wait nobody ends (self test)
// cudaFuncSetAttribute(MaxDynamicSharedMemorySize) once per kernel and device; returns a cudaError_t value.
int ensure_dynamic_smem(const void* kernel, int bytes);

}  // namespace detag

struct detag_state {
  int n = 0;
  long long d = 0;
  int K = 0;
  double eta = 0.0, alpha = 0.0;
  std::vector<int32_t> row_ptr, col_idx;
  std::vector<double> vals;
  std::vector<double> poly;  // P_K(M) when n <= 64
  bool circulant = false;    // every row of M is the previous one shifted by one
  int half_band = 0;         // of the circulant P_K(M): P[i][(i+delta) mod n] = 0 for |delta| > half_band
  double band[33] = {0};     // p(delta) at index delta + 16, valid when circulant and half_band <= 16
  std::vector<double> circ_row;  // first row of the circulant P_K(M) (kept when n <= kMaxSplitWorkers)
  // block-circulant structure with 8-worker blocks, symmetric in the block distance (tori): the per-frequency
  // 8 x 8 polynomial blocks in MMA fragment order
  bool torus = false;
  std::vector<double> torus_frag;
  detag::SplitPoly split, rows;   // 48 < n <= 256: P_K(M) for the integer tensor path's two kernels (empty: not taken)
  double reach = 0.0;             // of unstructured matrices beyond 128 workers: blocks of P_K(M) reached per 32 rows
  std::vector<unsigned char> image;  // the workspace up to the partial sums, as it is uploaded
  int variant_forced = DETAG_VARIANT_AUTO;
  int gradient_point = DETAG_GRADIENT_AT_NEW_MODEL;
  int algorithm = DETAG_ALGORITHM_DETAG;
  int gradient_source = DETAG_GRADIENT_SYNTHETIC;
  const float* g_ext = nullptr;
  unsigned spin_limit = 1u << 20;
  long long stall_after = -1;
  const char* launched[2] = {"", ""};  // detag_debug_kernel

  bool bound = false;
  long long ld = 0;
  float *x = nullptr, *y = nullptr, *g = nullptr;
  const float *a = nullptr, *c = nullptr;
  float* y_obs = nullptr;
  void* ws = nullptr;
  size_t ws_bytes = 0;
  int* d_status = nullptr;
  int* d_status_host = nullptr;  // status word of the staging area the last detag_step_host used
  double* d_result = nullptr;
  int32_t* d_row_ptr = nullptr;
  int32_t* d_col_idx = nullptr;
  double* d_vals = nullptr;
  double* d_poly = nullptr;
  double* d_torus = nullptr;
  const unsigned char* d_tables = nullptr;  // the workspace's beginning
  double* d_partials = nullptr;

  double sigma = 0.0;
  uint64_t seed = 0;
  long long coord_offset = 0;
  long long t = 0;

  // host-resident stepping: two internal streams and their events, created on first use
  cudaStream_t host_stream[2] = {nullptr, nullptr};
  struct CUevent_st* host_event[3] = {nullptr, nullptr, nullptr};

  // tensor maps of the launches seen so far, keyed by kernel family and buffers (a few entries, round robin)
  struct MapEntry {
    int family = 0;
    const void* ptr[5] = {nullptr, nullptr, nullptr, nullptr, nullptr};
    long long d = 0, ld = 0;
    detag::TensorMapSet maps;
  };
  std::vector<MapEntry> map_cache;
  size_t map_next = 0;

  int device = -1;
  int sm_count = 0;
  int smem_optin = 0;
  std::string err;
};

#endif  // DETAG_INTERNAL_H
