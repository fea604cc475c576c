// Launchers of the sm_103a kernels (host-callable, C++ linkage).
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>

#include <nvtx3/nvToolsExt.h>

#include "qt.h"

namespace qt {

// NVTX range for profilers (ncu --nvtx, nsys): a named span of host work and the
// launches it makes; costs a few ns when no tool is attached.
struct TraceRange {
  explicit TraceRange(const char* name) { nvtxRangePushA(name); }
  ~TraceRange() { nvtxRangePop(); }
  TraceRange(const TraceRange&) = delete;
  TraceRange& operator=(const TraceRange&) = delete;
};

// A launch parameter that depends on the device (SM count, occupancy, a
// kernel attribute set once): computed by f() the first time it is asked for
// with a given device current, then reused for that device.  f() must be
// idempotent (two threads may both compute it the first time).
class PerDevice {
 public:
  template <typename F>
  int get(F&& f) {
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return f();
    const int v = vals_[dev].load(std::memory_order_acquire);
    if (v != 0) return v - 1;
    const int r = f();
    vals_[dev].store(r + 1, std::memory_order_release);
    return r;
  }

 private:
  static constexpr int kMaxDevices = 64;
  std::atomic<int> vals_[kMaxDevices] = {};
};

// ---- device scratch sizes -------------------------------------------------
constexpr int kRedThreads = 256;          // threads of the reduction kernels
constexpr int kMaxRedBlocks = 152 * 8;    // upper bound of their grid
constexpr int kRdmMaxQ = 3;               // reduced density matrix: q <= 3
constexpr int kRdmMaxReals = 64;          // longest rdm result row
constexpr int kResultDoubles = 64;
constexpr int kPartialDoubles = kMaxRedBlocks * 64;
constexpr int kExpGroup = 16;             // Z masks per expectation pass
// CDF for sampling: chunk = 64 amplitudes (one warp, 128-bit loads),
// sub-block = 16 chunks, block = 64 sub-blocks
constexpr int kCdfChunkLog = 6, kCdfSubLog = 10, kCdfBlkLog = 16;

inline uint64_t cdf_num_sub(int n) { return ((1ull << n) + (1ull << kCdfSubLog) - 1) >> kCdfSubLog; }
inline uint64_t cdf_num_blk(int n) { return (cdf_num_sub(n) + 63) >> 6; }

constexpr float kRangeDown = 0x1p-64f;    // 2^34 amplitudes of 2^127 stay finite
struct Scratch {
  double* partial = nullptr;   // kPartialDoubles doubles (held as that many double-floats)
  double* result = nullptr;    // kResultDoubles doubles
  float* cdf_sub = nullptr;    // cdf_num_sub(n) floats
  double* cdf_cum = nullptr;   // cdf_num_blk(n) doubles
  // factor of the FP32 runs at their carry (a power of two): the results of
  // launch_rdm, launch_expect and launch_kraus_norms come out times it.
  // Double-floats have FP32's range, so the sums of a caller's state of norm^2
  // beyond 2^128 need kRangeDown
  float down = 1.f;
  float2* partials() const { return reinterpret_cast<float2*>(partial); }
};

// ---- kernels ---------------------------------------------------------------
// state <- U (2^k x 2^k row-major complex64, basis `targets` sorted ascending)
cudaError_t launch_apply(float2* psi, int n, int k, const uint32_t* targets, const float2* U,
                         cudaStream_t st);
// rho (the 4^q reals that rdm_unpack takes) of qubits Q into scr.result
cudaError_t launch_rdm(const float2* psi, int n, int q, const uint32_t* qubits, const Scratch& scr,
                       cudaStream_t st);
// the same on the host (blocks), where a density beyond FP32's range is read
// a second time with kRangeDown
cudaError_t read_rdm(const float2* psi, int n, int q, const uint32_t* qubits, Scratch scr, cudaStream_t st, double* r);
// Channels on 4 or 5 qubits, at least 2^kGramMinLog gather sets: P_i =
// <psi|K_i^dag K_i|psi> of nops operators.  scratch (kraus_scratch_bytes(q,
// nops) bytes of device memory, 16-byte aligned) begins with the results,
// nops x kraus_slices(q) doubles: the last kraus_error_slices(q) of row i sum
// to E_i^2 and the others to P_i, which is only good if E_i <= P_i (see
// k_kraus_trace).  From
// kraus_results(q, nops) doubles on come the operators as kraus_sort_columns writes them (K
// row-major (re, im) FP64, basis bit b <-> qubits[b]; 4^q complex64 each)
constexpr int kGramMinLog = 18;
inline bool kraus_by_gram(int n, int q) { return q <= 5 && n - q >= kGramMinLog; }
int kraus_slices(int q);
int kraus_error_slices(int q);
size_t kraus_results(int q, int nops);
size_t kraus_scratch_bytes(int q, int nops);
void kraus_sort_columns(int q, const uint32_t* qubits, const double* K, float2* out);
cudaError_t launch_kraus_probs(const float2* psi, int n, int q, const uint32_t* qubits, int nops, void* scratch,
                               cudaStream_t st);
// The other channels on 4..6 qubits, and operators that the above leaves: N and P_i = |K_i psi|^2 for kraus_group(q)
// operators (16, 4, 1 for q = 4, 5, 6; pad with zero matrices) into
// scr.result[0] (N) and scr.result[1..]; ops_dev: the operators, 2^q x 2^q
// row-major complex64 in device memory, basis bit b <-> qubits[b]
int kraus_group(int q);
cudaError_t launch_kraus_norms(const float2* psi, int n, int q, const uint32_t* qubits, int nops,
                               const float2* ops_dev, const Scratch& scr, cudaStream_t st);
// N = <psi|psi> and sum |psi_x|^2 (-1)^popc(x&mask) for nm <= 16 masks into scr.result[0..nm]
cudaError_t launch_expect(const float2* psi, int n, int nm, const uint64_t* masks,
                          const Scratch& scr, cudaStream_t st);
// S samples of trajectory traj into out (device)
cudaError_t launch_sample(const float2* psi, int n, uint64_t seed, uint64_t traj, uint32_t S,
                          uint64_t* out, const Scratch& scr, cudaStream_t st, const double* readout = nullptr);
// C(x) of every x as the sampler forms it (2^n doubles into out, device)
cudaError_t launch_cdf_values(const float2* psi, int n, const Scratch& scr, double* out, cudaStream_t st);
// 6-qubit fused gate on CUDA cores (FP32), matrix 64x64 row-major in device memory, n >= 13
cudaError_t launch_apply6_fp32(float2* psi, int n, const uint32_t* targets, const float2* udev, cudaStream_t st);
// per-block sums of |psi|^2 and |K psi|^2 (two double-floats a block) for one
// 64 x 64 operator (basis bit b <-> qubits[b]), n >= 6, times `down`
cudaError_t launch_norms64(const float2* psi, int n, const uint32_t* qubits, const float2* kdev, float down,
                           float2* partial, int* blocks, cudaStream_t st);
// multi-gate pass: up to kMultiGates fused gates (width <= 4, n >= 7 + width,
// targets ascending, matrix row-major) whose qubits, with the lowest kMultiLow,
// number at most kMultiBits, applied in order in one pass over the state;
// multi_fits: whether they are
constexpr int kMultiBits = 12, kMultiLow = 4, kMultiGates = 48, kMultiEntries = 2176;
constexpr int kMultiFewLog = 12;
struct MultiPiece {
  int k;
  uint32_t targets[4];
  const float2* u;
};
bool multi_fits(int n, int ng, const MultiPiece* pieces);
cudaError_t launch_multi(float2* psi, int n, int ng, const MultiPiece* pieces, cudaStream_t st);
// tensor-core path (split-TF32, k = 4..6, n >= k + 7): W is the real
// embedding of U, row-major [2^(k+1) x 2^(k+1)] FP32 in device memory; *err
// is set (nonzero) if a bounded wait in the kernel ran out
bool tc_supported(int n, int k);
cudaError_t launch_apply_tc(float2* psi, int n, int k, const uint32_t* targets, const float* wdev, int* err,
                            cudaStream_t st, uint32_t lbo = 0, uint32_t sbo = 0);
void real_embedding(int k, const float2* U, float* W);
// |0...0>
cudaError_t launch_init_state(float2* psi, int n, cudaStream_t st);
// Product-state preparation: psi[x] = H[x >> m] * L[x mod 2^m], each table the
// product of factor columns (U |0> of a fused gate on its own qubits) on the
// qubits below m (L) or from m up (H); qubits no factor holds are |0>.
constexpr int kFoldMax = 32;          // factors per table
constexpr int kFoldVals = 1024;       // factor values per table
constexpr int kFoldTableBits = 20;    // largest table: 2^20 entries
struct FoldSpec {
  float2 v[kFoldVals];                // factor columns, concatenated
  uint16_t off[kFoldMax];             // offset of factor f's 2^w values in v
  uint8_t w[kFoldMax];                // factor width (1..6)
  uint8_t q[kFoldMax][6];             // qubit of index bit b of factor f, relative to the table
  uint64_t zmask;                     // table bits that no factor holds (must be 0)
  int nf;                             // factors
};
// tables: 2^m + 2^(n-m) complex64 of device scratch; 1 <= m, n - m <= 20
cudaError_t launch_init_product(float2* psi, int n, int m, const FoldSpec& lo, const FoldSpec& hi,
                                float2* tables, cudaStream_t st);
// psi *= f
cudaError_t launch_scale(float2* psi, int n, float f, cudaStream_t st);

// unpack the reals of an rdm result into a row-major complex matrix
// rho[b][a] = sum psi_b conj(psi_a), basis bit b <-> qubits[b]
void rdm_unpack(int q, const uint32_t* qubits, const double* r, double* rho_interleaved);

int sm_count();
// binaryVersion / ptxVersion of the library's kernels on the current device
cudaError_t kernel_arch(int* binary_version, int* ptx_version);

}  // namespace qt
