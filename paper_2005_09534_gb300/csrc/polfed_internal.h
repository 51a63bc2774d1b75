// Internal declarations of the POLFED GB300 library (not part of the ABI).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/polfed.h"

namespace polfed {

// ----------------------------------------------------------------- errors
struct Error {
  int code;
  std::string msg;
};
void set_error(int code, const std::string& msg);
int fail(int code, const std::string& msg);  // set_error + return code
void clear_error();                          // an entry point starts with an empty message

#define PF_CUDA(call)                                                                          \
  do {                                                                                         \
    cudaError_t e_ = (call);                                                                   \
    if (e_ != cudaSuccess)                                                                     \
      return ::polfed::fail(POLFED_ECUDA, std::string(#call) + ": " + cudaGetErrorString(e_)); \
  } while (0)

#define PF_CHECK(call)          \
  do {                          \
    int rc_ = (call);           \
    if (rc_ != POLFED_OK) return rc_; \
  } while (0)

// ------------------------------------------------------------- counters
// Process-wide counters of kernel launches and of the step kernel's device
// time (CUDA events on the launching stream); calls report their deltas.
struct Counters {
  int64_t launches = 0;
  // step-kernel launches inside CUDA-event-timed runs (see StepTimer), in all
  // and by storage kind (index POLFED_F64 / POLFED_F32 / POLFED_DF64)
  int64_t step_launches = 0;
  double step_gpu_s = 0.0;
  double step_alg_bytes = 0.0;
  int64_t kind_launches[3] = {0, 0, 0};
  double kind_gpu_s[3] = {0.0, 0.0, 0.0};
  double kind_alg_bytes[3] = {0.0, 0.0, 0.0};
  // every step-kernel launch, timed or not (the timer reads its share from these)
  int64_t all_launches[3] = {0, 0, 0};
  double all_alg_bytes[3] = {0.0, 0.0, 0.0};
};
Counters& counters();
inline void count_launch(int64_t n = 1) { counters().launches += n; }
// count one step-kernel launch of storage kind `kind` moving `alg_bytes` algorithmic bytes
inline void count_step(int kind, double alg_bytes) {
  Counters& c = counters();
  c.launches++;
  c.all_launches[kind]++;
  c.all_alg_bytes[kind] += alg_bytes;
}

// Stream-ordered scratch of a call (freed with cudaFreeAsync), from a pool of the
// library's own: the default pool unmaps freed memory at the next synchronization,
// and mapping it again costs 70 us for a few MB, 2 ms for a GB.  The pool keeps at
// most 1/256 of the device's memory between calls, which other allocators cannot
// take: 1.1 GB here, what L = 24 needs.  Larger calls map the rest anew each time:
// L = 26, 32 FP32 columns, 40 steps, 84.5 ms, 82.3 with a pool that keeps all 4 GB.
// pool_trim gives back what is unused, as polfed_ctx_destroy and every allocation
// that fails do.
int scratch_alloc(void** p, size_t bytes, cudaStream_t s);
void pool_trim();
cudaError_t device_malloc(void** p, size_t bytes);  // cudaMalloc, once more after pool_trim

// -------------------------------------------------------------- binomials
// C(n, k) for 0 <= n, k <= 32 (C(32,16) < 2^31).
uint32_t binom_host(int n, int k);
void upload_binomials();  // __constant__ table, once per device

// ------------------------------------------------- Hamiltonian operator plan
// A term of Eq. (1) between sites i < j with coupling class l (1: J1, 2: J2).
struct Bond {
  int i, j, cls;
};

constexpr int kMaxBonds = 64;
constexpr int kMaxCross = 16;

// Split of the L bits into a low part (bits 0..b-1) and a high part (bits
// b..L-1).  Rows whose states share the high part s_hi form one contiguous
// "group"; rank(s) = T_hi[s_hi] + T_lo[s_lo] (combinatorial number system).
struct HamGeometry {
  int L, b, nh, n_up, periodic;
  int64_t dim;
  double J1, J2, Delta;
  double h[32];
  // literal terms of Eq. (1), classified by where their two sites lie
  int n_low1, n_low2;    // low bonds, class 1 first then class 2
  uint32_t low_mask[kMaxBonds];
  int n_high1, n_high2;  // high bonds (masks relative to bit b)
  uint32_t high_mask[kMaxBonds];
  int n_cross;           // one site in each part
  int cross_lo[kMaxCross], cross_hi[kMaxCross], cross_cls[kMaxCross];
  int cls_off[34];       // offset of popcount class c in the U_lo table
  int max_group;         // largest group (rows)
  int n_groups;          // valid groups
  int rec_stride;        // uint16 entries per neighbour record (16 or 32)
};

// Device tables of a geometry (owned by HamPlan).
struct HamTables {
  uint16_t* U_lo;   // [2^b] inverse of T_lo: U_lo[cls_off[c] + k] = k-th b-bit string with popcount c
  int32_t* T_hi;    // [2^nh] first row of group s_hi, -1 if the group is empty
  int32_t* order;   // [n_groups] groups, largest first
  double* F_lo;     // [2^b] diagonal part from low bonds and low fields (H units)
  double* F_hi;     // [2^nh] diagonal part from high bonds and high fields
  double* C_x;      // [2^n_cross] diagonal part from cross bonds by "differ" pattern
  // [2^b * rec_stride] per-row neighbour records, indexed by cls_off[c] + local
  // index; one table per lanes-per-row 1, 2, 4, 8 (entries are byte offsets
  // (local index + 1) * row bytes into a tile whose first row is zero):
  //   entry 0: bits of s_lo at the low sites of the cross bonds (bit k: bond k);
  //   entry 1: n1 | n2 << 8 (active low bonds of class 1 and 2);
  //   from entry 2: cross bond k's neighbour (s_lo with its low site flipped, in
  //   the neighbouring popcount class), 2 entries or 6 with J2; then the active
  //   class 1 neighbours (10 entries) and class 2, zero padded
  uint16_t* rec[4];
  // [n_groups] per-group constants in schedule order (see GroupRec)
  struct GroupRec* grec;
};

constexpr int kMaxHigh = 32;  // high bonds: L = 24 J1-J2 with b = 10 has 13 + 12 = 25
// Per-group constants (one group = rows sharing s_hi), precomputed per plan.
struct alignas(16) GroupRec {
  int r0, n_g, cls_base, n_hn1, n_hn, need_mask, pad0, pad1;
  int hn_base[kMaxHigh];  // first row of each neighbouring group through an antiparallel high bond
  int cr_base[8];         // first row of the group reached through cross bond k
  int cr_n[8];            // rows of that group (0 if no row of this group has the bond antiparallel)
};

int build_geometry(const polfed_model* m, int b_override, HamGeometry* g);

constexpr size_t kSliceSet = (size_t)96 << 20;  // of the 126 MB L2

class HamPlan {
 public:
  HamGeometry geo;
  HamTables tab{};
  void* dev = nullptr;       // one allocation for all tables
  void* dev_end = nullptr;
  int* err_flag = nullptr;   // set by a kernel whose bounded wait expired
  unsigned bar_base = 0;     // arrivals counted so far on the grid barrier (err_flag + 16)
  // per-precision alpha/beta-scaled tables (k_typed), indexed by dtype
  void* typed[3] = {nullptr, nullptr, nullptr};
  bool typed_ok[3] = {false, false, false};
  double typed_lo[3] = {0, 0, 0}, typed_hi[3] = {0, 0, 0};
  cudaStream_t stream = nullptr;
  bool stream_alloc = false;  // tables from cudaMallocAsync
  size_t slice_set = kSliceSet;  // bytes of the column slices that run in one launch; 0: one slice at a time

  // All of these only enqueue work on the stream.
  // kind >= 0: with the scaled tables of that storage type (prepare_typed in the same launch)
  int init(const polfed_model* m, cudaStream_t s, bool stream_ordered, int b_override = -1, int kind = -1,
           double e_lo = 0.0, double e_hi = 0.0);
  // tables (and typed_dst, kind >= 0) in caller memory, geo already set
  int bind(char* base, cudaStream_t s, int kind = -1, double e_lo = 0.0, double e_hi = 0.0, void* typed_dst = nullptr);
  int prepare_typed(int kind, double e_lo, double e_hi);  // alpha/beta-scaled tables
  void release();
  ~HamPlan() { release(); }
};

// Elements per slice for a precision and lanes-per-row.
int slice_width(int kind, int lpr);
size_t elem_bytes(int kind);  // internal storage element size (DF64: 8 = two floats)

// Filter engine over an arbitrary-width ABI block.  in/out are row-major
// dim x n_b of "abi_kind" (POLFED_F32: float, else double).
struct FilterScratch {
  void* xs = nullptr;     // slice buffers (dim x W each; see filter_scratch_bytes)
  float* flag = nullptr;  // [4] max |x|, max |y| (as float bits)
  size_t bytes = 0;
};
int filter_block(HamPlan& plan, int kind, const double* coeffs, int K, double invD, const void* in, void* out,
                 int n_b, int abi_kind, FilterScratch& scr, cudaStream_t s);
// FP32 filter with its own coefficients per column: out[:, j] = sum_n coef_j[n] T_n(H~) in[:, j].
// The block is filtered in slices of W = slice_width(POLFED_F32, choose_lpr(POLFED_F32, n_b)) columns;
// d_coef (device) holds, per slice q, (K + 1) rows of W floats:
// d_coef[(q (K + 1) + n) W + j - q W] = coefficient of column j at order n.  in/out as filter_block.
int filter_block_cols(HamPlan& plan, const float* d_coef, int K, const void* in, void* out, int n_b, int abi_kind,
                      FilterScratch& scr, cudaStream_t s);
// H~ of a block: needs no scratch where apply_direct holds
bool apply_direct(int kind, int abi_kind, int n_b, const void* in, const void* out);
int apply_block(HamPlan& plan, int kind, const void* in, void* out, int n_b, int abi_kind, FilterScratch& scr,
                cudaStream_t s);
// mu[2k] = t_k . t_k, mu[2k + 1] = t_{k+1} . t_k summed over n_b columns, t_{k+1} = 2 H~ t_k - t_{k-1}, k < half
// (device, overwritten).  t_odd: moment_scratch_bytes (float-float keeps t_n in FP64); part: room for the sums of
// kMaxMomentCtas CTAs of one step at least, more steps to a launch with more.  Synchronizes.
constexpr int kMaxMomentCtas = 304;  // the launch takes one per SM, and no more than these
int moment_steps(HamPlan& plan, int kind, const void* in, int n_b, int half, void* t_odd, void* part, size_t part_bytes,
                 double* mu, FilterScratch& scr, cudaStream_t s);
int moments_b(int kind, int L);  // low bits of a plan for moments, 0: the plan's own choice
size_t moment_scratch_bytes(const HamPlan& plan, int kind, int n_b);
size_t filter_scratch_bytes(const HamPlan& plan, int kind, int n_b);
int choose_lpr(int kind, int n_b);

// Batched filter: cooperative launches advance the Clenshaw recurrences of
// many (realization, 128-byte column slice) jobs, each with its own plan,
// order and coefficients (F32 or DF64 storage; all jobs J2 == 0 or all not).
constexpr int kBatchLpr = 8;  // 128-byte slices
struct BatchFilterItem {
  HamPlan* plan;          // prepare_typed(kind, ...) done
  const double* coef;     // host, K + 1 coefficients: Y = invD * sum_n coef[n] T_n(H~) X
  int K;
  double invD;
  const void* in;         // device, row-major dim x n_b (abi kind)
  void* out;              // device, row-major dim x n_b
  int n_b;
  bool bounds_error;      // out: output grew beyond the Chebyshev bound
};
struct BatchStats {
  int n_jobs = 0, n_steps = 0, grid = 0;
  double gpu_s = 0.0, alg_bytes = 0.0;
};
size_t batch_scratch_bytes(const std::vector<BatchFilterItem>& items, int kind);
int filter_batched(std::vector<BatchFilterItem>& items, int kind, int abi_kind, void* scratch, size_t bytes,
                   cudaStream_t s, int ctas_per_sm, BatchStats* st);

// Filter calls of the block-Lanczos driver can be routed through a hook (the
// batched runner's rendezvous).  Panels q = 0..npan-1: out[q] = invD sum_n
// coef[n] T_n(H~) in[q], each dim x S row-major FP64 on `s`.
struct FilterHook {
  virtual int filter(HamPlan& plan, int kind, const double* coef, int K, double invD, const double* const* in,
                     double* const* out, int npan, int S, cudaStream_t s) = 0;
  virtual int plan_b(int L) { return -1; }  // low/high split for the plans (-1 = default)
  // the caller launches its own kernels until resume() and sends no filter() meanwhile
  virtual void suspend() {}
  virtual void resume() {}
  virtual ~FilterHook() {}
};
// Context internals for the other translation units.
cudaStream_t ctx_stream(polfed_ctx* c);
void* ctx_solver(polfed_ctx* c);  // cusolverDnHandle_t
int ctx_device(polfed_ctx* c);

// polfed_eigs with an optional hook (nullptr = direct filter launches).
int eigs_impl(polfed_ctx* c, const polfed_model* model, double eps_target, int32_t N_ev, int32_t K, int32_t n_b,
              const polfed_opts* opts, double* evals, double* d_evecs, double* resid, polfed_stats* stats,
              FilterHook* hook);

// Chebyshev coefficients of Eq. (2) in FP64: c_n, n = 0..K, and D.
void cheb_coeffs(double sigma, int K, std::vector<double>& c, double& D);

// Kernel polynomial method: stochastic Chebyshev moments of H~ and the
// Jackson-damped fraction of the spectrum inside an interval.
constexpr int kMaxKpmMoments = 65536;
void jackson_coeffs(int N, std::vector<double>& g);
size_t kpm_buffer_bytes(const HamPlan& plan, int kind, int R);
// mu[n] = (1/R) sum_r r^T T_n(H~) r, n < n_mom (host out); r is row-major dim x R
// of float (kind POLFED_F32) or double.  Needs plan.prepare_typed(kind, ...), a
// buffer of kpm_buffer_bytes and filter scratch for R columns.
int kpm_moments(HamPlan& plan, int kind, const void* r, int R, int n_mom, double* mu, void* buf, FilterScratch& scr,
                cudaStream_t s);
double kpm_count_fraction(const double* mu, int n_mom, double x_a, double x_b);

// Basis kernel (polfed_basis_build).
int launch_basis(int L, int n_up, uint32_t* d_states, int64_t dim, cudaStream_t s);

}  // namespace polfed
