// hub_internal.cuh -- handle layout, error plumbing and device helpers shared by the
// library's translation units.  Not part of the public ABI (see include/hub.h).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/hub.h"

namespace hub {

constexpr int kMaxSites = 30;   // spin strings fit in uint32, two-spin index fits in int64
constexpr int kMaxBonds = 255;   // bond ids and per-row group lengths fit in uint8

// ---------------------------------------------------------------------------------------
// Errors: every entry point returns a code; the message goes to a thread-local string.
// ---------------------------------------------------------------------------------------
void set_error(const std::string &msg);
int fail(int code, const std::string &msg);
int cuda_fail(cudaError_t e, const char *what, const char *file, int line);

#define HUB_CUDA(call)                                                        \
  do {                                                                        \
    cudaError_t e_ = (call);                                                  \
    if (e_ != cudaSuccess) return ::hub::cuda_fail(e_, #call, __FILE__, __LINE__); \
  } while (0)

#define HUB_LAUNCH_CHECK() HUB_CUDA(cudaGetLastError())

// ---------------------------------------------------------------------------------------
// One-spin hopping matrix in CSR form (Sec. IV.A, Eqs. 9-10).
// ---------------------------------------------------------------------------------------
struct SpinCSR {
  int32_t *rowptr = nullptr;   // [count + 1]
  int32_t *col = nullptr;      // [nnz], ascending within a row
  double *val = nullptr;       // [nnz], -t_b * (-1)^(electrons strictly between the sites)
  uint32_t *scol = nullptr;    // [nnz], col | (sign bit << 31): -t_b = -t * sign for uniform t
  uint8_t *bond = nullptr;     // [nnz], bond id of the entry (gradients)
  int64_t nnz = 0;
  int32_t max_row = 0;
};

struct FastState;   // fast-path tables and scratch (hub_fast.cu)
struct K0State;     // k = 0 translation-sector tables (hub_k0.cu)
struct SmallState;  // single-launch Lanczos of small sectors (hub_small.cu)
struct FixState;    // fixed-point product and Lanczos (hub_fix.cu)

// Read-only view of everything a kernel needs, passed by value.
struct Ham {
  int M;
  int64_t n_up, n_dn;                 // count_up, count_dn
  const uint32_t *basis_up, *basis_dn;
  const int32_t *rp_up, *rp_dn;       // CSR row pointers
  const int32_t *col_up, *col_dn;
  const double *val_up, *val_dn;
  const uint32_t *scol_up, *scol_dn;  // signed columns (uniform-t kernels)
  const double *eps_up, *eps_dn;      // per-state site-energy sums (nullptr when eps == 0)
  int uniform_U;                      // 1: U_i = U0 for all i
  double U0;
  double U[kMaxSites];                // per-site U_i
  int uniform_t;                      // 1: all t_b equal to t0
  double t0;
  int has_eps;
};

// chained: a launch that need not wait for the kernel before it on the stream to drain; its blocks are
// placed while that one ends, and wait (after_previous, the first thing such a kernel does) for its
// results.  For rows of kernels of which most find on a device flag that there is nothing to do: a vector of
// the 13-site ring (6,6) that goes to the double-float kernels takes 146 us with plain launches, 142 chained,
// 115 chained with no more CTAs than are resident and with flags through L1 (120 in double-float alone).
template <typename... P, typename... A>
inline cudaError_t launch_kernel(bool chained, void (*kernel)(P...), dim3 grid, dim3 block, size_t smem,
                                 cudaStream_t s, A... args) {
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = block;
  c.dynamicSmemBytes = smem;
  c.stream = s;
  c.attrs = &attr;
  c.numAttrs = chained ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, static_cast<P>(args)...);
}
__device__ __forceinline__ void after_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
// A flag written by a kernel before this one, read after after_previous(): an ordinary load that the compiler
// can neither move nor make a read-only one.  (A volatile one goes past L1: 5 us in a kernel of 20 us.)
__device__ __forceinline__ int flag_of(const int *p) {
  int v;
  asm volatile("ld.global.b32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}

// Lane l of the warp: the warp's total of v[l % N].  Each of the first log2(N) exchanges sends one of
// a pair and keeps the other, so that N totals take N + 4 - log2(N) shuffles instead of 5 N.
template <int N, typename T>
__device__ __forceinline__ T warp_totals(T (&v)[N]) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int m = N / 2, o = 1; m > 0; m >>= 1, o <<= 1) {
    const bool odd = (lane & o) != 0;
#pragma unroll
    for (int k = 0; k < m; ++k) {
      const T keep = odd ? v[2 * k + 1] : v[2 * k], send = odd ? v[2 * k] : v[2 * k + 1];
      v[k] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  T t = v[0];
#pragma unroll
  for (int o = N; o < 32; o <<= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

// Scalars of the FP64 Lanczos recurrence on the device (hub_lanczos.cu).  The vectors are kept as they
// leave the update, r_j = beta_j q_j; inv = 1 / beta_j and c = beta_j / beta_{j-1} scale the next product.
struct F64Scal {
  double inv, c, alpha;
  double hist[2][2];                  // (alpha_j, beta_{j+1}) of the last two steps
  unsigned ticket[2];
};
struct F64Step {
  F64Scal *scal = nullptr;
  double *partials = nullptr;
  const double *prev = nullptr;       // may be the output
  double *psi = nullptr;
  double a = 0.0, b = 0.0, inv = 1.0, v = 0.0;   // second pass: alpha_j, beta_j, 1 / beta_{j+1}, v_j
};

// Adds the CTAs' values; true in the first thread of the last CTA to arrive, with *sum the total in
// a fixed order.  Leaves the ticket at zero.  All threads of all CTAs of the launch take part.
__device__ __forceinline__ bool grid_sum(double v, double *__restrict__ partials, unsigned *ticket, double *sum) {
  __shared__ double ws[32];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if (lane == 0) ws[warp] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int k = 0; k < nw; ++k) s += ws[k];
    partials[blockIdx.x] = s;
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
    if (last) *ticket = 0;
  }
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double t = 0.0;
  for (int k = threadIdx.x; k < (int)gridDim.x; k += blockDim.x) t += __ldcg(partials + k);
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if (lane == 0) ws[warp] = t;
  __syncthreads();
  if (threadIdx.x != 0) return false;
  t = 0.0;
  for (int k = 0; k < nw; ++k) t += ws[k];
  *sum = t;
  return true;
}
// The end of a step's first kernel: alpha_j from the parts of <r_j, w> / beta_j.
__device__ __forceinline__ void f64_step_alpha(const F64Step &L, double dot) {
  double sum;
  if (grid_sum(dot, L.partials, &L.scal->ticket[0], &sum)) L.scal->alpha = L.scal->inv * sum;
}

}  // namespace hub

// The handle behind the opaque hub_t.
struct hub_ctx {
  int device = 0;
  int M = 0;
  int N[2] = {0, 0};
  int64_t count[2] = {0, 0};
  bool shared = false;                 // N_up == N_dn: one basis and one CSR for both spins
  uint32_t *basis[2] = {nullptr, nullptr};
  uint64_t *binom = nullptr;           // device Pascal triangle, (kMaxSites+1)^2

  bool have_hop = false;
  int n_bonds = 0;
  std::vector<int32_t> bonds;
  std::vector<double> t, eps;
  hub::SpinCSR csr[2];
  double *eps_state[2] = {nullptr, nullptr};
  bool has_eps = false;

  bool have_U = false;
  bool uniform_U = true;
  double U0 = 0.0;
  std::vector<double> U;

  // Lanczos workspace (3 vectors), scalars, partial sums and the last run's coefficients.
  double *work[3] = {nullptr, nullptr, nullptr};
  double *psi_tmp = nullptr;
  double *d_scal = nullptr;            // [8] device scalars
  double *h_scal = nullptr;            // [8] pinned host mirror
  double *partials = nullptr;          // reduction partials
  int64_t partials_n = 0;
  std::vector<double> alpha, beta;

  // host-buffer apply; the second pair alternates with the first in hub_apply_host_many
  double *hx = nullptr, *hy = nullptr;
  double *hx2 = nullptr, *hy2 = nullptr;

  // |x0| of the last Lanczos run (the continued fraction of the Green's function needs it)
  double start_norm = 0.0;
  // second Lanczos pass: expand the eigenvector of T for the eigenvalue nearest psi_target
  // instead of the lowest one (hub_lanczos_ritz); psi_value records the value used
  bool psi_at_target = false;
  double psi_target = 0.0, psi_value = 0.0;
  // source index and sign per state of this handle's sector for hub_ladder
  int32_t *ladder_map = nullptr;
  int64_t ladder_cap = 0;

  // measurement: event pairs per kind (HUB_PROF_*), launch counters
  bool prof = false;
  static constexpr int kProfKinds = 4; // HUB_PROF_APPLY .. HUB_PROF_UPDATE
  std::vector<cudaEvent_t> ev_start[kProfKinds], ev_end[kProfKinds];
  int64_t n_launch[kProfKinds] = {0, 0, 0, 0};   // launches per kind since hub_profile(h, 1)
  int64_t n_timed[kProfKinds] = {0, 0, 0, 0};    // of which timed with an event pair
  int64_t n_kernels = 0;               // all kernels launched since hub_profile(h, 1)

  // fast path (double-float, two-pass apply) for uniform hopping and interaction
  hub::FastState *fast = nullptr;
  int mode = 0;                        // HUB_MODE_AUTO or HUB_MODE_FP64
  bool fail_waits = false;             // test hook: pass 1 reports a given-up wait (hub_test_fail_waits)

  // k = 0 sector of the translation i -> i-1 mod M (hub_set_symmetry); vectors are then in
  // row form, rows x cols (hub_k0.cu)
  hub::K0State *k0 = nullptr;

  // sectors of at most small_max_dim states run hub_lanczos_ground as one cooperative
  // kernel per batch of iterations (hub_small.cu); 0 turns that off
  int64_t small_max_dim = int64_t(1) << 18;
  hub::SmallState *small = nullptr;

  // fixed-point product and Lanczos (hub_fix.cu): tables, flags and vectors
  hub::FixState *fix = nullptr;

  // the last product's kernels (hub_last_route): HUB_ROUTE_*, or the one that the words of a path's own
  // flags decide
  int route = 0;
  const int *route_flag[2] = {nullptr, nullptr};   // device: nonzero for FP64, for double-float

  hub::Ham view() const;
};

namespace hub {

// Allocation helpers: on failure they set the message and return false.
bool dev_alloc(void **p, size_t bytes, const char *what);
void dev_free(void *p);
int ensure_partials(hub_ctx *h, int64_t n);

// Launch helpers.
int num_sms();
constexpr int kReduceThreads = 256;

// Deterministic FP64 reduction of partials[0..n) into *out (device), one block.
int reduce_partials(const double *partials, int n, double *out, int mode, cudaStream_t s);
// Same, in two fixed-order stages through tmp[ntmp] (for long partial lists).
int reduce_partials_2stage(const double *partials, int n, double *tmp, int ntmp, double *out, int mode,
                           cudaStream_t s);

// Apply entry used by Lanczos and the VJP (no argument checks).
int apply_launch(hub_ctx *h, const double *x, double *y, cudaStream_t s);
void set_route(hub_ctx *h, int route, const int *f64_flag = nullptr, const int *df_flag = nullptr);
// The FP64 product kernel of the full sector; with a gate it does nothing unless gate[0] != 0
// when it runs (a device flag written earlier on the stream).
int f64_apply(hub_ctx *h, const double *x, double *y, const int *gate, cudaStream_t s);
// Whether products of the handle's vectors go to the FP64 kernel; its grid; and the product with the
// Lanczos step around it (second: the pass that builds the Ritz vector).
bool f64_product(hub_ctx *h);
int64_t f64_grid(const hub::Ham &H);
int f64_apply_step(hub_ctx *h, const double *x, double *y, const hub::F64Step &L, bool second, cudaStream_t s);

// Fast path (hub_fast.cu).
bool fast_eligible(const hub_ctx *h);
int fast_build(hub_ctx *h);
void fast_release(hub_ctx *h);
int fast_apply_f64(hub_ctx *h, const double *x, double *y, cudaStream_t s);
int fast_apply_host(hub_ctx *h, const double *x_host, double *y_host, double *xd, double *yd, cudaStream_t s);
// True when the fast path's host-buffer apply runs in row chunks (staged pass 1, enough rows),
// the case fast_apply_host_many pipelines across vectors.
bool fast_host_pipelined(const hub_ctx *h);
int fast_apply_host_many(hub_ctx *h, int64_t n_vec, const double *x_host, double *y_host, double *const xd[2],
                         double *const yd[2], cudaStream_t s);
// The same product behind the fixed-point one: every kernel does nothing unless gate[0] != 0 when
// it runs; scale: the vector's power-of-two exponent and a zero.
int fast_apply_gated(hub_ctx *h, const double *x, double *y, const int *scale, const int *gate, cudaStream_t s);
// The first n <= 4 scratch vectors of the handle, each large enough for a vector in either order.
int fast_scratch(hub_ctx *h, int n, float **v);
void fast_release_scratch(hub_ctx *h);
// The handle's device error flag.
int *fast_err(const hub_ctx *h);
int fast_check_error(hub_ctx *h);
// Lowest eigenvalues of the successive tridiagonals T_1, T_2, ... of one Lanczos run (host),
// each by bisection on the Sturm count like tridiag_lowest, but started from a bracket around
// the previous value (by Cauchy interlacing the new one lies at or below it), widened until the
// count is 0 at its lower end and at least 1 at its upper end; both bisections end on the two
// adjacent doubles where the count steps from 0 to 1, so they return the same value.
struct LowestTracker {
  double last = 0.0, step = 0.0;
  int n = 0;
  double next(const double *a, const double *b, int k);
};
double tridiag_lowest(const double *a, const double *b, int k);

// Eigenvalue of the last run's T whose eigenvector the second Lanczos pass expands (E0, or the
// one nearest h->psi_target); also stored in h->psi_value.
double psi_eigenvalue(hub_ctx *h, double E0);
inline bool use_fast(const hub_ctx *h) {
  return h->mode == HUB_MODE_AUTO && h->fast && !h->k0 && fast_eligible(h);
}

// The double-float window (hub_fast.cu): biased FP64 exponents of the largest entry, and how far
// below it a nonzero entry may lie.
constexpr int kExpSpan = 80, kExpLo = 200, kExpHi = 1900;

// Fixed-point product and Lanczos (hub_fix.cu).
bool fix_apply_eligible(const hub_ctx *h);
int fix_apply(hub_ctx *h, const double *x, double *y, cudaStream_t s);
bool fix_lanczos_eligible(const hub_ctx *h);
int fix_lanczos(hub_ctx *h, const double *x0, int maxit, double tol, double *E0, double *psi_out, int *iters,
                cudaStream_t s);
void fix_release(hub_ctx *h);
// v /= |v| (hub_lanczos.cu)
int f64_normalise(hub_ctx *h, int64_t D, double *v, cudaStream_t s);

// Single-launch Lanczos of small sectors (hub_small.cu).
bool small_eligible(const hub_ctx *h);
int small_lanczos(hub_ctx *h, const double *x0, int maxit, double tol, double *E0, double *psi_out, int *iters,
                  cudaStream_t s);
int small_check_error(hub_ctx *h);
void small_release(hub_ctx *h);

// k = 0 sector (hub_k0.cu).
int64_t vec_len(const hub_ctx *h);   // length of a state vector in the handle's current layout
int k0_apply(hub_ctx *h, const double *x, double *y, cudaStream_t s);
int k0_project_inplace(hub_ctx *h, double *x, cudaStream_t s);
void k0_leave(hub_ctx *h);           // back to the full sector, vectors sized for it dropped
void k0_release(hub_ctx *h);

// Event pair around a launch of the given kind (no-op unless profiling).
int prof_mark(hub_ctx *h, int kind, bool begin, cudaStream_t s);

// Count kernel launches for the measurement hooks.
inline void count_launch(hub_ctx *h, int n = 1) {
  if (h->prof) h->n_kernels += n;
}

// Device helpers ------------------------------------------------------------------------
// Combinatorial number system (Sec. II, App. A).  binom[n * kB + k] = C(n, k);
// rank(s) = sum_j C(b_j, j) over the set bits b_1 < b_2 < ... of s (j = 1, 2, ...), the
// position of s in the ascending list of strings with its number of ones.
constexpr int kB = kMaxSites + 1;

__device__ __forceinline__ uint32_t rank_of(uint32_t s, const uint64_t *__restrict__ C) {
  uint32_t r = 0;
  int j = 1;
  while (s) {
    int b = __ffs(s) - 1;
    r += (uint32_t)C[b * kB + j];
    ++j;
    s &= s - 1;
  }
  return r;
}

// Diagonal of H at (u, d) (Sec. III.B): sum_i U_i bit_i(I_up & I_dn) + eps(I_up) + eps(I_dn).
__device__ __forceinline__ double diag_of(const Ham &H, uint32_t Iu, uint32_t Id, int64_t u, int64_t d) {
  double v;
  if (H.uniform_U) {
    v = H.U0 * (double)__popc(Iu & Id);
  } else {
    v = 0.0;
    for (uint32_t m = Iu & Id; m; m &= m - 1) v += H.U[__ffs(m) - 1];
  }
  if (H.has_eps) v += H.eps_up[u] + H.eps_dn[d];
  return v;
}

__host__ __device__ inline int popc32(uint32_t v) {
#ifdef __CUDA_ARCH__
  return __popc(v);
#else
  return __builtin_popcount(v);
#endif
}

}  // namespace hub
