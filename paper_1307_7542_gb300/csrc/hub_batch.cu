// hub_batch.cu -- many small ground-state problems in one persistent launch (K6).
//
// Sec. VIII: an exact-diagonalisation impurity solver repeats the ground-state search for
// every (N_up, N_dn) sector and every bath-parameter set.  Each such problem is small (for
// an 8-site impurity star the largest sector has 70 x 70 = 4900 states), so one problem per
// launch would be dominated by launch and synchronisation latency.  Here all problems are
// jobs of one kernel: persistent CTAs take jobs from an atomic queue (largest first), keep
// the job's two Lanczos vectors in shared memory and run the whole plain Lanczos
// iteration of Sec. IV / V inside the CTA.  The matrix-free product is Eq. 11 on the
// count_dn x count_up state matrix (Eq. count2): spin-up hops gather inside a row, spin-down
// hops combine rows, the diagonal comes from the set bits of I_up & I_dn (Sec. III.B); the
// hopping values -t_b * esign (Eq. 8) are formed on the fly from the job's parameter set.
// The one-spin bases and hopping structures of the particle numbers that occur are built once on the
// host and shared by all jobs.
#include <algorithm>
#include <cmath>
#include <numeric>
#include <vector>

#include "hub_internal.cuh"

namespace hub {

constexpr int kBatchMaxSites = 16;
constexpr int kBatchMaxDim = 8192;      // two FP64 vectors of this length in shared memory
#ifndef HUB_BATCH_THREADS
#define HUB_BATCH_THREADS 512            // threads per CTA of the large jobs (one job per CTA at a time)
#endif
constexpr int kBatchThreads = HUB_BATCH_THREADS;
constexpr int kBatchCheckEvery = 8;     // E0 of T_j is evaluated every this many iterations
#ifndef HUB_BATCH_SPLIT
#define HUB_BATCH_SPLIT 2048              // jobs of more states run in a launch of their own
#endif
// Jobs by size: each class is a launch of its own, its CTAs sized for its largest job.  Small jobs in
// small CTAs: more of them per SM, and shorter barriers and sums; all jobs of 64 sets of the 8-site
// star take 16.3 ms with 256 threads from 256 states on, 14.5 from 400, 13.1 from 2048 (192 or 512
// threads above: 13.4 and 14.3; 32 or 96 below: 14.0 and 13.3).
struct BatchClass {
  int above, threads;                  // jobs of more than `above` states, threads per CTA
};
constexpr int kBatchClasses = 2;
constexpr BatchClass kBatchClass[kBatchClasses] = {{HUB_BATCH_SPLIT, kBatchThreads}, {0, 64}};

struct BatchTables {
  const uint32_t *basis;     // all one-spin bases, N = 0..M, concatenated
  const int32_t *rp;         // row pointers (global entry offsets), concatenated
  const uint32_t *word;      // column | (2 bond + sign) << 16, entries concatenated
  const uint32_t *ell;       // the same as [entry][state] of each N, for lanes along the states
  int off_ell[kBatchMaxSites + 2];
  int off_basis[kBatchMaxSites + 2];   // start of N's basis in `basis`
  int off_rp[kBatchMaxSites + 2];      // start of N's row pointers in `rp`
  int count[kBatchMaxSites + 1];       // C(M, N)
};

struct BatchArgs {
  int M, n_bonds, n_jobs, maxit;
  double tol;
  const double *t, *U, *eps;           // per parameter set: [n_bonds], [M], [M] (eps may be null)
  const int32_t *job_nup, *job_ndn, *job_param, *order;
  int *counter;                        // work queue head (zeroed before the launch)
  double *E0;
  int32_t *iters, *status;
};

// Sum over the CTA (of warps that hold a nonzero value), the same in every thread.  The adds are few
// because they are FP64: five per warp with data, then one value per lane.
__device__ __forceinline__ double block_sum(double v, double *red) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
  if (__any_sync(0xffffffffu, v != 0.0))         // NaN too
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  __syncthreads();                     // red may still be read from the previous call
  if (lane == 0) red[wid] = v;
  __syncthreads();
  double s = lane < nw ? red[lane] : 0.0;
  for (int o = 16; o > 0; o >>= 1)
    if (o < nw) s += __shfl_xor_sync(0xffffffffu, s, o);
  return __shfl_sync(0xffffffffu, s, 0);
}

// Number of eigenvalues of the tridiagonal (a, b) smaller than x (Sturm sequence).
__device__ int sturm_count_dev(const double *a, const double *b, int k, double x) {
  int cnt = 0;
  double d = 1.0;
  for (int i = 0; i < k; ++i) {
    const double bb = i ? b[i - 1] * b[i - 1] : 0.0;
    d = (a[i] - x) - (i ? bb / d : 0.0);
    if (d == 0.0) d = -1e-300;
    if (d < 0.0) ++cnt;
  }
  return cnt;
}

// Whether x lies above the lowest eigenvalue: the leading minors p_i of T - x are not all positive.  Two
// multiply-adds per row and no divisions (the pivots d_i = p_i / p_{i-1} cost one each, some 15
// FP64 instructions on a unit that issues one per 16 cycles); the pair (p_i, p_{i-1}) is scaled every
// four rows.  Four rows cannot overflow or underflow for
// coefficients within 2^+-100 (the caller sees to it).
__device__ __forceinline__ bool above_lowest(const double *a, const double *b, int k, double x) {
  double p0 = 1.0, p1 = a[0] - x;
  bool neg = !(p1 > 0.0);
  for (int i = 1; i < k; ++i) {
    const double bb = b[i - 1] * b[i - 1];
    const double p2 = fma(a[i] - x, p1, -bb * p0);
    p0 = p1;
    p1 = p2;
    neg = neg || !(p2 > 0.0);
    if ((i & 3) == 0) {                      // 2^-e from p1's exponent e: normal while all are positive
      const double f = __hiloint2double((2046 - ((__double2hiint(p1) >> 20) & 0x7ff)) << 20, 0);
      p0 *= f;
      p1 *= f;
    }
  }
  return neg;
}

// Lowest eigenvalue of the k x k tridiagonal by 32-way multisection, one warp.  E_prev: the lowest
// eigenvalue of a leading block, which is an upper bound (NaN: none).  The first round then tries
// distances below it on a logarithmic scale, so that the bits that agree need no rounds: 4 to 8 rounds
// instead of 12 to 16.
__device__ double tri_lowest_warp(const double *a, const double *b, int k, double E_prev) {
  const int lane = threadIdx.x & 31;
  double lo = INFINITY, hi = -INFINITY;
  for (int i = lane; i < k; i += 32) {
    const double r = (i ? fabs(b[i - 1]) : 0.0) + (i < k - 1 ? fabs(b[i]) : 0.0);
    lo = fmin(lo, a[i] - r);
    hi = fmax(hi, a[i] + r);
  }
  for (int o = 16; o > 0; o >>= 1) {
    lo = fmin(lo, __shfl_xor_sync(0xffffffffu, lo, o));
    hi = fmax(hi, __shfl_xor_sync(0xffffffffu, hi, o));
  }
  if (k == 1) return a[0];
  const double range = hi - lo;
  const bool minors = range < 0x1p100 && range > 0x1p-100;
  auto above = [&](double x) { return minors ? above_lowest(a, b, k, x) : sturm_count_dev(a, b, k, x) >= 1; };
  if (E_prev > lo && E_prev < hi) {
    const double top = fmin(hi, E_prev + 1e-15 * range), x = top - (top - lo) * exp2(-1.6 * (double)(lane + 1));
    const unsigned ball = __ballot_sync(0xffffffffu, above(lane == 31 ? top : x));
    const int L = ball ? __ffs(ball) - 1 : 32;
    const double nhi = __shfl_sync(0xffffffffu, lane == 31 ? top : x, L & 31);
    const double nlo = __shfl_sync(0xffffffffu, x, max(L - 1, 0) & 31);
    if (L < 32) {
      if (L > 0) lo = nlo;
      hi = nhi;
    }
  }
  for (int round = 0; round < 16; ++round) {
    const double step = (hi - lo) / 32.0;
    const double x = lane == 31 ? hi : lo + step * (lane + 1);
    const unsigned ball = __ballot_sync(0xffffffffu, above(x));
    const int L = ball ? __ffs(ball) - 1 : 31;
    const double nhi = __shfl_sync(0xffffffffu, x, L);
    const double nlo = L == 0 ? lo : __shfl_sync(0xffffffffu, x, L - 1);
    if (!(nhi < hi || nlo > lo)) break;        // no progress at double precision
    lo = nlo;
    hi = nhi;
  }
  return 0.5 * (lo + hi);
}

// What bounds it is the FP64 unit: a multiply-add per hopping term, six operations per state for the
// diagonal and the recurrence.  A thread keeps a column u of the state matrix and takes rows d in pairs,
// so that a spin-up entry is loaded once for two rows by neighbouring lanes, a spin-down row's
// entries are the same for a warp's lanes, and sums over occupied sites come from tables.  The
// vectors stay as the update leaves them, r_j = beta_j q_j; the next product is scaled instead.
// 64 sets of the 8-site star (5184 jobs): 39 -> 13.1 ms (half the FP64 unit's rate; the rest is latency
// at barriers and the tail of the queue).
__global__ void __launch_bounds__(kBatchThreads, 1024 / kBatchThreads) k_batch_lanczos(const BatchTables T, const BatchArgs A) {
  extern __shared__ __align__(16) double sm[];
  __shared__ double red[32];
  __shared__ double s_U[2][256], s_eps[2][256];   // sums over the set bits of the low and the high byte
  __shared__ double s_t[2 * kMaxBonds];           // -t_b, t_b
  __shared__ int s_job, s_stop;
  __shared__ double s_E;
  // layout: w over r_{j-1} | r_j (D each), alpha | beta (maxit each)
  const int tid = threadIdx.x;
  const bool two = A.M > 8;
  for (;;) {
    if (tid == 0) s_job = atomicAdd(A.counter, 1);
    __syncthreads();
    const int slot = s_job;
    if (slot >= A.n_jobs) return;
    const int job = A.order[slot];
    const int Nu = A.job_nup[job], Nd = A.job_ndn[job], P = A.job_param[job];
    const int nu = T.count[Nu], nd = T.count[Nd], D = nu * nd;
    double *w = sm, *q = sm + D;               // w starts as r_{j-1}
    double *alpha = sm + 2 * D, *beta = alpha + A.maxit;
    for (int i = tid; i < 2 * A.n_bonds; i += blockDim.x) {
      const double t = A.t[(int64_t)P * A.n_bonds + (i >> 1)];
      s_t[i] = (i & 1) ? t : -t;
    }
    for (int i = tid; i < (two ? 512 : 256); i += blockDim.x) {
      double su = 0.0, se = 0.0;
      for (int k = 0; k < 8; ++k) {
        const int site = (i >> 8) * 8 + k;
        if (!((i >> k) & 1) || site >= A.M) continue;
        su += A.U[(int64_t)P * A.M + site];
        if (A.eps) se += A.eps[(int64_t)P * A.M + site];
      }
      s_U[i >> 8][i & 255] = su;
      s_eps[i >> 8][i & 255] = se;
    }
    const uint32_t *bu = T.basis + T.off_basis[Nu], *bd = T.basis + T.off_basis[Nd];
    const int32_t *rpu = T.rp + T.off_rp[Nu], *rpd = T.rp + T.off_rp[Nd];
    const uint32_t *ell = T.ell + T.off_ell[Nu];
    // start vector: SplitMix64 uniform [-1, 1) with counter (job << 32) | (element + 1)
    double nrm = 0.0;
    for (int n = tid; n < D; n += blockDim.x) {
      uint64_t z = (((uint64_t)job << 32) | (uint64_t)(n + 1)) * 0x9E3779B97F4A7C15ull;
      z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
      z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
      z ^= z >> 31;
      const double v = (double)(z >> 11) * (2.0 / 9007199254740992.0) - 1.0;
      q[n] = v;
      w[n] = 0.0;
      nrm = fma(v, v, nrm);
    }
    double inv = 1.0 / sqrt(block_sum(nrm, red)), c = 0.0;   // q_j = inv r_j; beta_{j-1} q_{j-1} = c r_{j-1}
    // columns of a sweep, rows side by side, and the thread's place
    const int cols = min(nu, (int)blockDim.x), side = (int)blockDim.x / cols;
    const int g = tid / cols, uc = tid - g * cols;
    double E_prev = NAN, E = 0.0;
    int status = HUB_ERR_NOCONV, j = 0;
    if (tid == 0) s_stop = 0;
    for (j = 0; j < A.maxit; ++j) {
      __syncthreads();
      // w = H q - beta_{j-1} q_{j-1}; alpha = <q, w>
      double dot = 0.0;
      for (int u = g < side ? uc : nu; u < nu; u += cols) {
        const uint32_t Iu = bu[u];
        const int hops = rpu[u + 1] - rpu[u];
        double eu = s_eps[0][Iu & 255];
        if (two) eu += s_eps[1][Iu >> 8];
        for (int d0 = g; d0 < nd; d0 += 2 * side) {
          const int d1 = d0 + side < nd ? d0 + side : d0;
          const int n0 = d0 * nu, n1 = d1 * nu;
          const uint32_t I0 = bd[d0], I1 = bd[d1];
          double g0 = s_U[0][Iu & I0 & 255] + (eu + s_eps[0][I0 & 255]);
          double g1 = s_U[0][Iu & I1 & 255] + (eu + s_eps[0][I1 & 255]);
          if (two) {
            g0 += s_U[1][(Iu & I0) >> 8] + s_eps[1][I0 >> 8];
            g1 += s_U[1][(Iu & I1) >> 8] + s_eps[1][I1 >> 8];
          }
          const double q0 = q[n0 + u], q1 = q[n1 + u];
          double a0 = g0 * q0, a1 = g1 * q1;
#pragma unroll 4
          for (int k = 0; k < hops; ++k) {
            const uint32_t e = ell[k * nu + u];
            const double t = s_t[e >> 16];
            a0 = fma(t, q[n0 + (int)(e & 0xffffu)], a0);
            if (d1 != d0) a1 = fma(t, q[n1 + (int)(e & 0xffffu)], a1);
          }
#pragma unroll 4
          for (int k = rpd[d0]; k < rpd[d0 + 1]; ++k) {
            const uint32_t e = T.word[k];
            a0 = fma(s_t[e >> 16], q[(int)(e & 0xffffu) * nu + u], a0);
          }
          a0 = fma(-c, w[n0 + u], inv * a0);
          w[n0 + u] = a0;
          dot = fma(q0, a0, dot);
          if (d1 != d0) {
#pragma unroll 4
            for (int k = rpd[d1]; k < rpd[d1 + 1]; ++k) {
              const uint32_t e = T.word[k];
              a1 = fma(s_t[e >> 16], q[(int)(e & 0xffffu) * nu + u], a1);
            }
            a1 = fma(-c, w[n1 + u], inv * a1);
            w[n1 + u] = a1;
            dot = fma(q1, a1, dot);
          }
        }
      }
      const double a = inv * block_sum(dot, red), ai = a * inv;
      double nn = 0.0;
      for (int n = tid; n < D; n += blockDim.x) {
        const double v = fma(-ai, q[n], w[n]);
        w[n] = v;
        nn = fma(v, v, nn);
      }
      const double b = sqrt(block_sum(nn, red));
      if (tid == 0) {
        alpha[j] = a;
        beta[j] = b;
      }
      const bool breakdown = b <= 1e-14 * fmax(1.0, fabs(a));
      const bool check = breakdown || j + 1 == A.maxit || ((j + 1) % kBatchCheckEvery == 0);
      if (check) {
        __syncthreads();
        if (tid < 32) {
          const double e = tri_lowest_warp(alpha, beta, j + 1, E_prev);
          if (tid == 0) {
            s_E = e;
            int stop = 0;
            if (breakdown) stop = 2;
            else if (A.tol > 0 && j + 1 > kBatchCheckEvery && fabs(e - E_prev) < A.tol) stop = 1;
            s_stop = stop;
          }
        }
        __syncthreads();
        E = s_E;
        if (s_stop) {
          status = s_stop == 2 ? HUB_CONVERGED_BREAKDOWN : HUB_OK;
          ++j;
          break;
        }
        E_prev = E;
      }
      // r_{j+1} = w; rotate
      c = b * inv;
      inv = 1.0 / b;
      double *t0 = q;
      q = w;
      w = t0;
    }
    if (A.tol <= 0 && status == HUB_ERR_NOCONV) status = HUB_OK;
    if (tid == 0) {
      A.E0[job] = E;
      A.iters[job] = j > A.maxit ? A.maxit : j;
      A.status[job] = status;
    }
    __syncthreads();
  }
}

}  // namespace hub

using namespace hub;

extern "C" int hub_batch_ground(int M, int n_bonds, const int32_t *bonds_host, int n_params, const double *t_host,
                                const double *U_host, const double *eps_host, int n_jobs, const int32_t *job_nup,
                                const int32_t *job_ndn, const int32_t *job_param, int maxit, double tol,
                                double *E0_host, int32_t *iters_host, int32_t *status_host, void *stream) {
  if (M < 1 || M > kBatchMaxSites) return fail(HUB_ERR_ARG, "hub_batch_ground: need 1 <= M <= 16");
  if (n_params < 1 || n_jobs < 0 || maxit < 1 || maxit > 1000)
    return fail(HUB_ERR_ARG, "hub_batch_ground: need n_params >= 1, n_jobs >= 0, 1 <= maxit <= 1000");
  if (!t_host || !U_host || (n_jobs && (!job_nup || !job_ndn || !job_param || !E0_host || !iters_host || !status_host)))
    return fail(HUB_ERR_ARG, "hub_batch_ground: NULL argument");
  if (n_jobs == 0) return HUB_OK;
  std::vector<int> cnt(M + 1);
  for (int N = 0; N <= M; ++N) {
    double c = 1.0;
    for (int k = 1; k <= N; ++k) c = c * (M - N + k) / k;
    cnt[N] = (int)std::llround(c);
  }
  int Dmax = 1;
  for (int k = 0; k < n_jobs; ++k) {
    const int a = job_nup[k], b = job_ndn[k], p = job_param[k];
    if (a < 0 || a > M || b < 0 || b > M || p < 0 || p >= n_params)
      return fail(HUB_ERR_ARG, "hub_batch_ground: job " + std::to_string(k) + " has a bad sector or parameter set");
    const int64_t D = (int64_t)cnt[a] * cnt[b];
    if (D > kBatchMaxDim)
      return fail(HUB_ERR_ARG, "hub_batch_ground: job " + std::to_string(k) + " has dimension " + std::to_string(D) +
                                   " > 8192; use hub_lanczos_ground");
    Dmax = std::max<int>(Dmax, (int)D);
  }
  for (int k = 0; k < n_params * M; ++k)
    if (!(U_host[k] == U_host[k])) return fail(HUB_ERR_ARG, "hub_batch_ground: U is NaN");

  // the regular set-up checks the bonds, on the smallest sector
  std::vector<double> ones(std::max(n_bonds, 1), 1.0);
  {
    hub_t h = nullptr;
    int rc = hub_basis(M, 0, 0, &h);
    if (rc) return rc;
    rc = hub_hopping(h, n_bonds, bonds_host, ones.data(), nullptr);
    hub_free(h);
    if (rc) return rc;
  }
  // one-spin bases (ascending) and hopping structures of the particle numbers that occur; built here,
  // since they are a few hundred entries and the set-up kernels took 0.35 ms per particle number
  std::vector<char> used(M + 1, 0);
  for (int k = 0; k < n_jobs; ++k) used[job_nup[k]] = used[job_ndn[k]] = 1;
  std::vector<uint32_t> basis, word, ell, rank((size_t)1 << M);
  std::vector<int32_t> rp;
  BatchTables T{};
  for (int N = 0; N <= M; ++N) {
    T.off_basis[N] = (int)basis.size();
    T.off_rp[N] = (int)rp.size();
    T.off_ell[N] = (int)ell.size();
    T.count[N] = cnt[N];
    if (!used[N]) continue;
    uint32_t n = 0;
    for (uint32_t I = 0; I < (uint32_t)1 << M; ++I)
      if (popc32(I) == N) {
        rank[I] = n++;
        basis.push_back(I);
      }
    size_t longest = 0;
    const size_t first = rp.size();
    for (uint32_t r = 0; r < n; ++r) {
      const uint32_t I = basis[T.off_basis[N] + r];
      const size_t base = word.size();
      rp.push_back((int32_t)base);
      for (int b = 0; b < n_bonds; ++b) {
        const int lo = std::min(bonds_host[2 * b], bonds_host[2 * b + 1]);
        const int hi = std::max(bonds_host[2 * b], bonds_host[2 * b + 1]);
        if (((I >> lo) & 1u) == ((I >> hi) & 1u)) continue;
        const uint32_t between = ((1u << hi) - 1u) & ~((2u << lo) - 1u);
        const uint32_t odd = (uint32_t)popc32(I & between) & 1u;      // Jordan-Wigner sign (Eq. 8)
        word.push_back(rank[I ^ (1u << lo) ^ (1u << hi)] | (2u * (uint32_t)b + odd) << 16);
      }
      std::sort(word.begin() + base, word.end(), [](uint32_t x, uint32_t y) { return (x & 0xffffu) < (y & 0xffffu); });
      longest = std::max(longest, word.size() - base);
    }
    rp.push_back((int32_t)word.size());
    ell.resize(ell.size() + (size_t)n * longest, 0u);
    for (uint32_t r = 0; r < n; ++r)
      for (int32_t k = rp[first + r]; k < rp[first + r + 1]; ++k)
        ell[T.off_ell[N] + (size_t)(k - rp[first + r]) * n + r] = word[k];
  }
  // largest jobs first
  std::vector<int32_t> order(n_jobs);
  std::iota(order.begin(), order.end(), 0);
  std::stable_sort(order.begin(), order.end(), [&](int32_t a, int32_t b) {
    return (int64_t)cnt[job_nup[a]] * cnt[job_ndn[a]] > (int64_t)cnt[job_nup[b]] * cnt[job_ndn[b]];
  });

  // device copies of everything (freed before returning)
  std::vector<void *> owned;
  auto up = [&](const void *src, size_t bytes, const char *what) -> void * {
    void *p = nullptr;
    if (!dev_alloc(&p, bytes, what)) return nullptr;
    owned.push_back(p);
    if (src && cudaMemcpy(p, src, bytes, cudaMemcpyHostToDevice) != cudaSuccess) return nullptr;
    return p;
  };
  auto release = [&]() {
    for (void *p : owned) dev_free(p);
  };
  BatchArgs A{};
  A.M = M;
  A.n_bonds = n_bonds;
  A.n_jobs = n_jobs;
  A.maxit = maxit;
  A.tol = tol;
  T.basis = (const uint32_t *)up(basis.data(), sizeof(uint32_t) * basis.size(), "batch bases");
  T.rp = (const int32_t *)up(rp.data(), sizeof(int32_t) * rp.size(), "batch row pointers");
  T.word = (const uint32_t *)up(word.data(), sizeof(uint32_t) * std::max<size_t>(word.size(), 1), "batch hopping entries");
  T.ell = (const uint32_t *)up(ell.data(), sizeof(uint32_t) * std::max<size_t>(ell.size(), 1), "batch hopping entries");
  A.t = (const double *)up(t_host, sizeof(double) * std::max(n_params * n_bonds, 1), "batch t");
  A.U = (const double *)up(U_host, sizeof(double) * n_params * M, "batch U");
  A.eps = eps_host ? (const double *)up(eps_host, sizeof(double) * n_params * M, "batch eps") : nullptr;
  A.job_nup = (const int32_t *)up(job_nup, sizeof(int32_t) * n_jobs, "batch jobs");
  A.job_ndn = (const int32_t *)up(job_ndn, sizeof(int32_t) * n_jobs, "batch jobs");
  A.job_param = (const int32_t *)up(job_param, sizeof(int32_t) * n_jobs, "batch jobs");
  A.order = (const int32_t *)up(order.data(), sizeof(int32_t) * n_jobs, "batch order");
  A.counter = (int *)up(nullptr, kBatchClasses * sizeof(int), "batch queues");
  A.E0 = (double *)up(nullptr, sizeof(double) * n_jobs, "batch E0");
  A.iters = (int32_t *)up(nullptr, sizeof(int32_t) * n_jobs, "batch iterations");
  A.status = (int32_t *)up(nullptr, sizeof(int32_t) * n_jobs, "batch status");
  if (!T.basis || !T.rp || !T.word || !T.ell || !A.t || !A.U || (eps_host && !A.eps) || !A.job_nup || !A.job_ndn ||
      !A.job_param || !A.order || !A.counter || !A.E0 || !A.iters || !A.status) {
    release();
    return fail(HUB_ERR_OOM, "hub_batch_ground: device allocation or upload failed");
  }
  // The shared memory of a CTA holds two vectors of the largest job it may take, so one
  // launch for every job would give the small ones the large ones' footprint (one CTA per SM
  // at the impurity star's 4900 states), and its threads are idle or short of work at the other
  // end.  The jobs (largest first) are therefore cut into classes, each a launch on a stream of
  // its own with CTAs sized for it, whose CTAs fill the SMs together (independent queues, no
  // waits between the launches).
  cudaStream_t s = (cudaStream_t)stream;
  auto dim_of = [&](int32_t j) { return (int64_t)cnt[job_nup[j]] * cnt[job_ndn[j]]; };
  cudaStream_t side[kBatchClasses] = {s, nullptr};
  cudaEvent_t ev_ready = nullptr, ev_done[kBatchClasses] = {nullptr, nullptr};
  int rc = HUB_OK;
  cudaError_t e = cudaMemsetAsync(A.counter, 0, kBatchClasses * sizeof(int), s);
  if (e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_ready, cudaEventDisableTiming);
  if (e == cudaSuccess) e = cudaEventRecord(ev_ready, s);
  if (e == cudaSuccess)
    e = cudaFuncSetAttribute(k_batch_lanczos, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)(sizeof(double) * (2 * (size_t)Dmax + 2 * (size_t)maxit)));
  for (int p = 0, first = 0; p < kBatchClasses && e == cudaSuccess; ++p) {
    int n = 0;
    while (first + n < n_jobs && dim_of(order[first + n]) > kBatchClass[p].above) ++n;
    if (n == 0) continue;
    const size_t smem = sizeof(double) * (2 * (size_t)dim_of(order[first]) + 2 * (size_t)maxit);
    const int threads = kBatchClass[p].threads;
    int per_sm = 1;
    if (p) e = cudaStreamCreateWithFlags(&side[p], cudaStreamNonBlocking);
    if (p && e == cudaSuccess) e = cudaEventCreateWithFlags(&ev_done[p], cudaEventDisableTiming);
    if (p && e == cudaSuccess) e = cudaStreamWaitEvent(side[p], ev_ready, 0);
    if (e == cudaSuccess) e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_batch_lanczos, threads, smem);
    if (e != cudaSuccess) break;
    BatchArgs Ap = A;
    Ap.n_jobs = n;
    Ap.order = A.order + first;
    Ap.counter = A.counter + p;
    const int grid = std::max(1, std::min(n, num_sms() * std::max(per_sm, 1)));
    k_batch_lanczos<<<grid, threads, smem, side[p]>>>(T, Ap);
    e = cudaGetLastError();
    if (p && e == cudaSuccess) e = cudaEventRecord(ev_done[p], side[p]);
    if (p && e == cudaSuccess) e = cudaStreamWaitEvent(s, ev_done[p], 0);
    first += n;
  }
  if (e == cudaSuccess) e = cudaMemcpyAsync(E0_host, A.E0, sizeof(double) * n_jobs, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(iters_host, A.iters, sizeof(int32_t) * n_jobs, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaMemcpyAsync(status_host, A.status, sizeof(int32_t) * n_jobs, cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) rc = cuda_fail(e, "hub_batch_ground", __FILE__, __LINE__);
  for (int p = 1; p < kBatchClasses; ++p) {
    if (side[p]) {
      cudaStreamSynchronize(side[p]);   // nothing of this call may outlive it
      cudaStreamDestroy(side[p]);
    }
    if (ev_done[p]) cudaEventDestroy(ev_done[p]);
  }
  if (ev_ready) cudaEventDestroy(ev_ready);
  release();
  if (rc) return rc;
  for (int k = 0; k < n_jobs; ++k)
    if (status_host[k] == HUB_ERR_NOCONV) {
      set_error("hub_batch_ground: some jobs reached maxit before |dE0| < tol");
      return HUB_ERR_NOCONV;
    }
  return HUB_OK;
}
