// hub_apply.cu -- the matrix-free Hamiltonian product (K3).
//
// Sec. IV.A, Eq. 11: H = I_dn (x) H_up + H_dn (x) I_up + H_U.  With the state stored as
// the count_dn x count_up row-major matrix X (Eq. count2; the vecold reshape of Sec.
// IV.A), the spin-up term is X H_up^T -- a gather inside one row of X -- and the
// spin-down term is H_dn X -- a combination of whole rows of X (Sec. IV.A: "vecnew =
// H_up x vecold" and "vecnew = vecold x H_dn^T", transposed to this row-major layout).
// The diagonal (Sec. III.B) is sum_i U_i bit_i(I_up & I_dn) + eps(I_up) + eps(I_dn),
// computed on the fly from popcount instead of Algorithm II's index_U tables.
//
// Kernel shape (FP64 path): a CTA takes two rows d of X and a chunk of columns u; each thread owns
// columns u and sums the H_up row of u (gathers from the two rows through L1; an entry's column and
// value are loaded once for both) and the H_dn rows of both d (coalesced loads of the neighbour rows
// X[d'][u], served from L2).  The FP64 unit bounds it: one multiply-add per term, at about 1/70 of the
// integer rate (12-site ring, every t and U its own, 853,776 states, 1.2e7 hops: 45 us, about 26 us of FP64
// issue).  Staging the two rows in shared memory gained nothing at any row length (1716 entries: 0.114 ms
// either way) and left an SM one CTA of 256 threads for rows of 6,000 to 12,800 entries: 4x4 (6,3), 8008
// entries, 0.46 ms staged, 0.29 ms not; 3x6 (5,4) 3.67 and 1.6 ms.
// Columns are cut at multiples of a warp, since a partial warp costs the unit a whole one.
#include "hub_internal.cuh"

namespace hub {

// The diagonal with the sums over doubly occupied sites from a table: one lookup per eight sites
// instead of one divergent read of the parameters per set bit.  (One per four sites costs up to seven
// FP64 additions a state: 13-site ring (6,6) 146 us against 135 us.)
__device__ __forceinline__ double f64_diag(const Ham &H, const double *s_U, uint32_t both, int64_t u, int64_t d) {
  double v;
  if (H.uniform_U) {
    v = H.U0 * (double)__popc(both);
  } else {
    v = s_U[both & 255];
    for (int k = 1; 8 * k < H.M; ++k) v += s_U[256 * k + ((both >> 8 * k) & 255)];
  }
  if (H.has_eps) v += H.eps_up[u] + H.eps_dn[d];
  return v;
}
// The Lanczos step around a product, in the same kernel (hub_lanczos.cu): see F64Step.
// kMode 0: y = H x.  kMode 1: y = inv (H x) - c prev and the CTA's part of inv <x, y>.
// kMode 2: psi += v x, y = (H x - a x - c prev) inv (second pass, known coefficients).
// gate: null, or a device flag; the kernel does nothing while gate[0] is 0 (the other paths
// pass their out-of-window flag, so that this kernel multiplies exactly the vectors they cannot).
template <int kMode, int kF64Rows>
__global__ void __launch_bounds__(256, 6) k_apply_f64(const Ham H, const double *__restrict__ x, double *y,
                                                   const int *__restrict__ gate, int chunks, const F64Step L) {
  if (gate) {
    after_previous();
    if (flag_of(gate) == 0) return;
  }
  // Sums of U_i over the set bits of each eight sites, from those of each four; only where U varies, since
  // the L1 that serves the gathers shrinks by it (uniform U, 17-site ring (7,2): 0.105 ms, with 9 KB 0.117).
  extern __shared__ double s_tab[];
  const double *s_U = s_tab + 128;
  if (!H.uniform_U) {
    for (int k = threadIdx.x; k < 128; k += blockDim.x) {
      double v = 0.0;
      for (int i = 0; i < 4; ++i)
        if (((k >> i) & 1) && (k >> 4) * 4 + i < H.M) v += H.U[(k >> 4) * 4 + i];
      s_tab[k] = v;
    }
    __syncthreads();
    for (int k = threadIdx.x; k < (H.M + 7) / 8 * 256; k += blockDim.x)
      s_tab[128 + k] = s_tab[(k >> 8) * 32 + (k & 15)] + s_tab[(k >> 8) * 32 + 16 + ((k >> 4) & 15)];
    __syncthreads();
  }
  const int64_t nu = H.n_up, nd = H.n_dn;
  const int64_t width = ((nu + chunks - 1) / chunks + 31) & ~(int64_t)31, items = (nd + kF64Rows - 1) / kF64Rows * chunks;
  double inv = 1.0, c = 0.0, dot = 0.0;
  if (kMode == 1) {
    inv = L.scal->inv;
    c = L.scal->c;
  }
  for (int64_t item = blockIdx.x; item < items; item += gridDim.x) {
    const int64_t d = item / chunks * kF64Rows, u0 = item % chunks * width, u1 = min(nu, u0 + width);
    const int rows = kF64Rows == 1 ? 1 : (int)min((int64_t)kF64Rows, nd - d);
    const double *__restrict__ r0 = x + d * nu, *__restrict__ r1 = rows > 1 ? r0 + nu : r0;
    const uint32_t Id0 = H.basis_dn[d], Id1 = rows > 1 ? H.basis_dn[d + 1] : 0u;
    const int32_t k0 = H.rp_dn[d], k1 = H.rp_dn[d + 1], k2 = rows > 1 ? H.rp_dn[d + 2] : k1;
    for (int64_t u = u0 + threadIdx.x; u < u1; u += blockDim.x) {
      const double x0 = r0[u], x1 = r1[u];
      const uint32_t Iu = H.basis_up[u];
      double acc0 = f64_diag(H, s_U, Iu & Id0, u, d) * x0;
      double acc1 = rows > 1 ? f64_diag(H, s_U, Iu & Id1, u, d + 1) * x1 : 0.0;
      const int32_t j0 = H.rp_up[u], j1 = H.rp_up[u + 1];
#pragma unroll 2
      for (int32_t k = j0; k < j1; ++k) {
        const int32_t e = H.col_up[k];
        const double v = H.val_up[k];
        acc0 = fma(v, r0[e], acc0);
        if (rows > 1) acc1 = fma(v, r1[e], acc1);
      }
#pragma unroll 4
      for (int32_t k = k0; k < k1; ++k) acc0 = fma(H.val_dn[k], x[(int64_t)H.col_dn[k] * nu + u], acc0);
#pragma unroll 4
      for (int32_t k = k1; k < k2; ++k) acc1 = fma(H.val_dn[k], x[(int64_t)H.col_dn[k] * nu + u], acc1);
#pragma unroll
      for (int r = 0; r < kF64Rows; ++r) {
        if (r >= rows) break;
        const int64_t o = (d + r) * nu + u;
        double v = r ? acc1 : acc0;
        const double xv = r ? x1 : x0;
        if (kMode == 1) {
          v = fma(-c, L.prev[o], inv * v);
          dot = fma(xv, v, dot);
        } else if (kMode == 2) {
          L.psi[o] = fma(L.v, xv, L.psi[o]);
          v = (fma(-L.a, xv, v) - L.b * L.prev[o]) * L.inv;
        }
        y[o] = v;
      }
    }
  }
  if (kMode == 1) f64_step_alpha(L, dot);
}

static int apply_kernels(hub_ctx *h, const double *x, double *y, cudaStream_t s);

constexpr int64_t kMaxTimed = 65536;

int prof_mark(hub_ctx *h, int kind, bool begin, cudaStream_t s) {
  if (!h->prof) return HUB_OK;
  int64_t &nt = h->n_timed[kind];
  if (begin) {
    if (nt >= kMaxTimed) return HUB_OK;
    if ((int64_t)h->ev_start[kind].size() <= nt) {
      cudaEvent_t e0, e1;
      HUB_CUDA(cudaEventCreate(&e0));
      HUB_CUDA(cudaEventCreate(&e1));
      h->ev_start[kind].push_back(e0);
      h->ev_end[kind].push_back(e1);
    }
    HUB_CUDA(cudaEventRecord(h->ev_start[kind][nt], s));
  } else {
    ++h->n_launch[kind];
    if (nt >= kMaxTimed) return HUB_OK;
    HUB_CUDA(cudaEventRecord(h->ev_end[kind][nt], s));
    ++nt;
  }
  return HUB_OK;
}

int apply_launch(hub_ctx *h, const double *x, double *y, cudaStream_t s) {
  int rc = prof_mark(h, HUB_PROF_APPLY, true, s);
  if (rc) return rc;
  if ((rc = apply_kernels(h, x, y, s))) return rc;
  return prof_mark(h, HUB_PROF_APPLY, false, s);
}

// Products of few terms go to the FP64 kernel: one launch.  Its 1.2e7 terms on the 12-site ring (6,6)
// take 44 us against 69 us for the fixed-point path, whose launches alone take 45 us; beyond
// about 2.2e7 terms (80 us) the FP64 unit costs more than the launches.
constexpr double kF64Terms = 2.2e7;
static bool f64_is_faster(const hub_ctx *h) {
  const double nu = (double)h->count[0], nd = (double)h->count[1];
  const double terms = (double)h->csr[0].nnz * nd + (double)h->csr[h->shared ? 0 : 1].nnz * nu + nu * nd;
  return !h->k0 && !h->fail_waits && terms <= kF64Terms;   // the test hook needs kernels that wait
}

static int apply_kernels(hub_ctx *h, const double *x, double *y, cudaStream_t s) {
  const Ham H = h->view();
  if (H.n_up == 0 || H.n_dn == 0) return HUB_OK;
  set_route(h, h->k0 ? HUB_ROUTE_SYM : HUB_ROUTE_FP64);
  if (h->k0) return k0_apply(h, x, y, s);
  if (f64_is_faster(h)) return f64_apply(h, x, y, nullptr, s);
  if (fix_apply_eligible(h)) {
    const int rc = fix_apply(h, x, y, s);
    if (rc != HUB_ERR_OOM) return rc;
    fast_release_scratch(h);          // its vectors do not fit (nor the double-float path's, the same ones)
    set_error("");
    set_route(h, HUB_ROUTE_FP64);
    return f64_apply(h, x, y, nullptr, s);
  }
  if (use_fast(h)) return fast_apply_f64(h, x, y, s);
  return f64_apply(h, x, y, nullptr, s);
}

void set_route(hub_ctx *h, int route, const int *f64_flag, const int *df_flag) {
  h->route = route;
  h->route_flag[0] = f64_flag;
  h->route_flag[1] = df_flag;
}

// Columns of a CTA: chunks of 256 and less where the row is short, so that a small matrix still makes
// several CTAs per SM; a quarter of a longer row.
static int f64_chunks(const Ham &H) { return (int)std::min<int64_t>(4, (H.n_up + 255) / 256); }
// Rows of a CTA: two, or one where rows are so narrow that a CTA has few threads at work (12 columns x 924
// rows: 8.1 us, 10.7 with two) or the matrix is so small that two would leave SMs idle (252 x 252: 7.6 us,
// 10.3 with two).
static int f64_rows(const Ham &H) {
  return H.n_up > 128 && (H.n_dn + 1) / 2 * f64_chunks(H) >= 2 * num_sms() ? 2 : 1;
}
int64_t f64_grid(const Ham &H) {
  const int rows = f64_rows(H);
  return std::min<int64_t>((H.n_dn + rows - 1) / rows * f64_chunks(H), (int64_t)num_sms() * 16);
}
bool f64_product(hub_ctx *h) {
  return !h->k0 && (f64_is_faster(h) || (!fix_apply_eligible(h) && !use_fast(h)));
}
template <int kMode>
static int f64_launch(hub_ctx *h, const double *x, double *y, const int *gate, const F64Step &L, cudaStream_t s) {
  const Ham H = h->view();
  count_launch(h);
  const int chunks = f64_chunks(H);
  const int64_t width = (H.n_up + chunks - 1) / chunks;
  const int threads = width > 128 ? 256 : (width > 64 ? 128 : 64);
  // behind the other paths' kernels (gate) it has nothing to do as a rule: no more CTAs than are resident
  const int grid = (int)(gate ? std::min<int64_t>(f64_grid(H), (int64_t)num_sms() * 6) : f64_grid(H));
  const size_t tab = H.uniform_U ? 0 : sizeof(double) * (128 + (size_t)(H.M + 7) / 8 * 256);
  HUB_CUDA(launch_kernel(gate && !h->prof, f64_rows(H) == 1 ? k_apply_f64<kMode, 1> : k_apply_f64<kMode, 2>, grid,
                         threads, tab, s, H, x, y, gate, chunks, L));
  return HUB_OK;
}
int f64_apply(hub_ctx *h, const double *x, double *y, const int *gate, cudaStream_t s) {
  return f64_launch<0>(h, x, y, gate, F64Step(), s);
}
int f64_apply_step(hub_ctx *h, const double *x, double *y, const F64Step &L, bool second, cudaStream_t s) {
  int rc = prof_mark(h, HUB_PROF_APPLY, true, s);
  if (rc || (rc = second ? f64_launch<2>(h, x, y, nullptr, L, s) : f64_launch<1>(h, x, y, nullptr, L, s))) return rc;
  return prof_mark(h, HUB_PROF_APPLY, false, s);
}

static int check_ready(const hub_ctx *h, const char *who) {
  if (!h) return fail(HUB_ERR_ARG, std::string(who) + ": NULL handle");
  if (!h->have_hop) return fail(HUB_ERR_STATE, std::string(who) + ": call hub_hopping first");
  if (!h->have_U) return fail(HUB_ERR_STATE, std::string(who) + ": call hub_set_U first");
  return HUB_OK;
}

int ready(const hub_ctx *h, const char *who) { return check_ready(h, who); }

}  // namespace hub

using namespace hub;

extern "C" int hub_apply(hub_t h, const double *x_dev, double *y_dev, void *stream) {
  int rc = check_ready(h, "hub_apply");
  if (rc) return rc;
  if (!x_dev || !y_dev) return fail(HUB_ERR_ARG, "hub_apply: NULL vector");
  const int64_t D = vec_len(h);
  if (x_dev < y_dev + D && y_dev < x_dev + D) return fail(HUB_ERR_ARG, "hub_apply: x and y overlap");
  return apply_launch(h, x_dev, y_dev, (cudaStream_t)stream);
}

// The FP64 device input and output vector of a host-buffer apply (x, y: hx and hy, or the
// second pair hx2 and hy2), allocated on first use.
static int host_apply_buffers(hub_ctx *h, double **x, double **y) {
  if (*x) return HUB_OK;
  const int64_t D = vec_len(h);
  if (!dev_alloc((void **)x, sizeof(double) * D, "host-apply input") ||
      !dev_alloc((void **)y, sizeof(double) * D, "host-apply output")) {
    dev_free(*x);
    *x = nullptr;
    return HUB_ERR_OOM;
  }
  return HUB_OK;
}

extern "C" int hub_last_route(hub_t h, int *route) {
  if (!h || !route) return fail(HUB_ERR_ARG, "hub_last_route: NULL argument");
  const int to[2] = {HUB_ROUTE_FP64, HUB_ROUTE_DF};
  *route = h->route;
  HUB_CUDA(cudaDeviceSynchronize());
  for (int k = 0; k < 2; ++k) {
    int flag = 0;
    if (h->route_flag[k]) HUB_CUDA(cudaMemcpy(&flag, h->route_flag[k], sizeof(int), cudaMemcpyDeviceToHost));
    if (flag) {
      *route = to[k];
      break;
    }
  }
  return HUB_OK;
}

extern "C" int hub_apply_host(hub_t h, const double *x_host, double *y_host, void *stream) {
  int rc = check_ready(h, "hub_apply_host");
  if (rc) return rc;
  if (!x_host || !y_host) return fail(HUB_ERR_ARG, "hub_apply_host: NULL vector");
  const int64_t D = vec_len(h);
  if ((rc = host_apply_buffers(h, &h->hx, &h->hy))) return rc;
  cudaStream_t s = (cudaStream_t)stream;
  if (use_fast(h) && fast_host_pipelined(h)) return fast_apply_host(h, x_host, y_host, h->hx, h->hy, s);
  HUB_CUDA(cudaMemcpyAsync(h->hx, x_host, sizeof(double) * D, cudaMemcpyHostToDevice, s));
  rc = apply_launch(h, h->hx, h->hy, s);
  if (rc) return rc;
  HUB_CUDA(cudaMemcpyAsync(y_host, h->hy, sizeof(double) * D, cudaMemcpyDeviceToHost, s));
  HUB_CUDA(cudaStreamSynchronize(s));
  return HUB_OK;
}

extern "C" int hub_apply_host_many(hub_t h, int64_t n_vec, const double *x_host, double *y_host, void *stream) {
  int rc = check_ready(h, "hub_apply_host_many");
  if (rc) return rc;
  if (n_vec < 0) return fail(HUB_ERR_ARG, "hub_apply_host_many: negative vector count");
  if (n_vec == 0) return HUB_OK;
  if (!x_host || !y_host) return fail(HUB_ERR_ARG, "hub_apply_host_many: NULL vector");
  const int64_t D = vec_len(h);
  if (D > 0 && n_vec > (int64_t)(SIZE_MAX / sizeof(double)) / D)
    return fail(HUB_ERR_ARG, "hub_apply_host_many: vector count too large");
  const uintptr_t xa = (uintptr_t)x_host, ya = (uintptr_t)y_host, bytes = (uintptr_t)(n_vec * D) * sizeof(double);
  if (xa != ya && xa < ya + bytes && ya < xa + bytes)
    return fail(HUB_ERR_ARG, "hub_apply_host_many: x and y overlap without being the same array");
  if (n_vec == 1 || !use_fast(h) || !fast_host_pipelined(h)) {   // one call per vector
    for (int64_t v = 0; v < n_vec; ++v)
      if ((rc = hub_apply_host(h, x_host + v * D, y_host + v * D, stream))) return rc;
    return HUB_OK;
  }
  if ((rc = host_apply_buffers(h, &h->hx, &h->hy)) || (rc = host_apply_buffers(h, &h->hx2, &h->hy2))) return rc;
  double *const xd[2] = {h->hx, h->hx2}, *const yd[2] = {h->hy, h->hy2};
  return fast_apply_host_many(h, n_vec, x_host, y_host, xd, yd, (cudaStream_t)stream);
}

extern "C" int hub_profile(hub_t h, int enable) {
  if (!h) return fail(HUB_ERR_ARG, "hub_profile: NULL handle");
  h->prof = enable != 0;
  if (h->prof) {
    for (int k = 0; k < hub_ctx::kProfKinds; ++k) h->n_launch[k] = h->n_timed[k] = 0;
    h->n_kernels = 0;
  }
  return HUB_OK;
}

extern "C" int hub_profile_read(hub_t h, int kind, double *ms, int64_t *launches, int64_t *kernel_launches) {
  if (!h || kind < 0 || kind >= hub_ctx::kProfKinds) return fail(HUB_ERR_ARG, "hub_profile_read: bad argument");
  double total = 0.0;
  for (int64_t k = 0; k < h->n_timed[kind]; ++k) {
    HUB_CUDA(cudaEventSynchronize(h->ev_end[kind][k]));
    float t = 0.f;
    HUB_CUDA(cudaEventElapsedTime(&t, h->ev_start[kind][k], h->ev_end[kind][k]));
    total += t;
  }
  const int64_t nt = h->n_timed[kind], nl = h->n_launch[kind];
  if (ms) *ms = nt ? total * (double)nl / (double)nt : 0.0;
  if (launches) *launches = nl;
  if (kernel_launches) *kernel_launches = h->n_kernels;
  return HUB_OK;
}

extern "C" int hub_set_mode(hub_t h, int mode) {
  if (!h || (mode != HUB_MODE_AUTO && mode != HUB_MODE_FP64)) return fail(HUB_ERR_ARG, "hub_set_mode: bad argument");
  h->mode = mode;
  return HUB_OK;
}

extern "C" int hub_test_fail_waits(hub_t h, int enable) {
  if (!h) return fail(HUB_ERR_ARG, "hub_test_fail_waits: NULL handle");
  h->fail_waits = enable != 0;
  return HUB_OK;
}

extern "C" int hub_check(hub_t h) {
  if (!h) return fail(HUB_ERR_ARG, "hub_check: NULL handle");
  HUB_CUDA(cudaDeviceSynchronize());
  const int rc = fast_check_error(h);
  return rc ? rc : small_check_error(h);
}
