// hub_grad.cu -- derivatives of H (K5): the bilinear forms a^T (dH/dtheta) b for every bond
// hopping t_b, on-site interaction U_i and site energy eps_i.
//
// With a = b = psi these are the Hellmann-Feynman gradients of E0 (per-bond hopping
// correlators, double occupancies, densities); with a = ybar, b = x they are the
// parameter cotangents of y = H x.  The derivative operators follow from Eq. 1:
//   dH/dt_b   = -sum_sigma (c+_i c_j + h.c.)   -> the hops of bond b in H_up and H_dn,
//                                                with the Jordan-Wigner sign of Eq. 8;
//   dH/dU_i   = n_{i up} n_{i dn}             -> bit i of (I_up & I_dn) (Sec. III.B);
//   dH/deps_i = n_{i up} + n_{i dn}.
//
// Every term of the product is one FP64 multiply-add here, so the FP64 unit bounds it; what has to
// be kept small is the work to sort the terms by parameter.  Two roles of CTAs (k_bilinear): for the
// spin-up hops a thread owns a position u and sums a[d][u] b[d][c] over many rows d, one register
// per entry c of u's hopping row; for the spin-down hops a warp owns a row d and 256 positions and
// sums eight entries of d's row at a time over them.  The sums then go to per-warp bins, and a
// second kernel adds the CTAs' partials in a fixed order.  Disordered 3x4 lattice at half filling
// (853,776 states, 2.2e7 terms, about 50 us of FP64 issue): 146 us, against 1406 us with one
// shared-memory FP64 atomic per spin-up term.
#include <algorithm>
#include <vector>

#include "hub_internal.cuh"

namespace hub {

int ready(const hub_ctx *h, const char *who);

struct GradArgs {
  int n_bonds;
  int n_par;            // n_bonds + 2M
  const uint8_t *bond_up, *bond_dn;
  int up_blocks;        // CTAs of the spin-up role, the first ones
  int max_up;           // entries of the longest spin-up hopping row
  int rows, stage;      // spin-up role: rows of an item; rows staged together (0: gathers from b itself)
};
constexpr int kGradThreads = 512, kGradWarps = kGradThreads / 32, kGradEntries = 8, kGradSeg = 256;
constexpr int kGradMaxBlocks = 608;      // partial sums kept per parameter

// Spin-up hops and the site energies' up part.  An item is kGradThreads positions x G.rows rows; eight
// entries of the positions' hopping rows at a time (the entry after the last is the position itself).
__device__ __forceinline__ void grad_up(const Ham &H, const GradArgs &G, const double *__restrict__ a,
                                        const double *__restrict__ b, double *__restrict__ bs,
                                        double *__restrict__ bins) {
  const int64_t nu = H.n_up, nd = H.n_dn;
  const int64_t cu = (nu + kGradThreads - 1) / kGradThreads, cd = (nd + G.rows - 1) / G.rows;
  for (int64_t item = blockIdx.x; item < cu * cd; item += G.up_blocks) {
    const int64_t u = item % cu * kGradThreads + threadIdx.x, d0 = item / cu * G.rows;
    const int64_t d1 = min(nd, d0 + G.rows);
    const bool live = u < nu;
    const int32_t j0 = live ? H.rp_up[u] : 0;
    const int hops = live ? H.rp_up[u + 1] - j0 : -1;
    for (int k0 = 0; k0 <= G.max_up; k0 += kGradEntries) {
      const int n = min(max(hops + 1 - k0, 0), kGradEntries);
      const int m = __reduce_max_sync(0xffffffffu, n);
      int idx[kGradEntries];
      double acc[kGradEntries];
#pragma unroll
      for (int e = 0; e < kGradEntries; ++e) {
        idx[e] = live ? (int)u : 0;
        if (e < n && k0 + e < hops) idx[e] = (int)(H.scol_up[j0 + k0 + e] & 0x7fffffffu);
        acc[e] = 0.0;
      }
      for (int64_t ds = d0; ds < d1; ds += max(G.stage, 1)) {
        const int S = (int)min((int64_t)max(G.stage, 1), d1 - ds);
        const double *__restrict__ row = b + ds * nu;
        if (G.stage) {
          __syncthreads();
#pragma unroll 8
          for (int64_t k = threadIdx.x; k < S * nu; k += kGradThreads) bs[k] = row[k];
          __syncthreads();
          row = bs;
        }
        for (int s = 0; s < S; ++s, row += nu) {
          const double av = live ? a[(ds + s) * nu + u] : 0.0;
#pragma unroll
          for (int e = 0; e < kGradEntries; ++e)
            if (e < m) acc[e] = fma(av, row[idx[e]], acc[e]);
        }
      }
#pragma unroll
      for (int e = 0; e < kGradEntries; ++e) {
        if (e >= n) continue;
        if (k0 + e < hops) {
          const int32_t k = j0 + k0 + e;
          atomicAdd(&bins[G.bond_up[k]], (H.scol_up[k] >> 31) ? acc[e] : -acc[e]);   // -(sign) a b
        } else {
          for (uint32_t i = H.basis_up[u]; i; i &= i - 1) atomicAdd(&bins[G.n_bonds + H.M + __ffs(i) - 1], acc[e]);
        }
      }
    }
  }
}

// Spin-down hops, interactions and the site energies' down part: per row d the entries are its hops
// (rows of b), its occupied sites (positions with that site occupied too) and one for the whole row.
__device__ __forceinline__ void grad_dn(const Ham &H, const GradArgs &G, const double *__restrict__ a,
                                        const double *__restrict__ b, double *__restrict__ bins) {
  const int64_t nu = H.n_up, nd = H.n_dn, segs = (nu + kGradSeg - 1) / kGradSeg;
  const int lane = threadIdx.x & 31, e_lane = lane & (kGradEntries - 1);
  const int64_t first = (int64_t)(blockIdx.x - G.up_blocks) * kGradWarps + (threadIdx.x >> 5);
  const int64_t step = (int64_t)(gridDim.x - G.up_blocks) * kGradWarps;
  for (int64_t item = first; item < nd * segs; item += step) {
    const int64_t d = item / segs, u0 = item % segs * kGradSeg, u1 = min(nu, u0 + kGradSeg);
    const double *__restrict__ arow = a + d * nu;
    const uint32_t Id = H.basis_dn[d];
    const int32_t j0 = H.rp_dn[d];
    const int hops = H.rp_dn[d + 1] - j0, sites = __popc(Id), all = hops + sites + 1;
    for (int k0 = 0; k0 < all; k0 += kGradEntries) {
      const int m = min(all - k0, kGradEntries), k = k0 + e_lane;
      int64_t from = d * nu;
      uint32_t mask = 0;
      if (k < hops)
        from = (int64_t)(H.scol_dn[j0 + k] & 0x7fffffffu) * nu;
      else if (k < hops + sites)
        mask = 1u << __fns(Id, 0, k - hops + 1);
      int64_t off[kGradEntries];
      uint32_t need[kGradEntries];
      double acc[kGradEntries];
#pragma unroll
      for (int e = 0; e < kGradEntries; ++e) {
        off[e] = __shfl_sync(0xffffffffu, from, e);
        need[e] = __shfl_sync(0xffffffffu, mask, e);
        acc[e] = 0.0;
      }
      for (int64_t u = u0 + lane; u < u1; u += 32) {
        const double av = arow[u];
        const uint32_t Iu = H.basis_up[u];
#pragma unroll
        for (int e = 0; e < kGradEntries; ++e)
          if (e < m && (Iu & need[e]) == need[e]) acc[e] = fma(av, b[off[e] + u], acc[e]);
      }
      const double v = warp_totals<kGradEntries>(acc);
      if (lane < m) {                        // the lanes' bins differ: a row's hops are of different bonds
        if (k < hops)
          bins[G.bond_dn[j0 + k]] += (H.scol_dn[j0 + k] >> 31) ? v : -v;
        else if (mask)
          bins[G.n_bonds + __ffs(mask) - 1] += v;
        else
          for (uint32_t i = Id; i; i &= i - 1) bins[G.n_bonds + H.M + __ffs(i) - 1] += v;
      }
      __syncwarp();
    }
  }
}

__global__ void __launch_bounds__(kGradThreads, 2) k_bilinear(const Ham H, GradArgs G, const double *__restrict__ a,
                                                              const double *__restrict__ b,
                                                              double *__restrict__ partials) {
  extern __shared__ double sm[];           // bins [warp][n_par], then staged rows of b
  for (int k = threadIdx.x; k < kGradWarps * G.n_par; k += kGradThreads) sm[k] = 0.0;
  __syncthreads();
  double *bins = sm + (threadIdx.x >> 5) * G.n_par;
  if ((int)blockIdx.x < G.up_blocks)
    grad_up(H, G, a, b, sm + kGradWarps * G.n_par, bins);
  else
    grad_dn(H, G, a, b, bins);
  __syncthreads();
  for (int k = threadIdx.x; k < G.n_par; k += kGradThreads) {
    double v = 0.0;
    for (int w = 0; w < kGradWarps; ++w) v += sm[w * G.n_par + k];
    partials[(int64_t)k * gridDim.x + blockIdx.x] = v;
  }
}

// out[k] = sum over blocks of partials[k][.], fixed order; one block per parameter.
__global__ void k_reduce_rows(const double *__restrict__ partials, int nblk, double *__restrict__ out) {
  __shared__ double s[256];
  const double *p = partials + (int64_t)blockIdx.x * nblk;
  double v = 0.0;
  for (int k = threadIdx.x; k < nblk; k += blockDim.x) v += p[k];
  s[threadIdx.x] = v;
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w) s[threadIdx.x] += s[threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0) out[blockIdx.x] = s[0];
}

// The launch: CTAs of both roles fill the SMs together (two of 512 threads each), half of them each.
struct GradLaunch {
  GradArgs G;
  int grid = 1;
  size_t smem = 0;
};
static GradLaunch grad_launch(const hub_ctx *h, const Ham &H) {
  const int half = std::min(num_sms(), kGradMaxBlocks / 2);   // CTAs of a role
  GradLaunch L;
  GradArgs &G = L.G;
  G.n_bonds = h->n_bonds;
  G.n_par = h->n_bonds + 2 * h->M;
  G.bond_up = h->csr[0].bond;
  G.bond_dn = h->csr[h->shared ? 0 : 1].bond;
  G.max_up = h->csr[0].max_row;
  const size_t bins = sizeof(double) * kGradWarps * G.n_par, row = sizeof(double) * (size_t)H.n_up;
  const size_t room = 220 * 1024 - 2 * 1024;
  G.stage = 0;
  if (bins + row <= room) G.stage = bins + row <= room / 2 ? (int)((room / 2 - bins) / row) : 1;
  const int64_t cu = (H.n_up + kGradThreads - 1) / kGradThreads;
  const int64_t cd = std::max<int64_t>(1, std::min<int64_t>(H.n_dn, half / std::max<int64_t>(cu, 1)));
  G.rows = (int)std::max<int64_t>(1, (H.n_dn + cd - 1) / cd);
  G.stage = std::min(G.stage, G.rows);
  L.smem = bins + row * (size_t)G.stage;
  G.up_blocks = (int)std::max<int64_t>(1, std::min<int64_t>(cu * ((H.n_dn + G.rows - 1) / G.rows), half));
  const int64_t items = H.n_dn * ((H.n_up + kGradSeg - 1) / kGradSeg);
  L.grid = G.up_blocks + (int)std::max<int64_t>(1, std::min<int64_t>((items + kGradWarps - 1) / kGradWarps, half));
  return L;
}
static int launch_bilinear(const Ham &H, const GradLaunch &L, const double *a, const double *b, double *P, double *out,
                           cudaStream_t s) {
  HUB_CUDA(cudaFuncSetAttribute(k_bilinear, cudaFuncAttributeMaxDynamicSharedMemorySize, 220 * 1024));
  k_bilinear<<<L.grid, kGradThreads, L.smem, s>>>(H, L.G, a, b, P);
  HUB_LAUNCH_CHECK();
  k_reduce_rows<<<L.G.n_par, 256, 0, s>>>(P, L.grid, out);
  HUB_LAUNCH_CHECK();
  return HUB_OK;
}

// Computes all n_bonds + 2M bilinear forms into host arrays.
static int bilinear(hub_ctx *h, const double *a, const double *b, double *dt, double *dU, double *de,
                    cudaStream_t s) {
  const Ham H = h->view();
  const GradLaunch L = grad_launch(h, H);
  const GradArgs &G = L.G;
  int rc = ensure_partials(h, (int64_t)G.n_par * L.grid + G.n_par);
  if (rc) return rc;
  double *P = h->partials, *out = h->partials + (int64_t)G.n_par * L.grid;
  if ((rc = launch_bilinear(H, L, a, b, P, out, s))) return rc;
  std::vector<double> host(G.n_par);
  HUB_CUDA(cudaMemcpyAsync(host.data(), out, sizeof(double) * G.n_par, cudaMemcpyDeviceToHost, s));
  HUB_CUDA(cudaStreamSynchronize(s));
  for (int k = 0; k < h->n_bonds; ++k)
    if (dt) dt[k] = host[k];
  for (int i = 0; i < h->M; ++i) {
    if (dU) dU[i] = host[h->n_bonds + i];
    if (de) de[i] = host[h->n_bonds + h->M + i];
  }
  return HUB_OK;
}

}  // namespace hub

using namespace hub;

extern "C" int hub_grad(hub_t h, const double *psi_dev, double *dE_dt_host, double *dE_dU_host,
                        double *dE_deps_host, void *stream) {
  int rc = ready(h, "hub_grad");
  if (rc) return rc;
  if (h->k0) return fail(HUB_ERR_STATE, "hub_grad: not available in the k = 0 sector (hub_set_symmetry)");
  if (!psi_dev) return fail(HUB_ERR_ARG, "hub_grad: psi is NULL");
  return bilinear(h, psi_dev, psi_dev, dE_dt_host, dE_dU_host, dE_deps_host, (cudaStream_t)stream);
}

extern "C" int hub_apply_vjp(hub_t h, const double *ybar_dev, const double *x_dev, double *xbar_dev,
                             double *tbar_host, double *Ubar_host, double *epsbar_host, void *stream) {
  int rc = ready(h, "hub_apply_vjp");
  if (rc) return rc;
  if (h->k0) return fail(HUB_ERR_STATE, "hub_apply_vjp: not available in the k = 0 sector (hub_set_symmetry)");
  if (!ybar_dev || (!x_dev && (tbar_host || Ubar_host || epsbar_host)))
    return fail(HUB_ERR_ARG, "hub_apply_vjp: NULL vector");
  cudaStream_t s = (cudaStream_t)stream;
  if (xbar_dev) {
    const int64_t D = h->count[0] * h->count[1];
    if (xbar_dev < ybar_dev + D && ybar_dev < xbar_dev + D) return fail(HUB_ERR_ARG, "hub_apply_vjp: xbar overlaps ybar");
    if ((rc = apply_launch(h, ybar_dev, xbar_dev, s))) return rc;
  }
  if (tbar_host || Ubar_host || epsbar_host) {
    if ((rc = bilinear(h, ybar_dev, x_dev, tbar_host, Ubar_host, epsbar_host, s))) return rc;
  } else {
    HUB_CUDA(cudaStreamSynchronize(s));
  }
  return HUB_OK;
}

// ---------------------------------------------------------------------------------------
// hub_grad_noalloc: the Hellmann-Feynman gradients with no memory allocation at call time.
// The per-block partial sums and the reduced results live in one file-scope device array
// of fixed size instead of the handle's lazily allocated scratch.
// ---------------------------------------------------------------------------------------
namespace hub {

constexpr int kNoAllocMaxParams = 160;   // n_bonds + 2M that fit the fixed array
constexpr int64_t kNoAllocDoubles = (int64_t)kGradMaxBlocks * kNoAllocMaxParams + kNoAllocMaxParams;

// 608 * 160 + 160 doubles = 779,520 bytes, held by every GPU that loads the library.
static __device__ __align__(256) double g_grad_scratch[kNoAllocDoubles];

// Device address of g_grad_scratch on the current device.  In host code the symbol
// g_grad_scratch is only a host-side stand-in; kernels must be given this address.  It is
// looked up on every call (a host-side lookup once the library's device code is loaded on
// the device), so a context that was torn down and created again never sees a stale
// address; the first call on a device may load that code, which places the array there.
static int noalloc_scratch(double **out) {
  void *p = nullptr;
  HUB_CUDA(cudaGetSymbolAddress(&p, g_grad_scratch));
  *out = static_cast<double *>(p);
  return HUB_OK;
}

}  // namespace hub

extern "C" int hub_grad_noalloc(hub_t h, const double *psi_dev, double *dE_dt_host, double *dE_dU_host,
                                double *dE_deps_host, void *stream) {
  int rc = ready(h, "hub_grad_noalloc");
  if (rc) return rc;
  if (h->k0) return fail(HUB_ERR_STATE, "hub_grad_noalloc: not available in the k = 0 sector (hub_set_symmetry)");
  if (!psi_dev) return fail(HUB_ERR_ARG, "hub_grad_noalloc: psi is NULL");
  const int n_par = h->n_bonds + 2 * h->M;
  if (n_par > kNoAllocMaxParams)
    return fail(HUB_ERR_ARG, "hub_grad_noalloc: n_bonds + 2*M = " + std::to_string(n_par) +
                                 " exceeds the fixed scratch capacity of " + std::to_string(kNoAllocMaxParams) +
                                 " parameters; use hub_grad");
  int dev = 0;
  HUB_CUDA(cudaGetDevice(&dev));
  if (dev != h->device) return fail(HUB_ERR_ARG, "hub_grad_noalloc: the handle's device is not the current device");
  double *scratch = nullptr;
  if ((rc = noalloc_scratch(&scratch))) return rc;

  const Ham H = h->view();
  const GradLaunch L = grad_launch(h, H);
  // every partial the reduction reads is written by this call's first kernel, and every
  // result by its second, so nothing needs clearing between calls
  double *P = scratch, *out = scratch + (int64_t)n_par * L.grid;
  cudaStream_t s = (cudaStream_t)stream;
  if ((rc = launch_bilinear(H, L, psi_dev, psi_dev, P, out, s))) return rc;
  if (dE_dt_host && h->n_bonds)
    HUB_CUDA(cudaMemcpyAsync(dE_dt_host, out, sizeof(double) * h->n_bonds, cudaMemcpyDeviceToHost, s));
  if (dE_dU_host)
    HUB_CUDA(cudaMemcpyAsync(dE_dU_host, out + h->n_bonds, sizeof(double) * h->M, cudaMemcpyDeviceToHost, s));
  if (dE_deps_host)
    HUB_CUDA(cudaMemcpyAsync(dE_deps_host, out + h->n_bonds + h->M, sizeof(double) * h->M, cudaMemcpyDeviceToHost, s));
  HUB_CUDA(cudaStreamSynchronize(s));
  return HUB_OK;
}
