// hub_fast.cu -- double-float products for uniform hopping: of vectors that the fixed-point path
// (hub_fix.cu) does not serve, and of host buffers in row chunks.
//
// The product is Eq. 11 of Sec. IV.A on the count_dn x count_up state matrix X (Eq.
// count2):  Y = X H_up^T + H_dn X + diag o X, with every hopping element -t * esign
// (Eq. 8) and diag = U popcount(I_up & I_dn) + eps(I_up) + eps(I_dn) (Sec. III.B).  The
// two hopping terms want different memory orders, so they run as two passes:
//
//   pass 1 (k_up): a CTA takes two rows (d0, d1) of X at a time.  Both rows are copied
//     whole into shared memory by bulk asynchronous copies (cp.async.bulk, completion on
//     an mbarrier), then each thread sums the H_up row of its column u for both rows from
//     shared memory (in-row gather) and adds the diagonal:
//     Z[d][u] = t S_up + diag X[d][u].
//   pass 2 (k_dn): tiles of 32 rows x 64 columns, launched strip-major (all tiles of one
//     column strip are adjacent in the grid), so the strip of X that the H_dn rows
//     combine -- count_dn x 64 values -- stays in L2 while the whole strip is processed
//     and X is read from HBM about once.  Each warp adds t S_dn to Z for its rows with
//     64-bit loads of whole rows of the strip.
//
// Vectors are double-float (hub_df.cuh), stored planar per row: row d of a vector is 2 ld
// floats, the ld high parts followed by the ld low parts (ld >= count_up, a multiple of 4,
// padding columns zero).  Both planes of a row start on 16-byte boundaries (bulk copies),
// and the two values a packed FP32x2 instruction combines always sit in adjacent words:
// (hi of row d0, hi of row d1) come from two 32-bit shared loads in pass 1, and the
// (hi, hi) / (lo, lo) pairs of columns u, u+1 from two 64-bit loads in pass 2, so no
// register shuffling is needed around the TwoSum chains.  Inside this file the columns of X
// are kept in "slot" order: spin-up states sorted by the lengths of their two hopping
// groups, so that the 32 rows of H_up a warp sums in pass 1 have nearly equal lengths
// (little divergence) while its loads and stores stay contiguous.  Pass 2 combines whole
// rows and does not care about column order.  Only the FP64 <-> double-float conversions
// at the boundary of this file map slots back to ranks.  The hopping rows are reordered by
// sign (entries adding x first, then entries subtracting x), so no per-term sign handling
// is needed, and columns are stored as uint16 when count <= 65536.
#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "hub_df.cuh"
#include "hub_internal.cuh"

namespace hub {

int ready(const hub_ctx *h, const char *who);
std::vector<double> tridiag_vector(const double *a, const double *b, int k, double lam);

// ---------------------------------------------------------------------------------------
// Small PTX wrappers: mbarrier and bulk copy (sm_90+).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}
__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}
__device__ __forceinline__ void fence_mbar_init() {
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ void fence_proxy_async() {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_g2s(void *dst, const void *src, uint32_t bytes, uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
          smem_u32(dst)),
      "l"(src), "r"(bytes), "r"(smem_u32(bar))
      : "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t *bar, uint32_t phase) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(phase)
      : "memory");
  return ok != 0;
}
// Bounded wait: gives up after ~2^24 polls (each poll may suspend the thread briefly).
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t *bar, uint32_t phase) {
  for (uint32_t it = 0; it < (1u << 24); ++it)
    if (mbar_try_wait(bar, phase)) return true;
  return false;
}

// ---------------------------------------------------------------------------------------
// Fast-path view (passed by value).
// ---------------------------------------------------------------------------------------
struct FastView {
  int64_t n_up, n_dn, ld;            // ld: plane length of a row (multiple of 4); row stride 2 ld
  const uint32_t *basis_up, *basis_dn;
  const int32_t *rp_up, *sp_up;      // row start and sign split of H_up
  const int32_t *rp_dn, *sp_dn;
  const void *col_up, *col_dn;       // uint16 or uint32 columns
  // H_up in sliced column-major form for pass 1.  Rows are placed in slots ordered by their
  // (add, sub) group lengths so that the 32 rows a warp handles have nearly equal lengths;
  // slot k holds row slot_row[k].  Each slice of 32 slots has, per group, a schedule of
  // steps: in one step every lane reads at most one of its entries, chosen so that at most
  // two lanes of the warp hit the same shared-memory bank (column mod 32).  A word holds the
  // columns of two steps (uint16) or one (uint32); the words of a slice are stored in
  // batches of four per lane, word i of batch b of slot k at off[k/32] + (b*32 + k%32)*4 + i,
  // so that one 16-byte load brings a lane 8 (uint16) or 4 (uint32) steps.  Idle steps
  // (schedule gaps, padding of the last word and batch) name a zero column (staged rows) or
  // the sentinel 0xffff / 0xffffffff (rows read through L2).
  const uint32_t *sl_add, *sl_sub;   // packed words
  const int32_t *sl_off_add, *sl_off_sub;
  const uint16_t *steps_add, *steps_sub;   // per slice: scheduled steps (entries per lane)
  uint32_t idle_word;                // a column word whose entries are all idle steps
  const int32_t *slot_row;           // spin-up rank held by slot k
  const uint32_t *basis_up_slot;     // spin-up strings in slot order
  int t_neg;                         // the kernels apply H / |t|: hopping sign(t), diagonal U k / |t|
  float2 Utab[32];                   // (U / |t|) k for k = popcount(I_up & I_dn)
  int *err;                          // device error flag (bounded waits)
  const int *gate;                   // null, or a device flag: the kernels do nothing while it is 0
  int fail_waits;                    // test hook: take the given-up-wait exit once the copies landed
};

template <typename Col>
__device__ __forceinline__ uint32_t colat(const void *c, int64_t k) {
  return (uint32_t)((const Col *)c)[k];
}

// ---------------------------------------------------------------------------------------
// Sign-split CSR: per row, entries with esign = -1 (element +t: add x) first, then the
// entries with esign = +1 (element -t: subtract x); columns ascending inside each group.
// ---------------------------------------------------------------------------------------
template <typename Col>
__global__ void k_split_csr(int64_t n, const int32_t *__restrict__ rp, const uint32_t *__restrict__ scol,
                            int32_t *__restrict__ sp, Col *__restrict__ col) {
  for (int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; r < n; r += (int64_t)gridDim.x * blockDim.x) {
    const int32_t a = rp[r], b = rp[r + 1];
    int32_t w = a;
    for (int32_t k = a; k < b; ++k)
      if (scol[k] >> 31) col[w++] = (Col)(scol[k] & 0x7fffffffu);
    sp[r] = w;
    for (int32_t k = a; k < b; ++k)
      if (!(scol[k] >> 31)) col[w++] = (Col)(scol[k] & 0x7fffffffu);
  }
}

// basis of the spin-up states in slot order
__global__ void k_to_slots(int64_t n, const int32_t *__restrict__ slot_row, const uint32_t *__restrict__ basis,
                           uint32_t *__restrict__ basis_slot) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    basis_slot[k] = basis[slot_row[k]];
}

// ---------------------------------------------------------------------------------------
// Conversions between the ABI's FP64 layout (row length n_up, rank order) and the planar
// double-float layout (slot order), with a power-of-two scale.
// ---------------------------------------------------------------------------------------
// The fast path holds a vector as double-floats scaled by 2^-shift, max |x| 2^-shift in
// [1, 2).  Its per-entry error bound (about 20 u^2 (|H||x|)_n, u = 2^-24) needs every
// term, product and sum it forms to keep 48 bits, i.e. FP32 low parts above the FP32
// subnormal range: with nonzero |x| 2^-shift >= 2^-80 and a diagonal coefficient U / |t|
// of 0 or in [2^-16, 2^16] (fast_eligible), every nonzero product is at least 2^-96, its
// low part at least 2^-120.  The scaled results must also map back into the FP64 range.
// The window:
// the largest biased FP64 exponent in [kExpLo, kExpHi] and every nonzero entry's exponent
// at most kExpSpan below it; FP64 subnormals, infinities and NaN are outside.  A vector
// outside the window is multiplied by the FP64 kernel instead.

// partials[block] = largest biased FP64 exponent of the block's elements (2047 for inf or
// NaN), partials[nblk + block] = smallest biased exponent among its nonzero elements (0 for
// an FP64 subnormal, 2048 if all are zero); nblk = gridDim.x
__global__ void k_exp_range(int64_t D, const double *__restrict__ x, int *__restrict__ partials) {
  int m = 0, n = 2048;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < D; k += (int64_t)gridDim.x * blockDim.x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x[k]);
    const int e = (int)((b >> 52) & 0x7ffu);
    m = max(m, e);
    if (b << 1) n = min(n, e);
  }
  for (int o = 16; o > 0; o >>= 1) {
    m = max(m, __shfl_xor_sync(0xffffffffu, m, o));
    n = min(n, __shfl_xor_sync(0xffffffffu, n, o));
  }
  __shared__ int wm[32], wn[32];
  if ((threadIdx.x & 31) == 0) {
    wm[threadIdx.x >> 5] = m;
    wn[threadIdx.x >> 5] = n;
  }
  __syncthreads();
  if (threadIdx.x < 32) {
    const bool in = threadIdx.x < (blockDim.x >> 5);
    int a = in ? wm[threadIdx.x] : 0, c = in ? wn[threadIdx.x] : 2048;
    for (int o = 16; o > 0; o >>= 1) {
      a = max(a, __shfl_xor_sync(0xffffffffu, a, o));
      c = min(c, __shfl_xor_sync(0xffffffffu, c, o));
    }
    if (threadIdx.x == 0) {
      partials[blockIdx.x] = a;
      partials[gridDim.x + blockIdx.x] = c;
    }
  }
}

// Range of partials[0 .. nblk) (stride: nblk to the minima, as k_exp_range writes them;
// n_sets such sets back to back).
__device__ __forceinline__ void range_of(const int *__restrict__ p, int nblk, int n_sets, int &emax, int &emin) {
  int a = 0, c = 2048;
  for (int s = 0; s < n_sets; ++s)
    for (int k = threadIdx.x; k < nblk; k += blockDim.x) {
      a = max(a, p[2 * s * nblk + k]);
      c = min(c, p[(2 * s + 1) * nblk + k]);
    }
  for (int o = 16; o > 0; o >>= 1) {
    a = max(a, __shfl_xor_sync(0xffffffffu, a, o));
    c = min(c, __shfl_xor_sync(0xffffffffu, c, o));
  }
  __shared__ int wa[32], wc[32];
  if ((threadIdx.x & 31) == 0) {
    wa[threadIdx.x >> 5] = a;
    wc[threadIdx.x >> 5] = c;
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < (int)(blockDim.x >> 5); ++k) {
      a = max(a, wa[k]);
      c = min(c, wc[k]);
    }
    emax = a;
    emin = c;
  }
}

__device__ __forceinline__ bool out_of_window(int emax, int emin) {
  return emax != 0 && (emax < kExpLo || emax > kExpHi || emin < emax - kExpSpan);
}

// One block: scale[0] = shift (max |x| 2^-shift in [1, 2); 0 for a zero vector), scale[1] =
// 1 if the vector lies outside the fast path's window (see kExpSpan).
__global__ void k_scale(const int *__restrict__ partials, int nblk, int *__restrict__ scale) {
  int emax = 0, emin = 2048;
  range_of(partials, nblk, 1, emax, emin);
  if (threadIdx.x == 0) {
    scale[0] = emax == 0 ? 0 : emax - 1023;
    scale[1] = out_of_window(emax, emin) ? 1 : 0;
  }
}

// Host-buffer product, after all chunks: n_sets exponent partial sets (one per chunk, the
// first one gave the scale used so far).  scale[2] = shift of the whole vector, scale[3] =
// its window flag; flag[0] = 2 if the whole vector lies outside the window, 1 if its
// largest exponent exceeds the first chunk's (convert again with scale[2]), else 0.
__global__ void k_scale_all(const int *__restrict__ partials, int nblk, int n_sets, int *__restrict__ scale,
                            int *__restrict__ flag) {
  int emax = 0, emin = 2048;
  range_of(partials, nblk, n_sets, emax, emin);
  if (threadIdx.x == 0) {
    const int shift = emax == 0 ? 0 : emax - 1023;
    const bool out = out_of_window(emax, emin);
    scale[2] = shift;
    scale[3] = out ? 1 : 0;
    flag[0] = out ? 2 : (shift != scale[0] ? 1 : 0);
  }
}

// out (planar, slot order) = 2^-shift x (FP64, rank order) for rows r0 .. r1 - 1, shift =
// scale[0] (0 when scale is null); one row per block and step
__global__ void k_f64_to_df(int64_t r0, int64_t r1, int64_t n_up, int64_t ld, const double *__restrict__ x,
                            const int *__restrict__ scale, const int32_t *__restrict__ slot_row,
                            float *__restrict__ out, const int *__restrict__ gate) {
  if (gate) {
    after_previous();
    if (flag_of(gate) == 0) return;
  }
  const int shift = scale ? scale[0] : 0;
  for (int64_t d = r0 + blockIdx.x; d < r1; d += gridDim.x) {
    float *__restrict__ row = out + d * 2 * ld;
    const double *__restrict__ xr = x + d * n_up;
    for (int64_t u = threadIdx.x; u < ld; u += blockDim.x) {
      const float2 v = u < n_up ? f64_to_df(xr[slot_row[u]], shift) : make_float2(0.f, 0.f);
      row[u] = v.x;
      row[ld + u] = v.y;
    }
  }
}

// y[d][u] (FP64, rank order) = tabs 2^shift v[d][slot_of[u]] (planar double-float, slot
// order) for rows r0 .. r1 - 1, shift = scale[0]; one row per block and step so that the
// gathers of a row are served from L1.  Nothing is written when scale[1] is set (the FP64
// kernel writes y instead).  tabs = |t|: the kernels applied H / |t|.
__global__ void k_unpermute(int64_t r0, int64_t r1, int64_t n_up, int64_t ld, const float *__restrict__ v,
                            const int32_t *__restrict__ slot_of, const int *__restrict__ scale, double tabs,
                            double *__restrict__ y, const int *__restrict__ gate) {
  if (gate) after_previous();
  if (flag_of(scale + 1) || (gate && flag_of(gate) == 0)) return;
  const int shift = scale[0];
  for (int64_t d = r0 + blockIdx.x; d < r1; d += gridDim.x) {
    const float *__restrict__ row = v + d * 2 * ld;
    for (int64_t u = threadIdx.x; u < n_up; u += blockDim.x) {
      const int32_t s = slot_of[u];
      const double val = df_to_f64(make_float2(row[s], row[ld + s]), shift);
      y[d * n_up + u] = tabs == 1.0 ? val : val * tabs;
    }
  }
}

// ---------------------------------------------------------------------------------------
// Pass 1: spin-up hops (in-row gather from shared memory) and the diagonal.  A CTA takes
// two rows (d0, d1) at a time: their four planes are staged (four bulk copies completing on
// one mbarrier), every column index is loaded once for both rows, and the two rows' TwoSum
// chains run as one packed FP32x2 chain.  While a pair is computed, the CTA's next pair is
// prefetched into L2.
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

// Staged planes: hi(d0), lo(d0), hi(d1), lo(d1) at k * kUpPlane floats (compile-time
// offsets, so the four loads of a term share one address; kUpPlane is a multiple of 32, so
// all planes have the same bank alignment).  Entries ld and ld + 1 of every plane are zero
// and serve as the column of idle schedule steps (adding zero is exact).
constexpr int kUpPlane = 14080;

#ifndef HUB_UP_PAIRED
#define HUB_UP_PAIRED 1   // 1: pass 1 sums with DfSumP (low parts of a word's two entries paired); 0: DfSum4
#endif
#ifndef HUB_UP_THREADS
#define HUB_UP_THREADS 1024   // threads of the pass-1 CTA (one CTA per SM; fewer leave more registers)
#endif
constexpr int kUpThreads = HUB_UP_THREADS;
static_assert(kUpThreads % 32 == 0 && kUpThreads >= 512 && kUpThreads <= 1024, "pass-1 CTA size");
template <typename Col>
__global__ void __launch_bounds__(kUpThreads, 1) k_up(const FastView F, const float *__restrict__ x,
                                                      float *__restrict__ z, int64_t p_begin, int64_t p_end) {
  if (F.gate) {
    after_previous();
    if (flag_of(F.gate) == 0) return;
  }
  extern __shared__ __align__(128) unsigned char smem_raw[];
  float *xs = reinterpret_cast<float *>(smem_raw);
  __shared__ __align__(8) uint64_t bar;
  __shared__ float2 utab[32];
  const int tid = threadIdx.x;
  const int64_t ld = F.ld;
  const uint32_t pbytes = (uint32_t)(ld * sizeof(float));
  if (tid < 32) utab[tid] = F.Utab[tid];
  if (tid < 8) xs[(tid >> 1) * kUpPlane + ld + (tid & 1)] = 0.f;
  if (tid == 0) {
    mbar_init(&bar, 1);
    fence_mbar_init();
  }
  __syncthreads();
  uint32_t phase = 0;
  for (int64_t p = p_begin + blockIdx.x; p < p_end; p += gridDim.x) {   // row pairs p_begin .. p_end - 1
    const int64_t d0 = 2 * p, d1 = (2 * p + 1 < F.n_dn) ? 2 * p + 1 : 2 * p;   // odd tail: same row twice
    if (tid == 0) {
      const float *r0 = x + d0 * 2 * ld, *r1 = x + d1 * 2 * ld;
      fence_proxy_async();
      mbar_expect_tx(&bar, 4 * pbytes);
      bulk_g2s(xs, r0, pbytes, &bar);
      bulk_g2s(xs + kUpPlane, r0 + ld, pbytes, &bar);
      bulk_g2s(xs + 2 * kUpPlane, r1, pbytes, &bar);
      bulk_g2s(xs + 3 * kUpPlane, r1 + ld, pbytes, &bar);
      const int64_t pn = p + gridDim.x;
      if (pn < p_end) {
        prefetch_l2(x + 2 * pn * 2 * ld, 2 * pbytes);
        if (2 * pn + 1 < F.n_dn) prefetch_l2(x + (2 * pn + 1) * 2 * ld, 2 * pbytes);
      }
    }
    if (!mbar_wait_bounded(&bar, phase)) {
      if (tid == 0) atomicExch(F.err, 1);
      mbar_wait_bounded(&bar, phase);      // give a late copy one more bounded chance to land
      return;
    }
    if (F.fail_waits) {                    // test hook: the same exit, after the copies landed
      if (tid == 0) atomicExch(F.err, 1);
      return;
    }
    phase ^= 1u;
    const uint32_t I0 = F.basis_dn[d0], I1 = F.basis_dn[d1];
    float *__restrict__ z0 = z + d0 * 2 * ld;
    float *__restrict__ z1 = z + d1 * 2 * ld;
    for (int64_t slot = tid; slot < ld; slot += blockDim.x) {
      if (slot >= F.n_up) {                        // padding columns of Z stay zero
        z0[slot] = 0.f;
        z0[ld + slot] = 0.f;
        z1[slot] = 0.f;
        z1[ld + slot] = 0.f;
        continue;
      }
#if HUB_UP_PAIRED
      DfSumP acc{0ull, 0ull, 0ull, {0ull, 0ull}};
#else
      DfSum4 acc{0ull, 0ull, 0ull, {0ull, 0ull, 0ull, 0ull}};
#endif
      const int64_t sl = slot >> 5, lane = slot & 31;
      const uint4 *__restrict__ wa = reinterpret_cast<const uint4 *>(F.sl_add + F.sl_off_add[sl]) + lane;
      const uint4 *__restrict__ wsb = reinterpret_cast<const uint4 *>(F.sl_sub + F.sl_off_sub[sl]) + lane;
      const int na = F.steps_add[sl], ns = F.steps_sub[sl];
      // the (hi d0, hi d1) and (lo d0, lo d1) pairs of staged column C (idle steps read the zero
      // column)
#define HUB_HI(C) pk2(xs[(C)], xs[(C) + 2 * kUpPlane])
#define HUB_LO(C) pk2(xs[(C) + kUpPlane], xs[(C) + 3 * kUpPlane])
#if HUB_UP_PAIRED
      // uint16: one word, both of its scheduled entries as a pair, the low parts to accumulator
      // J (alternating by the word's position in its batch); uint32 (one entry per word): the
      // batch's words x, y as one pair (accumulator 0) and z, w as another (accumulator 1), so
      // that either way an accumulator takes one pair sum per four scheduled entries
#define HUB_WORD(ADD, J, WD)                                                             \
  do {                                                                                   \
    const uint32_t ca_ = (WD) & 0xffffu, cb_ = (WD) >> 16;                               \
    sump_pair(acc, HUB_HI(ca_), HUB_LO(ca_), HUB_HI(cb_), HUB_LO(cb_), (ADD), (J));      \
  } while (0)
#define HUB_J(w) (w)
#else
      // one scheduled entry: J, the low-part accumulator, by the entry's position in its batch
#define HUB_TERM(ADD, J, C)                                                              \
  do {                                                                                   \
    if (ADD)                                                                             \
      sum4_add(acc, HUB_HI(C), HUB_LO(C), (J));                                          \
    else                                                                                 \
      sum4_sub(acc, HUB_HI(C), HUB_LO(C), (J));                                          \
  } while (0)
#define HUB_WORD(ADD, J, WD)                                                             \
  do {                                                                                   \
    if (sizeof(Col) == 2) {                                                              \
      HUB_TERM(ADD, (J), (WD) & 0xffffu);                                                \
      HUB_TERM(ADD, (J) + 1, (WD) >> 16);                                                \
    } else {                                                                             \
      HUB_TERM(ADD, (J), (WD));                                                          \
    }                                                                                    \
  } while (0)
#define HUB_J(w) (((w) * (sizeof(Col) == 2 ? 2 : 1)) & 3)
#endif
      // Full batches of four words run unguarded; the last batch is taken word by word
      // (a word's padding step reads the zero column).  N is uniform over the warp.
#define HUB_GROUP(ADD, W, N)                                                             \
  do {                                                                                   \
    constexpr int kPer = sizeof(Col) == 2 ? 8 : 4;       /* steps per batch */           \
    constexpr int kPerWord = sizeof(Col) == 2 ? 2 : 1;                                   \
    const int nst = (N), nb = (nst + kPer - 1) / kPer;                                   \
    uint4 qn = nb > 0 ? W[0] : make_uint4(0u, 0u, 0u, 0u);                               \
    for (int b = 0; b < nb; ++b) {                                                       \
      const uint4 q = qn;                                                                \
      if (b + 1 < nb) qn = W[(b + 1) * 32];     /* next batch's columns in flight */     \
      const int rem = nst - kPer * b;                                                    \
      if (HUB_UP_PAIRED && sizeof(Col) == 4) {                                           \
        HUB_PAIR32(ADD, 0, q.x, q.y, rem > 1);                                           \
        if (rem > 2) HUB_PAIR32(ADD, 1, q.z, q.w, rem > 3);                              \
      } else {                                                                           \
        HUB_WORD(ADD, HUB_J(0), q.x);                                                    \
        if (rem > kPerWord) HUB_WORD(ADD, HUB_J(1), q.y);                                \
        if (rem > 2 * kPerWord) HUB_WORD(ADD, HUB_J(2), q.z);                            \
        if (rem > 3 * kPerWord) HUB_WORD(ADD, HUB_J(3), q.w);                            \
      }                                                                                  \
    }                                                                                    \
  } while (0)
#if HUB_UP_PAIRED
      // two 32-bit words as one pair, or the first alone when the batch ends after it
#define HUB_PAIR32(ADD, J, WA, WB, BOTH)                                                 \
  do {                                                                                   \
    if (BOTH)                                                                            \
      sump_pair(acc, HUB_HI(WA), HUB_LO(WA), HUB_HI(WB), HUB_LO(WB), (ADD), (J));        \
    else                                                                                 \
      sump_one(acc, HUB_HI(WA), HUB_LO(WA), (ADD), (J));                                 \
  } while (0)
#else
#define HUB_PAIR32(ADD, J, WA, WB, BOTH) \
  do {                                   \
  } while (0)
#endif
      HUB_GROUP(true, wa, na);
      HUB_GROUP(false, wsb, ns);
#undef HUB_GROUP
#undef HUB_PAIR32
#undef HUB_WORD
#undef HUB_J
#undef HUB_TERM
#undef HUB_HI
#undef HUB_LO
      // Z = diag x + t' S for both rows (packed), t' = +-1
      f2x Sh, Sl;
#if HUB_UP_PAIRED
      sump_norm(acc, Sh, Sl);
#else
      sum4_norm(acc, Sh, Sl);
#endif
      if (F.t_neg) {
        Sh ^= kSign2;
        Sl ^= kSign2;
      }
      const uint32_t Iu = F.basis_up_slot[slot];
      const float2 dg0 = utab[__popc(Iu & I0)], dg1 = utab[__popc(Iu & I1)];
      f2x ph, pl, zh, zl;
      df2_mul(pk2(dg0.x, dg1.x), pk2(dg0.y, dg1.y), pk2(xs[slot], xs[slot + 2 * kUpPlane]),
              pk2(xs[slot + kUpPlane], xs[slot + 3 * kUpPlane]), ph, pl);
      df2_add(ph, pl, Sh, Sl, zh, zl);
      const float2 h = upk2(zh), l = upk2(zl);
      z0[slot] = h.x;
      z0[ld + slot] = l.x;
      if (d1 != d0) {
        z1[slot] = h.y;
        z1[ld + slot] = l.y;
      }
    }
    __syncthreads();
  }
}

// ---------------------------------------------------------------------------------------
// Rows too long to stage (e.g. C(18, 9) = 48620 columns, 194 KB per plane): pass 1 runs on
// the transposed matrix instead.  X^T is formed by a tiled transpose, the spin-up hops then
// combine whole rows of X^T exactly as pass 2 combines rows of X (k_dn in mode 2, diagonal
// in the epilogue), and the result is transposed back into Z.  Each transpose moves a
// vector once through HBM; gathers through L2 would instead touch two sectors per term.
// ---------------------------------------------------------------------------------------
constexpr int kTile = 32;

// dst[c][r] = src[r][c] for planar matrices: src has n_r rows (plane length ld_s, n_c valid
// columns), dst has n_c rows of plane length ld_d; dst columns n_r .. ld_d - 1 are zeroed.
// Block (32, 8): a 32 x 32 tile of both planes through shared memory.
__global__ void __launch_bounds__(256) k_transpose(int64_t n_r, int64_t n_c, int64_t ld_s, int64_t ld_d,
                                                   const float *__restrict__ src, float *__restrict__ dst,
                                                   const int *__restrict__ gate) {
  if (gate) {
    after_previous();
    if (flag_of(gate) == 0) return;
  }
  __shared__ float th[kTile][kTile + 1], tl[kTile][kTile + 1];
  const int tx = threadIdx.x, ty = threadIdx.y;
  const int64_t c0 = (int64_t)blockIdx.x * kTile, r0 = (int64_t)blockIdx.y * kTile;
#pragma unroll
  for (int j = 0; j < kTile; j += 8) {
    const int64_t r = r0 + ty + j, c = c0 + tx;
    const bool in = r < n_r && c < n_c;
    th[ty + j][tx] = in ? src[r * 2 * ld_s + c] : 0.f;
    tl[ty + j][tx] = in ? src[r * 2 * ld_s + ld_s + c] : 0.f;
  }
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kTile; j += 8) {
    const int64_t c = c0 + ty + j, r = r0 + tx;
    if (c < n_c && r < ld_d) {
      dst[c * 2 * ld_d + r] = th[tx][ty + j];
      dst[c * 2 * ld_d + ld_d + r] = tl[tx][ty + j];
    }
  }
}

// ---------------------------------------------------------------------------------------
// Pass 2: spin-down hops as combinations of whole rows of a column strip, plus the
// epilogue.  Tile = 32 rows x 64 columns; blockIdx.x = row tile (fast), blockIdx.y =
// column strip (slow), so consecutive blocks share a strip.  Lane l of a warp owns the
// columns u0 + 2l, u0 + 2l + 1 (one 64-bit load per plane and row), and sums both with one
// packed FP32x2 TwoSum chain.
// ---------------------------------------------------------------------------------------
#ifndef HUB_DN_LANE_COLS
#define HUB_DN_LANE_COLS 4   // columns per lane in pass 2 (2: 64-bit loads, 4: 128-bit loads)
#endif
constexpr int kDnRows = 32, kDnLaneCols = HUB_DN_LANE_COLS, kDnCols = 32 * kDnLaneCols, kDnThreads = 256;
#ifndef HUB_DN_BATCH
#define HUB_DN_BATCH 2   // strip rows whose loads are issued together in pass 2
#endif
#ifndef HUB_DN_MINB
#define HUB_DN_MINB 5    // resident pass-2 CTAs per SM that the register allocation aims for
#endif

// The hopping side a row-combination pass works on: the rows of the matrix it reads are the
// states of this side, its columns (n_cols valid of ld) the states of the other side.
struct Side {
  int64_t n_rows, n_cols, ld;
  const int32_t *rp, *sp;            // sign-split CSR of this side's hopping matrix
  const void *col;
  int64_t r_begin = 0;               // first row a launch covers (rows r_begin .. n_rows - 1)
};

__device__ __forceinline__ f2x ld2(const float *p) { return *reinterpret_cast<const f2x *>(p); }
__device__ __forceinline__ void st2(float *p, f2x v) { *reinterpret_cast<f2x *>(p) = v; }


// kLane packed pairs per lane: columns u .. u + 2 kLane - 1 (16-byte loads for even kLane)
template <int kLane>
struct Vec {
  f2x v[kLane];
};
template <int kLane>
__device__ __forceinline__ Vec<kLane> ldv(const float *p) {
  Vec<kLane> r;
  if (kLane % 2 == 0) {
#pragma unroll
    for (int i = 0; i < kLane / 2; ++i) {
      const float4 q = reinterpret_cast<const float4 *>(p)[i];
      r.v[2 * i] = pk2(q.x, q.y);
      r.v[(2 * i + 1) % kLane] = pk2(q.z, q.w);
    }
  } else {
    r.v[0] = *reinterpret_cast<const f2x *>(p);
  }
  return r;
}
template <int kLane>
__device__ __forceinline__ void stv(float *p, const Vec<kLane> &a) {
  if (kLane % 2 == 0) {
#pragma unroll
    for (int i = 0; i < kLane / 2; ++i) {
      const float2 x = upk2(a.v[2 * i]), y = upk2(a.v[(2 * i + 1) % kLane]);
      reinterpret_cast<float4 *>(p)[i] = make_float4(x.x, x.y, y.x, y.y);
    }
  } else {
    *reinterpret_cast<f2x *>(p) = a.v[0];
  }
}

// Strip rows k, k + 1 of one sign group (loads issued together) into the lane's accumulators
// as a pair whose low parts go to accumulator J.
template <int kLane, int J, bool kAdd, typename Col>
__device__ __forceinline__ void dn_pair(DfSumP (&acc)[kLane], const Side &S, const char *__restrict__ xh,
                                        const char *__restrict__ xl, int32_t k, uint32_t row_bytes) {
  Vec<kLane> vh[2], vl[2];
#pragma unroll
  for (int q = 0; q < 2; ++q) {
    const uint64_t o = (uint64_t)colat<Col>(S.col, k + q) * row_bytes;
    vh[q] = ldv<kLane>(reinterpret_cast<const float *>(xh + o));
    vl[q] = ldv<kLane>(reinterpret_cast<const float *>(xl + o));
  }
#pragma unroll
  for (int i = 0; i < kLane; ++i) sump_pair(acc[i], vh[0].v[i], vl[0].v[i], vh[1].v[i], vl[1].v[i], kAdd, J);
}

// The strip rows ka .. kb - 1 of one sign group (bounds warp-uniform): pairs of rows with
// their low parts into the two accumulators in turn (HUB_DN_BATCH = 4: two pairs' loads in
// flight together), a last single row into accumulator 1.
template <int kLane, bool kAdd, typename Col>
__device__ __forceinline__ void dn_group(DfSumP (&acc)[kLane], const Side &S, const char *__restrict__ xh,
                                         const char *__restrict__ xl, int32_t ka, int32_t kb, uint32_t row_bytes) {
  static_assert(HUB_DN_BATCH == 2 || HUB_DN_BATCH == 4, "HUB_DN_BATCH must be 2 or 4");
  int32_t k = ka;
  for (; k + 4 <= kb; k += 4) {
    if (HUB_DN_BATCH == 4) {
      Vec<kLane> vh[4], vl[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const uint64_t o = (uint64_t)colat<Col>(S.col, k + q) * row_bytes;
        vh[q] = ldv<kLane>(reinterpret_cast<const float *>(xh + o));
        vl[q] = ldv<kLane>(reinterpret_cast<const float *>(xl + o));
      }
#pragma unroll
      for (int i = 0; i < kLane; ++i) {
        sump_pair(acc[i], vh[0].v[i], vl[0].v[i], vh[1].v[i], vl[1].v[i], kAdd, 0);
        sump_pair(acc[i], vh[2].v[i], vl[2].v[i], vh[3].v[i], vl[3].v[i], kAdd, 1);
      }
    } else {
      dn_pair<kLane, 0, kAdd, Col>(acc, S, xh, xl, k, row_bytes);
      dn_pair<kLane, 1, kAdd, Col>(acc, S, xh, xl, k + 2, row_bytes);
    }
  }
  if (k + 2 <= kb) {
    dn_pair<kLane, 0, kAdd, Col>(acc, S, xh, xl, k, row_bytes);
    k += 2;
  }
  if (k < kb) {
    const uint64_t o = (uint64_t)colat<Col>(S.col, k) * row_bytes;
    const Vec<kLane> vh = ldv<kLane>(reinterpret_cast<const float *>(xh + o));
    const Vec<kLane> vl = ldv<kLane>(reinterpret_cast<const float *>(xl + o));
#pragma unroll
    for (int i = 0; i < kLane; ++i) sump_one(acc[i], vh.v[i], vl.v[i], kAdd, 1);
  }
}

// kMode 0: w (planar double-float, slot order; may alias z) = Z + t S_dn, for hub_apply
//          (the FP64 output in rank order is written afterwards by k_unpermute).
// kMode 2: pass 1 on X^T (side = spin up, rows of x are spin-up states, columns spin-down
//          states): w = t S_up + diag x, diag from the two basis strings (no z).
template <typename Col, int kMode>
__global__ void __launch_bounds__(kDnThreads, HUB_DN_MINB) k_dn(const FastView F, const Side S, const float *__restrict__ x,
                                                  const float *z, float *w) {
  if (F.gate) {
    after_previous();
    if (flag_of(F.gate) == 0) return;
  }
  constexpr int kLane = kDnLaneCols / 2;               // packed pairs per lane
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t ld = S.ld;
  __shared__ float2 utab[kMode == 2 ? 32 : 1];
  if (kMode == 2) {
    if (threadIdx.x < 32) utab[threadIdx.x] = F.Utab[threadIdx.x];
    __syncthreads();
  }
  const int64_t u = (int64_t)blockIdx.y * kDnCols + kDnLaneCols * lane;
  const int64_t r0 = S.r_begin + (int64_t)blockIdx.x * kDnRows;
  const uint32_t row_bytes = (uint32_t)(2 * ld * sizeof(float));
  const bool active = u < S.n_cols;                    // u + kDnLaneCols <= ld (see fast_build)
  const char *__restrict__ xh = reinterpret_cast<const char *>(x + u);
  const char *__restrict__ xl = reinterpret_cast<const char *>(x + ld + u);
  for (int rr = warp; rr < kDnRows; rr += kDnThreads / 32) {
    const int64_t d = r0 + rr;
    if (d >= S.n_rows) break;
    const int32_t k0 = S.rp[d], ks = S.sp[d], k1 = S.rp[d + 1];
    float *wr = w + d * 2 * ld;
    if (!active) {
      if (u < ld) {                                      // padding columns of w stay zero
        stv<kLane>(wr + u, Vec<kLane>{});
        stv<kLane>(wr + ld + u, Vec<kLane>{});
      }
      continue;
    }
    DfSumP acc[kLane];
#pragma unroll
    for (int i = 0; i < kLane; ++i) acc[i] = DfSumP{0ull, 0ull, 0ull, {0ull, 0ull}};
    dn_group<kLane, true, Col>(acc, S, xh, xl, k0, ks, row_bytes);
    dn_group<kLane, false, Col>(acc, S, xh, xl, ks, k1, row_bytes);
    Vec<kLane> yh, yl;
    if (kMode == 2) {
      // diag x for the columns (spin-down states) u .. u + kDnLaneCols - 1 of spin-up row d
      const float *xr = x + d * 2 * ld;
      const Vec<kLane> xvh = ldv<kLane>(xr + u), xvl = ldv<kLane>(xr + ld + u);
      const uint32_t Iu = F.basis_up[d];
#pragma unroll
      for (int i = 0; i < kLane; ++i) {
        float2 dg[2];
#pragma unroll
        for (int b = 0; b < 2; ++b) {
          const int64_t c = u + 2 * i + b;
          dg[b] = c < S.n_cols ? utab[__popc(Iu & F.basis_dn[c])] : make_float2(0.f, 0.f);
        }
        f2x Sh, Sl, ph, pl;
        sump_norm(acc[i], Sh, Sl);
        if (F.t_neg) {
          Sh ^= kSign2;
          Sl ^= kSign2;
        }
        df2_mul(pk2(dg[0].x, dg[1].x), pk2(dg[0].y, dg[1].y), xvh.v[i], xvl.v[i], ph, pl);
        df2_add(ph, pl, Sh, Sl, yh.v[i], yl.v[i]);
      }
    } else {
      const float *zr = z + d * 2 * ld;
      const Vec<kLane> zh = ldv<kLane>(zr + u), zl = ldv<kLane>(zr + ld + u);
#pragma unroll
      for (int i = 0; i < kLane; ++i) {
        f2x Sh, Sl;
        sump_norm(acc[i], Sh, Sl);
        if (F.t_neg) {
          Sh ^= kSign2;
          Sl ^= kSign2;
        }
        df2_add(zh.v[i], zl.v[i], Sh, Sl, yh.v[i], yl.v[i]);
      }
    }
    stv<kLane>(wr + u, yh);
    stv<kLane>(wr + ld + u, yl);
  }
}

// ---------------------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------------------
static int grid_vec() { return num_sms() * 4; }

struct FastState {
  bool built = false;
  bool col16 = true;
  int32_t *sp[2] = {nullptr, nullptr};
  uint32_t *sl_add = nullptr, *sl_sub = nullptr;
  int32_t *sl_off_add = nullptr, *sl_off_sub = nullptr;
  uint16_t *steps_add = nullptr, *steps_sub = nullptr;
  uint32_t idle_word = 0xffffffffu;
  int32_t *slot_row = nullptr, *slot_of = nullptr;
  uint32_t *basis_slot = nullptr;
  void *col[2] = {nullptr, nullptr};
  float *xdf = nullptr, *zdf = nullptr;      // hub_apply scratch (planar double-float)
  bool staged = true;                        // pass 1 stages rows; else it runs on X^T
  int acc_terms = 0;                         // most terms one low-part accumulator sums (error bound)
  int64_t ld_t = 0;                          // plane length of X^T rows (count_dn padded)
  float *xt = nullptr, *zt = nullptr;        // X^T and Z^T (rows too long to stage)
  int *d_range = nullptr;                    // exponent partials [2 G], then scale[4] (k_scale)
  int *d_err = nullptr;
  int64_t ld = 0;
  // pipelined host-buffer apply: copy stream, per-chunk events, exponent partials, flag
  cudaStream_t copy_stream = nullptr;
  std::vector<cudaEvent_t> events;
  int *d_range_chunks = nullptr, *d_flag = nullptr, *h_flag = nullptr;
  // the multi-vector form: a second copy stream (outputs) and its own events
  cudaStream_t copy_out_stream = nullptr;
  std::vector<cudaEvent_t> many_events;
};

static FastState *fast_of(const hub_ctx *h) { return h->fast; }

void fast_release(hub_ctx *h) {
  FastState *f = fast_of(h);
  if (!f) return;
  for (int s = 0; s < 2; ++s) {
    dev_free(f->sp[s]);
    dev_free(f->col[s]);
  }
  dev_free(f->xdf);
  dev_free(f->zdf);
  dev_free(f->xt);
  dev_free(f->zt);
  if (h->route == HUB_ROUTE_DF) set_route(h, HUB_ROUTE_NONE);     // its flag goes
  dev_free(f->d_range);
  dev_free(f->d_err);
  dev_free(f->d_range_chunks);
  dev_free(f->d_flag);
  if (f->h_flag) cudaFreeHost(f->h_flag);
  for (cudaEvent_t e : f->events) cudaEventDestroy(e);
  if (f->copy_stream) cudaStreamDestroy(f->copy_stream);
  for (cudaEvent_t e : f->many_events) cudaEventDestroy(e);
  if (f->copy_out_stream) cudaStreamDestroy(f->copy_out_stream);
  dev_free(f->sl_add);
  dev_free(f->sl_sub);
  dev_free(f->sl_off_add);
  dev_free(f->sl_off_sub);
  dev_free(f->steps_add);
  dev_free(f->steps_sub);
  dev_free(f->slot_row);
  dev_free(f->slot_of);
  dev_free(f->basis_slot);
  delete f;
  h->fast = nullptr;
}

// Plane length of a row: count_up rounded up to a multiple of 4 (16-byte plane starts) and
// of the columns a pass-2 lane loads at once.
static int64_t padded_ld(int64_t n_up) {
  const int64_t a = kDnLaneCols > 4 ? kDnLaneCols : 4;
  return (n_up + a - 1) / a * a;
}

// Parameter magnitudes the double-float window allows (0, or 2^-16 .. 2^16; see kExpSpan).
static bool in_param_range(double v) {
  const double a = std::fabs(v);
  return a == 0.0 || (a >= 0x1p-16 && a <= 0x1p16);
}

// Most terms (pass 2: pair sums) one low-part accumulator of a hopping sum may take: with
// N such additions the product's error is at most max(N + 10.1, 16) u^2 (|H||x|)_n,
// u = 2^-24, so N <= 15 keeps it, with the oracle's own FP64 rounding (2 u^2), below
// 1e-13 (|H||x|)_n = 28.1 u^2.  A row with F_add adding and F_sub subtracting entries gives
// N <= ceil(F_add/4) + ceil(F_sub/4) (9 for the 32-entry rows of the 4x4 lattice).
constexpr int kMaxAccTerms = 15;

// The fast path: uniform t != 0 and U, no site energies (the diagonal is then U k exactly),
// |t| and U / |t| in the parameter range, hopping rows short enough for kMaxAccTerms.
bool fast_eligible(const hub_ctx *h) {
  if (!h->have_hop || !h->have_U || !h->uniform_U || h->has_eps) return false;
  for (double tb : h->t)
    if (tb != h->t[0]) return false;
  if (h->t.empty() || h->t[0] == 0.0 || !in_param_range(h->t[0])) return false;
  if (!in_param_range(h->U0 / std::fabs(h->t[0]))) return false;
  if (h->count[0] <= 0 || h->count[1] <= 0) return false;
  if (h->fast && h->fast->acc_terms > kMaxAccTerms) return false;
  // element quads of a vector are indexed with 32-bit integers
  return h->count[1] * (padded_ld(h->count[0]) / 4) < ((int64_t)1 << 32);
}

// Build the sign-split CSR and double-float tables (called after hub_hopping).
int fast_build(hub_ctx *h) {
  fast_release(h);
  FastState *f = new (std::nothrow) FastState();
  if (!f) return fail(HUB_ERR_OOM, "fast path: host allocation failed");
  h->fast = f;
  f->col16 = h->count[0] <= 65536 && h->count[1] <= 65536;
  f->ld = padded_ld(h->count[0]);
  f->ld_t = padded_ld(h->count[1]);
  f->staged = f->ld + 2 <= kUpPlane;
  const size_t csz = f->col16 ? sizeof(uint16_t) : sizeof(uint32_t);
  for (int s = 0; s < 2; ++s) {
    if (s == 1 && h->shared) break;
    const SpinCSR &c = h->csr[s];
    const int64_t n = h->count[s];
    if (!dev_alloc((void **)&f->sp[s], sizeof(int32_t) * (n + 1), "split CSR") ||
        !dev_alloc(&f->col[s], csz * (size_t)std::max<int64_t>(c.nnz, 1), "split CSR columns"))
      return HUB_ERR_OOM;
    const int g = (int)std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 16);
    if (f->col16)
      k_split_csr<uint16_t><<<std::max(g, 1), 256>>>(n, c.rowptr, c.scol, f->sp[s], (uint16_t *)f->col[s]);
    else
      k_split_csr<uint32_t><<<std::max(g, 1), 256>>>(n, c.rowptr, c.scol, f->sp[s], (uint32_t *)f->col[s]);
    HUB_LAUNCH_CHECK();
  }
  // sliced, bank-scheduled H_up for pass 1 (built on the host from the sign-split CSR)
  {
    const int64_t n = h->count[0];
    const int64_t nsl = (n + 31) / 32;
    const int64_t nnz = h->csr[0].nnz;
    std::vector<int32_t> rp(n + 1), spv(n);
    std::vector<uint32_t> col(std::max<int64_t>(nnz, 1));
    HUB_CUDA(cudaMemcpy(rp.data(), h->csr[0].rowptr, sizeof(int32_t) * (n + 1), cudaMemcpyDeviceToHost));
    HUB_CUDA(cudaMemcpy(spv.data(), f->sp[0], sizeof(int32_t) * n, cudaMemcpyDeviceToHost));
    if (f->col16) {
      std::vector<uint16_t> c16(std::max<int64_t>(nnz, 1));
      if (nnz) HUB_CUDA(cudaMemcpy(c16.data(), f->col[0], sizeof(uint16_t) * nnz, cudaMemcpyDeviceToHost));
      for (int64_t k = 0; k < nnz; ++k) col[k] = c16[k];
    } else if (nnz) {
      HUB_CUDA(cudaMemcpy(col.data(), f->col[0], sizeof(uint32_t) * nnz, cudaMemcpyDeviceToHost));
    }
    // slots: rows ordered by (add length, sub length), stable (identity when pass 1 runs
    // on X^T, which has no use for the order)
    std::vector<int32_t> slot_row(n);
    for (int64_t r = 0; r < n; ++r) slot_row[r] = (int32_t)r;
    if (f->staged) std::stable_sort(slot_row.begin(), slot_row.end(), [&](int32_t a, int32_t b) {
      const int la = spv[a] - rp[a], lb = spv[b] - rp[b];
      const int sa = rp[a + 1] - spv[a], sb = rp[b + 1] - spv[b];
      return la != lb ? la > lb : sa > sb;
    });
    std::vector<int32_t> slot_of(n);
    for (int64_t k = 0; k < n; ++k) slot_of[slot_row[k]] = (int32_t)k;
    // terms per low-part accumulator: whole rows of a CSR (pass 2; pass 1 on X^T), or the
    // scheduled steps of a slice (staged pass 1, below)
    auto acc_of_rows = [](const std::vector<int32_t> &r, const std::vector<int32_t> &sp) {
      int m = 0;
      for (size_t k = 0; k + 1 < r.size(); ++k)
        m = std::max(m, (sp[k] - r[k] + 3) / 4 + (r[k + 1] - sp[k] + 3) / 4);
      return m;
    };
    {
      const int sd = h->shared ? 0 : 1;
      std::vector<int32_t> rpd(h->count[sd] + 1), spd(h->count[sd]);
      HUB_CUDA(cudaMemcpy(rpd.data(), h->csr[sd].rowptr, sizeof(int32_t) * rpd.size(), cudaMemcpyDeviceToHost));
      HUB_CUDA(cudaMemcpy(spd.data(), f->sp[sd], sizeof(int32_t) * spd.size(), cudaMemcpyDeviceToHost));
      f->acc_terms = acc_of_rows(rpd, spd);
      if (!f->staged) f->acc_terms = std::max(f->acc_terms, acc_of_rows(rp, spv));
    }
    const int g = (int)std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, (int64_t)num_sms() * 16));
    if (!dev_alloc((void **)&f->slot_row, sizeof(int32_t) * n, "slot order") ||
        !dev_alloc((void **)&f->slot_of, sizeof(int32_t) * n, "slot order") ||
        !dev_alloc((void **)&f->basis_slot, sizeof(uint32_t) * n, "basis in slot order"))
      return HUB_ERR_OOM;
    HUB_CUDA(cudaMemcpy(f->slot_row, slot_row.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice));
    HUB_CUDA(cudaMemcpy(f->slot_of, slot_of.data(), sizeof(int32_t) * n, cudaMemcpyHostToDevice));
    k_to_slots<<<g, 256>>>(n, f->slot_row, h->basis[0], f->basis_slot);
    HUB_LAUNCH_CHECK();
    if (f->staged) {
      // Per slice and group, the lanes' entries are scheduled into steps; the 32-bit loads of
      // one step cost as many shared-memory wavefronts as the most used bank (column mod 32)
      // has distinct columns in it.  Greedy: lanes with the most remaining entries first; each
      // takes a column already used in the step (a broadcast), else one of the most loaded bank
      // that is still under the cap.  Pass 1 is limited by both instruction issue (steps) and
      // shared-memory wavefronts: on the 4x4 lattice a cap of two columns per bank and step
      // runs fastest (steps within a few per cent of the longest lane); a cap of three saves
      // steps but costs 20 % in time, and an adaptive cap (the busiest bank's remaining load
      // over the remaining steps) saves 17 % of the wavefronts for 5 % more steps and runs 1 %
      // slower.
#ifndef HUB_BANK_CAP
#define HUB_BANK_CAP 2   // columns per bank and step: k > 0 fixed, 0 adaptive, -k adaptive capped at k
#endif
      constexpr int kBankCap = HUB_BANK_CAP;
      // idle steps: the zero entry after the staged row when rows are staged, else a sentinel
      const bool staged = f->ld + 2 <= kUpPlane;
      const uint32_t idle = staged ? (uint32_t)f->ld : (f->col16 ? 0xffffu : 0xffffffffu);
      f->idle_word = f->col16 ? (idle | (idle << 16)) : idle;
      const int pack = f->col16 ? 2 : 1;
      std::vector<uint16_t> st[2] = {std::vector<uint16_t>(nsl), std::vector<uint16_t>(nsl)};
      std::vector<int32_t> off[2] = {std::vector<int32_t>(nsl + 1, 0), std::vector<int32_t>(nsl + 1, 0)};
      std::vector<uint32_t> words[2];
      std::vector<std::vector<uint32_t>> warp_steps;  // [S][32] entries of one slice
      for (int64_t sl = 0; sl < nsl; ++sl) {
        for (int grp = 0; grp < 2; ++grp) {
          std::vector<uint32_t> rem[32];
          for (int l = 0; l < 32; ++l) {
            const int64_t slot = sl * 32 + l;
            if (slot >= n) continue;
            const int32_t r = slot_row[slot];
            const int32_t a = grp == 0 ? rp[r] : spv[r], b = grp == 0 ? spv[r] : rp[r + 1];
            for (int32_t k = a; k < b; ++k) rem[l].push_back((uint32_t)slot_of[col[k]]);
          }
          warp_steps.clear();
          std::vector<uint32_t> distinct;
          for (;;) {
            int lanes[32], nl = 0;
            size_t left = 0;
            distinct.clear();
            for (int l = 0; l < 32; ++l)
              if (!rem[l].empty()) {
                lanes[nl++] = l;
                left = std::max(left, rem[l].size());
                distinct.insert(distinct.end(), rem[l].begin(), rem[l].end());
              }
            if (!nl) break;
            std::sort(distinct.begin(), distinct.end());
            distinct.erase(std::unique(distinct.begin(), distinct.end()), distinct.end());
            int bankload[32] = {0};
            for (uint32_t c : distinct) ++bankload[c & 31];
            const int maxload = *std::max_element(bankload, bankload + 32);
            const int need = std::max(1, (int)((maxload + left - 1) / left));
            const int cap = kBankCap > 0 ? kBankCap : (kBankCap < 0 ? std::min(-kBankCap, need) : need);
            std::stable_sort(lanes, lanes + nl, [&](int a, int b) { return rem[a].size() > rem[b].size(); });
            std::vector<uint32_t> step(32, idle);
            uint32_t used_col[32][8];
            int used[32] = {0};
            auto in_step = [&](uint32_t c) {
              const int bk = c & 31;
              for (int i = 0; i < used[bk]; ++i)
                if (used_col[bk][i] == c) return true;
              return false;
            };
            for (int q = 0; q < nl; ++q) {
              const int l = lanes[q];
              int best = -1, best_shared = 0, best_load = 0, best_used = 0;
              for (int e = 0; e < (int)rem[l].size(); ++e) {
                const uint32_t c = rem[l][e];
                const int bk = c & 31;
                const int shared = in_step(c) ? 1 : 0;
                if (!shared && (used[bk] >= cap || used[bk] >= 8)) continue;
                const bool better = best < 0 || shared > best_shared ||
                                    (shared == best_shared && (bankload[bk] > best_load ||
                                                               (bankload[bk] == best_load && used[bk] < best_used)));
                if (better) {
                  best = e;
                  best_shared = shared;
                  best_load = bankload[bk];
                  best_used = used[bk];
                }
              }
              if (best < 0) continue;
              const uint32_t c = rem[l][best];
              step[l] = c;
              if (!best_shared) used_col[c & 31][used[c & 31]++] = c;
              rem[l].erase(rem[l].begin() + best);
            }
            warp_steps.push_back(step);
          }
          const int S = (int)warp_steps.size();
          if (S > 65535) return fail(HUB_ERR_ARG, "fast path: hopping row schedule too long");
          st[grp][sl] = (uint16_t)S;
          if (grp == 1) f->acc_terms = std::max(f->acc_terms, (st[0][sl] + 3) / 4 + (S + 3) / 4);
          const int nw = (S + pack - 1) / pack, nb = (nw + 3) / 4;
          off[grp][sl + 1] = off[grp][sl] + 32 * 4 * nb;
          for (int bt = 0; bt < nb; ++bt)
            for (int l = 0; l < 32; ++l)
              for (int i = 0; i < 4; ++i) {
                const int j = 4 * bt + i;
                uint32_t wd = f->idle_word;
                if (j < nw && pack == 2) {
                  const uint32_t lo = warp_steps[2 * j][l];
                  const uint32_t hi = 2 * j + 1 < S ? warp_steps[2 * j + 1][l] : idle;
                  wd = lo | (hi << 16);
                } else if (j < nw) {
                  wd = warp_steps[j][l];
                }
                words[grp].push_back(wd);
              }
        }
      }
      if (!dev_alloc((void **)&f->sl_off_add, sizeof(int32_t) * (nsl + 1), "slice offsets") ||
          !dev_alloc((void **)&f->sl_off_sub, sizeof(int32_t) * (nsl + 1), "slice offsets") ||
          !dev_alloc((void **)&f->sl_add, sizeof(uint32_t) * std::max<size_t>(words[0].size(), 1), "sliced columns") ||
          !dev_alloc((void **)&f->sl_sub, sizeof(uint32_t) * std::max<size_t>(words[1].size(), 1), "sliced columns") ||
          !dev_alloc((void **)&f->steps_add, sizeof(uint16_t) * nsl, "slice steps") ||
          !dev_alloc((void **)&f->steps_sub, sizeof(uint16_t) * nsl, "slice steps"))
        return HUB_ERR_OOM;
      HUB_CUDA(cudaMemcpy(f->sl_off_add, off[0].data(), sizeof(int32_t) * (nsl + 1), cudaMemcpyHostToDevice));
      HUB_CUDA(cudaMemcpy(f->sl_off_sub, off[1].data(), sizeof(int32_t) * (nsl + 1), cudaMemcpyHostToDevice));
      if (!words[0].empty())
        HUB_CUDA(cudaMemcpy(f->sl_add, words[0].data(), sizeof(uint32_t) * words[0].size(), cudaMemcpyHostToDevice));
      if (!words[1].empty())
        HUB_CUDA(cudaMemcpy(f->sl_sub, words[1].data(), sizeof(uint32_t) * words[1].size(), cudaMemcpyHostToDevice));
      HUB_CUDA(cudaMemcpy(f->steps_add, st[0].data(), sizeof(uint16_t) * nsl, cudaMemcpyHostToDevice));
      HUB_CUDA(cudaMemcpy(f->steps_sub, st[1].data(), sizeof(uint16_t) * nsl, cudaMemcpyHostToDevice));
    }
  }
  if (!dev_alloc((void **)&f->d_err, sizeof(int) * 4, "error flag")) return HUB_ERR_OOM;
  HUB_CUDA(cudaMemset(f->d_err, 0, sizeof(int) * 4));
  HUB_CUDA(cudaDeviceSynchronize());
  f->built = true;
  return HUB_OK;
}

static FastView fast_view(const hub_ctx *h, const FastState *f, const int *gate) {
  FastView v{};
  v.gate = gate;
  v.n_up = h->count[0];
  v.n_dn = h->count[1];
  v.ld = f->ld;
  v.basis_up = h->basis[0];
  v.basis_dn = h->basis[1];
  const int sd = h->shared ? 0 : 1;
  v.rp_up = h->csr[0].rowptr;
  v.sp_up = f->sp[0];
  v.rp_dn = h->csr[sd].rowptr;
  v.sp_dn = f->sp[sd];
  v.col_up = f->col[0];
  v.col_dn = f->col[sd];
  v.sl_add = f->sl_add;
  v.sl_sub = f->sl_sub;
  v.sl_off_add = f->sl_off_add;
  v.sl_off_sub = f->sl_off_sub;
  v.steps_add = f->steps_add;
  v.steps_sub = f->steps_sub;
  v.slot_row = f->slot_row;
  v.idle_word = f->idle_word;
  v.basis_up_slot = f->basis_slot;
  // The kernels apply H / |t| (hopping elements -sign(t) esign, exact), the caller's results
  // are scaled by |t| in FP64 (hub_apply) or through alpha, beta (Lanczos).
  const double t = h->t.empty() ? 1.0 : h->t[0];
  v.t_neg = t < 0.0;
  // host double -> double-float: hi = float(a), lo = float(a - hi)
  auto hdf = [](double a) {
    float hi = (float)a;
    return make_float2(hi, (float)(a - (double)hi));
  };
  const double u_scaled = h->U0 / std::fabs(t);
  for (int k = 0; k < 32; ++k) v.Utab[k] = hdf(u_scaled * (double)k);
  v.err = f->d_err;
  v.fail_waits = h->fail_waits ? 1 : 0;
  return v;
}

static size_t up_smem(const FastState *f) { return sizeof(float) * (3 * (size_t)kUpPlane + (size_t)f->ld + 2); }
constexpr size_t kMaxStage = 224 * 1024;
static_assert(sizeof(float) * 4 * kUpPlane <= kMaxStage, "four staged planes must fit");

// the spin-down side (pass 2 on X) and the spin-up side (pass 1 on X^T)
static Side side_dn(const hub_ctx *h, const FastState *f) {
  const int sd = h->shared ? 0 : 1;
  return Side{h->count[1], h->count[0], f->ld, h->csr[sd].rowptr, f->sp[sd], f->col[sd]};
}
static Side side_up(const hub_ctx *h, const FastState *f) {
  return Side{h->count[0], h->count[1], f->ld_t, h->csr[0].rowptr, f->sp[0], f->col[0]};
}

static dim3 dn_grid(const Side &S) {
  return dim3((unsigned)((S.n_rows - S.r_begin + kDnRows - 1) / kDnRows), (unsigned)((S.n_cols + kDnCols - 1) / kDnCols));
}

template <typename Col, int kMode>
static int launch_dn_t(const FastView &v, const Side &S, const float *x, const float *z, float *w, bool chained,
                       cudaStream_t s) {
  const dim3 g = dn_grid(S);
  if (g.y > 65535) return fail(HUB_ERR_ARG, "fast apply: too many column strips");
  HUB_CUDA(launch_kernel(chained, k_dn<Col, kMode>, g, kDnThreads, 0, s, v, S, x, z, w));
  return HUB_OK;
}

template <int kMode>
static int launch_dn(const FastState *f, const FastView &v, const Side &S, const float *x, const float *z, float *w,
                     bool chained, cudaStream_t s) {
  return f->col16 ? launch_dn_t<uint16_t, kMode>(v, S, x, z, w, chained, s)
                  : launch_dn_t<uint32_t, kMode>(v, S, x, z, w, chained, s);
}

// dst = src^T for planar matrices (see k_transpose)
static int transpose(int64_t n_r, int64_t n_c, int64_t ld_s, int64_t ld_d, const float *src, float *dst,
                     const int *gate, bool chained, cudaStream_t s) {
  const dim3 g((unsigned)((n_c + kTile - 1) / kTile), (unsigned)((ld_d + kTile - 1) / kTile));
  if (g.y > 65535) return fail(HUB_ERR_ARG, "fast apply: matrix too large to transpose");
  HUB_CUDA(launch_kernel(chained, k_transpose, g, dim3(kTile, 8), 0, s, n_r, n_c, ld_s, ld_d, src, dst, gate));
  return HUB_OK;
}

static int ensure_vec(float **p, int64_t n, const char *what);
static int64_t scratch_floats(const hub_ctx *h, const FastState *f);

// z <- pass 1 (x planar double-float); with staged rows, only the row pairs p0 .. p1 - 1
// (p1 < 0: all pairs).
static int run_up(hub_ctx *h, FastState *f, const float *x, float *z, cudaStream_t s, int64_t p0 = 0, int64_t p1 = -1,
                  const int *gate = nullptr) {
  const FastView v = fast_view(h, f, gate);
  const bool chained = gate && !h->prof;
  if (p1 < 0) p1 = (v.n_dn + 1) / 2;
  if (!f->staged && (p0 != 0 || p1 != (v.n_dn + 1) / 2)) return fail(HUB_ERR_STATE, "pass 1: partial range");
  if (p1 <= p0) return HUB_OK;
  int rc;
  if ((rc = prof_mark(h, HUB_PROF_UP, true, s))) return rc;
  if (f->staged) {
    count_launch(h);
    const int threads = v.n_up >= 4096 ? kUpThreads : (v.n_up >= 1024 ? 512 : (v.n_up >= 256 ? 256 : 128));
    const int grid = (int)std::min<int64_t>(p1 - p0, (int64_t)num_sms());
    const size_t smem = up_smem(f);
#define HUB_UP(C)                                                                                          \
  do {                                                                                                     \
    HUB_CUDA(cudaFuncSetAttribute(k_up<C>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kMaxStage));  \
    HUB_CUDA(launch_kernel(chained, k_up<C>, grid, threads, smem, s, v, x, z, p0, p1));                     \
  } while (0)
    if (f->col16) HUB_UP(uint16_t); else HUB_UP(uint32_t);
#undef HUB_UP
  } else {
    const int64_t Dt = scratch_floats(h, f);   // also fast_scratch's, which takes them as they are
    if ((rc = ensure_vec(&f->xt, Dt, "transposed x")) || (rc = ensure_vec(&f->zt, Dt, "transposed z"))) return rc;
    count_launch(h, 3);
    if ((rc = transpose(h->count[1], h->count[0], f->ld, f->ld_t, x, f->xt, gate, chained, s))) return rc;
    if ((rc = launch_dn<2>(f, v, side_up(h, f), f->xt, nullptr, f->zt, chained, s))) return rc;
    if ((rc = transpose(h->count[0], h->count[1], f->ld_t, f->ld, f->zt, z, gate, chained, s))) return rc;
  }
  return prof_mark(h, HUB_PROF_UP, false, s);
}

// pass 2 on the rows r0 .. r1 - 1 of X (r1 < 0: all rows)
static int run_dn(hub_ctx *h, FastState *f, const float *x, const float *z, float *w, cudaStream_t s, int64_t r0 = 0,
                  int64_t r1 = -1, const int *gate = nullptr) {
  const FastView v = fast_view(h, f, gate);
  count_launch(h);
  int rc = prof_mark(h, HUB_PROF_DN, true, s);
  if (rc) return rc;
  Side S = side_dn(h, f);
  S.r_begin = r0;
  if (r1 >= 0) S.n_rows = r1;
  if (S.n_rows <= S.r_begin) return prof_mark(h, HUB_PROF_DN, false, s);
  if ((rc = launch_dn<0>(f, v, S, x, z, w, gate && !h->prof, s))) return rc;
  return prof_mark(h, HUB_PROF_DN, false, s);
}

static int ensure_vec(float **p, int64_t n, const char *what) {
  if (*p) return HUB_OK;
  return dev_alloc((void **)p, sizeof(float) * n, what) ? HUB_OK : HUB_ERR_OOM;
}

static int row_grid(const hub_ctx *h) { return (int)std::min<int64_t>(h->count[1], (int64_t)num_sms() * 8); }

// Exponent partials and scale words of the handle: [2 G] partials, then scale[0..3].
static int *range_buf(FastState *f) {
  if (!f->d_range && !dev_alloc((void **)&f->d_range, sizeof(int) * (2 * grid_vec() + 4), "exponent partials"))
    return nullptr;
  return f->d_range;
}

// Floats of a scratch vector: a planar vector, or a fixed-point one in either order.
static int64_t scratch_floats(const hub_ctx *h, const FastState *f) {
  return 2 * std::max(h->count[1] * f->ld, h->count[0] * f->ld_t);
}

int fast_scratch(hub_ctx *h, int n, float **v) {
  FastState *f = fast_of(h);
  float **const all[4] = {&f->xdf, &f->zdf, &f->xt, &f->zt};
  for (int k = 0; k < n; ++k) {
    const int rc = ensure_vec(all[k], scratch_floats(h, f), "apply scratch");
    if (rc) return rc;
    v[k] = *all[k];
  }
  return HUB_OK;
}

static int fast_exp_range(hub_ctx *h, const double *x, int64_t D, int **part, int *nblk, cudaStream_t s) {
  FastState *f = fast_of(h);
  *nblk = grid_vec();
  if (!(*part = range_buf(f))) return HUB_ERR_OOM;
  count_launch(h);
  k_exp_range<<<*nblk, 256, 0, s>>>(D, x, *part);
  HUB_LAUNCH_CHECK();
  return HUB_OK;
}

void fast_release_scratch(hub_ctx *h) {
  FastState *f = fast_of(h);
  for (float **v : {&f->xdf, &f->zdf, &f->xt, &f->zt}) {
    dev_free(*v);
    *v = nullptr;
  }
}

int *fast_err(const hub_ctx *h) { return fast_of(h)->d_err; }

// Conversion, both passes and the un-permutation of a product whose scale is known.
static int df_apply(hub_ctx *h, FastState *f, const double *x, double *y, const int *scale, const int *gate,
                    cudaStream_t s) {
  int rc;
  count_launch(h);
  const bool chained = gate && !h->prof;
  HUB_CUDA(launch_kernel(chained, k_f64_to_df, row_grid(h), 256, 0, s, 0, h->count[1], h->count[0], f->ld, x, scale,
                         f->slot_row, f->xdf, gate));
  if ((rc = run_up(h, f, f->xdf, f->zdf, s, 0, -1, gate))) return rc;
  if ((rc = run_dn(h, f, f->xdf, f->zdf, f->zdf, s, 0, -1, gate))) return rc;
  count_launch(h);
  HUB_CUDA(launch_kernel(chained, k_unpermute, row_grid(h), 512, 0, s, 0, h->count[1], h->count[0], f->ld, f->zdf,
                         f->slot_of, scale, std::fabs(h->t[0]), y, gate));
  return HUB_OK;
}

int fast_apply_gated(hub_ctx *h, const double *x, double *y, const int *scale, const int *gate, cudaStream_t s) {
  FastState *f = fast_of(h);
  float *v[2];
  const int rc = fast_scratch(h, 2, v);
  return rc ? rc : df_apply(h, f, x, y, scale, gate, s);
}

// hub_apply on the double-float path: FP64 in, FP64 out.  A vector outside the double-float window
// (kExpSpan) is multiplied by the FP64 kernel instead: both are launched, the device-side
// flag scale[1] decides which one writes y, so the call stays asynchronous.
int fast_apply_f64(hub_ctx *h, const double *x, double *y, cudaStream_t s) {
  FastState *f = fast_of(h);
  if (!f || !f->built) return fail(HUB_ERR_STATE, "fast apply: not built");
  float *v[2];
  int *part = nullptr, G = 0, rc;
  if ((rc = fast_scratch(h, 2, v))) return rc;
  if ((rc = fast_exp_range(h, x, h->count[0] * h->count[1], &part, &G, s))) return rc;
  int *scale = part + 2 * G;
  count_launch(h);
  k_scale<<<1, 256, 0, s>>>(part, G, scale);
  HUB_LAUNCH_CHECK();
  set_route(h, HUB_ROUTE_DF, scale + 1);
  if ((rc = df_apply(h, f, x, y, scale, nullptr, s))) return rc;
  return f64_apply(h, x, y, scale + 1, s);
}

// Row chunks of the host-buffer apply.
constexpr int kHostChunks = 8;

// Row chunk bounds b[0..n] of n_dn rows with relative sizes w (boundaries even, so that no
// pass-1 row pair straddles two chunks; empty chunks dropped); returns n.
static int chunk_bounds(int64_t n_dn, const int (&w)[kHostChunks], int64_t *b) {
  int total = 0;
  for (int c = 0; c < kHostChunks; ++c) total += w[c];
  int n = 0, acc = 0;
  b[0] = 0;
  for (int c = 0; c < kHostChunks; ++c) {
    acc += w[c];
    const int64_t e = c + 1 == kHostChunks ? n_dn : std::min<int64_t>(n_dn, (n_dn * acc / total) & ~(int64_t)1);
    if (e > b[n]) b[++n] = e;
  }
  return n;
}

// Row chunks of a host-buffer apply: the input's last chunk and the output's first chunk are a
// quarter of the others (little pass-1 work is left once the last input chunk has landed, and
// the first output chunk is ready to go back early); per is the largest chunk.
struct HostChunks {
  int64_t bi[kHostChunks + 1], bo[kHostChunks + 1];
  int nci, nco;
  int64_t per;
};

static HostChunks host_chunks(int64_t n_dn) {
  static const int w_in[kHostChunks] = {4, 4, 4, 4, 4, 4, 4, 1}, w_out[kHostChunks] = {1, 4, 4, 4, 4, 4, 4, 4};
  HostChunks C;
  C.nci = chunk_bounds(n_dn, w_in, C.bi);
  C.nco = chunk_bounds(n_dn, w_out, C.bo);
  C.per = 0;
  for (int c = 0; c < C.nci; ++c) C.per = std::max(C.per, C.bi[c + 1] - C.bi[c]);
  for (int c = 0; c < C.nco; ++c) C.per = std::max(C.per, C.bo[c + 1] - C.bo[c]);
  return C;
}

// Scratch of the chunked host-buffer apply: double-float x and z, per-chunk exponent
// partials, the scale words, the route flag (device and pinned host) and the input copy stream.
static int host_pipe_buffers(hub_ctx *h, FastState *f) {
  float *v[2];
  const int rc = fast_scratch(h, 2, v);
  if (rc) return rc;
  if (!f->d_range_chunks &&
      !dev_alloc((void **)&f->d_range_chunks, sizeof(int) * 2 * grid_vec() * kHostChunks, "exponent partials"))
    return HUB_ERR_OOM;
  if (!range_buf(f)) return HUB_ERR_OOM;
  if (!f->d_flag && !dev_alloc((void **)&f->d_flag, sizeof(int), "scale flag")) return HUB_ERR_OOM;
  if (!f->h_flag) HUB_CUDA(cudaMallocHost((void **)&f->h_flag, sizeof(int)));
  if (!f->copy_stream) HUB_CUDA(cudaStreamCreateWithFlags(&f->copy_stream, cudaStreamNonBlocking));
  return HUB_OK;
}

static int ensure_events(std::vector<cudaEvent_t> &ev, int n) {
  while ((int)ev.size() < n) {
    cudaEvent_t e;
    HUB_CUDA(cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    ev.push_back(e);
  }
  return HUB_OK;
}

// Pass 1 of a host-buffer apply in the input's row chunks (bounds b[0..nc]): each chunk waits
// for its copy (ev_in[c]), then takes its exponent partials (the first chunk also fixes the
// conversion scale), its conversion to double-float and pass 1 on its row pairs.  Ends with
// the whole vector's scale and the route flag, copied to f->h_flag on s (0: converted with the
// right scale; 1: the largest exponent lies outside the first chunk, redo with the global
// scale; 2: outside the double-float window, FP64 kernel).  xd: the FP64 device input.
static int host_pass1(hub_ctx *h, FastState *f, const double *xd, const int64_t *b, int nc, int64_t per,
                      const cudaEvent_t *ev_in, cudaStream_t s) {
  const int64_t n_up = h->count[0];
  const int G = grid_vec();
  int *part = f->d_range_chunks;                 // 2 G exponent partials per chunk
  int *scale = f->d_range + 2 * G;                // [0, 1] first chunk's scale, [2, 3] the whole vector's
  const int rg = (int)std::min<int64_t>(per, (int64_t)num_sms() * 8);
  int rc;
  for (int c = 0; c < nc; ++c) {
    HUB_CUDA(cudaStreamWaitEvent(s, ev_in[c], 0));
    count_launch(h, c == 0 ? 3 : 2);
    k_exp_range<<<G, 256, 0, s>>>((b[c + 1] - b[c]) * n_up, xd + b[c] * n_up, part + 2 * c * G);
    if (c == 0) k_scale<<<1, 256, 0, s>>>(part, G, scale);
    k_f64_to_df<<<rg, 256, 0, s>>>(b[c], b[c + 1], n_up, f->ld, xd, scale, f->slot_row, f->xdf, nullptr);
    HUB_LAUNCH_CHECK();
    if ((rc = run_up(h, f, f->xdf, f->zdf, s, b[c] / 2, (b[c + 1] + 1) / 2))) return rc;
  }
  count_launch(h);
  k_scale_all<<<1, 256, 0, s>>>(part, G, nc, scale, f->d_flag);
  HUB_LAUNCH_CHECK();
  HUB_CUDA(cudaMemcpyAsync(f->h_flag, f->d_flag, sizeof(int), cudaMemcpyDeviceToHost, s));
  return HUB_OK;
}

// Route flag 1: conversion and pass 1 again, with the whole vector's scale.
static int host_redo(hub_ctx *h, FastState *f, const double *xd, cudaStream_t s) {
  int *scale = f->d_range + 2 * grid_vec();
  count_launch(h);
  k_f64_to_df<<<row_grid(h), 256, 0, s>>>(0, h->count[1], h->count[0], f->ld, xd, scale + 2, f->slot_row, f->xdf,
                                          nullptr);
  HUB_LAUNCH_CHECK();
  return run_up(h, f, f->xdf, f->zdf, s);
}

// Pass 2 in the output's row chunks (bounds b[0..nc]), so that each chunk's result goes back
// while the next is computed (every chunk reads the whole of X by strips; X is read from HBM
// once per chunk): run_dn and the un-permutation into the FP64 device output yd on s, then the
// chunk's copy to y_host on sc (ev_out[c] hands the chunk from s to sc).
static int host_pass2(hub_ctx *h, FastState *f, double *yd, double *y_host, const int64_t *b, int nc, int64_t per,
                      const cudaEvent_t *ev_out, cudaStream_t s, cudaStream_t sc) {
  const int64_t n_up = h->count[0];
  int *scale = f->d_range + 2 * grid_vec();
  const int rg = (int)std::min<int64_t>(per, (int64_t)num_sms() * 8);
  int rc;
  for (int c = 0; c < nc; ++c) {
    if ((rc = run_dn(h, f, f->xdf, f->zdf, f->zdf, s, b[c], b[c + 1]))) return rc;
    count_launch(h);
    k_unpermute<<<rg, 512, 0, s>>>(b[c], b[c + 1], n_up, f->ld, f->zdf, f->slot_of, scale + 2,
                                   std::fabs(h->t[0]), yd, nullptr);
    HUB_LAUNCH_CHECK();
    HUB_CUDA(cudaEventRecord(ev_out[c], s));
    HUB_CUDA(cudaStreamWaitEvent(sc, ev_out[c], 0));
    HUB_CUDA(cudaMemcpyAsync(y_host + b[c] * n_up, yd + b[c] * n_up, sizeof(double) * (b[c + 1] - b[c]) * n_up,
                             cudaMemcpyDeviceToHost, sc));
  }
  return HUB_OK;
}

// Sectors below this are multiplied in one piece (copy in, hub_apply, copy out): their copies take
// less than the chunks' launches.
constexpr int64_t kHostPipelineMin = (int64_t)1 << 22;

bool fast_host_pipelined(const hub_ctx *h) {
  const FastState *f = fast_of(h);
  return f && f->built && f->staged && h->count[1] >= 2 * kHostChunks &&
         h->count[0] * h->count[1] >= kHostPipelineMin;
}

// The chunked copies and passes of fast_apply_host: input chunks on the copy stream, pass 1
// per chunk, the route flag read on the host, pass 2 and the output chunks back on the copy
// stream.
static int pipeline_host(hub_ctx *h, FastState *f, const double *x_host, double *y_host, double *xd, double *yd,
                         cudaStream_t s, const HostChunks &C) {
  const int64_t n_up = h->count[0], n_dn = h->count[1];
  int rc;
  cudaStream_t sc = f->copy_stream;
  cudaEvent_t *ev_in = f->events.data(), *ev_out = ev_in + kHostChunks, ev_end = ev_in[2 * kHostChunks + 1];
  for (int c = 0; c < C.nci; ++c) {
    HUB_CUDA(cudaMemcpyAsync(xd + C.bi[c] * n_up, x_host + C.bi[c] * n_up,
                             sizeof(double) * (C.bi[c + 1] - C.bi[c]) * n_up, cudaMemcpyHostToDevice, sc));
    HUB_CUDA(cudaEventRecord(ev_in[c], sc));
  }
  if ((rc = host_pass1(h, f, xd, C.bi, C.nci, C.per, ev_in, s))) return rc;
  HUB_CUDA(cudaStreamSynchronize(s));
  set_route(h, *f->h_flag == 2 ? HUB_ROUTE_FP64 : HUB_ROUTE_DF);
  if (*f->h_flag == 2) {   // outside the double-float window: the FP64 kernel, one copy back
    if ((rc = f64_apply(h, xd, yd, nullptr, s))) return rc;
    HUB_CUDA(cudaMemcpyAsync(y_host, yd, sizeof(double) * n_dn * n_up, cudaMemcpyDeviceToHost, s));
    HUB_CUDA(cudaStreamSynchronize(s));
    return HUB_OK;
  }
  if (*f->h_flag == 1 && (rc = host_redo(h, f, xd, s))) return rc;
  if ((rc = host_pass2(h, f, yd, y_host, C.bo, C.nco, C.per, ev_out, s, sc))) return rc;
  HUB_CUDA(cudaEventRecord(ev_end, sc));
  HUB_CUDA(cudaStreamWaitEvent(s, ev_end, 0));
  HUB_CUDA(cudaStreamSynchronize(s));
  return HUB_OK;
}

// hub_apply_host on the fast path with staged rows.  The input arrives in row chunks on a copy
// stream while the compute stream converts each chunk and runs pass 1 on its row pairs; after
// pass 2 the output goes back in row chunks while later chunks are un-permuted.  The
// power-of-two scale of the conversion is taken from the first chunk's largest exponent; if
// the whole vector's largest exponent is larger, conversion and pass 1 are redone with it, so
// the result is that of these kernels on the whole vector (hub_apply itself runs sectors of this
// size in fixed point).  xd, yd: the handle's FP64 device buffers.
int fast_apply_host(hub_ctx *h, const double *x_host, double *y_host, double *xd, double *yd, cudaStream_t s) {
  FastState *f = fast_of(h);
  if (!f || !f->built) return fail(HUB_ERR_STATE, "fast apply: not built");
  const int64_t n_up = h->count[0], n_dn = h->count[1];
  if (!fast_host_pipelined(h)) return fail(HUB_ERR_STATE, "fast apply: no row-chunk pipeline for this sector");
  int rc;
  if ((rc = host_pipe_buffers(h, f))) return rc;
  // events: [kHostChunks] input chunks, [kHostChunks] output chunks, start, end
  if ((rc = ensure_events(f->events, 2 * kHostChunks + 2))) return rc;
  cudaStream_t sc = f->copy_stream;
  const cudaEvent_t ev_start = f->events[2 * kHostChunks];
  const HostChunks C = host_chunks(n_dn);
  HUB_CUDA(cudaEventRecord(ev_start, s));
  HUB_CUDA(cudaStreamWaitEvent(sc, ev_start, 0));
  rc = pipeline_host(h, f, x_host, y_host, xd, yd, s, C);
  if (rc) {   // no copy into or out of the caller's buffers may outlive the call
    cudaStreamSynchronize(sc);
    cudaStreamSynchronize(s);
  }
  return rc;
}


// hub_apply_host_many on the fast path with staged rows.  While the compute stream works on
// vector v, vector v + 1's rows come in on the input copy stream and vector v - 1's output goes
// back on the output copy stream (the host link carries both directions at once).  The FP64
// device buffers alternate between even and odd vectors (xd[v & 1], yd[v & 1]): an input
// buffer is refilled only after the compute stream has finished reading it (x_free), an output
// buffer is rewritten only after its copy to the host has ended (y_free).  Each vector takes
// the same kernels, scale and route as in fast_apply_host, so every result is bit for bit that
// of one hub_apply_host call.  The host waits once per vector, for its route flag after pass 1;
// the next vector's input copies are queued before that wait.
int fast_apply_host_many(hub_ctx *h, int64_t n_vec, const double *x_host, double *y_host, double *const xd[2],
                         double *const yd[2], cudaStream_t s) {
  FastState *f = fast_of(h);
  if (!fast_host_pipelined(h)) return fail(HUB_ERR_STATE, "fast apply: no row-chunk pipeline for this sector");
  const int64_t n_up = h->count[0], n_dn = h->count[1], D = n_up * n_dn;
  int rc;
  if ((rc = host_pipe_buffers(h, f))) return rc;
  if (!f->copy_out_stream) HUB_CUDA(cudaStreamCreateWithFlags(&f->copy_out_stream, cudaStreamNonBlocking));
  // events: [2][kHostChunks] input chunks (by buffer), [kHostChunks] output chunks,
  // x_free[2], y_free[2], start, end
  if ((rc = ensure_events(f->many_events, 3 * kHostChunks + 6))) return rc;
  cudaEvent_t *ev_in = f->many_events.data(), *ev_out = ev_in + 2 * kHostChunks, *x_free = ev_out + kHostChunks,
              *y_free = x_free + 2;
  const cudaEvent_t ev_start = y_free[2], ev_end = y_free[3];
  const HostChunks C = host_chunks(n_dn);
  cudaStream_t si = f->copy_stream, so = f->copy_out_stream;

  auto copy_in = [&](int64_t v) -> int {
    const int p = (int)(v & 1);
    if (v >= 2) HUB_CUDA(cudaStreamWaitEvent(si, x_free[p], 0));
    for (int c = 0; c < C.nci; ++c) {
      HUB_CUDA(cudaMemcpyAsync(xd[p] + C.bi[c] * n_up, x_host + v * D + C.bi[c] * n_up,
                               sizeof(double) * (C.bi[c + 1] - C.bi[c]) * n_up, cudaMemcpyHostToDevice, si));
      HUB_CUDA(cudaEventRecord(ev_in[p * kHostChunks + c], si));
    }
    return HUB_OK;
  };
  auto run = [&]() -> int {
    int rc;
    HUB_CUDA(cudaEventRecord(ev_start, s));
    HUB_CUDA(cudaStreamWaitEvent(si, ev_start, 0));
    HUB_CUDA(cudaStreamWaitEvent(so, ev_start, 0));
    if ((rc = copy_in(0))) return rc;
    for (int64_t v = 0; v < n_vec; ++v) {
      const int p = (int)(v & 1);
      if ((rc = host_pass1(h, f, xd[p], C.bi, C.nci, C.per, ev_in + p * kHostChunks, s))) return rc;
      if (v + 1 < n_vec && (rc = copy_in(v + 1))) return rc;
      HUB_CUDA(cudaStreamSynchronize(s));
      const int route = *f->h_flag;
      set_route(h, route == 2 ? HUB_ROUTE_FP64 : HUB_ROUTE_DF);
      if (route == 1 && (rc = host_redo(h, f, xd[p], s))) return rc;
      if (v >= 2) HUB_CUDA(cudaStreamWaitEvent(s, y_free[p], 0));
      if (route == 2) {   // outside the double-float window: the FP64 kernel, one copy back
        if ((rc = f64_apply(h, xd[p], yd[p], nullptr, s))) return rc;
        HUB_CUDA(cudaEventRecord(x_free[p], s));
        HUB_CUDA(cudaEventRecord(ev_out[0], s));
        HUB_CUDA(cudaStreamWaitEvent(so, ev_out[0], 0));
        HUB_CUDA(cudaMemcpyAsync(y_host + v * D, yd[p], sizeof(double) * D, cudaMemcpyDeviceToHost, so));
      } else {
        HUB_CUDA(cudaEventRecord(x_free[p], s));
        if ((rc = host_pass2(h, f, yd[p], y_host + v * D, C.bo, C.nco, C.per, ev_out, s, so))) return rc;
      }
      HUB_CUDA(cudaEventRecord(y_free[p], so));
    }
    HUB_CUDA(cudaEventRecord(ev_end, so));
    HUB_CUDA(cudaStreamWaitEvent(s, ev_end, 0));
    HUB_CUDA(cudaStreamSynchronize(s));
    return HUB_OK;
  };
  rc = run();
  if (rc) {   // no copy into or out of the caller's buffers may outlive the call
    cudaStreamSynchronize(si);
    cudaStreamSynchronize(so);
    cudaStreamSynchronize(s);
  }
  return rc;
}

int fast_check_error(hub_ctx *h) {
  FastState *f = fast_of(h);
  if (!f) return HUB_OK;
  int e = 0;
  HUB_CUDA(cudaMemcpy(&e, f->d_err, sizeof(int), cudaMemcpyDeviceToHost));
  if (e) {
    HUB_CUDA(cudaMemset(f->d_err, 0, sizeof(int)));
    return fail(HUB_ERR_TIMEOUT, "a bounded wait for a staged row gave up (row copy never completed)");
  }
  return HUB_OK;
}

}  // namespace hub
