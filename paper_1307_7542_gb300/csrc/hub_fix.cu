// hub_fix.cu -- the product (Eq. 11) and the Lanczos recurrence (Sec. IV, V) in 64-bit fixed
// point on the integer pipe, for uniform t and U without site energies.
//
// GB300 issues FP64 at about 1/70 of its integer rate, and a hopping term of the product is
// +-t x_m: with all entries of a vector on one power-of-two grid, x_m = X_m 2^e with X_m a
// 64-bit integer, a sum of terms is a sum of integers -- exact, and the same in any order.  What
// limits the product is then moving the terms.
//
// Each spin's hops run as one of two kernels.  Gathers (k_fix_gather): rows along which the spin
// varies are staged whole in shared memory, each thread sums the terms of its position; for up to
// kStageMax states.  Row combinations (k_fix_comb): the rows of the order along which the other
// spin varies are added and subtracted; for spins with more states.  Where both spins are of the
// same kind the vector is held in both orders (count_dn x count_up and its transpose), and whoever
// writes it -- the conversion of a caller's vector, the Lanczos update -- writes both, through a
// shared-memory tile; where they differ one order serves both passes.  The two passes write one
// contribution each, the second with the diagonal; k_fix_out or k_fix_update adds them.
//
// Grid.  |X_m| <= 2^B, B = min(56, 62 - hh), 2^hh >= the largest number of hopping terms of an
// entry, so that no sum overflows.  A rounded entry is off by at most 1/2 of 2^e: of the
// vector's largest entry 2^-B in a Lanczos run, 2^-(B-1) in a product.  Y is kept on the grid 2^(e + g), g >= 0 chosen for the diagonal.
//
// Lanczos vectors.  The vectors are kept unnormalised and monic, s_{j+1} = H s_j - alpha_j s_j -
// beta_j^2 s_{j-1} (q_j = s_j / |s_j|, beta_{j+1} = |s_{j+1}| / |s_j|), each on its own grid, so
// only shifts and two multiplications by a 55-bit coefficient are needed per entry, and the
// dot products <s_j, H s_j>, <s_j, s_{j-1}> and |s_{j+1}|^2 are integer sums (H s_j rounded to 7 bits
// fewer, the product of the lowest limbs to their high part, and left out of <s_j, s_{j-1}>): no
// result depends on the order in which blocks finish.  A rounding is 2^-56 of a vector's largest entry
// at most, so that an entry of rms size keeps 53 bits of a random start vector, 46 after sixty steps at 4x4 half
// filling, 45 to 41 of a 4x4 ground state with an electron added.  Its start vector uses the whole grid
// (k_fix_plan).  Largest error of alpha over the first steps against long double (12-site ring, 24 steps;
// in brackets with double-float vectors, which kept 48 bits of every entry): random start 3.7e-15
// (3.9e-14) at U = 4, 5.4e-15 (9.0e-14) at U = 7.25, all entries positive 4.3e-15 (4.3e-14), one entry of
// 400 rms 1.6e-14 (4.8e-14), one configuration 4.1e-15 (5.8e-14), a ground state 1.2e-13 (2.2e-12), an
// electron added to it 8.2e-14 (1.0e-13), at U = 12 8.7e-14 (1.7e-13).  Against FP64 vectors, whose own
// errors are of that size: 4x4 half filling, 60 steps, 1e-14 (9e-14) at U = 4, 4e-14 (3e-13) at U = 8;
// an electron added, 20 steps, 4e-14 (7e-14).
//
// Products for a caller (hub_apply) must keep every entry within 1e-13 (|H||x|)_n, which a grid
// fixed by the largest entry does not give where (|H||x|)_n is small.  k_fix_out sees the entry's
// two sums: if neither reaches the threshold that proves the bound, the entry's index is recorded
// and k_fix_entries recomputes it in FP64.  A vector with many small entries (a sample decides
// beforehand), or with more such entries than the list holds, is multiplied by the double-float
// or FP64 kernels instead, all on device flags, without a host round trip.
//
// Measured on the 4x4 cluster at half filling (1.66e8 states): a Lanczos step 4.12 ms (passes 1.32
// and 1.31, update 1.38) against 5.0 ms in double-float; a product 4.2 ms against 6.1 ms.
#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

#include "hub_internal.cuh"

namespace hub {

std::vector<double> tridiag_vector(const double *a, const double *b, int k, double lam);

typedef long long i64;
typedef unsigned long long u64;

constexpr int kFixMaxBits = 56;     // largest B
constexpr int kFixSpare = 2;        // bits beyond B that an update may use before k_fix_rescale
constexpr int kStageMax = 14384;    // longest rows that are staged: two of 115 KB
constexpr int kCombCols = 128;      // columns of a combination strip: four per lane
constexpr int kCombThreads = 256;
constexpr int kCombPairs = 3;       // pairs of rows loaded before the first is added
constexpr int kCombRows = 64;       // most rows of a tile
constexpr int kTileThreads = 256;
constexpr int kUpdateBlocks = 4;    // resident update CTAs per SM (64 registers a thread)
constexpr int kFixSlots = 64;       // copies of the accumulators (fewer collisions of atomics)
constexpr int kFixHist = 8;         // Lanczos steps recorded between two host read-backs
constexpr int kFixFrac = 4;         // fraction bits of the update's sums

// ctl words of a product (device): see k_fix_plan
enum { kCtlShift = 0, kCtlSkip = 1, kCtlDf = 2, kCtlF64 = 3, kCtlDfScale = 4, kCtlCount = 6, kCtlScale = 8, kCtlWords = 10 };
// Entries to recompute: a 64-bit count over two words, since any number of a vector's entries may ask for it.
__device__ __forceinline__ u64 *count_of(int *ctl) { return reinterpret_cast<u64 *>(ctl + kCtlCount); }

// One spin's hopping matrix as row combinations: a row's entries are ordered adding pairs,
// subtracting pairs, then the last adding and the last subtracting one where their numbers are odd.
struct CombLists {
  int R;                              // rows of a tile
  const int32_t *rp;                  // row starts
  const uint32_t *cnt;                // adding entries | subtracting entries << 16
  const uint32_t *word;               // entries: rows of the vector
};
// The same as gathers inside a row: slices of two groups of 16 positions whose schedules (see
// k_fix_schedule) are of nearly the same length; a group is four quads of consecutive positions.  A
// step's entry is 16 bits, the position and +-1 as the top two bits; a lane's 16 bytes are eight
// steps, at word[(l * cap + j / 8) * 32 + lane] for step j of slice l; meta[l * 32 + lane] = the lane's position
// | the slice's steps (even) << 16.
struct GatherLists {
  const uint4 *word;
  const uint32_t *meta;
  int cap, slices;
};

// Diagonal in fixed point: d = U n
struct FixDiag {
  int kind;                           // 0: zero; 1: n times an integer; 2: table of n
  int mul;                            // kind 1: U / tau
  int shift;                          // bits the (high) product is shifted right
  i64 tab[32];                        // kind 2, in units of tau 2^(dh - 62)
};

// One contribution to the product: rows x positions of one order of the vector.
struct FixPass {
  i64 n_rows, n_pos, ld;              // ld: row stride in entries
  const i64 *x;
  i64 *out;
  const uint32_t *bits_row, *bits_pos;
  FixDiag diag;                       // kind 0 in the pass that leaves the diagonal to the other
  int q, g;                           // 62 - B; bits the grid of the output is coarser by
  int t_neg;                          // uniform t < 0: the sums change sign
  int *err;                           // device error flag
  int fail_waits;                     // test hook
  int chained;                        // launch_kernel's
  const int *skip;                    // products: device flag, nothing to do
  u64 *acc;                           // Lanczos: dot product and maximum into these slots
  struct FixScal *scal;               // Lanczos, second pass of a step: its last block ends the step
  int second;
};

// Lanczos scalars on the device.
struct FixScal {
  double N;                           // |S_j|^2 (an integer on its grid)
  double alpha, beta2;                // of step j
  double overlap;                     // <S_j, S_{j-1}>
  double max_cur, max_prev;           // bounds on |S_j|, |S_{j-1}|
  int rel;                            // exponent of S_{j-1}'s grid minus that of S_j's
  int sh;                             // exponent of S_{j+1}'s grid minus that of S_j's
  i64 ma, mb;                         // coefficients of the update (55-bit mantissas) ...
  int sy, sa, sb;                     // ... and the shifts of its three terms (right, left, left)
  double bound, ratio;                // on |S_{j+1}| on its grid; the last step's max |S_{j+1}| / bound
  int rescale;                        // bits S_{j+1} is too large by
  int step, hist_n;
  unsigned ticket_dn, ticket_up;
  double hist[3 * kFixHist];          // (alpha_j, beta_{j+1}, |S_j|^2) of the steps since the last read-back
};
// Accumulators: [kFixSlots][kAcc] 64-bit words: hh and mid sums split in 32-bit halves, two maxima, and
// the sums of a second dot product
constexpr int kAcc = 10;

__device__ __forceinline__ i64 shr_any(i64 v, int s) {   // v 2^-s, truncated
  return s >= 0 ? v >> min(s, 63) : (i64)((u64)v << min(-s, 62));
}
// v = hi 2^28 + lo, -2^27 <= lo < 2^27
__device__ __forceinline__ void limbs28(i64 v, int &hi, int &lo) {
  lo = (int)((unsigned)v << 4) >> 4;
  hi = (int)((v - lo) >> 28);
}
// A vector whose rows are staged for gathers holds its entries as the two limbs, lo in the low word:
// a sum of 8 terms +-X is then one multiply-add by +-1 per limb and term, without carries.
__device__ __forceinline__ i64 limbs_pack(i64 v) {
  int h, l;
  limbs28(v, h, l);
  return (i64)(((u64)(unsigned)h << 32) | (unsigned)l);
}
__device__ __forceinline__ void limbs_of(i64 p, int &hi, int &lo) {
  lo = (int)p;
  hi = (int)((u64)p >> 32);
}
__device__ __forceinline__ i64 limbs_value(int hi, int lo) { return (i64)hi * (1 << 28) + lo; }
template <bool kLimb>
__device__ __forceinline__ i64 fix_store(i64 v) {
  return kLimb ? limbs_pack(v) : v;
}
template <bool kLimb>
__device__ __forceinline__ void fix_load(i64 p, int &hi, int &lo) {
  if (kLimb)
    limbs_of(p, hi, lo);
  else
    limbs28(p, hi, lo);
}
__device__ __forceinline__ void prefetch_l2(const void *p, uint32_t bytes) {   // multiples of 16
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}
__device__ __forceinline__ i64 int2_bits(int2 v) { return (i64)(((u64)(unsigned)v.y << 32) | (unsigned)v.x); }
__device__ __forceinline__ i64 entry_of(int2 v) { return int2_bits(v); }     // of a vector stored plainly
// Sum of products: hh 2^56 + mid 2^28
struct Dot {
  i64 hh, mid;
  __device__ __forceinline__ void add(int ah, int al, int bh, int bl) {   // 0 <= bl < 2^28, the others signed limbs
    hh += (i64)ah * bh;
    mid += (i64)ah * bl;
    mid += (i64)al * bh;
    mid += (i64)__mulhi(al << 4, bl);
  }
  // without the product of the low limbs: their signs are independent, so that it adds 2^-48 /
  // sqrt(D) of the squared norms
  __device__ __forceinline__ void add_high(int ah, int al, int bh, int bl) {
    hh += (i64)ah * bh;
    mid += (i64)ah * bl;
    mid += (i64)al * bh;
  }
  __device__ __forceinline__ void square(int ah, int al) {
    hh += (i64)ah * ah;
    mid += (i64)(2 * ah) * al;
    mid += (i64)__mulhi(al << 2, al << 2);
  }
};
// Dot sums with their halves apart, so that a thread can add any number of them
struct DotLong {
  i64 v[4];
  __device__ __forceinline__ void take(Dot &d) {
    v[0] += d.hh >> 32;
    v[1] += d.hh & 0xffffffffll;
    v[2] += d.mid >> 32;
    v[3] += d.mid & 0xffffffffll;
    d.hh = d.mid = 0;
  }
  __device__ __forceinline__ void take_squares(Dot &d) {   // sums of squares up to 2^64
    v[0] += (i64)((u64)d.hh >> 32) - (d.hh >> 32);
    take(d);
  }
};

// x = X 2^e rounded to the nearest integer X (an FP64 subnormal counts as zero)
__device__ __forceinline__ i64 f64_to_fix(double x, int e) {
  const u64 b = (u64)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0) return 0;
  const u64 m = (b & 0x000fffffffffffffull) | 0x0010000000000000ull;
  const int s = ex - 1075 - e;
  u64 v;
  if (s >= 0) {
    v = m << min(s, 8);
  } else {
    const int r = -s;
    v = r >= 55 ? 0ull : (m + (1ull << (r - 1))) >> r;
  }
  return (b >> 63) ? -(i64)v : (i64)v;
}

// x c 2^-31 = X 2^e rounded to the nearest integer X, |X| < 2^57 (Lanczos start vectors: see k_fix_plan)
__device__ __forceinline__ i64 f64_to_fix_scaled(double x, unsigned c, int e) {
  const u64 b = (u64)__double_as_longlong(x);
  const int ex = (int)((b >> 52) & 0x7ff);
  if (ex == 0) return 0;
  const u64 m = ((b & 0x000fffffffffffffull) | 0x0010000000000000ull) << 11;
  const u64 p = __umul64hi(m, (u64)c << 32);             // x c 2^-31 = p 2^(ex - 1085)
  const int r = e + 1085 - ex;                           // 7 and more
  const u64 v = r > 64 ? 0ull : ((p >> (r - 1)) + 1) >> 1;
  return (b >> 63) ? -(i64)v : (i64)v;
}

// v 2^e rounded to FP64 (results in the normal range)
__device__ __forceinline__ double fix_to_f64(i64 v, int e) {
  if (v == 0) return 0.0;
  const u64 sign = (u64)v & 0x8000000000000000ull;
  u64 m = v < 0 ? (u64)0 - (u64)v : (u64)v;
  const int lz = __clzll((i64)m);
  m <<= lz;
  u64 r = m >> 11;
  const unsigned rem = (unsigned)m & 0x7ffu;
  r += (rem > 0x400u || (rem == 0x400u && (r & 1ull))) ? 1ull : 0ull;
  const int E = 63 - lz + e + 1023;
  return __longlong_as_double((i64)(sign | (((u64)(unsigned)(E - 1) << 52) + r)));
}

// True in exactly one block, the last to arrive; all slots are then complete.  Leaves the
// ticket at zero.
__device__ __forceinline__ bool last_block(unsigned *ticket) {
  __shared__ bool last;
  if (threadIdx.x < 32) __threadfence();     // the adding threads
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  __syncthreads();
  if (last && threadIdx.x == 0) *ticket = 0;
  return last;
}

// ---------------------------------------------------------------------------------------
// Scale and route of a caller's vector, from the range of its exponents.  ctl[kCtlShift]: exponent of
// max |x|; [kCtlSkip]: not for this path; [kCtlF64] / [kCtlDf]: the FP64 / double-float kernels
// multiply it instead.  A vector outside the double-float window (kExp*) goes to FP64 as before.
// `wide` vectors -- more than one in eight of 4096 sampled entries below 2^-8 of the largest -- would
// fill the list of entries to recompute; random numbers have 2 % there (max 6 sigma), a ground
// state of the 12-site ring 40 % and more.  Only time depends on the sample: the list catches what
// it misses.  [kCtlScale]: 2^31 times a factor, from just below 1 to 2, that takes max |x| to just below
// the next power of two but one: a Lanczos run is free to scale its start vector, so that it uses the whole
// grid.  The last block to finish decides; it leaves the ticket at zero.
// ---------------------------------------------------------------------------------------
constexpr int kPlanThreads = 256, kPlanSamples = 4096;
struct FixRange {                     // what the blocks hand to the last one
  unsigned ticket;
  uint16_t sample[kPlanSamples];      // exponents of every D / kPlanSamples-th entry (0: none)
  int part[1];                        // top word of the largest magnitude, then smallest exponent, of each block
};
__global__ void __launch_bounds__(kPlanThreads) k_fix_plan(i64 D, const double *__restrict__ x, int df_ok,
                                                           FixRange *__restrict__ R, int *__restrict__ ctl) {
  __shared__ int wmax[kPlanThreads / 32], wmin[kPlanThreads / 32], sum;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, nblk = gridDim.x;
  const i64 first = blockIdx.x * (i64)kPlanThreads + tid, step = D > kPlanSamples ? D / kPlanSamples : 1;
  if (first < kPlanSamples)
    R->sample[first] = first * step < D ? (uint16_t)(((u64)__double_as_longlong(x[first * step]) >> 52) & 0x7ff) : 0;
  int a = 0, c = 2048;
  auto across = [&]() {               // the block's range, in every thread
    a = __reduce_max_sync(0xffffffffu, a);
    c = __reduce_min_sync(0xffffffffu, c);
    if (lane == 0) {
      wmax[warp] = a;
      wmin[warp] = c;
    }
    __syncthreads();
    for (int k = 0; k < kPlanThreads / 32; ++k) {
      a = max(a, wmax[k]);
      c = min(c, wmin[k]);
    }
  };
  for (i64 k = first; k < D; k += (i64)nblk * kPlanThreads) {
    const u64 b = (u64)__double_as_longlong(x[k]);
    const int top = (int)(b >> 32) & 0x7fffffff;
    a = max(a, top);
    if (b << 1) c = min(c, top >> 20);
  }
  across();
  if (tid == 0) {
    R->part[blockIdx.x] = a;
    R->part[nblk + blockIdx.x] = c;
    sum = 0;
  }
  __threadfence();                    // the samples are every thread's
  if (!last_block(&R->ticket)) return;
  __threadfence();
  a = 0;
  c = 2048;
  for (int k = tid; k < nblk; k += kPlanThreads) {
    a = max(a, __ldcg(R->part + k));
    c = min(c, __ldcg(R->part + nblk + k));
  }
  __syncthreads();
  across();
  const unsigned mant = ((unsigned)a & 0xfffffu) + 0x100001u;       // max |x| is below mant 2^-20 of its power of two
  a >>= 20;
  int n = 0;
  const int samples = (int)min(D, (i64)kPlanSamples);
  for (int k = tid; k < samples; k += kPlanThreads) n += __ldcg(R->sample + k) < a - 8 ? 1 : 0;
  atomicAdd(&sum, n);
  __syncthreads();
  if (tid != 0) return;
  const bool out = a != 0 && (a < kExpLo || a > kExpHi || c < a - kExpSpan);
  const bool wide = a == 0 || 8 * sum > samples;
  ctl[kCtlShift] = ctl[kCtlDfScale] = a == 0 ? 0 : a - 1023;
  ctl[kCtlDfScale + 1] = 0;
  ctl[kCtlScale] = (int)(unsigned)(((1ull << 52) - (1ull << 38)) / mant);
  ctl[kCtlSkip] = out || wide ? 1 : 0;
  *count_of(ctl) = 0;
  ctl[kCtlDf] = !out && wide && df_ok ? 1 : 0;
  ctl[kCtlF64] = out || (wide && !df_ok) ? 1 : 0;
}

// A thread's sums (N = 4: one dot product, 8: two) into the block's slot; vmax (top word of the
// largest magnitude) into maximum number `which`.
template <int N>
__device__ __forceinline__ void block_sums(i64 (&v)[N], unsigned vmax, int which, u64 *__restrict__ acc) {
  __shared__ i64 sv[N][32];
  __shared__ unsigned sm[32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = (int)(blockDim.x >> 5);
  const i64 total = warp_totals<N>(v);
  vmax = __reduce_max_sync(0xffffffffu, vmax);
  if (lane < N) sv[lane][warp] = total;
  if (lane == 0) sm[warp] = vmax;
  __syncthreads();
  if (warp == 0) {
    u64 *slot = acc + (size_t)(blockIdx.x % kFixSlots) * kAcc;
    if (lane < N) {
      i64 t = 0;
      for (int k = 0; k < nw; ++k) t += sv[lane][k];
      atomicAdd(slot + (lane < 4 ? lane : lane + 2), (u64)t);
    }
    vmax = __reduce_max_sync(0xffffffffu, lane < nw ? sm[lane] : 0u);
    if (lane == 0) atomicMax(slot + 4 + which, (u64)vmax);
  }
}

// hh 2^56 + mid 2^28 of summed halves as a double, exact to 2^-53 of the total
__device__ __forceinline__ double dot_value(const i64 *s) {
  const i64 mid_hi = s[2] + (s[3] >> 32), mid_lo = s[3] & 0xffffffffll;
  const i64 hh_hi = s[0] + (s[1] >> 32), hh_lo = s[1] & 0xffffffffll;
  return (double)hh_hi * 0x1p88 + ((double)hh_lo * 0x1p56 + ((double)mid_hi * 0x1p60 + (double)mid_lo * 0x1p28));
}
// Sums of the slots (first warp): the two dot products and bounds on the two maxima; the slots are
// left at zero for the next kernel.
struct SlotSums {
  double dot, dot2, max0, max1;
};
__device__ __forceinline__ SlotSums take_slots(u64 *acc) {
  __threadfence();
  i64 s[8] = {0, 0, 0, 0, 0, 0, 0, 0};
  unsigned m0 = 0, m1 = 0;
  for (int k = threadIdx.x; k < kFixSlots; k += 32) {
    u64 *p = acc + (size_t)k * kAcc;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      s[i] += (i64)__ldcg(p + i);
      s[4 + i] += (i64)__ldcg(p + 6 + i);
    }
    m0 = max(m0, (unsigned)__ldcg(p + 4));
    m1 = max(m1, (unsigned)__ldcg(p + 5));
    for (int i = 0; i < kAcc; ++i) p[i] = 0;
  }
  for (int o = 16; o > 0; o >>= 1)
#pragma unroll
    for (int i = 0; i < 8; ++i) s[i] += __shfl_xor_sync(0xffffffffu, s[i], o);
  return SlotSums{dot_value(s), dot_value(s + 4), ((double)__reduce_max_sync(0xffffffffu, m0) + 1.0) * 0x1p32,
                  ((double)__reduce_max_sync(0xffffffffu, m1) + 1.0) * 0x1p32};
}

// diag(row, position) X on the output's grid, X = xh 2^28 + xl
__device__ __forceinline__ i64 diag_term(const FixPass &P, const i64 *__restrict__ tab, uint32_t Ir, uint32_t Ip,
                                         int xh, int xl) {
  const FixDiag &G = P.diag;
  const uint32_t both = Ir & Ip;
  if (G.kind == 1) {
    const int k = G.mul * __popc(both);
    const i64 v = (i64)xl * k + ((i64)xh * k) * (1 << 28);
    return G.shift ? (v + (1ll << (G.shift - 1))) >> G.shift : v;
  }
  const i64 X = limbs_value(xh, xl);
  return shr_any(__mul64hi(tab[__popc(both)], (i64)((u64)X << P.q)), G.shift);
}

// An entry of a pass: hopping sum s, own entry X.  Returns the output; kLz: adds to the dot
// product <X, output 2^-7> and the maximum.  The output enters the dot product rounded to a multiple of
// 128, not cut off: 64 units too little in every entry add up where the entries of X have one sign
// (alpha of an all-positive vector off by 2e-15 of the operator's scale and more, now 2e-17; the
// bound on the sums leaves room for the 64).
template <bool kLz>
__device__ __forceinline__ i64 pass_entry(const FixPass &P, const i64 *__restrict__ tab, i64 s, int xh, int xl,
                                          uint32_t Ir, uint32_t Ip, Dot &dot, unsigned &vmax) {
  if (P.g) s = (s + (1ll << (P.g - 1))) >> P.g;
  if (P.diag.kind) s += diag_term(P, tab, Ir, Ip, xh, xl);
  if (kLz) {
    const i64 r = s + 64;
    const int yh = (int)((u64)r >> 32);
    dot.add(xh, xl, yh >> 3, (int)((unsigned)(r >> 7) & 0x0fffffffu));
    vmax = max(vmax, (unsigned)abs(yh));
  }
  return s;
}

// The end of a pass: sums into the slots; the last block of a step's second pass turns them into
// alpha_j and the coefficients of the update
//   S_{j+1} = 2^-sh (2^g (out_1 + out_2) - alpha S_j - beta^2 2^rel S_{j-1}),
// sh from a bound on its entries, which keeps them below 2^(B + kFixSpare), and from the part of the
// bound that the last step's largest entry reached (a third as a rule, nearly the same from step to
// step), so that they come to lie between 2^(B-1) and 2^B; where they do not, k_fix_rescale takes
// the spare bits off.
__device__ __forceinline__ void pass_end(const FixPass &P, const DotLong &dot, unsigned vmax) {
  i64 v[4] = {dot.v[0], dot.v[1], dot.v[2], dot.v[3]};
  block_sums<4>(v, vmax, P.second, P.acc);
  if (!P.second || !last_block(&P.scal->ticket_dn) || threadIdx.x >= 32) return;
  const SlotSums t = take_slots(P.acc);
  const double d = t.dot * 128.0, m0 = t.max0, m1 = t.max1;
  if (threadIdx.x != 0) return;
  FixScal &q = *P.scal;
  const int B = 62 - P.q;
  // alpha_j = <q_j, H q_j - beta_j q_{j-1}>: the overlap of S_j and S_{j-1} is rounding only, but
  // without its term it would double from step to step
  const double bp = ldexp(q.beta2, q.rel), G = (double)(1ll << P.g), alpha = (d * G - bp * q.overlap) / q.N;
  const double bound = (m0 + m1) * G + fabs(alpha) * q.max_cur + bp * q.max_prev;
  int sh = 0, least = 0, xa = 0, xb = 0;
  frexp(bound, &least);                    // bound < 2^least
  frexp(bound * fmin(1.0, 1.05 * q.ratio), &sh);
  sh = max(sh - B, least - B - kFixSpare);
  q.bound = ldexp(bound, -sh);
  const double fa = frexp(ldexp(alpha, -sh), &xa), fb = frexp(ldexp(bp, -sh), &xb);
  q.alpha = alpha;
  q.sh = sh;
  q.ma = (i64)ldexp(fa, 55);
  q.mb = (i64)ldexp(fb, 55);
  q.sy = sh - P.g - kFixFrac;
  q.sa = xa + kFixFrac + 1;                // fa 2^55 S 2^-56 2^sa = alpha 2^-sh S 2^kFixFrac
  q.sb = xb + kFixFrac + 1;
}

// ---------------------------------------------------------------------------------------
// Gathers: the hops of the positions' spin.  A CTA stages two rows of the vector whole in shared
// memory (bulk copies completing on an mbarrier), then each thread sums the hopping row of its
// position for both rows.  What bounds it is the shared-memory bandwidth, 8 bytes per term, so the
// schedule lets a half-warp's 16 eight-byte loads hit 16 different bank pairs (position mod
// 16), idle steps reading a zero of a bank left free.  Issue slots come next: a term's sign is a
// factor +-1 of one multiply-add per limb, which leaves the schedule free to mix signs (steps of one
// sign each save a third of the instructions but need 13 % more steps, and ran 20 % slower).
// ---------------------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_addr(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t phase) {   // bounded: about 2^24 polls
  for (uint32_t it = 0; it < (1u << 24); ++it) {
    uint32_t ok;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}"
        : "=r"(ok)
        : "r"(smem_addr(bar)), "r"(phase)
        : "memory");
    if (ok) return true;
  }
  return false;
}

// kPlane: entries from one staged row to the next (a constant, so that both rows' loads of a term
// share one address).  kLimb: entries stored as limbs.
template <int kPlane, bool kLz, bool kLimb>
__global__ void __launch_bounds__(1024, 1) k_fix_gather(const FixPass P, const GatherLists L) {
  extern __shared__ __align__(128) unsigned char smem[];
  int2 *const x0 = reinterpret_cast<int2 *>(smem), *const x1 = x0 + kPlane;   // entries ld .. ld + 15 are zero
  __shared__ __align__(8) uint64_t bar;
  __shared__ i64 utab[32];
  if (!kLz) {
    after_previous();
    if (flag_of(P.skip)) return;
  }
  const int tid = threadIdx.x, lane = tid & 31;
  if (tid < 32) {
    utab[tid] = P.diag.tab[tid];
    (tid < 16 ? x0 : x1)[P.ld + (tid & 15)] = make_int2(0, 0);     // idle steps read one of these
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&bar)) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
  const uint32_t bytes = (uint32_t)(P.ld * sizeof(i64));
  const i64 pairs = (P.n_rows + 1) / 2;
  const int n_pos = (int)P.n_pos;
  uint32_t phase = 0;
  DotLong dots{{0, 0, 0, 0}};
  unsigned vmax = 0;
  for (i64 p = blockIdx.x; p < pairs; p += gridDim.x) {
    const i64 r0 = 2 * p;
    const bool two = r0 + 1 < P.n_rows;
    const i64 *s0 = P.x + r0 * P.ld, *s1 = two ? s0 + P.ld : s0;   // odd tail: the same row twice
    if (tid == 0) {
      asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
      asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(&bar)), "r"(2 * bytes)
                   : "memory");
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                       smem_addr(x0)),
                   "l"(s0), "r"(bytes), "r"(smem_addr(&bar))
                   : "memory");
      asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                       smem_addr(x1)),
                   "l"(s1), "r"(bytes), "r"(smem_addr(&bar))
                   : "memory");
      const i64 pn = p + gridDim.x;           // the CTA's next pair into L2 meanwhile
      if (pn < pairs)
        prefetch_l2(P.x + 2 * pn * P.ld, 2 * pn + 1 < P.n_rows ? 2 * bytes : bytes);
    }
    const uint32_t I0 = P.diag.kind ? P.bits_row[r0] : 0u, I1 = P.diag.kind && two ? P.bits_row[r0 + 1] : I0;
    if (!mbar_wait(&bar, phase)) {
      if (tid == 0) atomicExch(P.err, 1);
      mbar_wait(&bar, phase);                 // give a late copy one more bounded chance to land
      return;
    }
    if (P.fail_waits) {                       // test hook: the same exit, after the copies landed
      if (tid == 0) atomicExch(P.err, 1);
      return;
    }
    phase ^= 1u;
    i64 *const o0 = P.out + r0 * P.ld, *const o1 = o0 + P.ld;
    Dot dot{0, 0};
    const int nw = (int)(blockDim.x >> 5);
    const uint4 *__restrict__ wp = L.word + (uint32_t)((tid >> 5) * L.cap * 32 + lane);
    int sl = tid >> 5;
    uint32_t meta = 0;
    uint4 qn = make_uint4(0u, 0u, 0u, 0u);
    if (sl < L.slices) {
      meta = L.meta[sl * 32 + lane];
      qn = wp[0];
    }
    for (; sl < L.slices; sl += nw) {
      const int s = (int)(meta & 0xffffu);
      int n = (int)(meta >> 16);
      const uint4 *__restrict__ w4 = wp;
      wp += (uint32_t)(nw * L.cap * 32);
      const bool more = sl + nw < L.slices;
      if (more) meta = L.meta[(sl + nw) * 32 + lane];
      i64 a0 = 0, a1 = 0;
#define FIX_TERM(ADDR, SGN)                                                  \
  do {                                                                       \
    const int2 *at_ = reinterpret_cast<const int2 *>(smem + (ADDR));         \
    const int2 u_ = at_[0], v_ = at_[kPlane];                                \
    const int s_ = (SGN);                                                    \
    if (kLimb) {                                                             \
      l0 = u_.x * s_ + l0;                                                   \
      h0 = u_.y * s_ + h0;                                                   \
      l1 = v_.x * s_ + l1;                                                   \
      h1 = v_.y * s_ + h1;                                                   \
    } else {                                                                 \
      a0 += s_ < 0 ? -entry_of(u_) : entry_of(u_);                           \
      a1 += s_ < 0 ? -entry_of(v_) : entry_of(v_);                           \
    }                                                                        \
  } while (0)
#define FIX_WORD(W)                                                          \
  do {                                                                       \
    const uint32_t w_ = (W);                                                 \
    FIX_TERM((w_ << 3) & 0x1fff8u, (int)(w_ << 16) >> 30);                   \
    FIX_TERM((w_ >> 13) & 0x1fff8u, (int)w_ >> 30);                          \
  } while (0)
      for (; n > 0; n -= 8) {
        const uint4 q = qn;
        int h0 = 0, l0 = 0, h1 = 0, l1 = 0;   // limb sums of 8 terms, below 2^31
        if (n >= 8) {
          w4 += 32;
          if (n > 8) qn = w4[0];              // next batch in flight
          FIX_WORD(q.x);
          FIX_WORD(q.y);
          FIX_WORD(q.z);
          FIX_WORD(q.w);
        } else {
          FIX_WORD(q.x);
          if (n > 2) FIX_WORD(q.y);
          if (n > 4) FIX_WORD(q.z);
        }
        if (kLimb) {
          a0 += limbs_value(h0, l0);
          a1 += limbs_value(h1, l1);
        }
      }
#undef FIX_WORD
#undef FIX_TERM
      if (more) qn = wp[0];                   // the next slice's first batch
      if (P.t_neg) {
        a0 = -a0;
        a1 = -a1;
      }
      if (s >= n_pos) continue;
      const uint32_t Ip = P.diag.kind ? P.bits_pos[s] : 0u;
      const int2 u = x0[s], v = x1[s];
      int uh, ul, vh, vl;
      fix_load<kLimb>(int2_bits(u), uh, ul);
      fix_load<kLimb>(int2_bits(v), vh, vl);
      o0[s] = pass_entry<kLz>(P, utab, a0, uh, ul, I0, Ip, dot, vmax);
      if (two) o1[s] = pass_entry<kLz>(P, utab, a1, vh, vl, I1, Ip, dot, vmax);
    }
    if (kLz) dots.take(dot);
    __syncthreads();
  }
  if (kLz) pass_end(P, dots, vmax);
}

// Schedules, built on the device by the five kernels below (blockIdx.y: the spin), without a copy to
// the host, beside the allocation of the scratch vectors: a handle's first product waits for them.  The
// first product of the 13-site ring (6,6) takes 0.28 ms (0.29 without a schedule, in double-float; 0.51
// with the groups made on the host), of 4x4 (2,8) 0.42 ms (0.30; 1.4).
//
// Groups of 16 positions: four quads of consecutive positions each (the outputs of a quad are one 32-byte
// sector), chosen greedily among the next 32 quads, longest rows first, so that the group's
// busiest bank stays low; or the quads in their own order where that needs no more steps.  At 4x4 1.17
// steps per entry of a row against 1.26.
constexpr int kSchedRow = 64;         // longest hopping row of the gather form
constexpr int kSchedMax = 2 * kSchedRow;
// Quads that a warp groups: more of them make better groups (4x4, 12,870 positions: 1.197 steps per entry with
// 64, 1.186 with 128, 1.171 with all), but take a quarter of a microsecond each, before the first product.
constexpr int kSegMax = 1024;
static int seg_quads(double D) { return D < 0x1p22 ? 64 : (D < 0x1p25 ? 256 : kSegMax); }
struct SchedSpin {
  int n, groups, idle, cap, seg;      // positions, groups (even), the position of a zero, most steps, seg_quads
  const int32_t *rp;
  const uint32_t *scol;
  uint32_t *load;                     // [4 groups][8] entries of a quad by bank, two counts a word
  uint32_t *len;                      // [4 groups] bytes: longest row of a quad
  uint16_t *sorted, *greedy;          // [4 groups] quads by length; grouped
  uint8_t *steps;                     // [2][groups] steps of the groups in natural order, and grouped
  uint32_t *total;                    // [2] their sums
  uint16_t *quad;                     // [4 groups] the groups' quads, longest groups first ...
  uint8_t *deg;                       // [groups] ... and their steps
  uint16_t *word;                     // the schedule (GatherLists)
  uint32_t *meta;
};
struct SchedArgs {
  SchedSpin spin[2];
};

__global__ void __launch_bounds__(256) k_fix_quads(const SchedArgs A) {
  const SchedSpin &S = A.spin[blockIdx.y];
  __shared__ uint32_t count[16][16];
  const int half = threadIdx.x >> 4, lane = threadIdx.x & 15, q = blockIdx.x * 16 + half;
  if (blockIdx.x == 0 && threadIdx.x < 2) S.total[threadIdx.x] = 0;
  count[half][lane] = 0;
  __syncthreads();
  const int r0 = min(4 * q, S.n), r1 = min(4 * q + 4, S.n);
  for (int32_t k = S.rp[r0] + lane; k < S.rp[r1]; k += 16) atomicAdd(&count[half][S.scol[k] & 15], 1u);
  __syncthreads();
  if (q >= 4 * S.groups) return;
  if (lane < 8) S.load[8 * q + lane] = count[half][2 * lane] | (count[half][2 * lane + 1] << 16);
  if (lane == 8) {
    int m = 0;
    for (int r = r0; r < r1; ++r) m = max(m, S.rp[r + 1] - S.rp[r]);
    reinterpret_cast<uint8_t *>(S.len)[q] = (uint8_t)m;
  }
}

// Place of byte i among the bytes of w, largest first and equal ones in their order.
__device__ __forceinline__ int place_desc(const uint32_t *w, int words, int i) {
  const uint32_t own = w[i >> 2], v = (own >> (8 * (i & 3))) & 255u, v4 = v * 0x01010101u;
  int above = 0;
  for (int k = 0; k < (i >> 2); ++k) above += __popc(__vcmpgeu4(w[k], v4));
  for (int k = (i >> 2) + 1; k < words; ++k) above += __popc(__vcmpgtu4(w[k], v4));
  above >>= 3;
  for (int j = 0; j < 4; ++j) {
    const uint32_t b = (own >> (8 * j)) & 255u;
    above += b > v || (b == v && j < (i & 3)) ? 1 : 0;
  }
  return above;
}

constexpr int kSchedQuads = (kStageMax + 31) / 32 * 8;       // most quads of a spin
__global__ void __launch_bounds__(256) k_fix_sort(const SchedArgs A) {
  const SchedSpin &S = A.spin[blockIdx.y];
  __shared__ uint32_t len[kSchedQuads / 4];
  for (int k = threadIdx.x; k < S.groups; k += 256) len[k] = S.len[k];
  __syncthreads();
  const int q = blockIdx.x * 256 + threadIdx.x;
  if (q < 4 * S.groups) S.sorted[place_desc(len, S.groups, q)] = (uint16_t)q;
}

__global__ void __launch_bounds__(32) k_fix_group(const SchedArgs A) {
  const SchedSpin &S = A.spin[blockIdx.y];
  __shared__ uint32_t load[kSegMax][9];
  __shared__ uint16_t id[kSegMax], left[kSegMax];
  __shared__ uint8_t len[kSegMax];
  const int lane = threadIdx.x, base = blockIdx.x * S.seg, n = min(S.seg, 4 * S.groups - base);
  if (n <= 0) return;
  const uint8_t *lens = reinterpret_cast<const uint8_t *>(S.len);
  for (int i = lane; i < n; i += 32) {
    const int q = S.sorted[base + i];
    id[i] = (uint16_t)q;
    len[i] = lens[q];
    left[i] = (uint16_t)i;
#pragma unroll
    for (int w = 0; w < 8; ++w) load[i][w] = S.load[8 * q + w];
  }
  __syncwarp();
  uint32_t natural = 0, greedy = 0;
  for (int g = 0, head = 0; 4 * g < n; ++g) {
    uint32_t sum[8];                             // two banks a word, at most 16 rows of kSchedRow entries: 2^10
#pragma unroll
    for (int w = 0; w < 8; ++w) sum[w] = 0;
    uint32_t most = 0;
    for (int k = 0; k < 4; ++k, ++head) {
      const int window = k ? min(32, n - head) : 1;
      const int own = lane < window ? left[head + lane] : 0;
      uint32_t m2[2] = {0, 0}, sq[4] = {0, 0, 0, 0};         // sq <= 2^20 in all: the group's entries squared
#pragma unroll
      for (int w = 0; w < 8; ++w) {
        const uint32_t t = sum[w] + load[own][w];
        m2[w & 1] = __vmaxu2(m2[w & 1], t);
        sq[w & 1] += (t & 0xffffu) * (t & 0xffffu);
        sq[2 + (w & 1)] += (t >> 16) * (t >> 16);
      }
      const uint32_t mm = __vmaxu2(m2[0], m2[1]), m = max(mm & 0xffffu, mm >> 16);
      const uint32_t key = lane < window ? (m << 21) | (sq[0] + sq[1] + sq[2] + sq[3]) : ~0u;
      const int at = __ffs(__ballot_sync(0xffffffffu, key == __reduce_min_sync(0xffffffffu, key))) - 1;
      const int pick = __shfl_sync(0xffffffffu, own, at);
      __syncwarp();
      if (lane < at) left[head + lane + 1] = (uint16_t)own;
      if (lane == 0) {
        left[head] = (uint16_t)pick;
        S.greedy[base + 4 * g + k] = id[pick];
      }
      __syncwarp();
#pragma unroll
      for (int w = 0; w < 8; ++w) sum[w] += load[pick][w];
      most = max(most, (uint32_t)len[pick]);
    }
#pragma unroll
    for (int w = 0; w < 8; ++w) most = max(most, max(sum[w] & 0xffffu, sum[w] >> 16));
    most = min(most, (uint32_t)S.cap);
    // the same of the group in natural order
    const int ng = base / 4 + g;
    uint32_t v = 0;
    if (lane < 16)
      for (int k = 0; k < 4; ++k) v += (S.load[8 * (4 * ng + k) + (lane >> 1)] >> (16 * (lane & 1))) & 0xffffu;
    else if (lane < 20)
      v = lens[4 * ng + lane - 16];
    v = min(__reduce_max_sync(0xffffffffu, v), (uint32_t)S.cap);
    if (lane == 0) {
      S.steps[ng] = (uint8_t)v;
      S.steps[S.groups + ng] = (uint8_t)most;
    }
    natural += v;
    greedy += most;
  }
  if (lane == 0) {
    atomicAdd(S.total, natural);
    atomicAdd(S.total + 1, greedy);
  }
}

// The groups by length, so that the two of a slice need nearly the same number of steps.
__global__ void __launch_bounds__(1024) k_fix_order(const SchedArgs A) {
  const SchedSpin &S = A.spin[blockIdx.y];
  __shared__ uint32_t deg[(kSchedQuads / 4 + 3) / 4];
  const bool greedy = S.total[1] < S.total[0];
  const int words = (S.groups + 3) / 4;
  for (int k = threadIdx.x; k < words; k += 1024) {
    uint32_t w = 0;
    for (int j = 0; j < 4 && 4 * k + j < S.groups; ++j)
      w |= (uint32_t)S.steps[(greedy ? S.groups : 0) + 4 * k + j] << (8 * j);
    deg[k] = w;
  }
  __syncthreads();
  for (int g = threadIdx.x; g < S.groups; g += 1024) {
    const int at = place_desc(deg, words, g);
    S.deg[at] = (uint8_t)(deg[g >> 2] >> (8 * (g & 3)));
    for (int k = 0; k < 4; ++k) S.quad[4 * at + k] = greedy ? S.greedy[4 * g + k] : (uint16_t)(4 * g + k);
  }
}

// Schedule of a group of 16 positions, the lanes of a half-warp: a colouring of the bipartite graph
// lanes x banks (position mod 16) whose edges are the group's entries -- no two edges of a lane or
// of a bank share a step.  By Koenig's theorem as many steps suffice as the largest degree has
// edges; they are found edge by edge, exchanging two colours along an alternating path where the
// lane and the bank have no free step in common.  A bank with more entries than cap steps takes
// the rest in steps of its lanes alone (conflicts, but the schedule stays bounded).  A warp per
// group, one lane of which colours, with the free steps of lanes and banks as bit masks: 93 us at 4x4
// (a thread per group and linear searches: 0.8 ms).
constexpr uint16_t kNoEntry = 0xffff;
__global__ void __launch_bounds__(32) k_fix_schedule(const SchedArgs A) {
  const SchedSpin &S = A.spin[blockIdx.y];
  const int g = blockIdx.x, lane = threadIdx.x, n = S.n;
  if (g >= S.groups) return;
  const uint16_t *__restrict__ quad = S.quad;
  const int32_t *__restrict__ rp = S.rp;
  const uint32_t *__restrict__ scol = S.scol;
  __shared__ uint16_t at[16][kSchedMax];         // entry of a lane at a step
  __shared__ int8_t who[16][kSchedMax];          // lane that reads a bank at a step
  __shared__ u64 free_l[16][2], free_b[16][2];   // free steps
  for (int k = lane; k < 16 * kSchedMax; k += 32) {
    at[k / kSchedMax][k % kSchedMax] = kNoEntry;
    who[k / kSchedMax][k % kSchedMax] = -1;
  }
  const int steps = S.deg[g];
  if (lane < 16)
    for (int h = 0; h < 2; ++h) {
      const int m = min(max(steps - 64 * h, 0), 64);
      free_l[lane][h] = free_b[lane][h] = m == 64 ? ~0ull : (1ull << m) - 1ull;
    }
  __syncwarp();
  auto first = [](u64 a, u64 b) { return a ? __ffsll((long long)a) - 1 : (b ? 63 + __ffsll((long long)b) : -1); };
  for (int l = 0; lane == 0 && l < 16; ++l) {
    const int r = quad[4 * g + (l >> 2)] * 4 + (l & 3);
    if (r >= n) continue;
    for (int32_t k = rp[r]; k < rp[r + 1]; ++k) {
      const uint32_t w = scol[k];
      const uint16_t v = (uint16_t)((w & 0x3fffu) | (w >> 31 ? 0x4000u : 0xc000u));     // esign -1 adds
      const int b = w & 15;
      // a step free for both, or one of the lane and one of the bank
      int x = first(free_l[l][0] & free_b[b][0], free_l[l][1] & free_b[b][1]), y = x;
      if (x < 0) {
        x = first(free_l[l][0], free_l[l][1]);
        y = first(free_b[b][0], free_b[b][1]);
      }
      bool ok = y >= 0;
      if (ok && x != y) {
        // exchange steps x and y along the path b -x- lane -y- bank -x- ...: frees step x of b
        int8_t pl[34], pb[34];
        uint16_t pv[34];
        int m = 0;
        for (int cb = b; ok;) {
          const int l1 = who[cb][x];
          if (l1 < 0) break;
          pl[m] = (int8_t)l1;
          pb[m] = (int8_t)cb;
          pv[m++] = at[l1][x];
          const uint16_t v2 = at[l1][y];
          if (v2 == kNoEntry) break;
          cb = v2 & 15;
          pl[m] = (int8_t)l1;
          pb[m] = (int8_t)cb;
          pv[m++] = v2;
          ok = who[cb][y] == l1 && m < 32;   // else it meets an entry without a bank of its own
        }
        for (int i = 0; ok && i < m; ++i) {
          const int t = i & 1 ? y : x;
          at[(int)pl[i]][t] = kNoEntry;
          who[(int)pb[i]][t] = -1;
          free_l[(int)pl[i]][t >> 6] |= 1ull << (t & 63);
          free_b[(int)pb[i]][t >> 6] |= 1ull << (t & 63);
        }
        for (int i = 0; ok && i < m; ++i) {
          const int t = i & 1 ? x : y;
          at[(int)pl[i]][t] = pv[i];
          who[(int)pb[i]][t] = pl[i];
          free_l[(int)pl[i]][t >> 6] &= ~(1ull << (t & 63));
          free_b[(int)pb[i]][t >> 6] &= ~(1ull << (t & 63));
        }
      }
      at[l][x] = v;                   // the lane has a free step: steps >= its entries
      free_l[l][x >> 6] &= ~(1ull << (x & 63));
      if (ok) {
        who[b][x] = (int8_t)l;
        free_b[b][x >> 6] &= ~(1ull << (x & 63));
      }
    }
  }
  __syncwarp();
  // into the slice's layout; idle lanes read the zero of a bank the step leaves free
  const int all = (S.deg[g & ~1] + 1) & ~1, half = g & 1;          // words hold two steps
  for (int j = lane; j < max(8, (all + 7) & ~7); j += 32) {
    int fb = 0;
    while (fb < 15 && who[fb][j] >= 0) ++fb;
    const uint16_t z = (uint16_t)((S.idle + ((fb - S.idle) & 15)) | 0x4000);
    uint16_t *out = S.word + ((((size_t)(g >> 1) * (S.cap / 8) + (j >> 3)) * 32 + 16 * half) * 8 + (j & 7));
    for (int l = 0; l < 16; ++l) out[8 * l] = at[l][j] == kNoEntry ? z : at[l][j];
  }
  if (lane < 16) S.meta[16 * g + lane] = (uint32_t)(quad[4 * g + (lane >> 2)] * 4 + (lane & 3)) | ((uint32_t)all << 16);
}

// ---------------------------------------------------------------------------------------
// Row combinations: the hops of the rows' spin, where its rows are too long to stage.  Tile = R rows x 128 columns; tiles of one column strip are adjacent in the
// grid, so that the strip of x (n_rows x 128 values, 13 MB at 4x4) stays in L2 while all its
// row tiles combine it.  A warp takes a row at a time, lane l the columns 2l, 2l + 1, 64 + 2l and
// 65 + 2l: every load is a coalesced 512-byte segment, the index, address and branch work of an
// entry is shared by 128 sums, and pairs of equal sign take one three-operand add per word.
// ---------------------------------------------------------------------------------------

// four columns of a lane
struct Quad {
  i64 v[4];
};
__device__ __forceinline__ Quad ld_quad(const char *__restrict__ p, uint32_t up) {
  const longlong2 a = *reinterpret_cast<const longlong2 *>(p), b = *reinterpret_cast<const longlong2 *>(p + up);
  return Quad{{a.x, a.y, b.x, b.y}};
}

// A hopping row (entries k0 ..) summed over the lane's columns into s.  w: the words of its first
// 32 entries, one per lane (loaded while the previous row was summed); longer rows take them 32
// at a time.  up: byte offset of the lane's second pair of columns (0 where it has none).
__device__ __forceinline__ void comb_row(const CombLists &S, const char *__restrict__ xb, uint32_t row_bytes, uint32_t up,
                                         int lane, int32_t k0, uint32_t cnt, uint32_t w, Quad &s) {
  constexpr int kP = kCombPairs;
  const int na = cnt & 0xffff, ns = cnt >> 16, all = na + ns;
  const int pa = na & ~1, pe = pa + (ns & ~1);
#pragma unroll
  for (int i = 0; i < 4; ++i) s.v[i] = 0;
  for (int base = 0; base < all; base += 32) {
    if (base) w = S.word[k0 + base + lane];
    const int n = min(32, all - base);
    const int np = min(max(pe - base, 0), n), ae = pa - base;    // paired entries here, adding ones first
    Quad o0, o1;                                                 // the odd ones
    const bool odd0 = np < n, odd1 = np + 1 < n;
    const uint32_t c0 = __shfl_sync(0xffffffffu, w, np & 31), c1 = __shfl_sync(0xffffffffu, w, (np + 1) & 31);
    if (odd0) o0 = ld_quad(xb + (u64)c0 * row_bytes, up);
    if (odd1) o1 = ld_quad(xb + (u64)c1 * row_bytes, up);
    for (int j = 0; j < np; j += 2 * kP) {
      Quad v[2 * kP];
#pragma unroll
      for (int t = 0; t < kP; ++t) {
        const uint32_t ca = __shfl_sync(0xffffffffu, w, j + 2 * t), cb = __shfl_sync(0xffffffffu, w, j + 2 * t + 1);
        if (j + 2 * t < np) {
          v[2 * t] = ld_quad(xb + (u64)ca * row_bytes, up);
          v[2 * t + 1] = ld_quad(xb + (u64)cb * row_bytes, up);
        }
      }
#pragma unroll
      for (int t = 0; t < kP; ++t) {
        if (j + 2 * t < ae) {
#pragma unroll
          for (int i = 0; i < 4; ++i) s.v[i] = s.v[i] + v[2 * t].v[i] + v[2 * t + 1].v[i];
        } else if (j + 2 * t < np) {
#pragma unroll
          for (int i = 0; i < 4; ++i) s.v[i] = s.v[i] - v[2 * t].v[i] - v[2 * t + 1].v[i];
        }
      }
    }
    if (odd0) {                       // the adding one, unless there is none
      if (na & 1) {
#pragma unroll
        for (int i = 0; i < 4; ++i) s.v[i] += o0.v[i];
      } else {
#pragma unroll
        for (int i = 0; i < 4; ++i) s.v[i] -= o0.v[i];
      }
    }
    if (odd1) {
#pragma unroll
      for (int i = 0; i < 4; ++i) s.v[i] -= o1.v[i];
    }
  }
}

template <bool kLz>
__global__ void __launch_bounds__(kCombThreads, 2) k_fix_comb(const FixPass P, const CombLists S) {
  constexpr int kWarps = kCombThreads / 32;
  __shared__ i64 utab[32];
  if (P.chained) after_previous();          // tested at run time: the Lanczos form without a test ran 10 % slower
  if (P.skip && flag_of(P.skip)) return;
  if (P.fail_waits) {                       // test hook: report as a given-up wait would
    if (threadIdx.x == 0) atomicExch(P.err, 1);
    return;
  }
  if (threadIdx.x < 32) utab[threadIdx.x] = P.diag.tab[threadIdx.x];
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const uint32_t tiles = (uint32_t)((P.n_rows + S.R - 1) / S.R);
  const uint32_t strip = blockIdx.x / tiles;
  const i64 r0 = (i64)(blockIdx.x - strip * tiles) * S.R;
  const int nr = (int)min((i64)S.R, P.n_rows - r0);
  // the lane's columns c, c + 1 and c + 64, c + 65; lanes past the last column repeat the first
  // one (their sums are dropped)
  const i64 c = (i64)strip * kCombCols + 2 * lane;
  const bool in[2] = {c < P.n_pos, c + 64 < P.n_pos}, second[2] = {c + 1 < P.n_pos, c + 65 < P.n_pos};
  const uint32_t row_bytes = (uint32_t)(P.ld * sizeof(i64)), up = in[1] ? 512u : 0u;
  const char *__restrict__ xb = reinterpret_cast<const char *>(P.x + (in[0] ? c : 0));
  uint32_t Ip[4] = {0, 0, 0, 0};
  if (P.diag.kind) {
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const i64 u = c + 64 * (i >> 1) + (i & 1);
      if (u < P.n_pos) Ip[i] = P.bits_pos[u];
    }
  }
  // the warp's rows are warp, warp + kWarps, ...: start, counts and words of the next one are
  // loaded while the current one is summed
  int32_t k0 = 0, k0n = 0;
  uint32_t cnt = 0, cntn = 0, w = 0;
  if (warp < nr) {
    k0 = S.rp[r0 + warp];
    cnt = S.cnt[r0 + warp];
    w = S.word[k0 + lane];                   // padded by 32 words
  }
  if (warp + kWarps < nr) {
    k0n = S.rp[r0 + warp + kWarps];
    cntn = S.cnt[r0 + warp + kWarps];
  }
  DotLong dots{{0, 0, 0, 0}};
  unsigned vmax = 0;
#pragma unroll 1
  for (int rr = warp; rr < nr; rr += kWarps) {
    Quad s;
    const i64 d = r0 + rr;
    uint32_t wn = 0, cnt2 = 0;
    int32_t k2 = 0;
    if (rr + kWarps < nr) wn = S.word[k0n + lane];
    if (rr + 2 * kWarps < nr) {
      k2 = S.rp[d + 2 * kWarps];
      cnt2 = S.cnt[d + 2 * kWarps];
    }
    comb_row(S, xb, row_bytes, up, lane, k0, cnt, w, s);
    if (P.t_neg) {
#pragma unroll
      for (int i = 0; i < 4; ++i) s.v[i] = -s.v[i];
    }
    k0 = k0n;
    cnt = cntn;
    w = wn;
    k0n = k2;
    cntn = cnt2;
    const uint32_t Ir = P.diag.kind ? P.bits_row[d] : 0u;
    Dot dot{0, 0};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      if (!in[h]) break;
      const i64 at = d * P.ld + c + 64 * h;
      const longlong2 xv = *reinterpret_cast<const longlong2 *>(P.x + at);
      int xh, xl;
      limbs28(xv.x, xh, xl);
      const i64 y0 = pass_entry<kLz>(P, utab, s.v[2 * h], xh, xl, Ir, Ip[2 * h], dot, vmax);
      i64 y1 = 0;
      if (second[h]) {
        limbs28(xv.y, xh, xl);
        y1 = pass_entry<kLz>(P, utab, s.v[2 * h + 1], xh, xl, Ir, Ip[2 * h + 1], dot, vmax);
      }
      *reinterpret_cast<longlong2 *>(P.out + at) = make_longlong2(y0, y1);
    }
    if (kLz) dots.take(dot);
  }
  if (kLz) pass_end(P, dots, vmax);
}

// ---------------------------------------------------------------------------------------
// Kernels that write both orders: tiles of 64 x 64 entries, rows read and written as 512-byte
// segments, the transposed copy through shared memory.  HBM-bound.
// ---------------------------------------------------------------------------------------

// T x T tile t of a transposed matrix (its rows c0 .., positions r0 ..) between memory and shared
// memory, which holds it as [row][position] of the untransposed one.  A thread has two entries of
// T / 2 T / 256 rows; an odd last position comes with the padding behind it.
template <int T>
struct TileBuf {
  i64 v[T][T + 1];
};
template <int T>
struct TileAt {                       // the thread's place: columns c, c + 1 of rows k0, k0 + kStep, ..
  static constexpr int kStep = 2 * kTileThreads / T;
  const int c = 2 * (int)(threadIdx.x % (T / 2)), k0 = (int)(threadIdx.x / (T / 2));
};
template <int T>
__device__ __forceinline__ void tile_in_t(TileBuf<T> &t, const i64 *__restrict__ m, i64 ldm, i64 r0, i64 c0, i64 n_r,
                                          i64 n_c) {
  const TileAt<T> at;
#pragma unroll
  for (int i = 0; i < T / TileAt<T>::kStep; ++i) {
    const int k = at.k0 + i * TileAt<T>::kStep;
    if (c0 + k < n_c && r0 + at.c < n_r) {
      const longlong2 v = *reinterpret_cast<const longlong2 *>(m + (c0 + k) * ldm + r0 + at.c);
      t.v[at.c][k] = v.x;
      t.v[at.c + 1][k] = v.y;
    }
  }
}
template <int T>
__device__ __forceinline__ void tile_out_t(const TileBuf<T> &t, i64 *__restrict__ m, i64 ldm, i64 r0, i64 c0, i64 n_r,
                                           i64 n_c) {
  const TileAt<T> at;
#pragma unroll
  for (int i = 0; i < T / TileAt<T>::kStep; ++i) {
    const int k = at.k0 + i * TileAt<T>::kStep;
    if (c0 + k < n_c && r0 + at.c < n_r)
      *reinterpret_cast<longlong2 *>(m + (c0 + k) * ldm + r0 + at.c) = make_longlong2(t.v[at.c][k], t.v[at.c + 1][k]);
  }
}
// Corner of a tile, rows of tiles in turn (numbered along strips of 24 tile columns, so that the tiles in
// work cover a square, the update took 1.60 ms instead of 1.44 at 4x4).
template <int T>
__device__ __forceinline__ void tile_at(uint32_t tile, i64 n_c, i64 *r0, i64 *c0) {
  const uint32_t tx = (uint32_t)((n_c + T - 1) / T), by = tile / tx;
  *c0 = (i64)(tile - by * tx) * T;
  *r0 = (i64)by * T;
}
template <int T>
__device__ __forceinline__ uint32_t tiles_of(i64 n_r, i64 n_c) {      // below 2^31 (fix_fits)
  return (uint32_t)(((n_c + T - 1) / T) * ((n_r + T - 1) / T));
}
__device__ __forceinline__ double2 ld_two(const double *p, bool vec, bool second) {
  if (vec) return *reinterpret_cast<const double2 *>(p);
  return make_double2(p[0], second ? p[1] : 0.0);
}

// X (stride ld) and XT (transposed, stride ldt), either may be null, from FP64 x (n_r x n_c) on the
// grid of ctl[kCtlShift].  acc != null: a Lanczos run's, scaled by ctl[kCtlScale]; also |X|^2 into the slots.
template <int T, bool kLimb, bool kTurns>
__global__ void __launch_bounds__(kTileThreads) k_fix_in(i64 n_r, i64 n_c, i64 ld, i64 ldt,
                                                         const double *__restrict__ x, const int *__restrict__ ctl,
                                                         int use_skip, int B, i64 *__restrict__ X,
                                                         i64 *__restrict__ XT, u64 *__restrict__ acc) {
  __shared__ TileBuf<T> t;
  if (use_skip) {
    after_previous();
    if (flag_of(ctl + kCtlSkip)) return;
  }
  const int e = ctl[kCtlShift] - (acc ? B - 1 : B - 2);
  const unsigned c = (unsigned)ctl[kCtlScale];
  const TileAt<T> at;
  const bool vec = (n_c & 1) == 0 && ((uintptr_t)x & 15) == 0;
  constexpr int kN = T / TileAt<T>::kStep;
  DotLong dots{{0, 0, 0, 0}};
  const uint32_t tiles = kTurns ? tiles_of<T>(n_r, n_c) : 0;
  uint32_t tile = blockIdx.x;
  do {
    i64 r0, c0;
    tile_at<T>(tile, n_c, &r0, &c0);
    const i64 u = c0 + at.c;
    const bool in = u < n_c, second = u + 1 < n_c;
    double2 xv[kN];
#pragma unroll
    for (int i = 0; i < kN; ++i) {
      const i64 d = r0 + at.k0 + i * TileAt<T>::kStep;
      xv[i] = make_double2(0.0, 0.0);
      if (d < n_r && in) xv[i] = ld_two(x + d * n_c + u, vec, second);
    }
    if (kTurns && XT && tile != blockIdx.x) __syncthreads();          // the tile before has been written out
    Dot dot{0, 0};
#pragma unroll
    for (int i = 0; i < kN; ++i) {
      const int k = at.k0 + i * TileAt<T>::kStep;
      i64 v[2];
      if (acc) {
        v[0] = f64_to_fix_scaled(xv[i].x, c, e);
        v[1] = f64_to_fix_scaled(xv[i].y, c, e);
      } else {
        v[0] = f64_to_fix(xv[i].x, e);
        v[1] = f64_to_fix(xv[i].y, e);
      }
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        if (acc) {
          int h, l;
          limbs28(v[j], h, l);
          dot.square(h, l);
        }
        v[j] = fix_store<kLimb>(v[j]);
        t.v[k][at.c + j] = v[j];
      }
      if (X && r0 + k < n_r && in) *reinterpret_cast<longlong2 *>(X + (r0 + k) * ld + u) = make_longlong2(v[0], v[1]);
    }
    if (XT) {
      __syncthreads();
      tile_out_t<T>(t, XT, ldt, r0, c0, n_r, n_c);
    }
    dots.take(dot);
    tile += gridDim.x;
  } while (kTurns && tile < tiles);
  if (acc) block_sums<4>(dots.v, 0u, 0, acc);
}

// Scalars of a Lanczos start: |S_1|^2 from k_fix_in's slots.
__global__ void k_fix_start(u64 *acc, int B, FixScal *q) {
  const double N = take_slots(acc).dot;
  if (threadIdx.x == 0) {
    q->N = N;
    q->overlap = 0.0;
    q->alpha = q->beta2 = 0.0;
    q->max_cur = ldexp(1.0, B);
    q->rescale = 0;
    q->max_prev = 0.0;
    q->ratio = 0.5;
    q->rel = q->sh = 0;
    q->step = q->hist_n = 0;
    q->ticket_dn = q->ticket_up = 0;
  }
}

__global__ void k_fix_rewind(FixScal *q) { q->hist_n = 0; }

// S_{j+1} over S_{j-1}, from the two contributions a (order of S) and b (kBt: the other order); kBt:
// S_{j+1} in the other order too, into ST (which may be b).  Adds |S_{j+1}|^2 and <S_{j+1}, S_j> and
// finds max |S_{j+1}|; the last block moves the scalars on.  Memory bounds it: 48 bytes per entry,
// 1.38 ms at 4x4 (5.8 TB/s; in double-float 1.35 ms for 40 bytes).  A CTA takes tiles in turn and
// adds up its sums once at the end (1.48 ms with a CTA per tile); more loads in flight per thread
// (unrolled by 2 to 8, with 64 or 80 registers) were slower, 1.48 to 1.56 ms.  psi != null: psi += v_j q_j first (v: the eigenvector of T;
// psi in the caller's order, rows and positions swapped if swap).
template <int T, bool kBt, bool kLimb, bool kPsi>
__global__ void __launch_bounds__(kTileThreads, kUpdateBlocks) k_fix_update(i64 n_r, i64 n_c, i64 ld, i64 ldt,
                                                             const i64 *__restrict__ a, const i64 *b,
                                                             const i64 *__restrict__ cur, i64 *__restrict__ prev,
                                                             i64 *ST, FixScal *__restrict__ q, u64 *__restrict__ acc,
                                                             const double *__restrict__ v, double *__restrict__ psi,
                                                             int swap, int B) {
  __shared__ TileBuf<T> t;
  int mah, mal, mbh, mbl;
  limbs28(q->ma, mah, mal);
  limbs28(q->mb, mbh, mbl);
  const int sy = q->sy, sa = q->sa, sb = q->sb;
  const bool plain_shifts = sy >= 0 && sy < 64 && sa >= 0 && sa <= 28 && sb >= 0 && sb <= 28;
  const double pc = kPsi ? v[q->step] / sqrt(q->N) : 0.0;
  DotLong dots{{0, 0, 0, 0}}, overs{{0, 0, 0, 0}};
  unsigned vmax = 0;
  const TileAt<T> at;
  const int c = at.c;
  const uint32_t tiles = tiles_of<T>(n_r, n_c);
  for (uint32_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    i64 r0, c0;
    tile_at<T>(tile, n_c, &r0, &c0);
    if (kBt) {
      if (tile != blockIdx.x) __syncthreads();            // the tile before has been written out
      tile_in_t<T>(t, b, ldt, r0, c0, n_r, n_c);
      __syncthreads();
    } else if (kPsi && swap && tile != blockIdx.x) {
      __syncthreads();
    }
    Dot dot{0, 0}, over{0, 0};
    const i64 u = c0 + c;
    const bool second = u + 1 < n_c;
#pragma unroll 1
    for (int k = at.k0, it = 0; k < T; k += TileAt<T>::kStep, ++it) {
      if (it == 4) dots.take_squares(dot);     // entries may reach 2^(B + kFixSpare): eight squares 2^63
      const i64 d = r0 + k;
      if (d >= n_r || u >= n_c) continue;
      const i64 o = d * ld + u;
      const longlong2 sc = *reinterpret_cast<const longlong2 *>(cur + o), sp = *reinterpret_cast<const longlong2 *>(prev + o);
      const longlong2 ya = *reinterpret_cast<const longlong2 *>(a + o);
      longlong2 yb;
      if (kBt)
        yb = make_longlong2(t.v[k][c], t.v[k][c + 1]);
      else
        yb = *reinterpret_cast<const longlong2 *>(b + o);
      const i64 y2[2] = {ya.x + yb.x, ya.y + yb.y};
      int ch[2], cl[2];
      fix_load<kLimb>(sc.x, ch[0], cl[0]);
      fix_load<kLimb>(sc.y, ch[1], cl[1]);
      i64 s[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        int ph, pl;
        fix_load<kLimb>(i ? sp.y : sp.x, ph, pl);
        // alpha S_j and beta^2 S_{j-1} from their limb products
        const i64 ah = (i64)ch[i] * mah, am = (i64)ch[i] * mal + (i64)cl[i] * mah + __mulhi(cl[i] << 2, mal << 2);
        const i64 bh = (i64)ph * mbh, bm = (i64)ph * mbl + (i64)pl * mbh + __mulhi(pl << 2, mbl << 2);
        i64 t3;
        if (plain_shifts)
          t3 = (y2[i] >> sy) - ((ah << sa) + (am >> (28 - sa))) - ((bh << sb) + (bm >> (28 - sb)));
        else
          t3 = shr_any(y2[i], sy) - (shr_any(ah, -sa) + shr_any(am, 28 - sa)) - (shr_any(bh, -sb) + shr_any(bm, 28 - sb));
        s[i] = (t3 + (1ll << (kFixFrac - 1))) >> kFixFrac;
      }
      if (!second) s[1] = 0;
      if (kPsi) {
        const i64 c2[2] = {limbs_value(ch[0], cl[0]), limbs_value(ch[1], cl[1])};
        if (!kBt && swap) {
          t.v[k][c] = c2[0];                    // written below, along the caller's rows
          t.v[k][c + 1] = c2[1];
        } else {
          psi[d * n_c + u] += pc * (double)c2[0];
          if (second) psi[d * n_c + u + 1] += pc * (double)c2[1];
        }
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        int h, l;
        limbs28(s[i], h, l);
        dot.square(h, l);
        over.add_high(h, l, ch[i], cl[i]);
        vmax = max(vmax, (unsigned)abs((int)(s[i] >> 32)));
        if (kLimb) s[i] = (i64)(((u64)(unsigned)h << 32) | (unsigned)l);
      }
      *reinterpret_cast<longlong2 *>(prev + o) = make_longlong2(s[0], s[1]);
      if (kBt) {
        t.v[k][c] = s[0];
        t.v[k][c + 1] = s[1];
      }
    }
    if (kBt) {
      __syncthreads();
      tile_out_t<T>(t, ST, ldt, r0, c0, n_r, n_c);
    } else if (kPsi && swap) {
      __syncthreads();
      const int r = (int)(threadIdx.x % T);
      for (int k = (int)(threadIdx.x / T); k < T; k += kTileThreads / T)
        if (c0 + k < n_c && r0 + r < n_r) psi[(c0 + k) * n_r + r0 + r] += pc * (double)t.v[r][k];
    }
    dots.take_squares(dot);
    overs.take(over);
  }
  i64 sums8[8];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    sums8[i] = dots.v[i];
    sums8[i + 4] = overs.v[i];
  }
  block_sums<8>(sums8, vmax, 0, acc);
  if (!last_block(&q->ticket_up) || threadIdx.x >= 32) return;
  const SlotSums sums = take_slots(acc);
  if (threadIdx.x == 0) {
    // bits to take off: entries below 2^B (1 - 2^-15), so that the top limbs of eight add up below 2^31
    int r = 0;
    while (r < kFixSpare && sums.max0 > ldexp(1.0 - 0x1p-15, B + r)) ++r;
    const double N = ldexp(sums.dot, -2 * r), b2 = ldexp(N / q->N, 2 * (q->sh + r));
    const int i = q->hist_n;
    if (i < kFixHist) {
      q->hist[3 * i] = q->alpha;
      q->hist[3 * i + 1] = sqrt(b2);
      q->hist[3 * i + 2] = q->N;
    }
    q->hist_n = i + 1;
    q->step += 1;
    q->N = N;
    q->beta2 = b2;
    q->rel = -(q->sh + r);
    q->max_prev = q->max_cur;
    q->max_cur = ldexp(sums.max0, -r) + 1.0;
    q->overlap = ldexp(sums.dot2, -r);
    q->rescale = r;
    q->ratio = sums.max0 / q->bound;
  }
}

// S_{j+1} (and its other order) 2^-rescale, rounded: nothing to do as a rule, so the grid is small (a
// 12-site ring step 44.3 us with 4 CTAs per SM, 45.1 with 16)
template <bool kLimb>
__global__ void __launch_bounds__(256) k_fix_rescale(const FixScal *__restrict__ q, i64 n, i64 *__restrict__ S, i64 nt,
                                                     i64 *__restrict__ ST) {
  const int r = q->rescale;
  if (r == 0) return;
  for (i64 k = blockIdx.x * (i64)blockDim.x + threadIdx.x; k < n + nt; k += (i64)gridDim.x * blockDim.x) {
    i64 *p = k < n ? S + k : ST + (k - n);
    int h, l;
    fix_load<kLimb>(*p, h, l);
    *p = fix_store<kLimb>((limbs_value(h, l) + (1ll << (r - 1))) >> r);
  }
}

// y (n_r x n_c, caller's order) = tabs 2^.. (a + b), a and b each in that order or (kAt, kBt) the other
// one.  An entry whose contributions' magnitudes -- a lower bound of (|H||x|)_n -- do
// not reach thr is recorded in list (see k_fix_entries).  Memory bounds it (24 bytes per entry, 0.59 ms
// at 4x4): 0.69 ms with four CTAs per SM and loads as they are needed, 0.85 ms with a tile's loads in
// registers first (116 of them, two CTAs); unrolled by 2 or 4, or five CTAs, 0 to 0.09 ms slower.
template <int T, bool kAt, bool kBt, bool kTurns>
__global__ void __launch_bounds__(kTileThreads, kUpdateBlocks) k_fix_out(i64 n_r, i64 n_c, i64 ld, i64 ldt,
                                                                         const i64 *__restrict__ a, const i64 *__restrict__ b, int eg, i64 thr, double tabs,
                                                          int *__restrict__ ctl, i64 *__restrict__ list, int cap,
                                                          double *__restrict__ y) {
  static_assert(T == 32 || !(kAt && kBt), "two tiles in 48 KB");
  __shared__ TileBuf<T> t;
  __shared__ TileBuf<kAt && kBt ? T : 2> t2;
  after_previous();
  if (flag_of(ctl + kCtlSkip)) return;
  const int e = ctl[kCtlShift] + eg;
  const TileAt<T> at;
  const bool vec = (n_c & 1) == 0 && ((uintptr_t)y & 15) == 0;
  const uint32_t tiles = kTurns ? tiles_of<T>(n_r, n_c) : 0;
  uint32_t tile = blockIdx.x;
  do {
    i64 r0, c0;
    tile_at<T>(tile, n_c, &r0, &c0);
    const i64 u = c0 + at.c;
    const bool second = u + 1 < n_c;
    if (kTurns && (kAt || kBt) && tile != blockIdx.x) __syncthreads();          // the tile before has been read
    if (kBt) tile_in_t<T>(t, b, ldt, r0, c0, n_r, n_c);
    if constexpr (kAt && kBt)
      tile_in_t<T>(t2, a, ldt, r0, c0, n_r, n_c);
    else if (kAt)
      tile_in_t<T>(t, a, ldt, r0, c0, n_r, n_c);
    if (kAt || kBt) __syncthreads();
#pragma unroll 1
    for (int k = at.k0; k < T; k += TileAt<T>::kStep) {
      const i64 d = r0 + k;
      if (d >= n_r || u >= n_c) continue;
      longlong2 va;
      if constexpr (kAt && kBt)
        va = make_longlong2(t2.v[k][at.c], t2.v[k][at.c + 1]);
      else
        va = kAt ? make_longlong2(t.v[k][at.c], t.v[k][at.c + 1]) : *reinterpret_cast<const longlong2 *>(a + d * ld + u);
      const longlong2 vb = kBt ? make_longlong2(t.v[k][at.c], t.v[k][at.c + 1])
                               : *reinterpret_cast<const longlong2 *>(b + d * ld + u);
      const i64 n = d * n_c + u;
      const i64 s0[2] = {va.x, va.y}, s1[2] = {vb.x, vb.y};
      double v[2];
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        v[j] = fix_to_f64(s0[j] + s1[j], e);
        if (tabs != 1.0) v[j] *= tabs;
        if ((j == 0 || second) && llabs(s0[j]) + llabs(s1[j]) < thr) {
          const u64 at_list = atomicAdd(count_of(ctl), 1ull);
          if (at_list < (u64)cap) list[at_list] = n + j;
        }
      }
      if (vec) {
        *reinterpret_cast<double2 *>(y + n) = make_double2(v[0], v[1]);
      } else {
        y[n] = v[0];
        if (second) y[n + 1] = v[1];
      }
    }
    tile += gridDim.x;
  } while (kTurns && tile < tiles);
}

// psi += v_j q_j alone (the last vector)
template <bool kLimb>
__global__ void k_fix_axpy(i64 n_r, i64 n_c, i64 ld, const i64 *__restrict__ cur, const FixScal *__restrict__ q,
                           const double *__restrict__ v, double *__restrict__ psi, int swap) {
  const double pc = v[q->step] / sqrt(q->N);
  const i64 D = n_r * n_c;
  for (i64 k = blockIdx.x * (i64)blockDim.x + threadIdx.x; k < D; k += (i64)gridDim.x * blockDim.x) {
    const i64 d = k / n_c, u = k - d * n_c;
    int hi, lo;
    fix_load<kLimb>(cur[d * ld + u], hi, lo);
    psi[swap ? u * n_r + d : k] += pc * (double)limbs_value(hi, lo);
  }
}

// The recorded entries in FP64, one warp each: hops gathered by the lanes.  More entries than
// the list holds: the whole vector goes to the double-float (or FP64) kernels.
__global__ void __launch_bounds__(256) k_fix_entries(const Ham H, const double *__restrict__ x, double *__restrict__ y,
                                                     int *__restrict__ ctl, const i64 *__restrict__ list, int cap,
                                                     int df_ok) {
  after_previous();
  if (flag_of(ctl + kCtlSkip)) return;
  const u64 all = *count_of(ctl);
  const int n = (int)min(all, (u64)cap);
  if (all > (u64)cap) {
    if (blockIdx.x == 0 && threadIdx.x == 0) ctl[df_ok ? kCtlDf : kCtlF64] = 1;
    return;
  }
  const int lane = threadIdx.x & 31;
  const int w0 = (int)((blockIdx.x * blockDim.x + threadIdx.x) >> 5), nw = (int)((gridDim.x * blockDim.x) >> 5);
  for (int k = w0; k < n; k += nw) {
    const i64 at = list[k], d = at / H.n_up, u = at - d * H.n_up;
    double v = lane == 0 ? diag_of(H, H.basis_up[u], H.basis_dn[d], u, d) * x[at] : 0.0;
    for (int32_t j = H.rp_up[u] + lane; j < H.rp_up[u + 1]; j += 32) v = fma(H.val_up[j], x[d * H.n_up + H.col_up[j]], v);
    for (int32_t j = H.rp_dn[d] + lane; j < H.rp_dn[d + 1]; j += 32)
      v = fma(H.val_dn[j], x[(i64)H.col_dn[j] * H.n_up + u], v);
    for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) y[at] = v;
  }
}

// Entry lists of a spin (see CombLists) from its CSR matrix.
__global__ void k_fix_lists(i64 n, const int32_t *__restrict__ rp, const uint32_t *__restrict__ scol,
                            uint32_t *__restrict__ cnt, uint32_t *__restrict__ word) {
  for (i64 r = blockIdx.x * (i64)blockDim.x + threadIdx.x; r < n; r += (i64)gridDim.x * blockDim.x) {
    const int32_t a = rp[r], b = rp[r + 1];
    int na = 0;
    for (int32_t k = a; k < b; ++k) na += (int)(scol[k] >> 31);
    const int ns = b - a - na, pa = na & ~1, pe = pa + (ns & ~1);
    int ia = 0, is = 0;
    for (int32_t k = a; k < b; ++k) {
      const bool add = (scol[k] >> 31) != 0;
      int at;
      if (add) {
        at = ia < pa ? ia : pe;
        ++ia;
      } else {
        at = is < (ns & ~1) ? pa + is : pe + (na & 1);
        ++is;
      }
      word[a + at] = scol[k] & 0x7fffffffu;
    }
    cnt[r] = (uint32_t)na | ((uint32_t)ns << 16);
  }
}

// ---------------------------------------------------------------------------------------
// Host side.
// ---------------------------------------------------------------------------------------
struct FixState {
  bool lists_ready = false;           // entry lists of the spins: gather schedule or row combinations
  uint32_t *cnt[2] = {nullptr, nullptr}, *word[2] = {nullptr, nullptr};
  uint16_t *sched[2] = {nullptr, nullptr};
  uint32_t *meta[2] = {nullptr, nullptr};
  int cap_steps[2] = {0, 0}, slices[2] = {0, 0};
  int *ctl = nullptr;
  FixRange *range = nullptr;          // in ctl's allocation
  i64 *list = nullptr;
  int cap = 0;
  u64 *acc = nullptr;
  FixScal *scal = nullptr, *h_scal = nullptr;
  i64 *vec[2] = {nullptr, nullptr};   // S_j, S_{j-1}
  double *v = nullptr;                // eigenvector of T
  int v_cap = 0;
  cudaStream_t gs = nullptr;
  cudaGraphExec_t graph[2] = {nullptr, nullptr};
  std::vector<unsigned char> graph_key;
  bool graph_failed = false;
};

void fix_release(hub_ctx *h) {
  FixState *f = h->fix;
  if (!f) return;
  for (int s = 0; s < 2; ++s) {
    dev_free(f->cnt[s]);
    dev_free(f->word[s]);
    dev_free(f->sched[s]);              // meta lies in the same allocation
    dev_free(f->vec[s]);
    if (f->graph[s]) cudaGraphExecDestroy(f->graph[s]);
  }
  if (h->route == HUB_ROUTE_FIX) set_route(h, HUB_ROUTE_NONE);    // its flags go
  dev_free(f->ctl);
  dev_free(f->list);
  dev_free(f->acc);
  dev_free(f->scal);
  if (f->h_scal) cudaFreeHost(f->h_scal);
  dev_free(f->v);
  if (f->gs) cudaStreamDestroy(f->gs);
  delete f;
  h->fix = nullptr;
}

static int ceil_log2(double v) {      // smallest n with v <= 2^n (v > 0)
  int n = 0;
  const double m = std::frexp(v, &n);
  return m == 0.5 ? n - 1 : n;
}

// What the fixed-point path needs to know about the model; ok == false: not for this path.
struct FixPlan {
  bool ok = false;
  bool gather[2] = {false, false};    // the spin's hops as gathers inside staged rows
  double tau = 1.0, units = 0.0;      // |t|; worst-case error of an entry in units of 2^e
  int hh = 0, B = 0, q = 0, g = 0, dh = 0;
  int kind = 0;
  bool limbs() const { return gather[0] && gather[1]; }   // the vectors' storage
};

static FixPlan fix_plan(const hub_ctx *h) {
  FixPlan p;
  if (h->mode != HUB_MODE_AUTO || h->k0 || !h->have_hop || !h->have_U || !h->fast) return p;
  if (h->count[0] <= 0 || h->count[1] <= 0) return p;
  // t uniform, U uniform, no site energies (the other models keep the 53-bit entries of the FP64
  // kernels, which the grid does not quite reach)
  if (!h->uniform_U || h->has_eps || h->t.empty()) return p;
  for (double t : h->t)
    if (t != h->t[0]) return p;
  p.tau = std::fabs(h->t[0]);
  if (!(p.tau >= 0x1p-500 && p.tau <= 0x1p500)) return p;
  const int rows = h->csr[0].max_row + h->csr[h->shared ? 0 : 1].max_row;
  for (int s = 0; s < 2; ++s)
    p.gather[s] = h->count[s] <= kStageMax && h->csr[h->shared ? 0 : s].max_row <= kSchedRow;
  p.hh = ceil_log2(std::max(rows, 1));
  p.B = std::min(kFixMaxBits, 62 - p.hh);
  p.q = 62 - p.B;
  const double r = h->U0 / p.tau, dmax = std::fabs(r) * std::min(h->N[0], h->N[1]);
  if (!std::isfinite(dmax) || dmax > 0x1p24) return p;
  if (dmax > 0.0) {
    p.kind = r == std::floor(r) && dmax <= std::ldexp(1.0, p.q) ? 1 : 2;
    p.dh = std::max(ceil_log2(dmax), -40);
    // |Y| <= 2^(B - g) (rows + dmax) < 2^63; the general diagonal's high product must not be
    // shifted left
    p.g = std::max(0, ceil_log2(1.07 * (std::max(rows, 1) + dmax)) + p.B - 63);
    if (p.kind == 2) p.g = std::max(p.g, p.dh + 2 - p.q);
  }
  // rounding of the entries (1/2 each), of the shift to Y's grid and of the diagonal's product (2^g
  // each at most)
  p.units = 0.5 * (rows + dmax) + (p.g || p.kind == 2 ? std::ldexp(2.0, p.g) : 0.0) + 1.0;
  p.ok = true;
  return p;
}

static FixState *fix_state(hub_ctx *h) {
  if (!h->fix) h->fix = new (std::nothrow) FixState();
  return h->fix;
}

// Row stride in entries: rows start on 32-byte sectors.
static i64 fix_ld(i64 n) { return (n + 3) & ~(i64)3; }
static int grid_of(i64 n) { return (int)std::max<i64>(1, std::min<i64>((n + 255) / 256, (i64)num_sms() * 16)); }

// Arrays of a spin's gather schedule and of what it is made from, in one allocation (a first product
// pays for each).
static int gather_arrays(FixState *f, int s, int n, int seg, const SpinCSR &c, SchedSpin *S) {
  const int slices = (n + 31) / 32, groups = 2 * slices;
  const int cap = std::min(kSchedMax, (2 * std::max(c.max_row, 1) + 7) / 8 * 8);
  size_t at = 0;
  auto take = [&](size_t bytes) {
    const size_t o = at;
    at += (bytes + 255) / 256 * 256;
    return o;
  };
  const size_t o_word = take(sizeof(uint16_t) * 32 * (size_t)slices * cap);
  const size_t o_meta = take(sizeof(uint32_t) * 32 * (size_t)slices);
  const size_t o_load = take(sizeof(uint32_t) * 8 * 4 * groups), o_len = take(4 * (size_t)groups);
  const size_t o_sorted = take(sizeof(uint16_t) * 4 * groups), o_greedy = take(sizeof(uint16_t) * 4 * groups);
  const size_t o_quad = take(sizeof(uint16_t) * 4 * groups), o_steps = take(2 * (size_t)groups);
  const size_t o_deg = take((size_t)groups), o_total = take(2 * sizeof(uint32_t));
  if (!f->sched[s] && !dev_alloc((void **)&f->sched[s], at, "gather schedule")) return HUB_ERR_OOM;
  char *base = (char *)f->sched[s];
  f->meta[s] = (uint32_t *)(base + o_meta);
  f->cap_steps[s] = cap;
  f->slices[s] = slices;
  *S = SchedSpin{n, groups, (int)fix_ld(n), cap, seg, c.rowptr, c.scol, (uint32_t *)(base + o_load),
                 (uint32_t *)(base + o_len), (uint16_t *)(base + o_sorted), (uint16_t *)(base + o_greedy),
                 (uint8_t *)(base + o_steps), (uint32_t *)(base + o_total), (uint16_t *)(base + o_quad),
                 (uint8_t *)(base + o_deg), f->sched[s], f->meta[s]};
  return HUB_OK;
}

// Tables of the plan, entry lists of the spins: enqueued on the legacy stream, to be waited for
// (fix_tables_wait) before the first launch that reads them.
static int fix_tables(hub_ctx *h, FixState *f, const FixPlan &p) {
  if (f->lists_ready) return HUB_OK;
  SchedArgs A{};
  int gathers = 0, groups = 0, segs = 0;
  for (int s = 0; s < (h->shared ? 1 : 2); ++s) {
    const SpinCSR &c = h->csr[s];
    const i64 nnz = c.nnz, n = h->count[s];
    if (p.gather[s]) {
      const int rc = gather_arrays(f, s, (int)n, seg_quads((double)h->count[0] * (double)h->count[1]), c, &A.spin[gathers]);
      if (rc) return rc;
      const SchedSpin &S = A.spin[gathers++];
      groups = std::max(groups, S.groups);
      segs = std::max(segs, (4 * S.groups + S.seg - 1) / S.seg);
      continue;
    }
    if ((!f->cnt[s] && !dev_alloc((void **)&f->cnt[s], sizeof(uint32_t) * n, "hopping entry counts")) ||
        (!f->word[s] && !dev_alloc((void **)&f->word[s], sizeof(uint32_t) * (nnz + 32), "hopping entries")))
      return HUB_ERR_OOM;
    HUB_CUDA(cudaMemsetAsync(f->word[s], 0, sizeof(uint32_t) * (nnz + 32), nullptr));
    k_fix_lists<<<grid_of(n), 256>>>(n, c.rowptr, c.scol, f->cnt[s], f->word[s]);
    HUB_LAUNCH_CHECK();
  }
  if (!gathers) return HUB_OK;
  k_fix_quads<<<dim3((4 * groups + 15) / 16, gathers), 256>>>(A);
  k_fix_sort<<<dim3((4 * groups + 255) / 256, gathers), 256>>>(A);
  k_fix_group<<<dim3(segs, gathers), 32>>>(A);
  k_fix_order<<<dim3(1, gathers), 1024>>>(A);
  k_fix_schedule<<<dim3(groups, gathers), 32>>>(A);
  HUB_LAUNCH_CHECK();
  return HUB_OK;
}
static int fix_tables_wait(FixState *f) {
  if (!f->lists_ready) HUB_CUDA(cudaStreamSynchronize(nullptr));
  f->lists_ready = true;
  return HUB_OK;
}

// A pass over the order of the vector whose rows are spin a's states.
static FixPass fix_pass(const hub_ctx *h, const FixState *f, const FixPlan &p, int a, bool diag) {
  const int b = 1 - a;
  FixPass P{};
  P.n_rows = h->count[a];
  P.n_pos = h->count[b];
  P.ld = fix_ld(P.n_pos);
  P.bits_row = h->basis[a];
  P.bits_pos = h->basis[b];
  P.q = p.q;
  P.g = p.g;
  P.t_neg = h->t[0] < 0.0;
  P.err = fast_err(h);
  P.fail_waits = h->fail_waits ? 1 : 0;
  if (!diag) return P;
  FixDiag &d = P.diag;
  d.kind = p.kind;
  if (p.kind == 1) {
    d.mul = (int)(h->U0 / p.tau);
    d.shift = p.g;
  }
  if (p.kind == 2) {
    d.shift = p.q - 2 - p.dh + p.g;
    for (int k = 0; k <= std::min(h->N[0], h->N[1]); ++k)
      d.tab[k] = (i64)std::llrint(std::ldexp(h->U0 * k / p.tau, 62 - p.dh));
  }
  return P;
}

// Rows of a combination tile, fewer where the grid would leave SMs idle (two CTAs each).
static int tile_rows(i64 n_rows, i64 n_cols) {
  const i64 strips = (n_cols + kCombCols - 1) / kCombCols;
  const i64 want = n_rows * strips / (2 * num_sms());
  return (int)std::min<i64>(kCombRows, std::max<i64>(1, want / 8) * 8);
}
static i64 comb_blocks(i64 n_rows, i64 n_cols) {
  const int R = tile_rows(n_rows, n_cols);
  return ((n_rows + R - 1) / R) * ((n_cols + kCombCols - 1) / kCombCols);
}
// Tiles of 64 x 64 entries, or 32 x 32 where the larger ones would leave SMs idle.
static bool small_tiles(const hub_ctx *h) { return h->count[0] * h->count[1] < (i64)64 * 64 * 8 * num_sms(); }
static i64 tile_blocks(const hub_ctx *h, i64 T) {
  return ((h->count[0] + T - 1) / T) * ((h->count[1] + T - 1) / T);
}
static i64 tile_blocks(const hub_ctx *h) { return tile_blocks(h, small_tiles(h) ? 32 : 64); }
// k_fix_in and k_fix_out: a CTA per tile, or (kTurns) as many as are resident, which take tiles in turn.  The
// first costs 8 us where the kernel finds nothing to do (2916 tiles) and 17 us with 7600; the second is
// slower where there is (4x4 half filling: 0.67 and 0.77 ms against 0.60 and 0.69; k_fix_out at 2916 tiles of
// 64 x 64 60 us against 54, k_fix_in 46 either way).
constexpr i64 kTurnTiles = 8192;
static bool in_turns(const hub_ctx *h) { return tile_blocks(h) <= kTurnTiles; }
static int in_blocks(const hub_ctx *h) {
  const i64 tiles = tile_blocks(h);
  return (int)(in_turns(h) ? std::min<i64>(tiles, (i64)(small_tiles(h) ? 8 : 3) * num_sms()) : tiles);
}
template <bool kTurns>
static auto in_kernel(const hub_ctx *h, bool limbs) {
  return limbs ? (small_tiles(h) ? k_fix_in<32, true, kTurns> : k_fix_in<64, true, kTurns>)
               : (small_tiles(h) ? k_fix_in<32, false, kTurns> : k_fix_in<64, false, kTurns>);
}
static auto in_kernel(const hub_ctx *h, bool limbs) { return in_turns(h) ? in_kernel<true>(h, limbs) : in_kernel<false>(h, limbs); }

// grids are one-dimensional, row strides in bytes 32-bit
static bool fix_fits(const hub_ctx *h) {
  const i64 lim = ((i64)1 << 31) - 1;
  for (int s = 0; s < 2; ++s)
    if (comb_blocks(h->count[s], h->count[1 - s]) > lim || fix_ld(h->count[s]) * 8 > (i64)0xffffffff) return false;
  return tile_blocks(h, 32) <= lim;
}

// out = the hops of the rows' (comb) or the positions' spin (gather) applied to P.x
static int launch_comb(const hub_ctx *h, const FixState *f, const FixPass &P, int a, cudaStream_t s) {
  const int t = h->shared ? 0 : a;
  CombLists L{tile_rows(P.n_rows, P.n_pos), h->csr[t].rowptr, f->cnt[t], f->word[t]};
  const int g = (int)comb_blocks(P.n_rows, P.n_pos);
  HUB_CUDA(launch_kernel(P.chained, P.acc ? k_fix_comb<true> : k_fix_comb<false>, g, kCombThreads, 0, s, P, L));
  return HUB_OK;
}
template <int kPlane, bool kLimb>
static int launch_gather_t(const FixPass &P, const GatherLists &L, cudaStream_t s) {
  static_assert(kPlane % 16 == 0, "both rows in the same banks");
  const size_t smem = 2 * sizeof(i64) * (size_t)kPlane;
  const int threads = kPlane > 2048 ? 1024 : (P.n_pos >= 256 ? 256 : 128);
  const i64 per_sm = std::max<i64>(1, std::min<i64>((i64)(220 * 1024 / smem), 1024 / threads));
  const int grid = (int)std::min<i64>((P.n_rows + 1) / 2, per_sm * num_sms());
  const auto k = P.acc ? k_fix_gather<kPlane, true, kLimb> : k_fix_gather<kPlane, false, kLimb>;
  HUB_CUDA(cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
  HUB_CUDA(launch_kernel(P.chained, k, grid, threads, smem, s, P, L));
  return HUB_OK;
}
template <int kPlane>
static int launch_gather_p(const FixPlan &p, const FixPass &P, const GatherLists &L, cudaStream_t s) {
  return p.limbs() ? launch_gather_t<kPlane, true>(P, L, s) : launch_gather_t<kPlane, false>(P, L, s);
}
static int launch_gather(const hub_ctx *h, const FixState *f, const FixPlan &p, const FixPass &P, int b, cudaStream_t s) {
  const int t = h->shared ? 0 : b;
  const GatherLists L{(const uint4 *)f->sched[t], f->meta[t], f->cap_steps[t] / 8, f->slices[t]};
  return P.ld + 16 <= 2048 ? launch_gather_p<2048>(p, P, L, s) : launch_gather_p<kStageMax + 16>(p, P, L, s);
}

// How the two spins' hops are run.  `a` is the spin whose states are the rows of the order the
// Lanczos vectors are kept in.
//   both as gathers: the positions' spin on that order, the rows' spin on the other one;
//   both as combinations: the rows' spin on that order, the positions' spin on the other one;
//   one of each: the gathered spin are the positions, both on that order, the other is not kept.
struct FixShape {
  int a = 1;                          // rows: spin down (the caller's order) unless only it gathers
  bool both = true;                   // two orders of the vector
};
static FixShape fix_shape(const FixPlan &p) {
  FixShape F;
  if (p.gather[0] != p.gather[1]) {
    F.both = false;
    F.a = p.gather[0] ? 1 : 0;
  }
  return F;
}

// The two contributions to the product of S (order of rows a; ST: the other order): out0 in the
// order of a, out1 in the other one if F.both, else in the same.  Where a pass gathers, its output
// may be its input.  lz: Lanczos sums into f->acc.
static int fix_product(hub_ctx *h, FixState *f, const FixPlan &p, const FixShape &F, const i64 *S, const i64 *ST,
                       i64 *out0, i64 *out1, const int *skip, bool lz, cudaStream_t s) {
  int rc;
  count_launch(h, 2);
  FixPass P0 = fix_pass(h, f, p, F.a, true), P1 = fix_pass(h, f, p, F.both ? 1 - F.a : F.a, false);
  P0.x = S;
  P0.out = out0;
  P1.x = F.both ? ST : S;
  P1.out = out1;
  P0.skip = P1.skip = skip;
  P0.chained = P1.chained = skip && !h->prof ? 1 : 0;
  if (lz) {
    P0.acc = P1.acc = f->acc;
    P0.scal = P1.scal = f->scal;
  }
  // one of each: the combination first, so that the gather may work in place
  const bool swap = !F.both;
  (swap ? P0 : P1).second = 1;
  for (int k = 0; k < 2; ++k) {
    const bool first = (k == 0) != swap;      // P0's turn
    const FixPass &P = first ? P0 : P1;
    // P0 runs the positions' spin where spins gather (and the rows' spin where both combine)
    const int rows = first || !F.both ? F.a : 1 - F.a;
    const bool gather = F.both ? p.gather[0] : first;
    const int kind = k == 0 ? HUB_PROF_UP : HUB_PROF_DN;
    if ((rc = prof_mark(h, kind, true, s))) return rc;
    if ((rc = gather ? launch_gather(h, f, p, P, 1 - rows, s) : launch_comb(h, f, P, rows, s))) return rc;
    if ((rc = prof_mark(h, kind, false, s))) return rc;
  }
  return HUB_OK;
}

// Scale and route words of x
static int plan_vector(hub_ctx *h, FixState *f, const double *x, i64 D, int df_ok, cudaStream_t s) {
  const int nblk = 4 * num_sms();
  if (!f->ctl) {
    const size_t words = 256;           // bytes, for the words and the padding behind them
    if (!dev_alloc((void **)&f->ctl, words + sizeof(FixRange) + 2 * sizeof(int) * nblk, "product flags")) return HUB_ERR_OOM;
    f->range = (FixRange *)((char *)f->ctl + words);
    HUB_CUDA(cudaMemsetAsync(f->range, 0, sizeof(unsigned), s));
  }
  count_launch(h);
  k_fix_plan<<<nblk, kPlanThreads, 0, s>>>(D, x, df_ok, f->range, f->ctl);
  HUB_LAUNCH_CHECK();
  return HUB_OK;
}

// Vectors of the handle's scratch a product needs: S, ST and, for combinations, their outputs.
static int scratch_vectors(const FixPlan &p, const FixShape &F) { return F.both && !p.gather[0] ? 4 : 2; }

// hub_apply in fixed point, the other kernels launched behind it on device flags.
bool fix_apply_eligible(const hub_ctx *h) {
  if (h->fail_waits) return false;    // the test hook exercises the double-float kernels' waits
  const FixPlan p = fix_plan(h);
  // an entry's worst-case error has to lie well inside the bound for vectors of ordinary shape
  return p.ok && p.units <= 128.0 && fix_fits(h);
}

int fix_apply(hub_ctx *h, const double *x, double *y, cudaStream_t s) {
  const FixPlan p = fix_plan(h);
  const FixShape F = fix_shape(p);
  FixState *f = fix_state(h);
  if (!f) return fail(HUB_ERR_OOM, "fixed-point apply: host allocation failed");
  int rc = fix_tables(h, f, p);
  if (rc) return rc;
  const i64 n_up = h->count[0], n_dn = h->count[1], D = n_up * n_dn;
  float *buf[4] = {nullptr, nullptr, nullptr, nullptr};
  if ((rc = fast_scratch(h, scratch_vectors(p, F), buf))) return rc;
  if (!f->list) {
    f->cap = (int)std::min<i64>(std::max<i64>(D / 64, 1024), (i64)1 << 24);
    if (!dev_alloc((void **)&f->list, sizeof(i64) * f->cap, "entries to recompute")) return HUB_ERR_OOM;
  }
  if ((rc = fix_tables_wait(f))) return rc;
  const int df_ok = use_fast(h) ? 1 : 0;
  if ((rc = plan_vector(h, f, x, D, df_ok, s))) return rc;
  set_route(h, HUB_ROUTE_FIX, f->ctl + kCtlF64, f->ctl + kCtlDf);
  // X: rows spin down (the caller's order); XT: rows spin up
  const bool cx = F.both || F.a == 1, ct = F.both || F.a == 0;
  i64 *X = (i64 *)buf[0], *XT = (i64 *)buf[1];
  const i64 ld = fix_ld(n_up), ldt = fix_ld(n_dn);
  const int *skip = f->ctl + kCtlSkip;
  count_launch(h, 3);
  const bool st = small_tiles(h);
  const bool chained = !h->prof;
  HUB_CUDA(launch_kernel(chained, in_kernel(h, p.limbs()), in_blocks(h), kTileThreads, 0, s, n_dn, n_up, ld, ldt, x,
                         f->ctl, 1, p.B, cx ? X : nullptr, ct ? XT : nullptr, nullptr));
  i64 *in0 = F.a == 1 ? X : XT, *in1 = F.a == 1 ? XT : X, *out0 = in0, *out1 = in1;   // gathers: in place
  if (F.both && !p.gather[0]) {
    out0 = (i64 *)buf[2];
    out1 = (i64 *)buf[3];
  }
  if ((rc = fix_product(h, f, p, F, in0, in1, out0, out1, skip, false, s))) return rc;
  const i64 thr = ((i64)std::ceil(p.units * 1.25e13) >> p.g) + 1;   // |error| <= units 2^e <= 0.8e-13 thr 2^(e + g)
  const int eg = p.g - (p.B - 2);
#define FIX_OUT(T, AT, BT, TURNS)                                                                                \
  HUB_CUDA(launch_kernel(chained, k_fix_out<T, AT, BT, TURNS>,                                                  \
                         (int)(TURNS ? std::min<i64>(tile_blocks(h, T), (i64)kUpdateBlocks * num_sms()) : tile_blocks(h, T)), \
                         kTileThreads, 0, s, n_dn, n_up, ld, ldt, out0, out1, eg, thr, p.tau, f->ctl, f->list, f->cap, y))
  const bool turns = tile_blocks(h, 32) <= kTurnTiles;
  if (F.both && st && turns)
    FIX_OUT(32, false, true, true);
  else if (F.both && st)
    FIX_OUT(32, false, true, false);
  else if (F.both)
    FIX_OUT(64, false, true, false);
  else if (F.a == 1)
    FIX_OUT(64, false, false, false);
  else if (turns)
    FIX_OUT(32, true, true, true);
  else
    FIX_OUT(32, true, true, false);
#undef FIX_OUT
  HUB_CUDA(launch_kernel(chained, k_fix_entries, num_sms() * 4, 256, 0, s, h->view(), x, y, f->ctl, f->list, f->cap,
                         df_ok));
  if (df_ok && (rc = fast_apply_gated(h, x, y, f->ctl + kCtlDfScale, f->ctl + kCtlDf, s))) return rc;
  return f64_apply(h, x, y, f->ctl + kCtlF64, s);
}

// ---------------------------------------------------------------------------------------
// Lanczos driver: three kernels per step, replayed as a graph (one per rotation of the two
// vectors), the scalars of the recurrence kept on the device.
// ---------------------------------------------------------------------------------------
bool fix_lanczos_eligible(const hub_ctx *h) { return fix_plan(h).ok && fix_fits(h); }

int fix_lanczos(hub_ctx *h, const double *x0, int maxit, double tol, double *E0, double *psi_out, int *iters,
                cudaStream_t s) {
  const FixPlan p = fix_plan(h);
  FixState *f = fix_state(h);
  if (!f) return fail(HUB_ERR_OOM, "fixed-point Lanczos: host allocation failed");
  int rc = fix_tables(h, f, p);
  if (rc) return rc;
  const FixShape F = fix_shape(p);
  const i64 n_up = h->count[0], n_dn = h->count[1], D = n_up * n_dn;
  const i64 n_r = h->count[F.a], n_c = h->count[1 - F.a], ld = fix_ld(n_c), ldt = fix_ld(n_r);
  // out0; the other order (its gather works in place) or out1; out1 of combinations in both orders
  const bool third = F.both && !p.gather[0];
  float *buf[4] = {nullptr, nullptr, nullptr, nullptr};
  if ((rc = fast_scratch(h, third ? 3 : 2, buf))) return rc;
  i64 *const out0 = (i64 *)buf[0], *const ST = (i64 *)buf[1], *const out1 = third ? (i64 *)buf[2] : ST;
  for (int k = 0; k < 2; ++k)
    if (!f->vec[k] && !dev_alloc((void **)&f->vec[k], sizeof(i64) * n_r * ld, "Lanczos vector")) return HUB_ERR_OOM;
  if ((!f->acc && !dev_alloc((void **)&f->acc, sizeof(u64) * kFixSlots * kAcc, "Lanczos sums")) ||
      (!f->scal && !dev_alloc((void **)&f->scal, sizeof(FixScal), "Lanczos scalars")))
    return HUB_ERR_OOM;
  if (!f->h_scal) HUB_CUDA(cudaMallocHost((void **)&f->h_scal, sizeof(FixScal)));
  if ((rc = fix_tables_wait(f))) return rc;
  const int ub = (int)std::min<i64>(tile_blocks(h), (i64)kUpdateBlocks * num_sms());
  const int swap = F.a == 0;
  const bool st32 = small_tiles(h);

  // S_1 = x0 on the grid of its largest entry
  auto start = [&]() -> int {
    int rc2 = plan_vector(h, f, x0, D, 0, s);
    if (rc2) return rc2;
    count_launch(h, 2);
    HUB_CUDA(cudaMemsetAsync(f->acc, 0, sizeof(u64) * kFixSlots * kAcc, s));
    HUB_CUDA(cudaMemsetAsync(f->vec[1], 0, sizeof(i64) * n_r * ld, s));
    in_kernel(h, p.limbs())<<<in_blocks(h), kTileThreads, 0, s>>>(
        n_dn, n_up, fix_ld(n_up), fix_ld(n_dn), x0, f->ctl, 0, p.B, swap ? nullptr : f->vec[0],
        swap ? f->vec[0] : (F.both ? ST : nullptr), f->acc);
    HUB_LAUNCH_CHECK();
    k_fix_start<<<1, 32, 0, s>>>(f->acc, p.B, f->scal);
    HUB_LAUNCH_CHECK();
    return HUB_OK;
  };
  // one step on (cur, prev): prev becomes S_{j+1}
  auto step = [&](i64 *cur, i64 *prev, double *psi, cudaStream_t st) -> int {
    int rc2 = prof_mark(h, HUB_PROF_APPLY, true, st);
    if (rc2 || (rc2 = fix_product(h, f, p, F, cur, ST, out0, out1, nullptr, true, st)) ||
        (rc2 = prof_mark(h, HUB_PROF_APPLY, false, st)) || (rc2 = prof_mark(h, HUB_PROF_UPDATE, true, st)))
      return rc2;
    count_launch(h);
#define FIX_UPDATE_T(T, BT, LIMB)                                                                                   \
  (psi ? k_fix_update<T, BT, LIMB, true> : k_fix_update<T, BT, LIMB, false>)<<<ub, kTileThreads, 0, st>>>(          \
      n_r, n_c, ld, ldt, out0, out1, cur, prev, ST, f->scal, f->acc, psi ? f->v : nullptr, psi, swap, p.B)
#define FIX_UPDATE(BT, LIMB)                                                                                        \
  do {                                                                                                              \
    if (st32)                                                                                                       \
      FIX_UPDATE_T(32, BT, LIMB);                                                                                   \
    else                                                                                                            \
      FIX_UPDATE_T(64, BT, LIMB);                                                                                   \
  } while (0)
    if (!F.both)
      FIX_UPDATE(false, false);
    else if (p.limbs())
      FIX_UPDATE(true, true);
    else
      FIX_UPDATE(true, false);
#undef FIX_UPDATE
#undef FIX_UPDATE_T
    HUB_LAUNCH_CHECK();
    count_launch(h);
    (p.limbs() ? k_fix_rescale<true> : k_fix_rescale<false>)<<<std::min(grid_of(D), 4 * num_sms()), 256, 0, st>>>(
        f->scal, n_r * ld, prev, F.both ? n_c * ldt : 0, ST);
    HUB_LAUNCH_CHECK();
    return prof_mark(h, HUB_PROF_UPDATE, false, st);
  };

  if ((rc = start())) return rc;
  int ctl[kCtlWords];
  HUB_CUDA(cudaMemcpyAsync(ctl, f->ctl, sizeof(ctl), cudaMemcpyDeviceToHost, s));
  HUB_CUDA(cudaMemcpyAsync(f->h_scal, f->scal, sizeof(FixScal), cudaMemcpyDeviceToHost, s));
  HUB_CUDA(cudaStreamSynchronize(s));
  h->start_norm = std::ldexp(std::sqrt(f->h_scal->N) / (unsigned)ctl[kCtlScale], 31 + ctl[kCtlShift] - (p.B - 1));
  if (ctl[kCtlShift] == 2047 - 1023 || !(f->h_scal->N > 0.0))          // N = 0: hub_green_coeffs looks at the norm
    return fail(HUB_ERR_ARG, "hub_lanczos_ground: start vector is zero or not finite");

  // graphs of one step, kept while their operands stay the same
  bool graphs = !h->prof && !f->graph_failed;
  if (graphs) {
    std::vector<unsigned char> key;
    auto add = [&](const void *q, size_t n) { key.insert(key.end(), (const unsigned char *)q, (const unsigned char *)q + n); };
    const FixPass P0 = fix_pass(h, f, p, F.a, true);
    const void *ptrs[8] = {out0, ST, out1, f->vec[0], f->vec[1], f->acc, f->scal, nullptr};
    add(&P0, sizeof(P0));
    add(ptrs, sizeof(ptrs));
    if (!f->graph[0] || key != f->graph_key) {
      bool ok = f->gs || cudaStreamCreateWithFlags(&f->gs, cudaStreamNonBlocking) == cudaSuccess;
      for (int k = 0; k < 2 && ok; ++k) {
        if (f->graph[k]) cudaGraphExecDestroy(f->graph[k]);
        f->graph[k] = nullptr;
        cudaGraph_t g = nullptr;
        ok = cudaStreamBeginCapture(f->gs, cudaStreamCaptureModeRelaxed) == cudaSuccess;
        if (!ok) break;
        const int r2 = step(f->vec[k], f->vec[1 - k], nullptr, f->gs);
        ok = cudaStreamEndCapture(f->gs, &g) == cudaSuccess && r2 == HUB_OK && g &&
             cudaGraphInstantiate(&f->graph[k], g, 0) == cudaSuccess;
        if (g) cudaGraphDestroy(g);
      }
      if (!ok) {
        for (int k = 0; k < 2; ++k) {
          if (f->graph[k]) cudaGraphExecDestroy(f->graph[k]);
          f->graph[k] = nullptr;
        }
        f->graph_failed = true;
        cudaGetLastError();
        set_error("");
      } else {
        f->graph_key = key;
      }
    }
    graphs = f->graph[0] != nullptr;
  }

  h->alpha.clear();
  h->beta.clear();
  // Small sectors run several steps per host read-back; steps past the stopping one are dropped.
  const int batch = D <= ((i64)1 << 21) ? kFixHist : 1;
  double E = 0.0, E_prev = 0.0;
  LowestTracker lowest;
  int status = HUB_ERR_NOCONV;
  bool done = false;
  for (int j = 0; j < maxit && !done;) {
    const int nb = std::min(batch, maxit - j);
    count_launch(h);
    k_fix_rewind<<<1, 1, 0, s>>>(f->scal);
    HUB_LAUNCH_CHECK();
    for (int b = 0; b < nb; ++b) {
      const int k = (j + b) & 1;
      if (graphs) {
        HUB_CUDA(cudaGraphLaunch(f->graph[k], s));
      } else if ((rc = step(f->vec[k], f->vec[1 - k], nullptr, s))) {
        return rc;
      }
    }
    HUB_CUDA(cudaMemcpyAsync(f->h_scal, f->scal, sizeof(FixScal), cudaMemcpyDeviceToHost, s));
    HUB_CUDA(cudaStreamSynchronize(s));
    for (int b = 0; b < nb; ++b) {
      const double a = p.tau * f->h_scal->hist[3 * b], be = p.tau * f->h_scal->hist[3 * b + 1];
      if (!std::isfinite(a) || !std::isfinite(be)) {
        if ((rc = fast_check_error(h))) return rc;
        return fail(HUB_ERR_CUDA, "hub_lanczos_ground: non-finite alpha/beta");
      }
      h->alpha.push_back(a);
      h->beta.push_back(be);
      if (tol > 0) E = lowest.next(h->alpha.data(), h->beta.data(), (int)h->alpha.size());   // else at the end
      if (tol > 0 && j + b > 0 && std::fabs(E - E_prev) < tol) {
        status = HUB_OK;
        done = true;
        break;
      }
      E_prev = E;
      if (be <= 1e-14 * std::fmax(1.0, std::fabs(a))) {
        status = HUB_CONVERGED_BREAKDOWN;
        done = true;
        break;
      }
    }
    j += nb;
  }
  if (tol <= 0 && status == HUB_ERR_NOCONV) status = HUB_OK;
  if (tol <= 0) E = tridiag_lowest(h->alpha.data(), h->beta.data(), (int)h->alpha.size());
  if ((rc = fast_check_error(h))) return rc;
  *E0 = E;
  const int k = (int)h->alpha.size();
  if (iters) *iters = k;

  if (psi_out) {
    // second pass: the same integer steps again, psi = sum_j v_j q_j
    const std::vector<double> vv = tridiag_vector(h->alpha.data(), h->beta.data(), k, psi_eigenvalue(h, E));
    if (f->v_cap < k) {
      dev_free(f->v);
      f->v = nullptr;
      f->v_cap = 0;
      if (!dev_alloc((void **)&f->v, sizeof(double) * k, "eigenvector of T")) return HUB_ERR_OOM;
      f->v_cap = k;
    }
    HUB_CUDA(cudaMemcpyAsync(f->v, vv.data(), sizeof(double) * k, cudaMemcpyHostToDevice, s));
    if ((rc = start())) return rc;        // reads x0, which psi may lie over
    HUB_CUDA(cudaMemsetAsync(psi_out, 0, sizeof(double) * D, s));
    for (int j = 0; j + 1 < k; ++j)
      if ((rc = step(f->vec[j & 1], f->vec[1 - (j & 1)], psi_out, s))) return rc;
    count_launch(h);
    (p.limbs() ? k_fix_axpy<true> : k_fix_axpy<false>)<<<grid_of(D), 256, 0, s>>>(
        n_r, n_c, ld, f->vec[(k - 1) & 1], f->scal, f->v, psi_out, swap);
    HUB_LAUNCH_CHECK();
    if ((rc = f64_normalise(h, D, psi_out, s))) return rc;
    HUB_CUDA(cudaStreamSynchronize(s));
    if ((rc = fast_check_error(h))) return rc;
  }
  if (status == HUB_ERR_NOCONV) set_error("hub_lanczos_ground: maxit reached before |dE0| < tol");
  return status;
}

}  // namespace hub
