// One pass of the block-MGS Arnoldi step over a range of vector elements:
// w -= sum_k h_k v_k for NB basis vectors, and the dots of the updated w with
// the next NN basis vectors (NN = 0, the last block: ||w||^2 and, while
// v_{j+1} shares the block, the dots with its own vectors).  Shared by the
// single-instance passes (rt_krylov.cu) and the batched ones (rt_batch.cu).
//
// What bounds it.  This GPU retires 1.88 FP64 multiply-adds per clock and SM
// (measured), and a dot and an update per basis element cost one each.  The
// update stays a chain of FP64 multiply-adds; the dots run on the integer
// pipe, which the FP64 pipe leaves idle: both factors are turned into 58-bit
// fixed-point numbers of two signed 29-bit digits and the digit products are
// summed exactly in 64-bit integers (four wide multiply-adds per product).  A
// probe of conversion and three digit products alone ran 2.5 products per
// clock and SM, and 1.86 with an FP64 multiply-add beside each: the integer
// work hides behind the FP64 pipe.
//
// Memory.  A CTA owns a contiguous range and streams tiles of kPassTile
// elements of w and of all basis vectors of the pass through a ring of
// shared-memory stages with bulk copies (bounded waits), so the registers hold
// no load in flight.
#pragma once

#include "rt_async.cuh"

namespace rt {
namespace {

// ------------------------------------------------------ fixed-point dots
// x = (a1 2^29 + a0) 2^(E - 1079) to within 2^(E - 1080): a1, a0 the signed
// 29-bit digits of x rounded to a multiple of 2^(E - 1079), for |x| below
// 2^(E - 1022) (biased exponent at most E, 64 <= E).  Zeros and subnormal
// numbers give digits of value zero.
__device__ __forceinline__ void fx_digits(uint32_t hi, uint32_t lo, int E, int& a1, int& a0) {
  const int sh = min(E + 4 - (int)((hi >> 20) & 0x7ff), 63);   // what is left past 2^-63 rounds to 0 below
  const uint64_t M = ((uint64_t)(__funnelshift_l(lo, hi, 11) | 0x80000000u) << 32) | (uint32_t)(lo << 11);
  const uint64_t G = M >> sh;   // |x| with its leading bit at 2^59 for exponent E
  // half a unit added to what is left of |x|; for a negative x the complement
  // (one less than -G) puts what the shift dropped on the right side of the
  // half, so that neither sign is rounded towards zero more often
  const uint32_t sg = (uint32_t)((int)hi >> 31);
  const uint64_t s64 = ((uint64_t)sg << 32) | sg;
  const uint64_t g = (G ^ s64) + 4;
  a0 = (int)(uint32_t)g >> 3;
  a1 = (int)(g >> 32) + (int)((uint32_t)g >> 31);
}

__device__ __forceinline__ int fx_exp(double x) { return (int)(((uint32_t)__double2hiint(x) >> 20) & 0x7ff); }

// a power of two, -1022 <= e <= 1023
__device__ __forceinline__ double fx_pow2(int e) { return __hiloint2double((e + 1023) << 20, 0); }

__device__ __forceinline__ double fx_warp_sum(double t) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  return t;
}

constexpr int kFxHead = 2;        // headroom (bits) over the first values' largest exponent
constexpr int kFxHeadMore = 3;    // the same when a later value did not fit
constexpr int kFxMinExp = 64;     // smallest scale: zeros and subnormal numbers shift out from 59 on
constexpr int kFxEpoch = 62;      // additions between two scalings: 62 products a lane fit the 64-bit sums

// ND dot products <w, v_d> of one warp, one element per lane and add(); the
// last NF of them on the FP64 pipe, the others on the integer pipe.  The
// scales (one exponent for w, one for the v_d) come from the warp's first
// values and are renewed when a value does not fit and after kFxEpoch
// additions; at each renewal the warp's integer sums are folded exactly into
// lane d's FP64 sum.  Infinities, NaN and values whose largest is below 2^-961
// (the scales end there) take the FP64 products; zeros and subnormal numbers
// have digits of value zero.
//
// SQ: dot 0 is <w, w> (v[0] is not read), from the digits of w twice and with
// w's scale twice.  What is left of w may be far smaller than the vectors v_d:
// on their scale its square would keep none of its digits.
template <int ND, int NF, bool SQ>
struct FixDot {
  static_assert(NF >= 0 && NF < ND, "at least one dot in fixed point");
  static constexpr int NI = ND - NF;
  static constexpr int D0 = SQ ? 1 : 0;   // first dot with a vector of its own
  long long hi[NI], mid[NI], low[NI];   // sums of the digit products a1 w1, a1 w0 + a0 w1, a0 w0
  double f[NF > 0 ? NF : 1];            // the lane's FP64 sums
  int Ew, Ev;
  int left;      // additions until the next renewal
  double acc;    // lane d < ND: the dot d of the folded additions

  __device__ __forceinline__ void clear() {
#pragma unroll
    for (int d = 0; d < NI; ++d) {
      hi[d] = 0;
      mid[d] = 0;
      low[d] = 0;
    }
  }

  __device__ __forceinline__ void init() {
    clear();
#pragma unroll
    for (int d = 0; d < NF; ++d) f[d] = 0.0;
    Ew = 0;
    Ev = 0;
    left = 0;
    acc = 0.0;
  }

  // the warp's integer sums into acc (warp-uniform call)
  __device__ __forceinline__ void fold() {
    const int lane = threadIdx.x & 31;
    int t2 = 0;
    unsigned t1 = 0, t0 = 0, f0 = 0;
#pragma unroll
    for (int d = 0; d < NI; ++d) {
      // the lane's sum T + f 2^-24 in units of 2^58 digit units (f truncated
      // to 24 bits: 2^-80 of the largest product the scales allow)
      const long long m = mid[d] + (low[d] >> 29);
      const long long T = hi[d] + (m >> 29);
      const unsigned rf = __reduce_add_sync(0xffffffffu, (unsigned)(m & 0x1fffffff) >> 5);
      const unsigned r0 = __reduce_add_sync(0xffffffffu, (unsigned)(T & 0xffffff));
      const unsigned r1 = __reduce_add_sync(0xffffffffu, (unsigned)((T >> 24) & 0xffffff));
      const int r2 = __reduce_add_sync(0xffffffffu, (int)(T >> 48));
      if (lane == d) {
        f0 = rf;
        t0 = r0;
        t1 = r1;
        t2 = r2;
      }
    }
    // (t2 2^48 + t1 2^24 + t0 + f0 2^-24) 2^58 2^(Ev - 1079) 2^(Ew - 1079)
    const long long top = ((long long)t2 << 24) + t1, bot = ((long long)t0 << 24) + f0;
    const double v = fma((double)top, 16777216.0, (double)bot * 5.9604644775390625e-08);
    // the power of two in two halves, so that neither overflows or underflows before the product does
    const int E = (SQ && lane == 0 ? Ew : Ev) + Ew - 2100;
    if (lane < NI) acc += v * fx_pow2(E >> 1) * fx_pow2(E - (E >> 1));
    clear();
  }

  // w: the lane's element of w; v[d]: its element of vector d
  __device__ __forceinline__ void add(double w, const double (&v)[ND]) {
    const int ew = fx_exp(w);
    int ev = 0;
#pragma unroll
    for (int d = D0; d < NI; ++d) ev = max(ev, fx_exp(v[d]));
#pragma unroll
    for (int d = 0; d < NF; ++d) f[d] = fma(w, v[NI + d], f[d]);
    if (!__all_sync(0xffffffffu, left > 0 && ew <= Ew && ev <= Ev)) {   // new scales
      const int head = left > 0 ? kFxHeadMore : kFxHead;
      if (Ew) fold();
      const int mw = __reduce_max_sync(0xffffffffu, ew), mv = __reduce_max_sync(0xffffffffu, ev);
      Ew = min(max(mw + head, kFxMinExp), 2046);
      Ev = min(max(mv + head, kFxMinExp), 2046);
      left = kFxEpoch;
      const bool f64 = max(mw, mv) == 2047 || (mw > 0 && mw + head < kFxMinExp) || (mv > 0 && mv + head < kFxMinExp);
      if (f64) {   // these elements in FP64
        left = 0;
        Ew = 0;
#pragma unroll
        for (int d = 0; d < NI; ++d) {
          const double t = fx_warp_sum(w * (SQ && d == 0 ? w : v[d]));
          if ((int)(threadIdx.x & 31) == d) acc += t;
        }
        return;
      }
      if (mw == 0 || (!SQ && mv == 0)) {   // nothing to add, and no scale for what follows
        left = 0;
        Ew = 0;
        return;
      }
    }
    --left;
    int w1, w0;
    fx_digits(__double2hiint(w), __double2loint(w), Ew, w1, w0);
    if (SQ) {
      hi[0] += (long long)w1 * w1;
      mid[0] += (long long)w1 * w0 * 2;
      low[0] += (long long)w0 * w0;
    }
#pragma unroll
    for (int d = D0; d < NI; ++d) {
      int a1, a0;
      fx_digits(__double2hiint(v[d]), __double2loint(v[d]), Ev, a1, a0);
      hi[d] += (long long)a1 * w1;
      mid[d] += (long long)a1 * w0;
      mid[d] += (long long)a0 * w1;
      low[d] += (long long)a0 * w0;
    }
  }

  // the warp's dots: lane d < ND holds dot d
  __device__ __forceinline__ double finish() {
    if (Ew) fold();
#pragma unroll
    for (int d = 0; d < NF; ++d) {
      const double t = fx_warp_sum(f[d]);
      if ((int)(threadIdx.x & 31) == NI + d) acc = t;
    }
    return acc;
  }
};

// ------------------------------------------------------------ block pass
// A CTA is kPassWarps consumer warps, one element per lane and tile, and one
// producer warp that fills the ring: the consumers never meet at a barrier
// inside the loop, so the FP64 phase of one warp overlaps the integer phase
// of another, and the producer runs ahead into the next tiles while the
// coefficients of the pass are still being formed.
constexpr int kPassWarps = 8;
constexpr int kPassTile = 32 * kPassWarps;
constexpr int kPassThreads = kPassTile + 32;
constexpr int kPassMaxStages = 8;
constexpr int kPassSmem = 110592;                 // ring bytes per CTA: two CTAs share an SM
constexpr int kPassDynSmem = kPassSmem + 128;

template <int B, int NB, int NN>
struct PassShape {
  static_assert(NB >= 0 && NB <= B && NN >= 0 && NN <= B && NB + NN > 0 && B <= kGramMax, "block shape");
  static_assert(NN == 0 || NB == 0 || NB == B, "only the last block is short");
  static constexpr int NG = NN == 0 && NB < B ? NB : 0;        // Gram dots of the last block
  static constexpr int ND = NN > 0 ? NN : 1 + NG;              // dots of the pass
  // dots on the FP64 pipe: a dot costs either pipe about the same time, so
  // they fill what the NB updates leave of it (the first kernel of a step,
  // with no update, ran at half the memory rate with all its dots in integers)
  static constexpr int NF = ND > NB ? (ND - NB) / 2 : 0;
  static constexpr bool SQ = NN == 0;                          // dot 0 is ||w||^2
  static constexpr int NV = 1 + NB + NN;                       // vectors of a stage, w first
  static constexpr int STAGE = NV * kPassTile * (int)sizeof(double);
  static constexpr int NST = kPassSmem / STAGE < kPassMaxStages ? kPassSmem / STAGE : kPassMaxStages;
  static_assert(NST >= 2 && NV <= 32, "at least two stages, one producer lane per vector");
};

// The CTA's ring: stages from a 128-byte aligned base, a full and an empty
// barrier each; `used` counts the tiles taken so far (stage and parity follow
// from it; the producer and the consumers each keep their own copy).
struct PassRing {
  unsigned char* base;
  uint64_t* full;
  uint64_t* empty;
  unsigned used;
  volatile int* dead;   // shared: a wait gave up, nothing waits any more
};

__device__ __forceinline__ void pass_wait(const PassRing& R, uint64_t* bar, uint32_t parity) {
  if (!*R.dead && !mbar_wait(bar, parity)) *R.dead = 1;
}

// barrier of the consumer warps
__device__ __forceinline__ void pass_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kPassTile) : "memory"); }

// sets up the ring in the CTA's dynamic shared memory (all threads)
__device__ __forceinline__ void pass_ring_init(PassRing& R, unsigned char* dyn, uint64_t* bars, int* dead, int nst) {
  R.base = dyn + ((128 - (smem_u32(dyn) & 127)) & 127);
  R.full = bars;
  R.empty = bars + kPassMaxStages;
  R.used = 0;
  R.dead = dead;
  if (threadIdx.x == 0) {
    *dead = 0;
    for (int s = 0; s < nst; ++s) {
      mbar_init(&R.full[s], 1);
      mbar_init(&R.empty[s], kPassWarps);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  __syncthreads();
}

// tile q of the nt tiles of the range [lo, hi): first element and element
// count (even).  rev: the tiles run from the top of the range downwards.
__device__ __forceinline__ void pass_tile(int64_t lo, int64_t hi, int q, int nt, int rev, int64_t& e0, int& cnt) {
  e0 = lo + (int64_t)(rev ? nt - 1 - q : q) * kPassTile;
  cnt = (int)(hi - e0 < kPassTile ? hi - e0 : kPassTile);
}
__device__ __forceinline__ int pass_tiles(int64_t lo, int64_t hi) {
  return (int)((hi - lo + kPassTile - 1) / kPassTile);
}

// The producer warp's operands: lane 0 copies w, lane 1 + k the k-th basis
// vector (the block's, then the next block's).
struct PassSrc {
  const double* p;   // this lane's vector (element 0); lanes past the last: NULL
  uint64_t policy;
};
template <int B, int NB, int NN>
__device__ __forceinline__ PassSrc pass_src(const double* w, const double* vb, const double* vn, int64_t N) {
  const int lane = threadIdx.x & 31;
  PassSrc s;
  s.p = lane == 0 ? w : lane <= NB ? vb + (int64_t)(lane - 1) * N : lane <= NB + NN ? vn + (int64_t)(lane - 1 - NB) * N
                                                                                    : nullptr;
  // the block's vectors are not read again in this step
  s.policy = lane >= 1 && lane <= NB ? policy_evict_first() : policy_evict_normal();
  return s;
}

// producer warp: the copies of one tile into its stage; with_v announces the
// bytes of the whole stage and copies the basis vectors, with_w copies w
template <int B, int NB, int NN>
__device__ __forceinline__ void pass_issue(const PassRing& R, unsigned slot, const PassSrc& S0, int64_t e0, int cnt,
                                           bool with_v, bool with_w) {
  using S = PassShape<B, NB, NN>;
  const int lane = threadIdx.x & 31;
  const uint32_t bytes = (uint32_t)cnt * 8;
  if (with_v && lane == 0) mbar_expect_tx(&R.full[slot], bytes * S::NV);
  __syncwarp();
  if (lane < S::NV && (lane == 0 ? with_w : with_v))
    bulk_load(R.base + (size_t)slot * S::STAGE + (size_t)lane * kPassTile * 8, S0.p + e0, bytes, &R.full[slot],
              S0.policy);
}

// producer warp: the tiles of [lo, hi) from tile `from` on; false once a wait
// gave up (nothing more is copied then).  R.used counts the tiles issued.
template <int B, int NB, int NN>
__device__ __forceinline__ bool pass_produce(PassRing& R, const PassSrc& S0, int64_t lo, int64_t hi, int rev,
                                             int from) {
  using S = PassShape<B, NB, NN>;
  const int nt = pass_tiles(lo, hi);
  int q = from;
  for (; q < nt; ++q) {
    const unsigned u = R.used + q, slot = u % S::NST;
    if (u >= (unsigned)S::NST) pass_wait(R, &R.empty[slot], (u / S::NST - 1) & 1);
    if (__any_sync(0xffffffffu, *R.dead)) break;
    int64_t e0;
    int cnt;
    pass_tile(lo, hi, q, nt, rev, e0, cnt);
    pass_issue<B, NB, NN>(R, slot, S0, e0, cnt, true, true);
  }
  R.used += q;
  return q == nt;
}

// producer warp, before it leaves: the copies it issued land (one bound for
// all of them).  The consumers take every tile, but one that gave up a wait
// goes on without the copies, and none may write the CTA's shared memory after
// its end.
__device__ __forceinline__ void pass_drain(const PassRing& R, unsigned nst) {
  const unsigned long long t0 = gtimer();
  for (unsigned p = R.used > nst ? R.used - nst : 0; p < R.used; ++p)
    while (!mbar_try_wait(&R.full[p % nst], (p / nst) & 1))
      if (gtimer() - t0 > kWaitNs) return;
}

// consumer warps: the pass over [lo, hi); h: the block's coefficients; the
// warp's dots are added to D
template <int B, int NB, int NN>
using PassDots = FixDot<PassShape<B, NB, NN>::ND, PassShape<B, NB, NN>::NF, PassShape<B, NB, NN>::SQ>;
template <int B, int NB, int NN>
__device__ __forceinline__ void pass_consume(PassRing& R, double* __restrict__ w, int64_t lo, int64_t hi, int rev,
                                             const double* h, PassDots<B, NB, NN>& D) {
  using S = PassShape<B, NB, NN>;
  const int nt = pass_tiles(lo, hi);
  const int t = threadIdx.x;
  for (int q = 0; q < nt; ++q) {
    const unsigned u = R.used + q, slot = u % S::NST;
    int64_t e0;
    int cnt;
    pass_tile(lo, hi, q, nt, rev, e0, cnt);
    pass_wait(R, &R.full[slot], (u / S::NST) & 1);
    const double* st = reinterpret_cast<const double*>(R.base + (size_t)slot * S::STAGE);
    // lanes past a short tile's end take its last element with w = 0
    const bool in = t < cnt;
    const int ti = min(t, cnt - 1);
    double wi = st[ti];
    double b[NB > 0 ? NB : 1], v[S::ND];
#pragma unroll
    for (int k = 0; k < NB; ++k) b[k] = st[(1 + k) * kPassTile + ti];
    if (NN > 0) {
#pragma unroll
      for (int k = 0; k < NN; ++k) v[k] = st[(1 + NB + k) * kPassTile + ti];
    }
    __syncwarp();
    if ((t & 31) == 0) mbar_arrive(&R.empty[slot]);   // the warp has its operands
#pragma unroll
    for (int k = 0; k < NB; ++k) wi = fma(-h[k], b[k], wi);
    if (NB > 0 && in) w[e0 + t] = wi;
    wi = in ? wi : 0.0;
    if (NN == 0) {   // v[0] stands for w itself
#pragma unroll
      for (int k = 0; k < S::NG; ++k) v[1 + k] = b[k];
    }
    D.add(wi, v);
  }
  R.used += nt;
}

// the CTA's dots from its consumer warps' (lane d of each: dot d), summed
// over the warps in a fixed order; consumer thread d < nd gets dot d
__device__ __forceinline__ double pass_block_dots(double warp_dot, int nd) {
  __shared__ double red[kGramMax][kPassWarps];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  pass_sync();
  if (lane < nd) red[lane][warp] = warp_dot;
  pass_sync();
  double s = 0.0;
  if ((int)threadIdx.x < nd) {
    double v[kPassWarps];
#pragma unroll
    for (int q = 0; q < kPassWarps; ++q) v[q] = red[threadIdx.x][q];
#pragma unroll
    for (int o = kPassWarps / 2; o > 0; o >>= 1)
#pragma unroll
      for (int q = 0; q < o; ++q) v[q] += v[q + o];
    s = v[0];
  }
  return s;
}

}  // namespace
}  // namespace rt
