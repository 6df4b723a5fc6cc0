// Device code shared by the single-instance kernels (rt_operator.cu) and the
// batched kernels (rt_batch.cu): the quadrature of one height, the formal
// solver's sweep along one ray, the FP32 step coefficients.
#pragma once

#include "rt_common.cuh"
#include "rt_convert.cuh"

namespace rt {
namespace {

constexpr int kMomThreads = 256;      // threads of the batch's quadratures and the FP32 one on many heights
constexpr int kMom32Threads = 512;    // threads of the FP32 quadrature on few heights
constexpr int kMaxTiles = 8;     // FP32 kernel: up to 256 threads per CTA (255 registers a lane)
constexpr int kMaxTilesRay = 16; // FP64 formal solver on rays: depth tiles per ray group (one warp each)
constexpr int kMaxTiles64 = 32;  // FP64 formal solver on pairs of rays: the same
constexpr int kRing = 8;         // prefetch depth of the FP64 formal-solver kernel (steps)
constexpr int kRing32 = 8;       // the same of the FP32 kernel (one lane carries I and Q), FP32 vectors
constexpr int kRing32D = 4;      // ... and FP64 vectors
constexpr int kMinSteps32 = 32;  // shortest depth tile of the FP32 kernel (steps)

enum KMode { KM_PLAIN = 0, KM_JACOBI = 1, KM_LOCAL_LAMBDA = 2, KM_RHS = 3 };

template <typename T>
__device__ __forceinline__ T warp_sum(T v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

template <typename To, typename From>
__device__ __forceinline__ To vcast(From x) {
  if constexpr (sizeof(To) == 4 && sizeof(From) == 8) return to_f32(x);
  else if constexpr (sizeof(To) == 8 && sizeof(From) == 4) return to_f64(x);
  else return x;
}

// beta* (coefficient of S_k in I_k) of ray r = m*Nnu + p at height k: the
// beta of the step ending at k; with the DELO-parabolic downwind coefficients
// cg (else NULL) also e_k times the gamma of the step before, whose downwind
// node is k.  col = coef_col(r, ...) and cstride: the table column and row
// length (coef_col).
__device__ __forceinline__ double beta_star(const double* __restrict__ cb, int k, int m, int64_t col,
                                            int64_t cstride, int Ns, int Nh,
                                            const double* __restrict__ ce = nullptr,
                                            const double* __restrict__ cg = nullptr) {
  if (m < Nh) {
    if (k == 0) return 0.0;
    double b = cb[(int64_t)(k - 1) * cstride + col];
    if (cg && k >= 2) b += ce[(int64_t)(k - 1) * cstride + col] * cg[(int64_t)(k - 2) * cstride + col];
    return b;
  }
  if (k == Ns - 1) return 0.0;
  double b = cb[(int64_t)k * cstride + col];
  if (cg && k <= Ns - 3) b += ce[(int64_t)k * cstride + col] * cg[(int64_t)(k + 1) * cstride + col];
  return b;
}

// ----------------------------------------------------------------- K1: T∘J
// MODE: KM_PLAIN z = x; KM_JACOBI z = x * dinv; KM_LOCAL_LAMBDA z = x and
// sigma_k <- M_k^{-1} sigma_k.

// FP32 quadrature of height k by the whole block (THREADS threads) as flat dot
// products over its rays, with the per-ray weights w0 = hat-w_m
// hat-w_p, w1 = w0 T201_m, w2 = w0 T202_m (wray, [3][nray]):
//     J00 = sum_r w0 I_r,   J20 = sum_r (w1 I_r + w2 Q_r).
// NORM: the input is x * inv, written to xout in the input's precision as
// each element is read (the GMRES normalisation of the batched solver).  A
// warp per direction row, as before, left lanes idle on short rows and half
// of its loads predicated off (32 uneven atmospheres: 139 us a launch).  U: rays
// whose loads are issued before their sums.
template <typename TI, int MODE, int THREADS, int U, bool NORM = false>
__device__ __forceinline__ void moments_flat32(const TI* __restrict__ x, const double* __restrict__ dinv,
                                               const float* __restrict__ wray, const float* __restrict__ t201,
                                               const float* __restrict__ t202, const double* __restrict__ Minv,
                                               int Ns, int Nmu, int64_t nray, float xi, float xiW2,
                                               float* __restrict__ S, int k, double inv = 1.0,
                                               TI* __restrict__ xout = nullptr) {
  constexpr int nw = THREADS / 32;
  const int64_t oI = (int64_t)k * nray, oQ = ((int64_t)Ns + k) * nray;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float a0 = 0.f, a1 = 0.f;
#pragma unroll (U == 1 ? 4 : 1)
  for (int64_t r0 = threadIdx.x; r0 < nray; r0 += U * THREADS) {
    TI xI[U], xQ[U];
    double dI[U], dQ[U];
    float w0[U], w1[U], w2[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t r = r0 + u * THREADS < nray ? r0 + u * THREADS : r0;
      xI[u] = x[oI + r];
      xQ[u] = x[oQ + r];
      if (MODE == KM_JACOBI) {
        dI[u] = dinv[oI + r];
        dQ[u] = dinv[oQ + r];
      }
      w0[u] = wray[r];
      w1[u] = wray[nray + r];
      w2[u] = wray[2 * nray + r];
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int64_t r = r0 + u * THREADS;
      if (u > 0 && r >= nray) continue;
      if (NORM) {
        xI[u] = (TI)(xI[u] * inv);
        xQ[u] = (TI)(xQ[u] * inv);
        xout[oI + r] = xI[u];
        xout[oQ + r] = xQ[u];
      }
      float vI = vcast<float>(xI[u]), vQ = vcast<float>(xQ[u]);
      if (MODE == KM_JACOBI) {
        vI *= to_f32(dI[u]);
        vQ *= to_f32(dQ[u]);
      }
      a0 = fmaf(w0[u], vI, a0);
      a1 = fmaf(w1[u], vI, a1);
      a1 = fmaf(w2[u], vQ, a1);
    }
  }
  a0 = warp_sum(a0);
  a1 = warp_sum(a1);
  __shared__ float red[2][nw];
  __shared__ float sig[2];
  if (lane == 0) { red[0][warp] = a0; red[1][warp] = a1; }
  __syncthreads();
  if (threadIdx.x == 0) {
    float a = 0.f, b = 0.f;
    for (int w = 0; w < nw; ++w) { a += red[0][w]; b += red[1][w]; }
    float s0 = xi * a, s2 = xiW2 * b;
    if (MODE == KM_LOCAL_LAMBDA) {
      const double* Mi = Minv + 4 * k;
      const float u0 = (float)Mi[0] * s0 + (float)Mi[1] * s2;
      const float u2 = (float)Mi[2] * s0 + (float)Mi[3] * s2;
      s0 = u0;
      s2 = u2;
    }
    sig[0] = s0;
    sig[1] = s2;
  }
  __syncthreads();
  for (int m = threadIdx.x; m < Nmu; m += blockDim.x) {
    S[(int64_t)k * Nmu + m] = sig[0] + t201[m] * sig[1];
    S[((int64_t)Ns + k) * Nmu + m] = t202[m] * sig[1];
  }
}

// the end of the FP64 quadrature of height k: the CTA's sums of a0 (J00) and
// a1 (J20) in a fixed order, then sigma and S
template <int MODE>
__device__ __forceinline__ void moments_finish64(double a0, double a1, const double* __restrict__ t201,
                                                 const double* __restrict__ t202, const double* __restrict__ Minv,
                                                 int Ns, int Nmu, double xi, double xiW2, double* __restrict__ S,
                                                 int k) {
  // transposed warp sum: lanes 0-15 get the sum of a0, lanes 16-31 of a1
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const bool h16 = lane & 16;
  double t = (h16 ? a1 : a0) + __shfl_xor_sync(0xffffffffu, h16 ? a0 : a1, 16);
#pragma unroll
  for (int o = 8; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  __shared__ double red[2][32];
  __shared__ double sig[2];
  if ((lane & 15) == 0) red[lane >> 4][warp] = t;
  __syncthreads();
  if (threadIdx.x == 0) {
    const int nw = blockDim.x >> 5;
    double j00 = 0.0, j20 = 0.0;
    for (int w = 0; w < nw; ++w) {
      j00 += red[0][w];
      j20 += red[1][w];
    }
    double s0 = xi * j00, s2 = xiW2 * j20;
    if (MODE == KM_LOCAL_LAMBDA) {
      const double* Mi = Minv + 4 * k;
      const double u0 = Mi[0] * s0 + Mi[1] * s2;
      const double u2 = Mi[2] * s0 + Mi[3] * s2;
      s0 = u0;
      s2 = u2;
    }
    sig[0] = s0;
    sig[1] = s2;
  }
  __syncthreads();
  for (int m = threadIdx.x; m < Nmu; m += blockDim.x) {
    S[(int64_t)k * Nmu + m] = sig[0] + t201[m] * sig[1];
    S[((int64_t)Ns + k) * Nmu + m] = t202[m] * sig[1];
  }
}

// FP64 quadrature of height k as flat dot products over its rays (the CTA's
// threads stride over r): with the per-ray weights w0 = hat-w_m hat-w_p,
// w1 = w0 T201_m, w2 = w0 T202_m (wray, [3][nray]),
//     J00 = sum_r w0 I_r,   J20 = sum_r (w1 I_r + w2 Q_r),
// then S of every direction.  Every FP64 operation is useful work: no
// lane idles on a short row and there is one reduction per height (the FP64
// pipe bounds this kernel).  Any block size that is a multiple of 32.
// WJ (Jacobi mode): wray holds per-element weights [3][Ns][nray], the
// per-ray weights times the inverse diagonal of the element (I, I, Q), so
// the scaling of x costs no operation here.  NORM: the input is x * inv,
// also written to xout (the GMRES normalisation of NormIn).
template <int MODE, bool WJ = false, bool NORM = false>
__device__ __forceinline__ void moments_flat64(const double* __restrict__ x, const double* __restrict__ dinv,
                                               const double* __restrict__ wray, const double* __restrict__ t201,
                                               const double* __restrict__ t202, const double* __restrict__ Minv,
                                               int Ns, int Nmu, int64_t nray, double xi, double xiW2,
                                               double* __restrict__ S, int k, double inv = 1.0,
                                               double* __restrict__ xout = nullptr) {
  const double* __restrict__ xI = x + (int64_t)k * nray;
  const double* __restrict__ xQ = x + ((int64_t)Ns + k) * nray;
  const double* __restrict__ dI = MODE == KM_JACOBI && !WJ ? dinv + (int64_t)k * nray : nullptr;
  const double* __restrict__ dQ = MODE == KM_JACOBI && !WJ ? dinv + ((int64_t)Ns + k) * nray : nullptr;
  const int64_t plane = (int64_t)Ns * nray;
  const double* __restrict__ w0 = WJ ? wray + (int64_t)k * nray : wray;
  const double* __restrict__ w1 = WJ ? w0 + plane : wray + nray;
  const double* __restrict__ w2 = WJ ? w0 + 2 * plane : wray + 2 * nray;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
#pragma unroll 4
  for (int64_t r = threadIdx.x; r < nray; r += blockDim.x) {
    double vI = xI[r], vQ = xQ[r];
    if (NORM) {
      vI *= inv;
      vQ *= inv;
      xout[(int64_t)k * nray + r] = vI;
      xout[((int64_t)Ns + k) * nray + r] = vQ;
    }
    if (MODE == KM_JACOBI && !WJ) {
      vI *= dI[r];
      vQ *= dQ[r];
    }
    a0 = fma(w0[r], vI, a0);
    a1 = fma(w1[r], vI, a1);
    a2 = fma(w2[r], vQ, a2);
  }
  moments_finish64<MODE>(a0, a1 + a2, t201, t202, Minv, Ns, Nmu, xi, xiW2, S, k);
}

// moments_flat64 for a profile symmetric on the frequency grid, modes PLAIN
// and LOCAL_LAMBDA: the rays (+-mu, p) and (+-mu, Nnu-1-p) have the same
// weights, so the four values are added first: 9 operations for 8 elements
// (I and Q) instead of 12.  The FP64 pipe bounds it on large problems.
template <int MODE, bool NORM = false>
__device__ __forceinline__ void moments_pair64(const double* __restrict__ x, const double* __restrict__ wray,
                                               const double* __restrict__ t201, const double* __restrict__ t202,
                                               const double* __restrict__ Minv, int Ns, int Nmu, int64_t nray,
                                               double xi, double xiW2, double* __restrict__ S, int k,
                                               double inv = 1.0, double* __restrict__ xout = nullptr) {
  const int Nh = Nmu / 2, Nnu = (int)(nray / Nmu), np = pair_count(Nnu);
  const int64_t oI = (int64_t)k * nray, oQ = ((int64_t)Ns + k) * nray;
  double a0 = 0.0, a1 = 0.0, a2 = 0.0;
  for (int q = threadIdx.x; q < Nh * np; q += blockDim.x) {
    const int mm = q / np, p = q - mm * np, p2 = Nnu - 1 - p;
    const int up = (Nh + mm) * Nnu, dn = (Nh - 1 - mm) * Nnu;
    const int r[4] = {up + p, dn + p, up + p2, dn + p2};
    const int n = p == p2 ? 2 : 4;   // the middle frequency is its own mirror
    double vI[4], vQ[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      vI[i] = i < n ? x[oI + r[i]] : 0.0;
      vQ[i] = i < n ? x[oQ + r[i]] : 0.0;
    }
    if (NORM) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        vI[i] *= inv;
        vQ[i] *= inv;
        if (i < n) {
          xout[oI + r[i]] = vI[i];
          xout[oQ + r[i]] = vQ[i];
        }
      }
    }
    const double sI = (vI[0] + vI[1]) + (vI[2] + vI[3]), sQ = (vQ[0] + vQ[1]) + (vQ[2] + vQ[3]);
    a0 = fma(wray[r[0]], sI, a0);
    a1 = fma(wray[nray + r[0]], sI, a1);
    a2 = fma(wray[2 * nray + r[0]], sQ, a2);
  }
  moments_finish64<MODE>(a0, a1 + a2, t201, t202, Minv, Ns, Nmu, xi, xiW2, S, k);
}

// --------------------------------------------------------------- K2: Lambda
// 2^a by the hardware's approximate exponential (a <= 0 here)
__device__ __forceinline__ float ex2_approx(float a) {
  float r;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(a));
  return r;
}

constexpr double kLn2 = 0.69314718055994530942;
constexpr float kSeriesD2 = (float)(0.5 / kLn2);

// (-1)^n ln2^(n+1) / (n+2)!: the series of beta / D2 in powers of D2
constexpr double pow_ln2(int k) { return k == 0 ? 1.0 : kLn2 * pow_ln2(k - 1); }
constexpr double fact(int k) { return k <= 1 ? 1.0 : k * fact(k - 1); }
constexpr float kB(int n) { return (float)((n % 2 ? -1.0 : 1.0) * pow_ln2(n + 1) / fact(n + 2)); }

// DELO-linear coefficients of two steps in FP32 from D2 = Delta / ln 2 and iD = 1
// / Delta, one step in each half of the packed FP32 instructions: one series where
// Delta < 1/2 (h = beta / Delta, from which alpha follows with its relative
// accuracy), the closed forms above; both are evaluated and one is selected.  Half
// of a step's instructions are its coefficients.  The register-ring solver (sweep)
// gains over one step at a time (N_s = 333, 10 x 55 rays: 20.5 -> 17.1 us an
// apply); the staged one (rt_tma.cu), which waits on memory, does not.
__device__ __forceinline__ void delo_coeffs2(float2 D2, float2 iD, float2& e, float2& al, float2& be) {
  auto two = [](float c) { return make_float2(c, c); };
  e = make_float2(ex2_approx(-D2.x), ex2_approx(-D2.y));
  float2 hb = two(kB(7));
  hb = __ffma2_rn(hb, D2, two(kB(6)));
  hb = __ffma2_rn(hb, D2, two(kB(5)));
  hb = __ffma2_rn(hb, D2, two(kB(4)));
  hb = __ffma2_rn(hb, D2, two(kB(3)));
  hb = __ffma2_rn(hb, D2, two(kB(2)));
  hb = __ffma2_rn(hb, D2, two(kB(1)));
  hb = __ffma2_rn(hb, D2, two(kB(0)));
  const float2 bs = __fmul2_rn(hb, D2);
  const float2 nonep = __ffma2_rn(D2, two(-(float)kLn2), two(-1.0f));
  const float2 as = __fmul2_rn(D2, __ffma2_rn(nonep, hb, two((float)kLn2)));
  const float2 q = __ffma2_rn(e, __fmul2_rn(iD, two(-1.0f)), iD);
  const float2 bt = __ffma2_rn(q, two(-1.0f), two(1.0f)), at = __ffma2_rn(e, two(-1.0f), q);
  be = make_float2(D2.x < kSeriesD2 ? bs.x : bt.x, D2.y < kSeriesD2 ? bs.y : bt.y);
  al = make_float2(D2.x < kSeriesD2 ? as.x : at.x, D2.y < kSeriesD2 ? as.y : at.y);
}

// FP32 step coefficients from Delta, implicit Euler and trapezoidal
template <int FS>
__device__ __forceinline__ void coeffs32(float D, float& e, float& al, float& be) {
  if (FS == RT_FS_IMPLICIT_EULER) {
    e = __frcp_rn(1.0f + D);
    al = 0.0f;
    be = D * e;
  } else {
    const float h = 0.5f * D, q = __frcp_rn(1.0f + h);
    e = (1.0f - h) * q;
    al = h * q;
    be = al;
  }
}

// coefficients of two steps from their Delta
template <int FS>
__device__ __forceinline__ void coeffs32x2(float D0, float D1, float2& e, float2& al, float2& be) {
  if constexpr (FS == RT_FS_DELO_LINEAR) {
    constexpr float c = (float)(1.0 / kLn2);
    delo_coeffs2(make_float2(D0 * c, D1 * c), make_float2(__fdividef(1.0f, D0), __fdividef(1.0f, D1)), e, al, be);
  } else {
    coeffs32<FS>(D0, e.x, al.x, be.x);
    coeffs32<FS>(D1, e.y, al.y, be.y);
  }
}

struct FormalArgs {
  const void* x;          // input vector (TV)
  const double* dinv;     // Jacobi inverse diagonal (KM_JACOBI)
  const double* ce;       // FP64 coefficient tables [(Ns-1)][nray]
  const double* ca;
  const double* cb;
  const double* cg;       // DELO-parabolic: downwind coefficient table (else NULL)
  int64_t cstride;        // columns of the FP64 tables (coef_col)
  int cshare;             // CoefShare
  int64_t npair;          // FP64, CS_PAIR: lanes (direction, frequency pair); else 0
  const float* dtau32;    // FP32: interval optical depths
  const float* r32;       // FP32: per-ray scale phi_hat/|mu|
  const void* S;          // source functions (TC) [2][Ns][Nmu]
  void* y;                // output vector (TV)
  int Ns, Nmu, Nnu;
  int64_t nray, nd;       // rays per Stokes parameter, downward rays
  int ngd;                // ray groups of downward rays
  int ntile;              // depth tiles per group (warps per CTA)
  double inflow_bottom;   // KM_RHS: I entering at the bottom (mu > 0)
  const int* kstop;       // graph early exit (NULL: run)
  int step;
};

// One lane: NS Stokes parameters (s0 .. s0+NS-1) of ray r, depth steps
// [j0, j1) in marching order (node index j; height k = j for downward rays,
// Ns-1-j for upward rays).  PHASE 0 composes the tile map (E, B) with zero
// inflow; PHASE 2 composes only B (E, a product of the e coefficients, comes
// from a table); PHASE 1 sweeps from the inflow I and writes the output.
// FP64 with FS = RT_FS_DELO_PARABOLIC: each step also takes gamma times S at
// the downwind node (read from the ring, which then holds one node past the
// tile; gamma is 0 on the last interval of a ray).
template <typename TC, typename TV, int FS, int MODE, int PHASE, int NS, int RING>
__device__ __forceinline__ void sweep(const FormalArgs& A, int s0, bool down, int64_t r, int m, bool active, int j0,
                                      int j1, TC (&I)[NS], TC& E) {
  constexpr bool PARA = sizeof(TC) == 8 && FS == RT_FS_DELO_PARABOLIC;
  const int Ns = A.Ns;
  const int64_t nray = A.nray;
  const int64_t plane = (int64_t)Ns * nray;
  const TC* __restrict__ Sm = reinterpret_cast<const TC*>(A.S) + (int64_t)s0 * Ns * A.Nmu + m;
  const int64_t sstride = (int64_t)Ns * A.Nmu;
  const TV* __restrict__ x = reinterpret_cast<const TV*>(A.x) + (int64_t)s0 * plane;
  TV* __restrict__ y = reinterpret_cast<TV*>(A.y) + (int64_t)s0 * plane;
  const double* __restrict__ dinv = A.dinv + (int64_t)s0 * plane;
  const float rs = (sizeof(TC) == 4) ? A.r32[r] : 0.0f;
  const int64_t col = coef_col(r, A.Nmu / 2, A.Nnu, A.cshare), cstride = A.cstride;
  auto height = [&](int j) { return down ? j : Ns - 1 - j; };
  auto interval = [&](int j) { return down ? j - 1 : Ns - 1 - j; };
  TC sp[NS];
#pragma unroll
  for (int q = 0; q < NS; ++q) sp[q] = Sm[q * sstride + (int64_t)height(j0 - 1) * A.Nmu];  // upwind source
  // gamma of the step before j0 (its downwind node is the tile's first node)
  TC gp = 0;
  if (PARA && j0 >= 2) gp = (TC)A.cg[(int64_t)interval(j0 - 1) * cstride + col];
  // register ring of the next RING steps
  TC re[RING], ra[RING], rb[RING], rg[RING], rsv[RING][NS];
  // as loaded: converted on loading, an FP64 vector made the FP32 solver wait
  // for each load at once (32 atmospheres through the batch: 141 -> 125 ms)
  TV rx[RING][NS];
  double rd[RING][NS];
  if (PARA) {
#pragma unroll
    for (int u = 0; u < RING; ++u)
#pragma unroll
      for (int q = 0; q < NS; ++q) rsv[u][q] = 0;
  }
  auto load = [&](int u, int j) {
    if (j < j1) {
      const int k = height(j), i = interval(j);
      if (sizeof(TC) == 8) {
        const int64_t c = (int64_t)i * cstride + col;
        re[u] = (TC)A.ce[c];
        ra[u] = (TC)A.ca[c];
        rb[u] = (TC)A.cb[c];
        if (PARA) rg[u] = (TC)A.cg[c];
      } else {
        re[u] = (TC)A.dtau32[i];   // Delta = dtau_i * r_ray; coefficients formed at use
      }
#pragma unroll
      for (int q = 0; q < NS; ++q) {
        rsv[u][q] = Sm[q * sstride + (int64_t)k * A.Nmu];
        if (PHASE == 1 && MODE != KM_RHS) {
          const int64_t o = q * plane + (int64_t)k * nray + r;
          rx[u][q] = x[o];
          if (MODE == KM_JACOBI) rd[u][q] = dinv[o];
        }
      }
    } else if (PARA && j == j1 && j < Ns) {
      // the downwind node of the tile's last step
#pragma unroll
      for (int q = 0; q < NS; ++q) rsv[u][q] = Sm[q * sstride + (int64_t)height(j) * A.Nmu];
    }
  };
  static_assert(RING % 2 == 0, "the FP32 coefficients are formed for two steps at once");
  float2 e2, al2, be2;   // FP32: steps u (even) and u + 1
  auto step = [&](int u, int j) {
    TC e, al, be;
    if (sizeof(TC) == 8) {
      e = re[u];
      al = ra[u];
      be = rb[u];
    } else {
      if (u % 2 == 0) coeffs32x2<FS>((float)re[u] * rs, (float)re[(u + 1) % RING] * rs, e2, al2, be2);
      e = (TC)(u % 2 ? e2.y : e2.x);
      al = (TC)(u % 2 ? al2.y : al2.x);
      be = (TC)(u % 2 ? be2.y : be2.x);
    }
    if (PHASE == 0) E *= e;
    const int64_t o = (int64_t)height(j) * nray + r;
#pragma unroll
    for (int q = 0; q < NS; ++q) {
      const TC sk = rsv[u][q];
      // beta S_k, plus gamma S_next for DELO-parabolic
      const TC cur = PARA ? fma(be, sk, rg[u] * rsv[(u + 1) % RING][q]) : be * sk;
      if (PHASE != 1) {
        I[q] = fma(e, I[q], fma(al, sp[q], cur));
      } else if (MODE == KM_LOCAL_LAMBDA) {
        // y = (x + beta* S) - I.  DELO-linear: x - (e I_prev + alpha S_prev).
        // DELO-parabolic (beta* = beta + e gamma_prev, gamma_prev S_k being
        // part of I_prev): x - (e (I_prev - gamma_prev S_k) + alpha S_prev + gamma S_next)
        if (PARA) {
          const TC t = fma(e, fma(-gp, sk, I[q]), fma(al, sp[q], rg[u] * rsv[(u + 1) % RING][q]));
          if (active) y[q * plane + o] = vcast<TV>(vcast<TC>(rx[u][q]) - t);
          I[q] = fma(fma(e, gp, be), sk, t);
        } else {
          const TC t = fma(e, I[q], al * sp[q]);
          if (active) y[q * plane + o] = vcast<TV>(vcast<TC>(rx[u][q]) - t);
          I[q] = fma(be, sk, t);
        }
      } else {
        I[q] = fma(e, I[q], fma(al, sp[q], cur));
        if (active) {
          if (MODE == KM_RHS) y[q * plane + o] = vcast<TV>(I[q]);
          else if (MODE == KM_JACOBI) y[q * plane + o] = vcast<TV>(vcast<TC>(rx[u][q]) * vcast<TC>(rd[u][q]) - I[q]);
          else y[q * plane + o] = vcast<TV>(vcast<TC>(rx[u][q]) - I[q]);
        }
      }
      sp[q] = sk;
    }
    if (PARA) gp = rg[u];
  };
#pragma unroll
  for (int u = 0; u < RING; ++u) load(u, j0 + u);
  int jb = j0;
  // full rounds: every step of the round and every refill is in range, so the
  // round is straight-line code the compiler can interleave across steps
  for (; jb + 2 * RING <= j1; jb += RING) {
#pragma unroll
    for (int u = 0; u < RING; ++u) {
      step(u, jb + u);
      load(u, jb + u + RING);
    }
  }
  for (; jb < j1; jb += RING) {
#pragma unroll
    for (int u = 0; u < RING; ++u) {
      if (jb + u < j1) {
        step(u, jb + u);
        load(u, jb + u + RING);
      }
    }
  }
}

}  // namespace
}  // namespace rt
