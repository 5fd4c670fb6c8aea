// Stage solve of the FP64 mode for more than kDenseSolveMaxNq coefficients per
// Chebyshev parity (k_solve_seg).  (The mixed mode keeps the unsegmented
// recurrence: its FP32 transforms turn a different rounding of a solve into
// differences of the size of their own error.)
//
// Systems and phases as in k_solve (rbc_kernels.cu): per (state, Fourier mode,
// parity) the temperature system, then streamfunction or mean flow; the UL
// factors turn each into a backward and a forward recurrence over nq rows.
// Here a column (mode, real or imaginary part) is cut into S segments of LR
// rows, a thread per (segment, column), everything of a thread's rows in
// registers:
//   A  right-hand side of its rows;
//   B  backward recurrence with nothing coming in from the next segment;
//   C  one thread per column carries the first D values of each segment
//      through all segments (the response to what comes in is linear: the
//      tables hold each row's response phi);
//   D  correction of its rows, boundary-row sums, forward recurrence from zero;
//   E  one thread per column: boundary unknowns, the last D values of each
//      segment carried forward (responses theta);
//   F  correction: the solution; G  dt L X_i into the later RK accumulators.
//
// Bound: the FP64 pipe (2 operations per clock and SM; a warp instruction holds
// its sub-partition for 64 clocks whatever its active lanes, and that is also
// the latency of a dependent one).  The recurrences over all nq rows kept one
// warp per block, on one of the four sub-partitions, busy with two dependent
// operations per row while the others waited; cut into segments they run on
// all warps, with one dependent operation per row and about S more per column.
// The accumulators are read and written once (phase G) instead of twice.
// LR depends on the grid only, so a state gives the same bits in any batch.
// Measured (GB300, per launch, unsegmented before): 256 x 64, 32 states
// 133 -> 85 us, 8 states 83 -> 32 us, one state 37 -> 23 us; 512 x 128, 3 states
// 155 -> 46 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "rbc_internal.h"

namespace rbc {

namespace {

enum { KT = 0, KP = 1, KU = 2 };

__device__ __forceinline__ size_t soff(const Grid& g, int f, int n, int m) {
  return ((size_t)(f * g.Nz + n) * g.nm + m) * 2;
}
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

template <int KIND> struct Sys {
  static constexpr int D = (KIND == KP) ? 2 : 1;
  static __device__ __forceinline__ const SegFactors& fac(const Tables& tb) {
    return KIND == KT ? tb.segT : KIND == KP ? tb.segP : tb.segU;
  }
};

// A thread's column: parity, mode, part, column of the tile, segment, its first
// row, rows per parity of the tables (a multiple of LR).
struct Col {
  int p, m, c, col, s, r0, NR;
};

// What a thread keeps of its rows of one system.
template <int LR> struct Seg {
  double b[LR];    // right-hand side, then the eliminated values, then the solution
  double r[LR];    // r_i of the tau rows
  double fv[LR];   // tapped explicit terms
  double mx[LR];   // stage 1: M X_n
};

// The global data of a system's right-hand side: explicit terms of the rows and
// their D neighbours on either side, accumulated right-hand sides.
template <int LR, int D> struct Loads {
  double w[LR + 2 * D], ri[LR];
};

// index of (row, component) in a table [2][NR][n][nmod]
template <int KIND> __device__ __forceinline__ size_t tix(const Grid& g, const Col& k, int row, int n, int j) {
  const size_t e = (size_t)(k.p * k.NR + row) * n + j;
  return KIND == KU ? e : e * g.nm + k.m;
}

// coefficients r0 - D .. r0 + LR + D - 1 of a state array (0 outside)
template <int LR, int D>
__device__ __forceinline__ void load_window(const Grid& g, const Col& k, int f, const double* A, double* w) {
#pragma unroll
  for (int i = 0; i < LR + 2 * D; ++i) {
    const int n = k.r0 - D + i;
    w[i] = (n >= 0 && n < g.nq) ? A[soff(g, f, 2 * n + k.p, k.m) + k.c] : 0.0;
  }
}
template <int LR, int D>
__device__ __forceinline__ void load_rhs(const Grid& g, const Col& k, int f, int stage, const double* F, const double* R,
                                         size_t S, Loads<LR, D>& ld) {
  load_window<LR, D>(g, k, f, F, ld.w);
#pragma unroll
  for (int i = 0; i < LR; ++i) {
    const int t = k.r0 - D + i;   // tau row
    ld.ri[i] = (stage > 1 && t >= 0 && t < g.nq - D) ? R[(size_t)(stage - 1) * S + soff(g, f, 2 * t + k.p, k.m) + k.c] : 0.0;
  }
}

// conversion taps of the explicit terms (S2, S4) and mass-matrix taps (S2, lap_k
// in C^(4)) of row i: sum over the 2 D + 1 coefficients around it
template <int KIND, int LR>
__device__ __forceinline__ double tap_f(const Grid& g, const Tables& tb, const Col& k, int i, const double* w) {
  constexpr int D = Sys<KIND>::D;
  const double* s = (KIND == KP ? tb.seg_s4 : tb.seg_s2) + (size_t)(k.p * k.NR + k.r0 + i) * (2 * D + 1);
  double v = 0.0;
#pragma unroll
  for (int j = 0; j <= 2 * D; ++j) v = fma(__ldg(s + j), w[i + j], v);
  return v;
}
template <int KIND, int LR>
__device__ __forceinline__ double tap_m(const Grid& g, const Tables& tb, const Col& k, int i, const double* w) {
  if (KIND != KP) return tap_f<KIND, LR>(g, tb, k, i, w);
  const double* s = tb.seg_mp + (size_t)(k.p * k.NR + k.r0 + i) * 5 * g.nm + k.m;
  double v = 0.0;
#pragma unroll
  for (int j = 0; j < 5; ++j) v = fma(__ldg(s + (size_t)j * g.nm), w[i + j], v);
  return v;
}

template <int KIND, int LR>
__device__ __forceinline__ void phase_a(const Grid& g, const Tables& tb, const Col& k, int stage, const double* X,
                                        Loads<LR, Sys<KIND>::D>& ld, const double* Ts, int W, double cpl, Seg<LR>& q) {
  constexpr int D = Sys<KIND>::D, NW = LR + 2 * D;
#pragma unroll
  for (int i = 0; i < LR; ++i) {
    const double v = tap_f<KIND, LR>(g, tb, k, i, ld.w);
    q.fv[i] = KIND == KP ? v : -v;
  }
  if (stage == 1) {
    load_window<LR, D>(g, k, KIND == KT ? 0 : 1, X, ld.w);
#pragma unroll
    for (int i = 0; i < LR; ++i) q.mx[i] = ld.ri[i] = tap_m<KIND, LR>(g, tb, k, i, ld.w);
  }
  const double a = __ldg(tb.dtae + stage * 5 + stage - 1);   // dt AE[stage][stage - 1]
#pragma unroll
  for (int i = 0; i < LR; ++i) q.b[i] = q.r[i] = fma(a, q.fv[i], ld.ri[i]);
  if (KIND == KP) {
    // + gamma dt (-i k Pr Ra) S4 T_i: the other part's column of T
    double w[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      const int n = k.r0 - D + i;
      w[i] = (n >= 0 && n < g.nq) ? Ts[n * W + (k.col ^ 1)] : 0.0;
    }
    const double ck = (k.c == 0 ? cpl : -cpl) * (g.kfac * k.m);
#pragma unroll
    for (int i = 0; i < LR; ++i) q.b[i] = fma(ck, tap_f<KP, LR>(g, tb, k, i, w), q.b[i]);
  }
}

// backward recurrence; phc, thc: this segment's responses of its first, last D rows for phases C, E
template <int KIND, int LR>
__device__ __forceinline__ void phase_b(const Grid& g, const Tables& tb, const Col& k, Seg<LR>& q, double* carry,
                                        double* phc, double* thc, int SW) {
  constexpr int D = Sys<KIND>::D;
  const SegFactors& f = Sys<KIND>::fac(tb);
#pragma unroll
  for (int j = 0; j < D; ++j)
#pragma unroll
    for (int i = 0; i < D; ++i) {
      phc[(j * D + i) * SW] = __ldg(f.phi + tix<KIND>(g, k, k.r0 + j, D, i));
      thc[(j * D + i) * SW] = __ldg(f.theta + tix<KIND>(g, k, k.r0 + LR - D + j, D, i));
    }
#pragma unroll
  for (int i = LR - 2; i >= 0; --i) {
    double v = q.b[i];
    if (D == 2 && i + 2 < LR) v = fma(-__ldg(f.beta + tix<KIND>(g, k, k.r0 + i, D, 1)), q.b[i + 2 < LR ? i + 2 : 0], v);
    q.b[i] = fma(-__ldg(f.beta + tix<KIND>(g, k, k.r0 + i, D, 0)), q.b[i + 1], v);
  }
#pragma unroll
  for (int j = 0; j < D; ++j) carry[j * SW] = q.b[j];
}

// one thread per column: what comes into each segment from the next one
template <int D>
__device__ __forceinline__ void phase_c(int S, int W, const double* carry, const double* phc, double* in, int SW) {
  double v[D];
#pragma unroll
  for (int j = 0; j < D; ++j) {
    v[j] = 0.0;
    in[j * SW + (S - 1) * W] = 0.0;
  }
#pragma unroll 4
  for (int s = S - 1; s > 0; --s) {
    double u[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
      u[j] = carry[j * SW + s * W];
#pragma unroll
      for (int i = 0; i < D; ++i) u[j] = fma(phc[(j * D + i) * SW + s * W], v[i], u[j]);
    }
#pragma unroll
    for (int j = 0; j < D; ++j) {
      v[j] = u[j];
      in[j * SW + (s - 1) * W] = v[j];
    }
  }
}

template <int KIND, int LR>
__device__ __forceinline__ void phase_d(const Grid& g, const Tables& tb, const Col& k, Seg<LR>& q, const double* in,
                                        double* bdp, double* carry, int SW) {
  constexpr int D = Sys<KIND>::D;
  const SegFactors& f = Sys<KIND>::fac(tb);
  double vi[D], bd[D];
#pragma unroll
  for (int j = 0; j < D; ++j) {
    vi[j] = in[j * SW];
    bd[j] = 0.0;
  }
#pragma unroll
  for (int i = 0; i < LR; ++i) {
    double v = q.b[i];
#pragma unroll
    for (int j = 0; j < D; ++j) v = fma(__ldg(f.phi + tix<KIND>(g, k, k.r0 + i, D, j)), vi[j], v);
#pragma unroll
    for (int j = 0; j < D; ++j) bd[j] = fma(-__ldg(f.multD + tix<KIND>(g, k, k.r0 + i, D, j)), v, bd[j]);
    // forward recurrence from zero: x_r = invd_r b_r - sum_j (invd_r Lb_r[j]) x_{r-D+j}
    v *= __ldg(f.invd + tix<KIND>(g, k, k.r0 + i, 1, 0));
    if (D == 2 && i >= 2) v = fma(-__ldg(f.ilb + tix<KIND>(g, k, k.r0 + i, D, 0)), q.b[i >= 2 ? i - 2 : 0], v);
    if (i >= 1) v = fma(-__ldg(f.ilb + tix<KIND>(g, k, k.r0 + i, D, D - 1)), q.b[i >= 1 ? i - 1 : 0], v);
    q.b[i] = v;
  }
#pragma unroll
  for (int j = 0; j < D; ++j) {
    bdp[j * SW] = bd[j];
    carry[j * SW] = q.b[LR - D + j];
  }
}

// one thread per column: boundary unknowns, then the values that come into each segment
template <int KIND>
__device__ __forceinline__ void phase_e(const Grid& g, const Tables& tb, const Col& k, int S, int W, const double* bdp,
                                        const double* carry, const double* thc, double* in, int SW) {
  constexpr int D = Sys<KIND>::D;
  const SegFactors& f = Sys<KIND>::fac(tb);
  double di[D * D], bd[D], v[D];
#pragma unroll
  for (int e = 0; e < D * D; ++e) {
    const size_t at = (size_t)k.p * D * D + e;
    di[e] = __ldg(f.Dinv + (KIND == KU ? at : at * g.nm + k.m));
  }
#pragma unroll
  for (int j = 0; j < D; ++j) {
    double a = 0.0, b = 0.0;   // two partial sums: shorter chain
    for (int s = 0; s + 1 < S; s += 2) {
      a += bdp[j * SW + s * W];
      b += bdp[j * SW + (s + 1) * W];
    }
    if (S & 1) a += bdp[j * SW + (S - 1) * W];
    bd[j] = a + b;
  }
  if (KIND == KT && k.m == 0 && k.c == 0) bd[0] += t_wall_rhs(g, k.p);
#pragma unroll
  for (int j = 0; j < D; ++j) {
    double x = 0.0;
#pragma unroll
    for (int i = 0; i < D; ++i) x = fma(di[j * D + i], bd[i], x);
    v[j] = x;
    in[j * SW] = x;
  }
#pragma unroll 4
  for (int s = 0; s < S - 1; ++s) {
    double u[D];
#pragma unroll
    for (int j = 0; j < D; ++j) {
      u[j] = carry[j * SW + s * W];
#pragma unroll
      for (int i = 0; i < D; ++i) u[j] = fma(thc[(j * D + i) * SW + s * W], v[i], u[j]);
    }
#pragma unroll
    for (int j = 0; j < D; ++j) {
      v[j] = u[j];
      in[j * SW + (s + 1) * W] = v[j];
    }
  }
}

template <int KIND, int LR>
__device__ __forceinline__ bool phase_f(const Grid& g, const Tables& tb, const Col& k, Seg<LR>& q, const double* in, int SW,
                                        double* xs, int W, double* Xo) {
  constexpr int D = Sys<KIND>::D;
  const SegFactors& f = Sys<KIND>::fac(tb);
  const int fd = KIND == KT ? 0 : 1;
  double vi[D];
#pragma unroll
  for (int j = 0; j < D; ++j) vi[j] = in[j * SW];
  bool ok = true;
#pragma unroll
  for (int i = 0; i < LR; ++i) {
    double v = q.b[i];
#pragma unroll
    for (int j = 0; j < D; ++j) v = fma(__ldg(f.theta + tix<KIND>(g, k, k.r0 + i, D, j)), vi[j], v);
    const int r = k.r0 + i;
    if (r < g.nq) {
      xs[r * W + k.col] = v;
      Xo[soff(g, fd, 2 * r + k.p, k.m) + k.c] = v;
      ok = ok && finite_bits(v);
    }
  }
  return ok;
}

// R_l += dt AE[l][stage-1] F + (AI[l][stage] / gamma) (M X_i - r_i) for the later stages l
template <int KIND, int LR>
__device__ __forceinline__ void phase_g(const Grid& g, const Tables& tb, const Col& k, int stage, const Seg<LR>& q,
                                        const double* xs, int W, double* R, size_t S) {
  constexpr int D = Sys<KIND>::D, NW = LR + 2 * D;
  const int f = KIND == KT ? 0 : 1;
  double w[NW];
#pragma unroll
  for (int i = 0; i < NW; ++i) {
    const int n = k.r0 - D + i;
    w[i] = (n >= 0 && n < g.nq) ? xs[n * W + k.col] : 0.0;
  }
  double lx[LR];
#pragma unroll
  for (int i = 0; i < LR; ++i) lx[i] = tap_m<KIND, LR>(g, tb, k, i, w) - q.r[i];
#pragma unroll
  for (int l = 2; l <= 4; ++l)
    if (l > stage && l <= g.ns) {
      const double ae = __ldg(tb.dtae + l * 5 + stage - 1), ai = __ldg(tb.dtae + 26 + l * 5 + stage);
      double* Rl = R + (size_t)(l - 1) * S;
      double old[LR];
#pragma unroll
      for (int i = 0; i < LR; ++i) {
        const int t = k.r0 - D + i;
        old[i] = stage == 1 ? q.mx[i] : (t >= 0 && t < g.nq - D) ? Rl[soff(g, f, 2 * t + k.p, k.m) + k.c] : 0.0;
      }
#pragma unroll
      for (int i = 0; i < LR; ++i) {
        const int t = k.r0 - D + i;
        if (t >= 0 && t < g.nq - D) Rl[soff(g, f, 2 * t + k.p, k.m) + k.c] = fma(ai, lx[i], fma(ae, q.fv[i], old[i]));
      }
    }
}

template <int LR>
__global__ void __launch_bounds__(512) k_solve_seg(Grid g, Tables tb, double* X, double* Xs, const double* F, double* R,
                                                   size_t S, const double* wT, double* nu, int* flags, int* err, int B,
                                                   int stage, int tms, const double* ra, const int* nsteps,
                                                   const int* step) {
  extern __shared__ double sbuf[];
  pdl_wait();
  const int stepidx = nsteps ? *step : 0;
  const int mt = (g.nm + tms - 1) / tms;
  const int b = blockIdx.x / (2 * mt), rem = blockIdx.x - b * 2 * mt;
  const int p = rem / mt, m0 = (rem - p * mt) * tms;
  if (b >= B || !(nsteps == nullptr || stepidx < nsteps[b])) return;   // uniform per block
  // a transform of this state gave up waiting (the tensor-core kernels): leave
  // the state as it was at the start of the failing step
  if (flags[b] & kFlagTimeout) return;
  const int nq = g.nq, W = 2 * tms, NS = (nq + LR - 1) / LR, SW = NS * W;
  const int lw = __ffs(W) - 1;
  double* Tx = sbuf;                 // [nq][W] T_i, then kept for the coupling
  double* Px = Tx + (size_t)nq * W;  // [nq][W] psi or U
  double* carry = Px + (size_t)nq * W;   // [2][NS][W]
  double* in = carry + 2 * SW;           // [2][NS][W]
  double* bdp = in + 2 * SW;             // [2][NS][W]
  double* phc = bdp + 2 * SW;            // [4][NS][W] responses of the segments' first rows
  double* thc = phc + 4 * SW;            // [4][NS][W] and of their last rows
  double* X0 = X + (size_t)b * S;
  double* Xo = (stage == g.ns) ? X0 : Xs + (size_t)b * S;   // stiffly accurate: last stage = new state
  const double* Fb = F + (size_t)b * S;
  double* Rb = R + (size_t)b * 4 * S;
  const double cpl = __ldg(tb.dtae + 25) * (ra ? ra[b] : g.Ra);   // ((gamma dt) Pr) Ra
  if (stage == 1 && m0 == 0 && p == 1 && threadIdx.x < 32 && nu != nullptr) {
    // Nu_V(t_n) (Eq. 9) of the step-start state, as in k_solve; the odd
    // coefficients read here belong to this block, which overwrites them only
    // after the barriers below (a one-stage scheme writes X0 here)
    const int lane = threadIdx.x;
    double cond = 0.0, adv = 0.0;
    for (int n = 2 * lane + 1; n < g.Nz; n += 64) cond -= 2.0 * *(X0 + soff(g, 0, n, 0));
    for (int jz = lane; jz < g.Mz; jz += 32) adv = fma(__ldg(tb.cc + jz), *(wT + (size_t)b * g.Mz + jz), adv);
#pragma unroll
    for (int sh = 16; sh > 0; sh >>= 1) {
      cond += __shfl_down_sync(0xffffffffu, cond, sh);
      adv += __shfl_down_sync(0xffffffffu, adv, sh);
    }
    if (lane == 0) nu[b] += ((stepidx == 0) ? 0.5 : 1.0) * g.dt * (cond + 0.5 * adv);
  }
  Col k;
  k.p = p;
  k.s = threadIdx.x >> lw;
  k.col = threadIdx.x & (W - 1);
  k.m = m0 + k.col / 2;
  k.c = k.col & 1;
  k.r0 = k.s * LR;
  k.NR = NS * LR;
  const bool on = k.s < NS && k.m < g.nm;
  const int at = k.s * W + k.col;   // (segment, column) of the exchange arrays
  bool ok = true;
  Seg<LR> q;
  Loads<LR, 1> lt;
  Loads<LR, 2> lp;   // also the mean flow's, one row further in
  // short segments: all global reads of both systems at once (one latency)
  constexpr bool kAhead = LR <= 4;
  if (on) {
    load_rhs<LR, 1>(g, k, 0, stage, Fb, Rb, S, lt);
    if (kAhead && k.m != 0) load_rhs<LR, 2>(g, k, 1, stage, Fb, Rb, S, lp);
  }
  auto system = [&](auto kind_m, auto kind_0) {
    constexpr int K = decltype(kind_m)::value, K0 = decltype(kind_0)::value;   // m >= 1, m = 0
    double* xs = K == KT ? Tx : Px;
    const bool zero = K != K0 && k.m == 0;
    if (on) {
      if (zero) {
        load_rhs<LR, 1>(g, k, 1, stage, Fb, Rb, S, lt);
        phase_a<K0, LR>(g, tb, k, stage, X0, lt, Tx, W, cpl, q);
        phase_b<K0, LR>(g, tb, k, q, carry + at, phc + at, thc + at, SW);
      } else {
        if constexpr (K == KT) {
          phase_a<K, LR>(g, tb, k, stage, X0, lt, Tx, W, cpl, q);
        } else {
          if (!kAhead) load_rhs<LR, 2>(g, k, 1, stage, Fb, Rb, S, lp);
          phase_a<K, LR>(g, tb, k, stage, X0, lp, Tx, W, cpl, q);
        }
        phase_b<K, LR>(g, tb, k, q, carry + at, phc + at, thc + at, SW);
      }
    }
    __syncthreads();
    if (on && k.s == 0) {
      if (zero)
        phase_c<Sys<K0>::D>(NS, W, carry + k.col, phc + k.col, in + k.col, SW);
      else
        phase_c<Sys<K>::D>(NS, W, carry + k.col, phc + k.col, in + k.col, SW);
    }
    __syncthreads();
    if (on) {
      if (zero)
        phase_d<K0, LR>(g, tb, k, q, in + at, bdp + at, carry + at, SW);
      else
        phase_d<K, LR>(g, tb, k, q, in + at, bdp + at, carry + at, SW);
    }
    __syncthreads();
    if (on && k.s == 0) {
      if (zero)
        phase_e<K0>(g, tb, k, NS, W, bdp + k.col, carry + k.col, thc + k.col, in + k.col, SW);
      else
        phase_e<K>(g, tb, k, NS, W, bdp + k.col, carry + k.col, thc + k.col, in + k.col, SW);
    }
    __syncthreads();
    if (on) {
      const bool o = zero ? phase_f<K0, LR>(g, tb, k, q, in + at, SW, xs, W, Xo) : phase_f<K, LR>(g, tb, k, q, in + at, SW, xs, W, Xo);
      ok = ok && o;
    }
    __syncthreads();
    if (on && stage < g.ns) {
      if (zero)
        phase_g<K0, LR>(g, tb, k, stage, q, xs, W, Rb, S);
      else
        phase_g<K, LR>(g, tb, k, stage, q, xs, W, Rb, S);
    }
  };
  system(std::integral_constant<int, KT>(), std::integral_constant<int, KT>());
  system(std::integral_constant<int, KP>(), std::integral_constant<int, KU>());
  if (!ok) {
    atomicOr(flags + b, kFlagNonFinite);
    atomicOr(err, kFlagNonFinite);
  }
}

size_t seg_smem(const Grid& g, int tms) {
  const int LR = solve_seg_rows(g.nq), NS = (g.nq + LR - 1) / LR;
  return ((size_t)2 * g.nq + 14 * NS) * 2 * tms * sizeof(double);
}
int seg_threads(const Grid& g, int tms) {
  const int LR = solve_seg_rows(g.nq), NS = (g.nq + LR - 1) / LR;
  return (NS * 2 * tms + 31) / 32 * 32;
}

// Modes per block: as many as fill 256 threads, fewer while the launch would
// leave SMs without two blocks (a state alone spreads over them).
int seg_tile(const Grid& g, int B) {
  int tms = 16;
  while (tms > 1 && (seg_threads(g, tms) > 256 || (long)B * 2 * ((g.nm + tms - 1) / tms) < 2L * 152)) tms >>= 1;
  return tms;
}

template <int LR>
cudaError_t launch_seg(const Grid& g, const Tables& t, const Work& w, double* X, int B, int stage, double* nu, int tms,
                       cudaStream_t s) {
  const int mt = (g.nm + tms - 1) / tms;
  return launch_pdl(w.pdl != 0, k_solve_seg<LR>, (unsigned)(B * 2 * mt), seg_threads(g, tms), seg_smem(g, tms), s, g, t, X,
                    w.Xs, w.F, w.R, state_doubles(g), w.wT, nu, w.flags, w.err, B, stage, tms, w.ra, w.nsteps, w.step);
}

}  // namespace

cudaError_t configure_solve_seg(const Grid& g) {
  (void)g;
  cudaError_t e = cudaSuccess;
  auto allow = [&](auto* fn) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  };
  allow(k_solve_seg<4>);
  allow(k_solve_seg<8>);
  return e;
}

cudaError_t launch_solve_seg(const Grid& g, const Tables& t, const Work& w, double* X, int B, int stage, double* nu,
                             cudaStream_t s) {
  int tms = (w.shapes && w.shapes->solve_tms > 0) ? w.shapes->solve_tms : seg_tile(g, B);
  while (tms > 1 && (seg_threads(g, tms) > 512 || seg_smem(g, tms) > 200 * 1024)) tms >>= 1;   // pinned tiles of the largest grids
  if (solve_seg_rows(g.nq) == 4) return launch_seg<4>(g, t, w, X, B, stage, nu, tms, s);
  return launch_seg<8>(g, t, w, X, B, stage, nu, tms, s);
}

}  // namespace rbc
