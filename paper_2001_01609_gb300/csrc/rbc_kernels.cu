// CUDA kernels of the fine/coarse propagator for sm_103a.
//
// One RK443 stage (Sec. 3.2, Sec. 3.6) of B batched time slices is four
// launches:
//   z inverse  Chebyshev coefficients -> fields at the 3/2-padded Lobatto points,
//              with the Fourier-mode factors ik (k_zinv; mixed from Nz = 64:
//              rbc_tcgen05.cu);
//   rows       per padded z-row: packed inverse real FFTs in x, advective products,
//              one packed forward FFT, truncation to the kept modes, x-means
//              (FP64: rbc_rows_f64.cu; mixed: rbc_rows_f32.cu);
//   z forward  the products to T coefficients n < Nz (files as the inverse; k_zfwd);
//   solve      per (slice, Fourier mode, Chebyshev parity): RK443 right-hand
//              side in tau rows, solve of the implicit system (temperature first,
//              then streamfunction with the implicit buoyancy coupling), RK
//              accumulator updates, Nu_V accumulation (small grids: k_solve_dense;
//              else k_solve; FP64 in both modes).
// Here also: the step loop's counters, diagnostics, statistics, transfers between
// grids, norms and the Parareal correction.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdint>
#include <cstring>
#include <type_traits>

#include "rbc_internal.h"

namespace rbc {

// IMEX Runge-Kutta pairs of Ascher, Ruuth & Spiteri (1997), [scheme][i][j]:
// coefficient of stage j in stage i, stage 0 explicit, zero-padded to 5 x 5.
// RK443 is the paper's (Sec. 3.2, Sec. 3.6); ARS(2,2,2) and ARS(1,1,1) are the
// lower-order coarse steppers of Sec. 3.6.  Filled by upload_schemes().
__constant__ double c_AE[3][5][5];
__constant__ double c_AI[3][5][5];

void scheme_tableau(int scheme, double AE[5][5], double AI[5][5], int* ns, double* gamma) {
  for (int i = 0; i < 5; ++i)
    for (int j = 0; j < 5; ++j) AE[i][j] = AI[i][j] = 0.0;
  if (scheme == RBC_RK222) {
    // gamma = 1 - 1/sqrt(2): second order and L-stable; delta = 1 - 1/(2 gamma)
    const double gm = 1.0 - 1.0 / std::sqrt(2.0), dl = 1.0 - 1.0 / (2.0 * gm);
    AI[1][1] = gm;
    AI[2][1] = 1.0 - gm;
    AI[2][2] = gm;
    AE[1][0] = gm;
    AE[2][0] = dl;
    AE[2][1] = 1.0 - dl;
    *ns = 2;
    *gamma = gm;
  } else if (scheme == RBC_RK111) {
    // explicit Euler for the nonlinear terms, implicit Euler for the linear ones
    AI[1][1] = 1.0;
    AE[1][0] = 1.0;
    *ns = 1;
    *gamma = 1.0;
  } else {
    const double ae[5][5] = {{0, 0, 0, 0, 0},
                             {1.0 / 2, 0, 0, 0, 0},
                             {11.0 / 18, 1.0 / 18, 0, 0, 0},
                             {5.0 / 6, -5.0 / 6, 1.0 / 2, 0, 0},
                             {1.0 / 4, 7.0 / 4, 3.0 / 4, -7.0 / 4, 0}};
    const double ai[5][5] = {{0, 0, 0, 0, 0},
                             {0, 1.0 / 2, 0, 0, 0},
                             {0, 1.0 / 6, 1.0 / 2, 0, 0},
                             {0, -1.0 / 2, 1.0 / 2, 1.0 / 2, 0},
                             {0, 3.0 / 2, -3.0 / 2, 1.0 / 2, 1.0 / 2}};
    for (int i = 0; i < 5; ++i)
      for (int j = 0; j < 5; ++j) {
        AE[i][j] = ae[i][j];
        AI[i][j] = ai[i][j];
      }
    *ns = 4;
    *gamma = 0.5;
  }
}


cudaError_t upload_schemes() {
  double ae[3][5][5], ai[3][5][5];
  for (int sc = 0; sc < 3; ++sc) {
    int ns;
    double gm;
    scheme_tableau(sc, ae[sc], ai[sc], &ns, &gm);
  }
  cudaError_t e = cudaMemcpyToSymbol(c_AE, ae, sizeof(ae));
  if (e == cudaSuccess) e = cudaMemcpyToSymbol(c_AI, ai, sizeof(ai));
  return e;
}

__device__ __forceinline__ double2 ld2(const double* p) { return *reinterpret_cast<const double2*>(p); }
__device__ __forceinline__ void st2(double* p, double2 v) { *reinterpret_cast<double2*>(p) = v; }
__device__ __forceinline__ double2 operator+(double2 a, double2 b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ double2 operator-(double2 a, double2 b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ double2 operator*(double s, double2 a) { return make_double2(s * a.x, s * a.y); }
// Roundings written out (explicit fma): the bits do not depend on how the
// compiler would contract a*b + c*d in each kernel that inlines this.
__device__ __forceinline__ double2 cmul(double2 a, double2 b) {
  return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ double2 conj2(double2 a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ double2 times_i(double2 a) { return make_double2(-a.y, a.x); }

// Complex element (f, n, m) of a state, in doubles.
__device__ __forceinline__ size_t soff(const Grid& g, int f, int n, int m) {
  return ((size_t)(f * g.Nz + n) * g.nm + m) * 2;
}

__device__ __forceinline__ bool slice_active_at(const int* nsteps, int stepidx, int b) {
  return nsteps == nullptr || stepidx < nsteps[b];
}


// ---------------------------------------------------------------------------
// Real-type generic complex helpers for the transform kernels, which run in
// FP64 (RBC_FP64) or in FP32 (RBC_MIXED); the state, the explicit terms F and
// the stage solve stay FP64 in both modes.
// ---------------------------------------------------------------------------
template <typename T> struct Cx;
template <> struct Cx<double> { using t = double2; };
template <> struct Cx<float> { using t = float2; };
template <typename T> using C2 = typename Cx<T>::t;

__device__ __forceinline__ float2 operator+(float2 a, float2 b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ float2 operator-(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ float2 operator*(float s, float2 a) { return make_float2(s * a.x, s * a.y); }
__device__ __forceinline__ float2 cmul(float2 a, float2 b) {
  return make_float2(fmaf(a.x, b.x, -(a.y * b.y)), fmaf(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ float2 conj2(float2 a) { return make_float2(a.x, -a.y); }
__device__ __forceinline__ float2 times_i(float2 a) { return make_float2(-a.y, a.x); }

template <typename T> __device__ __forceinline__ C2<T> mk2(T x, T y);
template <> __device__ __forceinline__ double2 mk2<double>(double x, double y) { return make_double2(x, y); }
template <> __device__ __forceinline__ float2 mk2<float>(float x, float y) { return make_float2(x, y); }
template <typename T> __device__ __forceinline__ C2<T> ldc(const T* p) { return *reinterpret_cast<const C2<T>*>(p); }
template <typename T> __device__ __forceinline__ void stc(T* p, C2<T> v) { *reinterpret_cast<C2<T>*>(p) = v; }
template <typename T> __device__ __forceinline__ C2<T> cvt2(double2 a) { return mk2<T>((T)a.x, (T)a.y); }

// ---------------------------------------------------------------------------
// z inverse transform (k_zinv).  Block per (slice, padded row pair j / Mz-1-j,
// tile of 32 modes) with kp warps; warp w accumulates the coefficients n of its
// share of [0, Nz), and the kp partial sums are added in a fixed order.
// Even/odd split: the padded points are symmetric, s_{Mz-1-j} = -s_j, and
// T_n^(q)(-s) = (-1)^(n+q) T_n^(q)(s), so the sums E, O over even and odd n at
// s_j give f^(q)(s_j) = E + O and f^(q)(-s_j) = (-1)^q (E - O): half the
// multiply-adds of evaluating both rows.  psi-slot operators V, VD, VD^2, VD^3
// (d/ds) and T-slot V, VD; the epilogue forms, with d/dz = 2 d/ds, d/dx = ik:
//   u = d_z psi (m = 0: U),  w = -ik psi,  d_x omega, d_z omega (omega = -lap psi,
//   m = 0: omega = -U'),  d_x u,  d_z u,  T,  d_x T,  d_z T.
// Output Z[b][field][j][m] (complex, real type T), fields in that order.
// ---------------------------------------------------------------------------
// Field f (0..8, as listed above) of one output point from the operator sums
// P[q] = d^q psi / ds^q (q < 4), t0 = T, t1 = dT/ds.  The roundings are written
// out (explicit fma), so every kernel that forms a field gets the same bits.
template <typename T>
__device__ __forceinline__ C2<T> zinv_field(int f, int m, T k, const C2<T>* P, C2<T> t0, C2<T> t1) {
  using V = C2<T>;
  const T zero = 0;
  const V z = mk2<T>(zero, zero);
  switch (f) {
    case 0: return m == 0 ? mk2<T>(P[0].x, zero) : (T)2 * P[1];                 // u (m = 0: U)
    case 1: return m == 0 ? z : -k * times_i(P[0]);                             // w = -ik psi
    case 2: {                                                                   // d_x omega
      if (m == 0) return z;
      const T kk = k * k;                                                       // omega = k^2 psi - 4 d2(psi)
      const V om = mk2<T>(fma(kk, P[0].x, (T)-4 * P[2].x), fma(kk, P[0].y, (T)-4 * P[2].y));
      return k * times_i(om);
    }
    case 3: {                                                                   // d_z omega
      if (m == 0) return mk2<T>((T)-4 * P[2].x, zero);
      const T kk2 = ((T)2 * k) * k;                                             // 2 k^2 d(psi) - 8 d3(psi)
      return mk2<T>(fma(kk2, P[1].x, (T)-8 * P[3].x), fma(kk2, P[1].y, (T)-8 * P[3].y));
    }
    case 4: return m == 0 ? z : k * times_i((T)2 * P[1]);                       // d_x u
    case 5: return m == 0 ? mk2<T>((T)2 * P[1].x, zero) : (T)4 * P[2];          // d_z u
    case 6: return t0;                                                          // T
    case 7: return m == 0 ? z : k * times_i(t0);                                // d_x T
    case 8: return (T)2 * t1;                                                   // d_z T
    default: return z;
  }
}

// Fields of one output row (j, m); half = 0: fields 0-3, 1: fields 4-8, -1: all.
template <typename T>
__device__ __forceinline__ void zinv_store(const Grid& g, T* Zb, int j, int m, T k, const C2<T>* P, C2<T> t0,
                                           C2<T> t1, int half) {
  const size_t fs = (size_t)g.Mz * g.nm * 2;
  T* zb = Zb + ((size_t)j * g.nm + m) * 2;
  const int f0 = half == 1 ? 4 : 0, f1 = half == 0 ? 4 : 9;
  for (int f = f0; f < f1; ++f) stc<T>(zb + f * fs, zinv_field<T>(f, m, k, P, t0, t1));
}

template <typename T>
__device__ __forceinline__ void zinv_item(const Grid& g, const T* __restrict__ Bz, const double* __restrict__ X, size_t S,
                          T* __restrict__ Z, int B, const int* nsteps, const int* step, int blk, int kp) {
  using V = C2<T>;
  extern __shared__ __align__(16) unsigned char zsm[];
  V* part = reinterpret_cast<V*>(zsm);                 // [kp][12][32] when kp > 1
  const int Mh = (g.Mz + 1) / 2;
  const int mt = (g.nm + 31) / 32;
  const int b = blk / (Mh * mt);
  const int rem = blk - b * Mh * mt;
  const int j = rem / mt, m0 = (rem - j * mt) * 32;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int m = m0 + lane;
  const bool valid = m < g.nm;
  const bool wact = w < kp;                            // warps beyond kp, if any, idle
  const double* Xb = X + (size_t)b * S;
  const T* bq[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) bq[q] = Bz + (size_t)(q * g.Mz + j) * g.Nz;
  // share of the coefficient pairs (n, n+1) of this warp
  const int npair = g.Nz / 2;
  const int per = (npair + kp - 1) / kp;
  const int p0 = w * per, p1 = min(npair, p0 + per);
  if (kp > 1 && B <= kPdlMaxBatch && lane < 4) {   // table entries into L1 while the launch before this one finishes
    float t;
    asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(t) : "l"(Bz + (size_t)(lane * g.Mz + j) * g.Nz + min(2 * p0, g.Nz - 1)));
  }
  pdl_wait();
  // a state or two alone look at whether they are active once their values are on their
  // way; in a batch the blocks hide each other's latency, and states that have taken
  // their steps shall cost nothing (64 x 32, 23 states of 0 to 9 steps, all launches in
  // FP64: 2904 us, 3121 with the values of all states loaded first; even steps alike)
  const int now = nsteps ? *step : 0, last = nsteps ? nsteps[b] : 1;   // (the grid is exact: b < B)
  if ((kp == 1 || B > kPdlMaxBatch) && now >= last) return;
  V E[6], O[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) E[q] = O[q] = mk2<T>(0, 0);
  if (valid && wact) {
#pragma unroll 4
    for (int pp = p0; pp < p1; ++pp) {
      const int n = 2 * pp;
#pragma unroll
      for (int par = 0; par < 2; ++par) {
        const V xp = cvt2<T>(ld2(Xb + soff(g, 1, n + par, m)));
        const V xt = cvt2<T>(ld2(Xb + soff(g, 0, n + par, m)));
        V* A = par ? O : E;
        T v[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) v[q] = __ldg(bq[q] + n + par);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          A[q].x = fma(v[q], xp.x, A[q].x);
          A[q].y = fma(v[q], xp.y, A[q].y);
        }
        A[4].x = fma(v[0], xt.x, A[4].x);
        A[4].y = fma(v[0], xt.y, A[4].y);
        A[5].x = fma(v[1], xt.x, A[5].x);
        A[5].y = fma(v[1], xt.y, A[5].y);
      }
    }
  }
  if (now >= last) return;   // uniform per block
  const T k = (T)(g.kfac * m);
  T* Zb = Z + (size_t)b * 9 * g.Mz * g.nm * 2;
  const int jr = g.Mz - 1 - j;
  if (kp > 1) {
    if (wact) {
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        part[(w * 12 + q) * 32 + lane] = E[q];
        part[(w * 12 + 6 + q) * 32 + lane] = O[q];
      }
    }
    __syncthreads();
    // accumulator a (E_0..5, O_0..5) is summed by warp a % kp, over the warps'
    // partial sums in warp order, into the first warp's slot
    for (int a = w; a < 12; a += kp) {
      V e = part[a * 32 + lane];
      for (int ww = 1; ww < kp; ++ww) e = e + part[(ww * 12 + a) * 32 + lane];
      part[a * 32 + lane] = e;
    }
    __syncthreads();
    if (!valid) return;
    // epilogue: warps take (row, half of the fields); with 2 warps one row each
    const int nt = kp >= 4 ? 4 : kp;
    for (int task = w; task < 4; task += nt) {
      const int row = task & 1, half = task >> 1;
      if (row == 1 && jr == j) continue;
      V Ev[6], Ov[6];
#pragma unroll
      for (int q = 0; q < 6; ++q) {
        Ev[q] = part[q * 32 + lane];
        Ov[q] = part[(6 + q) * 32 + lane];
      }
      V P[4];
      if (row == 0) {
#pragma unroll
        for (int q = 0; q < 4; ++q) P[q] = Ev[q] + Ov[q];
        zinv_store<T>(g, Zb, j, m, k, P, Ev[4] + Ov[4], Ev[5] + Ov[5], half);
      } else {
#pragma unroll
        for (int q = 0; q < 4; ++q) P[q] = ((q & 1) ? (T)-1 : (T)1) * (Ev[q] - Ov[q]);
        zinv_store<T>(g, Zb, jr, m, k, P, Ev[4] - Ov[4], (T)-1 * (Ev[5] - Ov[5]), half);
      }
    }
    return;
  }
  if (w != 0 || !valid) return;
  V P[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) P[q] = E[q] + O[q];
  zinv_store<T>(g, Zb, j, m, k, P, E[4] + O[4], E[5] + O[5], -1);
  if (jr != j) {
#pragma unroll
    for (int q = 0; q < 4; ++q) P[q] = ((q & 1) ? (T)-1 : (T)1) * (E[q] - O[q]);
    zinv_store<T>(g, Zb, jr, m, k, P, E[4] - O[4], (T)-1 * (E[5] - O[5]), -1);
  }
}

template <typename T>
__global__ void __launch_bounds__(256) k_zinv(Grid g, const T* __restrict__ Bz, const double* __restrict__ X, size_t S,
                                              T* __restrict__ Z, int B, const int* nsteps, const int* step) {
  zinv_item<T>(g, Bz, X, S, Z, B, nsteps, step, blockIdx.x, blockDim.x / 32);
}

// Warps sharing the coefficient sum of one k_zinv row pair.  It fixes the order
// of the floating-point additions, so it depends on the grid only (every batch
// size gives the same bits): small grids, whose single-state launches are
// latency-bound, split the sum over up to 8 warps; large grids keep one warp.
static int zinv_warps(const Grid& g) {
  if ((long)g.Nx * g.Nz > 8192) return 1;
  int kp = 1;
  while (kp < 8 && (g.Nz / 2) / (2 * kp) >= 2) kp *= 2;
  return kp;
}

// Deterministic block sum: the fixed tree red[t] += red[t + s], s = blockDim/2
// down to 1 (blockDim a power of two, at least 32).  Levels s >= 32 go through
// shared memory, the last five through warp shuffles with the same pairings.
__device__ double block_sum(double v, double* red) {
  red[threadIdx.x] = v;
  __syncthreads();
  for (int s = blockDim.x / 2; s >= 32; s >>= 1) {
    if ((int)threadIdx.x < s) red[threadIdx.x] += red[threadIdx.x + s];
    __syncthreads();
  }
  if (threadIdx.x < 32) {
    double x = red[threadIdx.x];
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) x += __shfl_down_sync(0xffffffffu, x, s);
    if (threadIdx.x == 0) red[0] = x;
  }
  __syncthreads();
  const double r = red[0];
  __syncthreads();
  return r;
}

// ---------------------------------------------------------------------------
// z forward transform (k_zfwd): F[b][f][n][m] = sum_j W[n][j] Q[b][f][j][m], n < Nz.
// W[n][Mz-1-j] = (-1)^n W[n][j] (symmetric points), so with the folds
// Ev_j = Q_j + Q_{Mz-1-j}, Od_j = Q_j - Q_{Mz-1-j} (the middle row, for odd Mz,
// once in Ev) F_n = sum_{j < ceil(Mz/2)} W[n][j] (n even ? Ev : Od)_j.  Block per
// (slice, field, tile of tm modes, chunk of the n range): the folds are staged
// in shared memory once per block and reused by every n of the chunk.  F is
// written in FP64 for the stage solve.
// ---------------------------------------------------------------------------
template <typename T>
__device__ __forceinline__ void zfwd_item(const Grid& g, const T* __restrict__ W, const T* __restrict__ Q, double* __restrict__ F,
                          size_t S, int B, int tm, int nch, const int* nsteps, const int* step, int blk) {
  using V = C2<T>;
  extern __shared__ __align__(16) unsigned char fsm[];
  V* fold = reinterpret_cast<V*>(fsm);                 // [2][Mh][tm]
  const int Mh = (g.Mz + 1) / 2;
  const int mt = (g.nm + tm - 1) / tm;
  const int per_b = 2 * mt * nch;
  const int b = blk / per_b;
  int rem = blk - b * per_b;
  const int ch = rem % nch;
  rem /= nch;
  const int f = rem / mt, m0 = (rem - f * mt) * tm;
  const int ng = blockDim.x >> (__ffs(tm) - 1);
  const int mi = threadIdx.x & (tm - 1), n0 = threadIdx.x / tm;
  const int nper = (g.Nz + nch - 1) / nch;
  const int nlo = ch * nper, nhi = min(g.Nz, nlo + nper);
  if (B <= kPdlMaxBatch) {   // the first table row into L1 while the launch before this one finishes
    float t;
    const T* wr = W + (size_t)min(nlo + n0, g.Nz - 1) * g.Mz;
    for (int jh = mi * 32; jh < Mh; jh += tm * 32) asm volatile("ld.global.nc.f32 %0, [%1];" : "=f"(t) : "l"(wr + jh));
  }
  pdl_wait();
  const int now = nsteps ? *step : 0, last = nsteps ? nsteps[b] : 1;   // (the grid is exact: b < B)
  if (B > kPdlMaxBatch && now >= last) return;                         // as in zinv_item
  const size_t qs = (size_t)g.Mz * g.nm * 2;
  const T* q = Q + (size_t)(b * 2 + f) * qs;
  const int ltm = __ffs(tm) - 1;             // tm is a power of two
  for (int it = threadIdx.x; it < Mh * tm; it += blockDim.x) {
    const int jh = it >> ltm, mi = it & (tm - 1), m = m0 + mi;
    V ev = mk2<T>(0, 0), od = mk2<T>(0, 0);
    if (m < g.nm) {
      const V a = ldc<T>(q + ((size_t)jh * g.nm + m) * 2);
      const int jr = g.Mz - 1 - jh;
      if (jr != jh) {
        const V c = ldc<T>(q + ((size_t)jr * g.nm + m) * 2);
        ev = a + c;
        od = a - c;
      } else {
        ev = a;
      }
    }
    fold[(size_t)jh * tm + mi] = ev;
    fold[(size_t)(Mh + jh) * tm + mi] = od;
  }
  if (now >= last) return;   // uniform per block
  __syncthreads();
  const int m = m0 + mi;
  if (m >= g.nm) return;
  for (int n = nlo + n0; n < nhi; n += ng) {
    const V* src = fold + (size_t)((n & 1) ? Mh : 0) * tm + mi;
    const T* wr = W + (size_t)n * g.Mz;
    V acc = mk2<T>(0, 0);
#pragma unroll 4
    for (int jh = 0; jh < Mh; ++jh) {
      const T wv = __ldg(wr + jh);
      const V v = src[(size_t)jh * tm];
      acc.x = fma(wv, v.x, acc.x);
      acc.y = fma(wv, v.y, acc.y);
    }
    st2(F + (size_t)b * S + soff(g, f, n, m), make_double2((double)acc.x, (double)acc.y));
  }
}

template <typename T>
__global__ void k_zfwd(Grid g, const T* __restrict__ W, const T* __restrict__ Q, double* __restrict__ F, size_t S,
                       int B, int tm, int nch, const int* nsteps, const int* step) {
  zfwd_item<T>(g, W, Q, F, S, B, tm, nch, nsteps, step, blockIdx.x);
}

static int zfwd_tile(const Grid& g, int B, size_t es) {
  const int Mh = (g.Mz + 1) / 2;
  int tm = 32;
  while (tm > 1 && (size_t)B * 2 * ((g.nm + tm - 1) / tm) < 2 * 152) tm >>= 1;
  while (tm > 4 && (size_t)2 * Mh * tm * 2 * es > 200 * 1024) tm >>= 1;
  return tm;
}
static int zfwd_chunks(const Grid& g, int B, int tm) {
  const long blocks = (long)B * 2 * ((g.nm + tm - 1) / tm);
  int nch = 1;
  while (nch < 8 && blocks * nch < 4L * 152 && g.Nz / (2 * nch) >= 128 / tm) nch *= 2;
  return nch;
}
static size_t zfwd_smem(const Grid& g, int B, size_t es) {
  return (size_t)2 * ((g.Mz + 1) / 2) * zfwd_tile(g, B, es) * 2 * es;
}

// ---------------------------------------------------------------------------
// Stage solve (k_solve) of grids with nq > kDenseSolveMaxNq (smaller grids:
// k_solve_dense).  Block per (slice,
// Chebyshev parity p, tile of tms Fourier modes); a column is one (mode m,
// real/imaginary part c) pair -- the stage matrices are real, so the two parts
// are independent systems except for the implicit buoyancy coupling -i k Pr Ra T
// (the imaginary part of T feeds the real part of psi and vice versa).  Per
// system (T first, then psi for m >= 1 or the mean flow U for m = 0):
//   phase 1 (all threads, NB consecutive tau rows of one column each): right-hand
//           side of the stage, updates of the later RK accumulators;
//   phase 2 (one warp, a column per lane): backward elimination with the UL
//           factors;
//   phase 3 (same warp): boundary block, forward substitution;
//   phase 4 (all threads): the solution to memory, dt L X_i = (M X_i - r_i) / gamma
//           into the later accumulators.
// In phases 2 and 3 a second warp copies the factors of RC steps at a time into
// shared memory, two chunks ahead, and sums the boundary rows one chunk behind;
// a third solves the mean flow of the tile that holds mode 0.  The temperature's
// and the second system's values share one array of nq + 2 rows of 2 tms doubles:
// row i of the latter lies two rows lower, in rows that phase 1, going up, has
// read.  A second array, or (RG) this stage's accumulator, which phase 1 has read,
// holds r_i.
//
// Bound: the FP64 pipe (2 operations per clock and SM) when blocks fill it, else
// the recurrences: ten dependent warp instructions of 64 clocks per row.
// Measured (GB300, per launch; before, all rows' factors from L2 by the recurring
// warp, three arrays and 256 threads of 125 registers, two blocks per SM; same
// bits): 1024 x 256, 32 states 1650 -> 1042 us, one state 240 -> 103 us; 512 x 128,
// 64 states 810 -> 515 us, 3 states 154 -> 64 us; 256 x 64, 32 states 137 -> 100 us,
// 8 states 83 -> 42 us, one state 37 -> 28 us.  Recurrences in segments on all warps
// took 922, 46, 87, 32 and 24 us (1024 x 256 with 32 states; 512 x 128 with 3; 256 x
// 64 with 32, 8, 1) and are not used: their roundings differ, and a mixed step or the
// defect of a converging Parareal run turns that into differences of the size of its
// own error.
// ---------------------------------------------------------------------------
enum { KT = 0, KP = 1, KU = 2 };

template <int KIND>
struct Sys {
  static constexpr int D = (KIND == KP) ? 2 : 1;
  static constexpr int LAM = 2 * D;
  static __device__ __forceinline__ const double* multB(const Tables& tb) {
    return KIND == KT ? tb.T_multB : KIND == KP ? tb.P_multB : tb.U_multB;
  }
  static __device__ __forceinline__ const double* multD(const Tables& tb) {
    return KIND == KT ? tb.T_multD : KIND == KP ? tb.P_multD : tb.U_multD;
  }
  static __device__ __forceinline__ const double* Dinv(const Tables& tb) {
    return KIND == KT ? tb.T_Dinv : KIND == KP ? tb.P_Dinv : tb.U_Dinv;
  }
  static __device__ __forceinline__ const double* Lb(const Tables& tb) {
    return KIND == KT ? tb.T_Lb : KIND == KP ? tb.P_Lb : tb.U_Lb;
  }
  static __device__ __forceinline__ const double* invd(const Tables& tb) {
    return KIND == KT ? tb.T_invd : KIND == KP ? tb.P_invd : tb.U_invd;
  }
  static __device__ __forceinline__ double tapF(const Grid& g, const Tables& tb, int p, int t, int j) {
    return KIND == KP ? __ldg(tb.s4 + (p * g.nq + t) * 5 + j) : __ldg(tb.s2 + (p * g.nq + t) * 3 + j);
  }
  static __device__ __forceinline__ double tapM(const Grid& g, const Tables& tb, int p, int t, int j, int m) {
    return KIND == KP ? __ldg(tb.mp + ((size_t)(p * g.nq + t) * 5 + j) * g.nm + m)
                      : __ldg(tb.s2 + (p * g.nq + t) * 3 + j);
  }
};

// finite, from the exponent bits (an FP64 comparison would occupy the FP64 pipe)
__device__ __forceinline__ bool finite_bits(double v) { return (__double2hiint(v) & 0x7ff00000) != 0x7ff00000; }

// What a thread of k_solve works on: its column, and its state's arrays.
struct SolveCol {
  int p, m, c, col, W;
  double cpl;        // gamma dt Pr Ra k, negated in the imaginary part's column
  const double* F;   // explicit terms
  const double* X;   // step-start state
  double* R;         // accumulated right-hand sides
  double* Xo;
  size_t S;
};

// phase 1 for tau rows t0 .. t0 + NB - 1 of a column: r_i, and the right-hand
// side bv of the system (psi: with the buoyancy of T, row r of it at T[r W])
template <int KIND, int NB>
__device__ __forceinline__ void solve_rhs(const Grid& g, const Tables& tb, int stage, const SolveCol& k, int t0,
                                          const double* T, double* r, double* bv) {
  using SY = Sys<KIND>;
  constexpr int NW = NB + SY::LAM;
  const int nq = g.nq, nt = nq - SY::D, ns = g.ns;
  const int f = (KIND == KT) ? 0 : 1;
  const size_t rs = soff(g, 0, 2, 0);                         // coefficients n, n + 2
  const size_t o0 = soff(g, f, 2 * t0 + k.p, k.m) + k.c;
  if (t0 >= nt) return;
  double fw[NW], ri[NB], Rl[NB][3];
#pragma unroll
  for (int i = 0; i < NW; ++i) fw[i] = (t0 + i < nq) ? k.F[o0 + i * rs] : 0.0;
  if (stage == 1) {
    double xw[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) xw[i] = (t0 + i < nq) ? k.X[o0 + i * rs] : 0.0;
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      const int t = t0 + i;
      double mx = 0.0;
#pragma unroll
      for (int j = 0; j <= SY::LAM; ++j)
        if (t + j < nq && t < nt) mx = fma(SY::tapM(g, tb, k.p, t, j, k.m), xw[i + j], mx);
      ri[i] = mx;
    }
  } else {
#pragma unroll
    for (int i = 0; i < NB; ++i) {
      ri[i] = (t0 + i < nt) ? k.R[(size_t)(stage - 1) * k.S + o0 + i * rs] : 0.0;
#pragma unroll
      for (int l = 0; l < 3; ++l)
        Rl[i][l] = (t0 + i < nt && l + 2 > stage && l + 2 <= ns) ? k.R[(size_t)(l + 1) * k.S + o0 + i * rs] : 0.0;
    }
  }
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int t = t0 + i;
    if (t >= nt) break;
    double fv = 0.0;
#pragma unroll
    for (int j = 0; j <= SY::LAM; ++j)
      if (t + j < nq) fv = fma(SY::tapF(g, tb, k.p, t, j), fw[i + j], fv);
    if (KIND != KP) fv = -fv;
    r[i] = fma(__ldg(tb.dtae + stage * 5 + stage - 1), fv, ri[i]);
#pragma unroll
    for (int l = 0; l < 3; ++l)
      if (l + 2 > stage && l + 2 <= ns)
        k.R[(size_t)(l + 1) * k.S + o0 + i * rs] =
            fma(__ldg(tb.dtae + (l + 2) * 5 + stage - 1), fv, stage == 1 ? ri[i] : Rl[i][l]);
    bv[i] = r[i];
    if (KIND == KP) {
      // + gamma dt (-i k Pr Ra) S4 T_i: real part + k.. Im(S4 T), imaginary part - k.. Re(S4 T)
      double st = 0.0;
#pragma unroll
      for (int j = 0; j <= 4; ++j)
        if (t + j < nq) st = fma(SY::tapF(g, tb, k.p, t, j), T[(t + j) * k.W + (k.col ^ 1)], st);
      bv[i] = fma(k.cpl, st, bv[i]);
    }
  }
}

// phase 4 for coefficients (and tau rows) t0 .. t0 + NB - 1 of a column; row i of
// the solution at x[i W], r_i at r[i W] or (RG) in the accumulator of this stage
template <int KIND, int NB, bool RG>
__device__ __forceinline__ bool solve_lx(const Grid& g, const Tables& tb, int stage, const SolveCol& k, int t0,
                                         const double* x, const double* r) {
  using SY = Sys<KIND>;
  constexpr int NW = NB + SY::LAM;
  const int nq = g.nq, nt = nq - SY::D, ns = g.ns;
  const int f = (KIND == KT) ? 0 : 1;
  const size_t rs = soff(g, 0, 2, 0);
  const size_t o0 = soff(g, f, 2 * t0 + k.p, k.m) + k.c;
  double xw[NW], Rl[NB][3], rg[NB];
  bool ok = true;
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    if (RG) rg[i] = (t0 + i < nt && stage < ns) ? k.R[(size_t)(stage - 1) * k.S + o0 + i * rs] : 0.0;
#pragma unroll
    for (int l = 0; l < 3; ++l)
      Rl[i][l] = (t0 + i < nt && l + 2 > stage && l + 2 <= ns) ? k.R[(size_t)(l + 1) * k.S + o0 + i * rs] : 0.0;
  }
#pragma unroll
  for (int i = 0; i < NW; ++i) xw[i] = (t0 + i < nq) ? x[(t0 + i) * k.W + k.col] : 0.0;
#pragma unroll
  for (int i = 0; i < NB; ++i) {
    const int t = t0 + i;
    if (t < nq) {
      k.Xo[o0 + i * rs] = xw[i];
      ok = ok && finite_bits(xw[i]);
    }
    if (stage < ns && t < nt) {
      double mx = 0.0;
#pragma unroll
      for (int j = 0; j <= SY::LAM; ++j)
        if (t + j < nq) mx = fma(SY::tapM(g, tb, k.p, t, j, k.m), xw[i + j], mx);
      const double lx2 = g.inv_gamma * (mx - (RG ? rg[i] : r[t * k.W + k.col]));   // dt (L X_i + coupling)
#pragma unroll
      for (int l = 0; l < 3; ++l)
        if (l + 2 > stage && l + 2 <= ns)
          k.R[(size_t)(l + 1) * k.S + o0 + i * rs] = fma(c_AI[g.scheme][l + 2][stage], lx2, Rl[i][l]);
    }
  }
  return ok;
}

// Phases 2 and 3 of a tile by two warps.  Chunk j of the sequence (RC steps
// backward, then RC forward) lies in ring[j % 3]: the first warp works on chunk j
// while the second sums the boundary rows of chunk j - 1 and chunks j + 1 and
// j + 2 are on their way.  Both warps pass the barrier before every chunk and
// two at the turn, so neither waits for more than the other's chunk.
constexpr int RC = 4;
__host__ __device__ constexpr int solve_ring(int tms) { return RC * 4 * tms; }   // doubles per chunk

__device__ __forceinline__ void pair_sync() {
  __syncwarp();
  asm volatile("bar.sync 1, 64;" ::: "memory");
}

template <int KIND>
__device__ __forceinline__ void solve_helper(const Grid& g, const Tables& tb, int p, int m0, int tms, const double* y,
                                             double* ring, double* bdx) {
  using SY = Sys<KIND>;
  constexpr int D = SY::D;
  const int nq = g.nq, W = 2 * tms, lt = __ffs(tms) - 1, lane = threadIdx.x & 31;
  const int nb = (nq - D + RC - 1) / RC;
  const double *mB = SY::multB(tb), *mD = SY::multD(tb), *Lb = SY::Lb(tb), *iv = SY::invd(tb);
  // backward chunk: [step][2 D][mode], multipliers of the rows below, then of the
  // boundary rows; forward: [step][D + 1][mode], L and the inverse diagonal
  auto load = [&](int j) {
    double* dst = ring + (j % 3) * solve_ring(tms);
    const bool back = j < nb;
    const int per = back ? 2 * D : D + 1, r0 = back ? nq - 1 - j * RC : D + (j - nb) * RC;
    if (j < 2 * nb)
      for (int e = lane; e < RC * per * tms; e += 32) {
        const int mode = e & (tms - 1), q = e >> lt, st = q / per, w = q - st * per;
        const int row = back ? r0 - st : r0 + st;
        if (row < D || row >= nq) continue;
        const size_t rw = (size_t)(p * nq + row);
        const double* src = back ? (w < D ? mB : mD) + (rw * D + (w < D ? w : w - D)) * g.nm
                                 : (w < D ? Lb + (rw * D + w) * g.nm : iv + rw * g.nm);
        const unsigned d = (unsigned)__cvta_generic_to_shared(dst + e);
        asm volatile("cp.async.ca.shared.global [%0], [%1], 8;" ::"r"(d), "l"(src + m0 + mode) : "memory");
      }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  const bool on = lane < W && (KIND != KP || m0 + (lane >> 1) > 0);
  double bd[D];
#pragma unroll
  for (int q = 0; q < D; ++q) bd[q] = 0.0;
  auto boundary = [&](int j) {
    if (on) {
      const double* f = ring + (j % 3) * solve_ring(tms) + (lane >> 1);
#pragma unroll
      for (int st = 0; st < RC; ++st) {
        const int row = nq - 1 - j * RC - st;
        if (row < D) break;
        const double v = y[row * W + lane];
#pragma unroll
        for (int q = 0; q < D; ++q) bd[q] = fma(-f[(st * 2 * D + D + q) * tms], v, bd[q]);
      }
    }
    __syncwarp();
  };
  load(0);
  load(1);
  for (int j = 0; j < nb; ++j) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    pair_sync();                       // chunk j is here; the rows of chunk j - 1 are final
    if (j > 0) boundary(j - 1);
    load(j + 2);
  }
  pair_sync();
  boundary(nb - 1);
  if (on)
#pragma unroll
    for (int q = 0; q < D; ++q) bdx[q * W + lane] = bd[q];
  pair_sync();
  for (int j = nb; j < 2 * nb; ++j) {
    asm volatile("cp.async.wait_group 1;" ::: "memory");
    pair_sync();
    load(j + 2);
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
}

template <int KIND>
__device__ __forceinline__ void solve_recurrence(const Grid& g, const Tables& tb, int p, int m0, int tms, double* y,
                                                 const double* ring, const double* bdx) {
  using SY = Sys<KIND>;
  constexpr int D = SY::D;
  const int nq = g.nq, W = 2 * tms, lane = threadIdx.x & 31, m = m0 + (lane >> 1);
  const int nb = (nq - D + RC - 1) / RC;
  const bool on = lane < W && (KIND != KP || m > 0);   // (mode 0: solve_mean)
  double Di[D][D], pend[D], win[D];
#pragma unroll
  for (int r = 0; r < D; ++r) {
    pend[r] = win[r] = 0.0;
#pragma unroll
    for (int q = 0; q < D; ++q) Di[r][q] = on ? __ldg(SY::Dinv(tb) + ((size_t)(p * D * D) + r * D + q) * g.nm + m) : 0.0;
  }
  for (int j = 0; j < nb; ++j) {
    pair_sync();
    if (on) {
      const double* f = ring + (j % 3) * solve_ring(tms) + (lane >> 1);
      const int r0 = nq - 1 - j * RC;
      double mb[RC][D], v[RC];
#pragma unroll
      for (int st = 0; st < RC; ++st) {
        const bool in = r0 - st >= D;
        v[st] = in ? y[(r0 - st) * W + lane] : 0.0;
#pragma unroll
        for (int q = 0; q < D; ++q) mb[st][q] = in ? f[(st * 2 * D + q) * tms] : 0.0;
      }
#pragma unroll
      for (int st = 0; st < RC; ++st) {
        if (r0 - st < D) break;
        const double bc = __dadd_rn(v[st], pend[0]);
        y[(r0 - st) * W + lane] = bc;
#pragma unroll
        for (int q = 0; q < D - 1; ++q) pend[q] = fma(-mb[st][D - 1 - q], bc, pend[q + 1]);
        pend[D - 1] = __dmul_rn(-mb[st][0], bc);
      }
    }
  }
  pair_sync();
  pair_sync();
  if (on) {
    // boundary rows: parity combinations of the wall values (Eq. 6) or slopes (Eq. 7)
    double bd[D];
#pragma unroll
    for (int q = 0; q < D; ++q) bd[q] = bdx[q * W + lane];
    if (KIND == KT && m == 0 && (lane & 1) == 0) bd[0] += t_wall_rhs(g, p);
#pragma unroll
    for (int r = 0; r < D; ++r) {
      double x = 0.0;
#pragma unroll
      for (int q = 0; q < D; ++q) x = fma(Di[r][q], bd[q], x);
      win[r] = x;
      y[r * W + lane] = x;
    }
  }
  for (int j = nb; j < 2 * nb; ++j) {
    pair_sync();
    if (on) {
      const double* f = ring + (j % 3) * solve_ring(tms) + (lane >> 1);
      const int r0 = D + (j - nb) * RC;
      double lb[RC][D], iv[RC], v[RC];
#pragma unroll
      for (int st = 0; st < RC; ++st) {
        const bool in = r0 + st < nq;
        v[st] = in ? y[(r0 + st) * W + lane] : 0.0;
        iv[st] = in ? f[(st * (D + 1) + D) * tms] : 0.0;
#pragma unroll
        for (int q = 0; q < D; ++q) lb[st][q] = in ? f[(st * (D + 1) + q) * tms] : 0.0;
      }
#pragma unroll
      for (int st = 0; st < RC; ++st) {
        if (r0 + st >= nq) break;
        double v2 = v[st];
#pragma unroll
        for (int q = 0; q < D; ++q) v2 = fma(-lb[st][q], win[q], v2);
        const double x = iv[st] * v2;
        y[(r0 + st) * W + lane] = x;
#pragma unroll
        for (int q = 0; q < D - 1; ++q) win[q] = win[q + 1];
        win[D - 1] = x;
      }
    }
  }
}

// Phases 2 and 3 of the mean flow, one column (part c of mode 0) per lane.
__device__ __forceinline__ void solve_mean(const Grid& g, const Tables& tb, int p, int W, double* y) {
  const int nq = g.nq, lane = threadIdx.x & 31;
  if (lane >= 2) return;
  const double *mB = tb.U_multB + p * nq, *mD = tb.U_multD + p * nq, *Lb = tb.U_Lb + p * nq, *iv = tb.U_invd + p * nq;
  double pend = 0.0, bd = 0.0;
#pragma unroll 8
  for (int r = nq - 1; r >= 1; --r) {
    const double bc = __dadd_rn(y[r * W + lane], pend);
    y[r * W + lane] = bc;
    pend = __dmul_rn(-__ldg(mB + r), bc);
    bd = fma(-__ldg(mD + r), bc, bd);
  }
  double x = fma(__ldg(tb.U_Dinv + p), bd, 0.0);
  y[lane] = x;
#pragma unroll 8
  for (int r = 1; r < nq; ++r) {
    x = __ldg(iv + r) * fma(-__ldg(Lb + r), x, y[r * W + lane]);
    y[r * W + lane] = x;
  }
}

// Nu_V(t_n) (Eq. 9) of the step-start state: wall temperature difference of
// the mean profile + Clenshaw-Curtis integral of <wT>_x; trapezoid weight.
// The first warp of the block of the odd coefficients of mode 0 sums it: each
// lane a strided share of both sums, then a fixed shuffle tree (the order
// depends on the grid only).  That block overwrites these coefficients only
// after its barriers (a one-stage scheme writes X0 itself).
__device__ __forceinline__ void nu_integral(const Grid& g, const Tables& tb, const double* X0, const double* wT,
                                            double* nu, int b, int stepidx) {
  if (threadIdx.x >= 32 || nu == nullptr) return;
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

constexpr int kSolveThreads = 128;
constexpr int kSolveSmem = 140 * 1024;   // nq = 256, 16 modes

template <int NB, bool RG>
__global__ void __launch_bounds__(kSolveThreads, 5) k_solve(Grid g, Tables tb, double* X, double* Xs, const double* F,
                                                            double* R, size_t S, const double* wT, double* nu, int* flags,
                                                            int* err, int B, int stage, int tms, const double* ra,
                                                            const int* nsteps, const int* step) {
  extern __shared__ double sbuf[];
  pdl_wait();
  const int stepidx = nsteps ? *step : 0;
  const int mt = (g.nm + tms - 1) / tms;       // tms divides nm: both are powers of two
  const int b = blockIdx.x / (2 * mt), rem = blockIdx.x - b * 2 * mt, p = rem / mt, m0 = (rem - p * mt) * tms;
  if (b >= B || !slice_active_at(nsteps, stepidx, b)) return;   // uniform per block
  // a transform of this state gave up waiting (the tensor-core kernels): leave
  // the state as it was at the start of the failing step
  if (flags[b] & kFlagTimeout) return;
  const int nq = g.nq, W = 2 * tms, lw = __ffs(W) - 1, warp = threadIdx.x >> 5;
  SolveCol k;
  k.p = p;
  k.W = W;
  k.col = threadIdx.x & (W - 1);
  k.m = m0 + k.col / 2;
  k.c = k.col & 1;
  const double cpl0 = __ldg(tb.dtae + 25) * (ra ? ra[b] : g.Ra);
  // (+-1) gamma dt Pr Ra k with the roundings of that left-to-right product:
  // the sign is exact, so it may come last
  k.cpl = (k.c == 0 ? cpl0 : -cpl0) * (g.kfac * k.m);
  double* X0 = X + (size_t)b * S;
  k.F = F + (size_t)b * S;
  k.X = X0;
  k.R = R + (size_t)b * 4 * S;
  k.Xo = (stage == g.ns) ? X0 : Xs + (size_t)b * S;   // stiffly accurate: last stage = new state
  k.S = S;
  double* y2 = sbuf;                           // psi / U: rows of W
  double* T = y2 + 2 * W;                      // T: row i where row i + 2 of psi goes
  double* rr = T + (size_t)nq * W;             // [nq][W] r_i, if not RG
  double* ring = rr + (RG ? 0 : (size_t)nq * W);   // [3] chunks of factors
  double* bdx = ring + 3 * solve_ring(tms);    // [2][W] boundary rows
  const int rows = NB * (kSolveThreads >> lw), mine = NB * ((int)threadIdx.x >> lw);   // rows per round
  // The warps of the recurrences: blocks of an SM take different ones (those
  // resident together are about 152 apart), since a warp's number fixes its
  // sub-partition and with it the FP64 pipe.
  const int first = (int)((blockIdx.x / 152 + blockIdx.x) & 3);
  if (stage == 1 && m0 == 0 && p == 1) nu_integral(g, tb, X0, wT, nu, b, stepidx);

  // r_i of tau row t for phase 4 (the accumulator of this stage has been read)
  auto keep_r = [&](int f, int t, double r) {
    if (RG)
      k.R[(size_t)(stage - 1) * S + soff(g, f, 2 * t + p, k.m) + k.c] = r;
    else
      rr[t * W + k.col] = r;
  };

  for (int t0 = mine; t0 < nq; t0 += rows) {
    double r[NB], bv[NB];
    solve_rhs<KT, NB>(g, tb, stage, k, t0, nullptr, r, bv);
#pragma unroll
    for (int i = 0; i < NB; ++i)
      if (t0 + i < nq - 1) {
        keep_r(0, t0 + i, r[i]);
        T[(t0 + i + 1) * W + k.col] = bv[i];
      }
  }
  __syncthreads();
  if (warp == first)
    solve_recurrence<KT>(g, tb, p, m0, tms, T, ring, bdx);
  else if (warp == (first ^ 1))
    solve_helper<KT>(g, tb, p, m0, tms, T, ring, bdx);
  __syncthreads();
  bool ok = true;
  for (int t0 = mine; t0 < nq; t0 += rows) ok = solve_lx<KT, NB, RG>(g, tb, stage, k, t0, T, rr) && ok;
  for (int tb0 = 0; tb0 < nq; tb0 += rows) {   // every thread: the barrier below
    const int t0 = tb0 + mine;
    double r[NB], bv[NB];
    if (k.m == 0)
      solve_rhs<KU, NB>(g, tb, stage, k, t0, nullptr, r, bv);
    else
      solve_rhs<KP, NB>(g, tb, stage, k, t0, T, r, bv);
    const int D = k.m == 0 ? 1 : 2;
    __syncthreads();                           // rows up to tb0 + rows - 1 of T have been read
#pragma unroll
    for (int i = 0; i < NB; ++i)
      if (t0 + i < nq - D) {
        keep_r(1, t0 + i, r[i]);
        y2[(t0 + i + D) * W + k.col] = bv[i];
      }
  }
  __syncthreads();
  if (warp == first)
    solve_recurrence<KP>(g, tb, p, m0, tms, y2, ring, bdx);
  else if (warp == (first ^ 1))
    solve_helper<KP>(g, tb, p, m0, tms, y2, ring, bdx);
  else if (warp == (first ^ 2) && m0 == 0)
    solve_mean(g, tb, p, W, y2);
  __syncthreads();
  for (int t0 = mine; t0 < nq; t0 += rows)
    ok = (k.m == 0 ? solve_lx<KU, NB, RG>(g, tb, stage, k, t0, y2, rr) : solve_lx<KP, NB, RG>(g, tb, stage, k, t0, y2, rr)) && ok;
  if (!ok) {
    atomicOr(flags + b, kFlagNonFinite);
    atomicOr(err, kFlagNonFinite);
  }
}

// ---------------------------------------------------------------------------
// Stage solve of small grids (k_solve_dense, nq <= kDenseSolveMaxNq), both modes:
// x = Ainv b with the dense inverses, one thread per (row r, column), which is
// tau row r of the right-hand side, row r of the product and tau row r of
// dt L X_i in turn.  Everything a thread needs from global memory is fetched at
// the start, the rows of Ainv before the launch before it has finished; r_i and
// the later accumulators stay in registers between the right-hand side and
// dt L X_i.
// Bound: latency (one trip to memory, then about 50 FP64 instructions in a
// row; blocks of one mode leave one warp per sub-partition).  Measured (GB300,
// a whole stage; as phases of k_solve, each with its own trips to memory,
// before): 128 x 32, one state 33.6 -> 31.3 us in FP64, 25.7 -> 23.2 us in mixed
// precision; 64 x 32, 23 states 49.5 -> 46.1 us and 41.0 -> 37.3 us.
// ---------------------------------------------------------------------------
constexpr int kDenseThreads = 256;   // rows times columns of a tile

__global__ void __launch_bounds__(kDenseThreads) k_solve_dense(Grid g, Tables tb, double* X, double* Xs, const double* F,
                                                               double* R, size_t S, const double* wT, double* nu,
                                                               int* flags, int* err, int B, int stage, int tms,
                                                               const double* ra, const int* nsteps, const int* step) {
  constexpr int NQ = kDenseSolveMaxNq;
  __shared__ double y[kDenseThreads], xT[kDenseThreads];   // [nq][W]: right-hand side; solution
  const int nq = g.nq, W = 2 * tms, lw = __ffs(W) - 1, mt = (g.nm + tms - 1) / tms;
  const int b = blockIdx.x / (2 * mt), rem = blockIdx.x - b * 2 * mt, p = rem / mt, m0 = (rem - p * mt) * tms;
  const int t = threadIdx.x >> lw, col = threadIdx.x & (W - 1), m = m0 + col / 2, c = col & 1;
  const bool on = t < nq && m < g.nm;
  double a[NQ];
  auto fetch_inv = [&](const double* inv, int nmod, int mi) {
    const double* row = inv + ((size_t)p * nq + t) * nq * nmod + mi;
#pragma unroll
    for (int q = 0; q < NQ; ++q) a[q] = (on && q < nq) ? __ldg(row + (size_t)q * nmod) : 0.0;
  };
  fetch_inv(tb.T_inv, g.nm, m);
  pdl_wait();
  const int stepidx = nsteps ? *step : 0;
  if (b >= B || !slice_active_at(nsteps, stepidx, b)) return;   // uniform per block
  if (flags[b] & kFlagTimeout) return;                          // as in k_solve
  double* X0 = X + (size_t)b * S;
  double* Xo = (stage == g.ns) ? X0 : Xs + (size_t)b * S;
  const double* Fb = F + (size_t)b * S;
  double* Rb = R + (size_t)b * 4 * S;
  const double Ra = ra ? ra[b] : g.Ra;
  const double cpl = (c == 0 ? __ldg(tb.dtae + 25) * Ra : -(__ldg(tb.dtae + 25) * Ra)) * (g.kfac * m);
  const int ns = g.ns;

  // tau row t of field f: taps of F, of X (stage 1) or the accumulated r_i, later accumulators
  struct Row {
    double f[5], x[5], R[3];
  } rows[2];
#pragma unroll
  for (int f = 0; f < 2; ++f) {
    const int lam = f == 1 && m != 0 ? 4 : 2, nt = nq - lam / 2;
    Row& w = rows[f];
    const bool mine = on && t < nt;
    const size_t ro = soff(g, f, 2 * t + p, m) + c;
#pragma unroll
    for (int j = 0; j < 5; ++j) {
      const bool in = mine && j <= lam && t + j < nq;
      w.f[j] = in ? Fb[soff(g, f, 2 * (t + j) + p, m) + c] : 0.0;
      w.x[j] = in && stage == 1 ? X0[soff(g, f, 2 * (t + j) + p, m) + c] : 0.0;
    }
    if (stage > 1 && mine) w.x[0] = Rb[(size_t)(stage - 1) * S + ro];
#pragma unroll
    for (int l = 0; l < 3; ++l)
      w.R[l] = (mine && stage > 1 && l + 2 > stage && l + 2 <= ns) ? Rb[(size_t)(l + 1) * S + ro] : 0.0;
  }
  if (stage == 1 && m0 == 0 && p == 1) nu_integral(g, tb, X0, wT, nu, b, stepidx);

  bool ok = true;
  auto system = [&](auto kind, int f) {
    constexpr int KIND = decltype(kind)::value;
    using SY = Sys<KIND>;
    Row& w = rows[f];
    const bool mine = on && t < nq - SY::D;
    double r = 0.0;
    if (mine) {
      double fv = 0.0;
#pragma unroll
      for (int j = 0; j <= SY::LAM; ++j)
        if (t + j < nq) fv = fma(SY::tapF(g, tb, p, t, j), w.f[j], fv);
      if (KIND != KP) fv = -fv;
      if (stage == 1) {
        double mx = 0.0;
#pragma unroll
        for (int j = 0; j <= SY::LAM; ++j)
          if (t + j < nq) mx = fma(SY::tapM(g, tb, p, t, j, m), w.x[j], mx);
        r = fma(__ldg(tb.dtae + 5), fv, mx);
#pragma unroll
        for (int l = 0; l < 3; ++l)
          if (l + 2 <= ns) w.R[l] = fma(__ldg(tb.dtae + (l + 2) * 5), fv, mx);
      } else {
        r = fma(__ldg(tb.dtae + stage * 5 + stage - 1), fv, w.x[0]);
#pragma unroll
        for (int l = 0; l < 3; ++l)
          if (l + 2 > stage && l + 2 <= ns) w.R[l] = fma(__ldg(tb.dtae + (l + 2) * 5 + stage - 1), fv, w.R[l]);
      }
      double bv = r;
      if (KIND == KP) {
        double st = 0.0;
#pragma unroll
        for (int j = 0; j <= 4; ++j)
          if (t + j < nq) st = fma(__ldg(tb.s4 + (p * nq + t) * 5 + j), xT[(t + j) * W + (col ^ 1)], st);
        bv = fma(cpl, st, bv);
      }
      y[(t + SY::D) * W + col] = bv;
    }
    // boundary rows of b: the mean temperature's wall values (Eq. 6) or slopes
    // (Eq. 7) in parity combinations; zero for T at m >= 1, psi and U
    if (on && t < SY::D) y[t * W + col] = (KIND == KT && m == 0 && c == 0) ? t_wall_rhs(g, p) : 0.0;
    return r;
  };
  // rows of the product, dt L X_i into the later accumulators
  auto finish = [&](auto kind, int f, double r) {
    constexpr int KIND = decltype(kind)::value;
    using SY = Sys<KIND>;
    if (!(on && t < nq - SY::D && stage < ns)) return;
    double mx = 0.0;
#pragma unroll
    for (int j = 0; j <= SY::LAM; ++j)
      if (t + j < nq) mx = fma(SY::tapM(g, tb, p, t, j, m), xT[(t + j) * W + col], mx);
    const double lx2 = g.inv_gamma * (mx - r);
    const size_t ro = soff(g, f, 2 * t + p, m) + c;
#pragma unroll
    for (int l = 0; l < 3; ++l)
      if (l + 2 > stage && l + 2 <= ns) Rb[(size_t)(l + 1) * S + ro] = fma(c_AI[g.scheme][l + 2][stage], lx2, rows[f].R[l]);
  };
  auto product = [&](int f) {
    if (!on) return;
    double acc0 = 0.0, acc1 = 0.0;                       // two partial sums: shorter chain
#pragma unroll
    for (int q = 0; q < NQ; q += 2) {
      if (q < nq) acc0 = fma(a[q], y[q * W + col], acc0);
      if (q + 1 < nq) acc1 = fma(a[q + 1], y[(q + 1) * W + col], acc1);
    }
    const double x = acc0 + acc1;
    xT[t * W + col] = x;
    Xo[soff(g, f, 2 * t + p, m) + c] = x;
    ok = ok && finite_bits(x);
  };
  using T_ = std::integral_constant<int, KT>;
  using P_ = std::integral_constant<int, KP>;
  using U_ = std::integral_constant<int, KU>;
  const double rT = system(T_(), 0);
  __syncthreads();
  product(0);
  if (m == 0)
    fetch_inv(tb.U_inv, 1, 0);
  else
    fetch_inv(tb.P_inv, g.nm, m);
  __syncthreads();
  finish(T_(), 0, rT);
  const double rP = m == 0 ? system(U_(), 1) : system(P_(), 1);
  __syncthreads();
  product(1);
  __syncthreads();
  if (m == 0)
    finish(U_(), 1, rP);
  else
    finish(P_(), 1, rP);
  if (!ok) {
    atomicOr(flags + b, kFlagNonFinite);
    atomicOr(err, kFlagNonFinite);
  }
}

// shared memory of a k_solve block: T and psi, r_i (unless rg), factors, boundary rows
static size_t solve_smem(const Grid& g, int tms, bool rg) {
  return ((size_t)((rg ? 1 : 2) * g.nq + 4) * 2 * tms + 3 * solve_ring(tms)) * 8;
}
constexpr size_t kSolveFive = 44 * 1024;   // five blocks per SM
// r_i goes to global memory where the block would not fit five times beside it
static bool solve_rg(const Grid& g, int tms) { return tms >= 8 && solve_smem(g, tms, false) > kSolveFive; }
// Modes per k_solve block.  Every column's arithmetic is independent of the
// tiling.  A small batch (a coarse sweep) takes small tiles and spreads over the
// SMs instead of leaving most of them idle; a large one the largest tile of which
// five blocks share an SM, since a recurrence costs as much for 16 columns as for
// 32.  With 128 coefficients per parity that takes r_i out of shared memory (1024
// x 256, 32 states: 1042 us; kept there, 1117 with 8 modes and 1330 with 16); with
// up to 64 it fits (512 x 128, 64 states: 515 us, in global memory 523).
static int solve_tile(const Grid& g, int B) {
  int tms = 16;
  while (tms > 1 && (long)B * 2 * ((g.nm + tms - 1) / tms) < 2L * 152) tms >>= 1;
  if (tms > g.nm) tms = g.nm;
  while (tms > 1 && solve_smem(g, tms, solve_rg(g, tms)) > kSolveFive) tms >>= 1;
  return tms;
}

// The shapes of a launch: the tuned ones where set, else the heuristics.
static int solve_tms_of(const Grid& g, const Shapes* sh, int B) {
  int tms = (sh && sh->solve_tms > 0) ? sh->solve_tms : solve_tile(g, B);
  while (tms > g.nm || (g.nq <= kDenseSolveMaxNq && g.nq * 2 * tms > kDenseThreads)) tms >>= 1;
  return tms;
}
static int zfwd_tm_of(const Grid& g, const Shapes* sh, int B, size_t es) {
  return (sh && sh->zfwd_tm > 0) ? sh->zfwd_tm : zfwd_tile(g, B, es);
}
static int zfwd_nch_of(const Grid& g, const Shapes* sh, int B, int tm) {
  return (sh && sh->zfwd_nch > 0) ? sh->zfwd_nch : zfwd_chunks(g, B, tm);
}
Shapes resolved_shapes(const Grid& g, const Tables& t, const Shapes& sh, int B) {
  Shapes r;
  r.solve_tms = solve_tms_of(g, &sh, B);
  if (t.tcW_hi[0] == nullptr) {
    r.zfwd_tm = zfwd_tm_of(g, &sh, B, g.mixed ? 4 : 8);
    r.zfwd_nch = zfwd_nch_of(g, &sh, B, r.zfwd_tm);
  }
  if (g.mixed)
    r.rows_cl = rows_f32_per_block(g, sh, B);
  else
    rows_f64_form(g, sh, B, &r.rows_cl, &r.rows_threads, &r.rows_lean);
  return r;
}
bool shapes_valid(const Grid& g, const Shapes& sh, size_t es) {
  if (sh.solve_tms > 0 && (sh.solve_tms > 16 || (sh.solve_tms & (sh.solve_tms - 1)) ||
                           solve_smem(g, sh.solve_tms, false) > 200 * 1024))
    return false;
  if (sh.zfwd_tm > 0 && (sh.zfwd_tm > 32 || (sh.zfwd_tm & (sh.zfwd_tm - 1)) ||
                         (size_t)2 * ((g.Mz + 1) / 2) * sh.zfwd_tm * 2 * es > 200 * 1024))
    return false;
  if (sh.zfwd_nch > 0 && (sh.zfwd_nch > 8 || (sh.zfwd_nch & (sh.zfwd_nch - 1)))) return false;
  if (es == 8 && sh.rows_cl == 1 && rows_f64_cl_bytes(g) > 200 * 1024) return false;
  if (sh.rows_threads != 0 && sh.rows_threads != 256 && sh.rows_threads != 512 && sh.rows_threads != 1024)
    return false;
  if (sh.rows_lean < -1 || sh.rows_lean > 1 || (es == 8 && sh.rows_lean == 1 && !rows_f64_batched(g))) return false;
  return true;
}

__global__ void k_advance(int* step) {
  pdl_wait();
  *step += 1;
}

// Body end of the device-side step loop: the loop ends once every state of the
// batch has taken its steps (maxs is written by the host before each launch).
// cancel (may be null): a word another stream sets to stop the loop early
// (work whose result is no longer wanted, e.g. a speculative Parareal iteration)
__global__ void k_advance_loop(int* step, const int* maxs, const int* cancel, cudaGraphConditionalHandle loop) {
  pdl_wait();
  const int s = *step + 1;
  *step = s;
  const bool stop = cancel != nullptr && *(const volatile int*)cancel != 0;
  cudaGraphSetConditional(loop, (s < *maxs && !stop) ? 1u : 0u);
}

static inline unsigned nblk(long n, int t) { return (unsigned)((n + t - 1) / t); }

static std::atomic<unsigned long long> g_launches{0};
unsigned long long launches_so_far() { return g_launches.load(); }
void add_launches(unsigned long long n) { g_launches.fetch_add(n); }
static inline void count(int n = 1) { g_launches.fetch_add(n); }

cudaError_t Prof::fold() {
  for (size_t i = 0; i < used; ++i) {
    float t = 0.f;
    cudaError_t e = cudaEventSynchronize(ev[2 * i + 1]);
    if (e != cudaSuccess) return e;
    e = cudaEventElapsedTime(&t, ev[2 * i], ev[2 * i + 1]);
    if (e != cudaSuccess) return e;
    ms[kind[i]] += t;
  }
  used = 0;
  return cudaSuccess;
}

void Prof::begin(int k, cudaStream_t s) {
  if (used * 2 + 2 > ev.size()) {
    if (ev.size() >= 8192) {
      fold();
    } else {
      for (int i = 0; i < 256; ++i) {
        cudaEvent_t e;
        cudaEventCreate(&e);
        ev.push_back(e);
      }
      kind.resize(ev.size() / 2);
    }
  }
  kind[used] = k;
  cudaEventRecord(ev[2 * used], s);
}

void Prof::end(int k, cudaStream_t s, double fl, double by) {
  cudaEventRecord(ev[2 * used + 1], s);
  ++used;
  launches[k] += 1;
  flops[k] += fl;
  bytes[k] += by;
}

// Tiles and threads of the L2 norms (see k_l2_diff).
constexpr int kCorrTile = 8;
constexpr int kCorrThreads = 256;
__global__ void k_l2_diff(Grid g, const double* __restrict__ gram, const double* A, const double* Bm, double* out, int ncta);

// Algorithmic work of one launch over B slices (all active).
static double zinv_flops(const Grid& g, int B) { return 24.0 * B * ((g.Mz + 1) / 2) * g.nm * g.Nz; }
static double zinv_bytes(const Grid& g, int B, size_t es) {
  return 8.0 * B * state_doubles(g) + (double)es * B * z_doubles(g);
}
static double rows_flops(const Grid& g, int B) {
  return (double)B * g.Mz * (6.0 * 5.0 * g.Mx * std::log2((double)g.Mx) + 10.0 * g.Mx);
}
static double rows_bytes(const Grid& g, int B, size_t es) {
  return (double)es * B * (z_doubles(g) + q_doubles(g)) + 8.0 * B * g.Mz;
}
static double zfwd_flops(const Grid& g, int B) { return 4.0 * B * g.Nz * g.nm * ((g.Mz + 1) / 2) * 2.0; }
static double zfwd_bytes(const Grid& g, int B, size_t es = 8) {
  return (double)es * B * q_doubles(g) + 8.0 * B * state_doubles(g);
}
// stage solve: per (m, parity) about 60 flops per coefficient row for T and psi;
// reads F, X and up to four accumulators, writes X and the accumulators
static double solve_flops(const Grid& g, int B) { return 120.0 * B * g.nm * 2.0 * g.nq * 2.0; }
static double solve_bytes(const Grid& g, int B) { return 8.0 * B * state_doubles(g) * 10.0; }

// The dynamic shared-memory allowances only ever grow, so that a later handle
// on a smaller grid does not shrink them below an earlier one's need.
template <typename F>
static cudaError_t allow_smem(F* fn, int need, int& allowed) {
  if (need <= allowed) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, need);
  if (e == cudaSuccess) allowed = need;
  return e;
}

cudaError_t configure_kernels(const Grid& g) {
  // k_l2_diff: tiles of up to 512 coefficients, clusters of up to 16 blocks
  cudaError_t l2 = cudaFuncSetAttribute(k_l2_diff, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                        kCorrTile * 512 * (int)sizeof(double2));
  if (l2 == cudaSuccess) l2 = cudaFuncSetAttribute(k_l2_diff, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  if (l2 != cudaSuccess) return l2;
  static int a_zfwd_d = 48 * 1024, a_zfwd_f = 48 * 1024;
  cudaError_t e = g.mixed ? configure_rows_f32(g) : configure_rows_f64(g);
  if (e == cudaSuccess && g.nq > kDenseSolveMaxNq)
    for (auto* fn : {k_solve<1, false>, k_solve<2, false>, k_solve<4, false>, k_solve<4, true>})
      if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, kSolveSmem);
  if (e == cudaSuccess)
    e = g.mixed ? allow_smem(k_zfwd<float>, (int)std::max(zfwd_smem(g, 1, 4), zfwd_smem(g, 1 << 20, 4)), a_zfwd_f)
                : allow_smem(k_zfwd<double>, (int)std::max(zfwd_smem(g, 1, 8), zfwd_smem(g, 1 << 20, 8)), a_zfwd_d);
  return e;
}

// z inverse on the CUDA cores.
template <typename T>
static cudaError_t launch_zinv(bool pdl, const Grid& g, const T* Bz, const Work& w, const double* X, int B, const int* ns,
                               cudaStream_t s) {
  const int kp = zinv_warps(g);
  const unsigned blocks = (unsigned)(B * ((g.Mz + 1) / 2) * ((g.nm + 31) / 32));
  return launch_pdl(pdl, k_zinv<T>, blocks, 32 * kp, kp > 1 ? (size_t)kp * 12 * 32 * 2 * sizeof(T) : 0, s, g, Bz, X,
                    state_doubles(g), reinterpret_cast<T*>(w.Z), B, ns, w.step);
}

// z inverse and row kernel.
static cudaError_t launch_transforms(const Grid& g, const Tables& t, const Work& w, const double* X, int B, const int* ns,
                                     Prof* pf, cudaStream_t s) {
  const size_t es = g.mixed ? sizeof(float) : sizeof(double);
  if (pf) pf->begin(RBC_KERNEL_ZINV, s);
  cudaError_t e;
  if (t.tcA_psi_hi != nullptr)
    e = launch_zinv_tc(g, t, w, X, B, ns, s);          // tensor cores, TF32 or BF16 with split compensation
  else
    e = g.mixed ? launch_zinv<float>(w.pdl != 0, g, t.zinv32, w, X, B, ns, s)
                : launch_zinv<double>(w.pdl != 0, g, t.zinv, w, X, B, ns, s);
  if (e != cudaSuccess) return e;
  if (pf) pf->end(RBC_KERNEL_ZINV, s, zinv_flops(g, B), zinv_bytes(g, B, es));
  if (pf) pf->begin(RBC_KERNEL_ROWS, s);
  e = g.mixed ? launch_rows_f32(g, t, w, B, ns, s) : launch_rows_f64(g, t, w, B, ns, s);
  if (pf) pf->end(RBC_KERNEL_ROWS, s, rows_flops(g, B), rows_bytes(g, B, es));
  return e;
}

cudaError_t launch_explicit(const Grid& g, const Tables& t, const Work& w, const double* X, int B, bool all_active,
                            cudaStream_t s) {
  const int* ns = all_active ? nullptr : w.nsteps;
  Prof* pf = (w.prof && w.prof->on && !all_active) ? w.prof : nullptr;
  const cudaError_t e = launch_transforms(g, t, w, X, B, ns, pf, s);
  if (e != cudaSuccess) return e;
  count(2);
  return cudaGetLastError();
}

template <typename T>
static cudaError_t launch_zfwd(const Grid& g, const T* W, const Work& w, int B, cudaStream_t s) {
  const size_t S = state_doubles(g), es = sizeof(T);
  const int tm = zfwd_tm_of(g, w.shapes, B, es);
  const int mt = (g.nm + tm - 1) / tm;
  const int nch = zfwd_nch_of(g, w.shapes, B, tm);
  const size_t smem = (size_t)2 * ((g.Mz + 1) / 2) * tm * 2 * es;
  return launch_pdl(w.pdl != 0, k_zfwd<T>, (unsigned)(B * 2 * mt * nch), 128, smem, s, g, W,
                    reinterpret_cast<const T*>(w.Q), w.F, S, B, tm, nch, w.nsteps, w.step);
}

cudaError_t launch_stage(const Grid& g, const Tables& t, const Work& w, double* X, int B, int stage, double* nu,
                         cudaStream_t s) {
  const size_t S = state_doubles(g);
  const double* Xin = (stage == 1) ? X : w.Xs;
  cudaError_t e = launch_explicit(g, t, w, Xin, B, false, s);
  if (e != cudaSuccess) return e;
  Prof* pf = (w.prof && w.prof->on) ? w.prof : nullptr;
  if (pf) pf->begin(RBC_KERNEL_ZFWD, s);
  if (g.mixed && t.tcW_hi[0] != nullptr)
    e = launch_zfwd_tc(g, t, w, B, s);                 // tensor cores, TF32 or BF16 with split compensation
  else
    e = g.mixed ? launch_zfwd<float>(g, t.zfwd32, w, B, s) : launch_zfwd<double>(g, t.zfwd, w, B, s);
  if (e != cudaSuccess) return e;
  if (pf) pf->end(RBC_KERNEL_ZFWD, s, zfwd_flops(g, B), zfwd_bytes(g, B, g.mixed ? 4 : 8));
  if (pf) pf->begin(RBC_KERNEL_SOLVE, s);
  const bool dense = g.nq <= kDenseSolveMaxNq;
  const int tms = solve_tms_of(g, w.shapes, B);
  const int mtiles = (g.nm + tms - 1) / tms;
  // tau rows per thread and round: four share the loads of a window; fewer while
  // a round would not give every thread of the block a row
  const int items = g.nq * 2 * tms;
  const bool rg = solve_rg(g, tms);
  auto* kernel = dense                        ? k_solve_dense
                 : rg                         ? k_solve<4, true>
                 : items >= 4 * kSolveThreads ? k_solve<4, false>
                 : items >= 2 * kSolveThreads ? k_solve<2, false>
                                              : k_solve<1, false>;
  e = launch_pdl(w.pdl != 0, kernel, (unsigned)(B * 2 * mtiles), dense ? (items + 31) / 32 * 32 : kSolveThreads,
                 dense ? 0 : solve_smem(g, tms, rg), s, g,
                 t, X, w.Xs, w.F, w.R, S, w.wT, nu, w.flags, w.err, B, stage, tms, w.ra, w.nsteps, w.step);
  if (e != cudaSuccess) return e;
  if (pf) pf->end(RBC_KERNEL_SOLVE, s, solve_flops(g, B), solve_bytes(g, B));
  count(2);
  return cudaGetLastError();
}

cudaError_t launch_advance(const Work& w, cudaStream_t s) {
  launch_pdl(w.pdl != 0, k_advance, 1, 1, 0, s, w.step);
  count();
  return cudaGetLastError();
}

cudaError_t launch_advance_loop(const Work& w, cudaGraphConditionalHandle loop, cudaStream_t s) {
  launch_pdl(w.pdl != 0, k_advance_loop, 1, 1, 0, s, w.step, w.maxs, w.cancel, loop);
  count();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Diagnostics.
// ---------------------------------------------------------------------------
__global__ void k_nu_final(Grid g, const double* cc, const double* X, size_t S, const double* wT, double* nu,
                           const int* nsteps, const int* flags, int B) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B || nsteps[b] <= 0 || (flags[b] & kFlagTimeout)) return;
  const double* X0 = X + (size_t)b * S;
  double cond = 0.0;
  for (int n = 1; n < g.Nz; n += 2) cond -= 2.0 * X0[soff(g, 0, n, 0)];
  double adv = 0.0;
  for (int jz = 0; jz < g.Mz; ++jz) adv = fma(cc[jz], wT[(size_t)b * g.Mz + jz], adv);
  nu[b] += 0.5 * g.dt * (cond + 0.5 * adv);
}

cudaError_t launch_nu_final(const Grid& g, const Tables& t, const Work& w, const double* X, int B, double* nu,
                            cudaStream_t s) {
  cudaError_t e = launch_explicit(g, t, w, X, B, true, s);
  if (e != cudaSuccess) return e;
  k_nu_final<<<nblk(B, 128), 128, 0, s>>>(g, t.cc, X, state_doubles(g), w.wT, nu, w.nsteps, w.flags, B);
  count();
  return cudaGetLastError();
}

// (Nu_V, Nu_b, Nu_t) of one state whose <wT>_x profile is in wT[0..Mz).
__global__ void k_nusselt(Grid g, const double* cc, const double* X, const double* wT, double* out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  double cond = 0.0, nb = 0.0, nt = 0.0;
  for (int n = 0; n < g.Nz; ++n) {
    const double a = X[soff(g, 0, n, 0)];
    if (n & 1) cond -= 2.0 * a;
    const double n2 = (double)n * n;
    nb -= 2.0 * a * ((n & 1) ? n2 : -n2);   // -dT/dz at z = -1/2: T_n'(-1) = (-1)^(n+1) n^2
    nt -= 2.0 * a * n2;                     // -dT/dz at z = +1/2: T_n'(1) = n^2
  }
  double adv = 0.0;
  for (int jz = 0; jz < g.Mz; ++jz) adv = fma(cc[jz], wT[jz], adv);
  out[0] = cond + 0.5 * adv;
  out[1] = nb;
  out[2] = nt;
}

cudaError_t launch_nusselt(const Grid& g, const Tables& t, const Work& w, const double* X, double* out3,
                           cudaStream_t s) {
  cudaError_t e = launch_explicit(g, t, w, X, 1, true, s);
  if (e != cudaSuccess) return e;
  k_nusselt<<<1, 32, 0, s>>>(g, t.cc, X, w.wT, out3);
  count();
  return cudaGetLastError();
}

// Consistency-check averages of Sec. 2.2, pass 1.  Z holds the FP64 z inverse
// of every state (fields u, w, d_x omega, d_z omega, ..., T, ... at the padded rows).  Block per (state, padded row j): x-means by Parseval over the kept
// modes (weight 1 for m = 0, 2 otherwise; Re(a conj b) for a pair of fields):
//   u^2 + w^2,   u.lap u = -u d_z omega + w d_x omega,   w T,
//   (T - <T>_x)^2 (modes m >= 1),   <T>_x = Re T_0(s_j).
// rows[b][q][j], q = 0..4 in that order.
__global__ void __launch_bounds__(128) k_diag_rows(Grid g, const double* __restrict__ Z, double* __restrict__ rows) {
  __shared__ double red[128];
  const int b = blockIdx.x / g.Mz, j = blockIdx.x - b * g.Mz;
  const size_t fs = (size_t)g.Mz * g.nm * 2;
  const double* zb = Z + (size_t)b * 9 * fs + (size_t)j * g.nm * 2;
  double ke = 0.0, ep = 0.0, wt = 0.0, tv = 0.0;
  for (int m = threadIdx.x; m < g.nm; m += blockDim.x) {
    const double c = m == 0 ? 1.0 : 2.0;
    const double2 u = ld2(zb + 2 * m), w = ld2(zb + fs + 2 * m);
    const double2 dxo = ld2(zb + 2 * fs + 2 * m), dzo = ld2(zb + 3 * fs + 2 * m);
    const double2 t = ld2(zb + 6 * fs + 2 * m);
    ke += c * (u.x * u.x + u.y * u.y + w.x * w.x + w.y * w.y);
    ep += c * (w.x * dxo.x + w.y * dxo.y - u.x * dzo.x - u.y * dzo.y);
    wt += c * (w.x * t.x + w.y * t.y);
    if (m > 0) tv += 2.0 * (t.x * t.x + t.y * t.y);
  }
  ke = block_sum(ke, red);
  ep = block_sum(ep, red);
  wt = block_sum(wt, red);
  tv = block_sum(tv, red);
  if (threadIdx.x == 0) {
    double* r = rows + (size_t)b * 5 * g.Mz + j;
    r[0] = ke;
    r[g.Mz] = ep;
    r[2 * g.Mz] = wt;
    r[3 * g.Mz] = tv;
    r[4 * g.Mz] = zb[6 * fs];
  }
}

// Pass 2, block per state: <f>_V = (1/2) sum_j cc_j <f>_x(s_j) (Lz = 1) for the
// first three rows, the Nusselt numbers of Eqs. 9-11 (conduction part of Nu_V
// and the wall slopes from the mean temperature coefficients), the profiles.
__global__ void __launch_bounds__(128) k_diag_final(Grid g, const double* __restrict__ cc, const double* __restrict__ X,
                                                    const double* __restrict__ rows, double* __restrict__ out) {
  __shared__ double red[128];
  const int b = blockIdx.x;
  const double* r = rows + (size_t)b * 5 * g.Mz;
  double s0 = 0.0, s1 = 0.0, s2 = 0.0;
  for (int j = threadIdx.x; j < g.Mz; j += blockDim.x) {
    const double c = cc[j];
    s0 += c * r[j];
    s1 += c * r[g.Mz + j];
    s2 += c * r[2 * g.Mz + j];
  }
  s0 = block_sum(s0, red);
  s1 = block_sum(s1, red);
  s2 = block_sum(s2, red);
  double* o = out + (size_t)b * (6 + 2 * g.Mz);
  if (threadIdx.x == 0) {
    const double* Xb = X + (size_t)b * state_doubles(g);
    double cond = 0.0, nb = 0.0, nt = 0.0;
    for (int n = 0; n < g.Nz; ++n) {
      const double a = Xb[soff(g, 0, n, 0)];
      if (n & 1) cond -= 2.0 * a;
      const double n2 = (double)n * n;
      nb -= 2.0 * a * ((n & 1) ? n2 : -n2);
      nt -= 2.0 * a * n2;
    }
    o[0] = 0.5 * s0;
    o[1] = 0.5 * s1;
    o[2] = 0.5 * s2;
    o[3] = cond + 0.5 * s2;
    o[4] = nb;
    o[5] = nt;
  }
  for (int j = threadIdx.x; j < g.Mz; j += blockDim.x) {
    o[6 + j] = r[4 * g.Mz + j];
    o[6 + g.Mz + j] = r[3 * g.Mz + j];
  }
}

cudaError_t launch_diagnostics(const Grid& g, const Tables& t, const Work& w, const double* X, int B, double* out,
                               cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  // FP64 z inverse of all states (no step mask), whatever the handle's precision
  cudaError_t e = launch_zinv<double>(false, g, t.zinv, w, X, B, nullptr, s);
  if (e != cudaSuccess) return e;
  k_diag_rows<<<(unsigned)(B * g.Mz), 128, 0, s>>>(g, w.Z, w.Q);
  k_diag_final<<<(unsigned)B, 128, 0, s>>>(g, t.cc, X, w.Q, out);
  count(3);
  return cudaGetLastError();
}

// Sampled quantities of the time statistics of Sec. 2.2, in place over B rows
// of rbc_diagnostics (6 + 2 Mz each): the characteristic speed
// <u^2 + w^2>_V^(1/2) replaces <u^2 + w^2>_V, and the plane mean of T^2,
// <(T - <T>_x)^2>_x + <T>_x^2, replaces the plane variance.
__global__ void k_stat_sample(Grid g, double* d, int B) {
  const int D = 6 + 2 * g.Mz;
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long)B * D) return;
  const int i = (int)(idx % D);
  if (i == 0) {
    d[idx] = sqrt(d[idx]);
  } else if (i >= 6 + g.Mz) {
    const double tm = d[idx - g.Mz];
    d[idx] = __dadd_rn(d[idx], __dmul_rn(tm, tm));
  }
}

// Trapezoid rule over one sampling interval: acc += h2 (prev + cur), h2 = half
// the interval; then prev = cur (n values).
__global__ void k_stat_accum(double* acc, double* prev, const double* cur, double h2, long n) {
  const long i = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const double c = cur[i];
  acc[i] = __dadd_rn(acc[i], __dmul_rn(h2, __dadd_rn(prev[i], c)));
  prev[i] = c;
}

// a += b (n values)
__global__ void k_add(double* a, const double* b, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) a[i] += b[i];
}

cudaError_t launch_stat_sample(const Grid& g, double* d, int B, cudaStream_t s) {
  const long n = (long)B * (6 + 2 * g.Mz);
  k_stat_sample<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(g, d, B);
  count();
  return cudaGetLastError();
}

cudaError_t launch_stat_accum(double* acc, double* prev, const double* cur, double h2, long n, cudaStream_t s) {
  k_stat_accum<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(acc, prev, cur, h2, n);
  count();
  return cudaGetLastError();
}

cudaError_t launch_add(double* a, const double* b, int n, cudaStream_t s) {
  k_add<<<(unsigned)((n + 127) / 128), 128, 0, s>>>(a, b, n);
  count();
  return cudaGetLastError();
}

// Squared L2(Omega) norms of temperature fields (the defect norm of Sec. 3.7):
// ||T||^2 = (Lx / 2) sum_m w_m Re(conj(c_m) . Gram c_m), w = 1 for m = 0, 2
// otherwise (Parseval in x), Gram the exact Chebyshev Gram matrix (z in
// [-1/2, 1/2]).  The sum runs over tiles of kCorrTile Fourier modes in tile
// order, each tile's terms summed by the block in a fixed order, with explicit
// roundings; rbc_l2_diff and the fused Parareal correction share this order,
// so both give the same bits.

// w Re(conj(di) . s) added to acc, s = sum_j gram_ij d_j
__device__ __forceinline__ double l2_term(double acc, double w, double2 di, double2 s) {
  return fma(w, fma(di.x, s.x, __dmul_rn(di.y, s.y)), acc);
}
__device__ __forceinline__ double2 gram_acc(double2 s, double gij, double2 dj) {
  return make_double2(fma(gij, dj.x, s.x), fma(gij, dj.y, s.y));
}

// ||A_b - B_b||^2 (or ||A_b||^2 when Bm is null) of the temperature field of nst
// states.  A cluster of ncta blocks per state: block c sums the tiles c, c + ncta,
// ... (differences staged once in shared memory) and leaves each tile's sum in
// the first block, which adds them in tile order.  The result does not depend
// on ncta, and no scratch outlives the call.
// Bound: the FP64 pipe, Nz / 2 complex-by-real multiply-adds per coefficient (15 us
// for 16 states of 256 x 64).  One block per state that walked over all tiles and
// formed each difference Nz / 2 times left 136 of 152 SMs idle: the two norms,
// correction and restriction of 16 such states took 729 us together, now 76.
constexpr int kMaxTiles = 64;   // nm <= 512
__global__ void __launch_bounds__(kCorrThreads) k_l2_diff(Grid g, const double* __restrict__ gram, const double* A,
                                                          const double* Bm, double* out, int ncta) {
  namespace cg = cooperative_groups;
  extern __shared__ double2 sd[];             // [kCorrTile][Nz]: the tile's modes
  __shared__ double red[kCorrThreads];
  __shared__ double tile_sum[kMaxTiles];      // the first block's holds all tiles
  cg::cluster_group cl = cg::this_cluster();
  const int b = blockIdx.x / ncta, c = blockIdx.x - b * ncta;
  const size_t S = state_doubles(g);
  const double* a = A + (size_t)b * S;
  const double* bb = Bm ? Bm + (size_t)b * S : nullptr;
  double* sums = cl.map_shared_rank(tile_sum, 0);
  const int tiles = (g.nm + kCorrTile - 1) / kCorrTile;
  cl.sync();                                  // every block runs before its memory is written
  for (int t = c; t < tiles; t += ncta) {
    const int m0 = t * kCorrTile, tm = min(kCorrTile, g.nm - m0);
    for (int it = threadIdx.x; it < tm * g.Nz; it += blockDim.x) {
      const int dm = it % tm, i = it / tm;
      double2 d = ld2(a + soff(g, 0, i, m0 + dm));
      if (bb) d = d - ld2(bb + soff(g, 0, i, m0 + dm));
      sd[dm * g.Nz + i] = d;
    }
    __syncthreads();
    double acc = 0.0;
    for (int it = threadIdx.x; it < tm * g.Nz; it += blockDim.x) {
      const int dm = it % tm, i = it / tm;
      const double2* d = sd + dm * g.Nz;
      double2 s = {0.0, 0.0};
#pragma unroll 4
      for (int jn = (i & 1); jn < g.Nz; jn += 2) s = gram_acc(s, __ldg(gram + (size_t)i * g.Nz + jn), d[jn]);
      acc = l2_term(acc, m0 + dm == 0 ? 1.0 : 2.0, d[i], s);
    }
    acc = block_sum(acc, red);                // (ends with a barrier: sd may be rewritten)
    if (threadIdx.x == 0) sums[t] = acc;
  }
  cl.sync();
  if (c == 0 && threadIdx.x == 0) {
    double tot = 0.0;
    for (int t = 0; t < tiles; ++t) tot += tile_sum[t];
    out[b] = 0.5 * g.Lx * tot;
  }
}

// Blocks per state: one per tile up to a cluster of 16, eight from 38 states on, where
// 38 x 8 already makes two blocks per SM.  More than eight, the portable size, only
// where the stream has the whole GPU (not in an SM partition, `confined`); fewer where
// the device cannot place one such cluster.  (With eight, 256 x 64, one state takes 27
// us instead of 16.5, 1024 x 256, one state 1170 instead of 591.)
bool l2_large_clusters(const Grid& g, int nst) { return nst < 38 && g.nm > 8 * kCorrTile; }

cudaError_t launch_l2_diff(const Grid& g, const Tables& t, const double* A, const double* Bm, int nst, double* out,
                           bool confined, cudaStream_t s) {
  if (nst <= 0) return cudaSuccess;
  const int tiles = (g.nm + kCorrTile - 1) / kCorrTile;
  int ncta = l2_large_clusters(g, nst) && !confined ? 16 : 8;
  while (ncta > tiles) ncta /= 2;
  cudaLaunchConfig_t cfg{};
  cfg.blockDim = kCorrThreads;
  cfg.dynamicSmemBytes = (size_t)kCorrTile * g.Nz * sizeof(double2);
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  for (;; ncta /= 2) {
    cfg.gridDim = (unsigned)(nst * ncta);
    at[0].val.clusterDim.x = (unsigned)ncta;
    int fit = 0;
    if (ncta == 1) break;
    if (cudaOccupancyMaxActiveClusters(&fit, k_l2_diff, &cfg) == cudaSuccess && fit > 0) break;
    cudaGetLastError();   // (a size that the device refuses)
  }
  cudaError_t e = cudaLaunchKernelEx(&cfg, k_l2_diff, g, t.gram, A, Bm, out, ncta);
  count();
  return e == cudaSuccess ? cudaGetLastError() : e;
}

// ---------------------------------------------------------------------------
// Native grid <-> spectral state.
// ---------------------------------------------------------------------------
// modes[fld][j][m] = (1/Nx) sum_i g[fld][j][i] exp(-i k_m x_i)
__global__ void k_grid_to_modes(Grid g, const double2* twn, const double* grid, double* modes) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 3L * g.Nz * g.nm) return;
  const int m = idx % g.nm;
  const int j = (idx / g.nm) % g.Nz;
  const int fld = idx / ((long)g.nm * g.Nz);
  const double* row = grid + ((size_t)fld * g.Nz + j) * g.Nx;
  double2 acc = {0.0, 0.0};
  for (int i = 0; i < g.Nx; ++i) {
    const double2 w = twn[((long)m * i) % g.Nx];
    acc.x = fma(row[i], w.x, acc.x);
    acc.y = fma(row[i], w.y, acc.y);
  }
  st2(modes + idx * 2, (1.0 / g.Nx) * acc);
}

// coefficients by exact interpolation; psi_m = i w_m / k (m >= 1), U = <u>_x.
__global__ void k_modes_to_state(Grid g, const double* Wn, const double* modes, double* X) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long)g.Nz * g.nm) return;
  const int m = idx % g.nm, n = idx / g.nm;
  double2 c[3];
  for (int fld = 0; fld < 3; ++fld) {
    double2 acc = {0.0, 0.0};
    for (int j = 0; j < g.Nz; ++j) {
      const double2 v = ld2(modes + (((size_t)fld * g.Nz + j) * g.nm + m) * 2);
      const double wv = Wn[(size_t)n * g.Nz + j];
      acc.x = fma(wv, v.x, acc.x);
      acc.y = fma(wv, v.y, acc.y);
    }
    c[fld] = acc;
  }
  double2 T = c[0];
  double2 P;
  if (m == 0) {
    T.y = 0.0;
    P = make_double2(c[1].x, 0.0);
  } else {
    const double k = g.kfac * m;
    P = (1.0 / k) * times_i(c[2]);
  }
  st2(X + soff(g, 0, n, m), T);
  st2(X + soff(g, 1, n, m), P);
}

cudaError_t launch_set_state(const Grid& g, const Tables& t, const double* gT, const double* gu, const double* gw,
                             double* scratch, double* X, cudaStream_t s) {
  // gT, gu, gw are consecutive [3][Nz][Nx] in device scratch (gT points at it)
  (void)gu;
  (void)gw;
  double* modes = scratch;
  k_grid_to_modes<<<nblk(3L * g.Nz * g.nm, 128), 128, 0, s>>>(g, t.twn, gT, modes);
  k_modes_to_state<<<nblk((long)g.Nz * g.nm, 128), 128, 0, s>>>(g, t.Wn, modes, X);
  count(2);
  return cudaGetLastError();
}

// native-point mode values of T, u, w: modes[fld][j][m]
__global__ void k_state_to_modes(Grid g, const double* Vn, const double* Vn1, const double* X, double* modes) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (long)g.Nz * g.nm) return;
  const int m = idx % g.nm, j = idx / g.nm;
  double2 T = {0, 0}, P = {0, 0}, P1 = {0, 0};
  for (int n = 0; n < g.Nz; ++n) {
    const double v = Vn[(size_t)j * g.Nz + n], v1 = Vn1[(size_t)j * g.Nz + n];
    const double2 xt = ld2(X + soff(g, 0, n, m)), xp = ld2(X + soff(g, 1, n, m));
    T = T + v * xt;
    P = P + v * xp;
    P1 = P1 + v1 * xp;
  }
  double2 u, w;
  if (m == 0) {
    u = make_double2(P.x, 0.0);
    w = make_double2(0.0, 0.0);
  } else {
    const double k = g.kfac * m;
    u = 2.0 * P1;
    w = -k * times_i(P);
  }
  const size_t fsz = (size_t)g.Nz * g.nm * 2;
  st2(modes + 0 * fsz + idx * 2, T);
  st2(modes + 1 * fsz + idx * 2, u);
  st2(modes + 2 * fsz + idx * 2, w);
}

// grid[fld][j][i] = Re c_0 + 2 sum_{m>=1} Re(c_m exp(i k_m x_i))
__global__ void k_modes_to_grid(Grid g, const double2* twn, const double* modes, double* grid) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= 3L * g.Nz * g.Nx) return;
  const int i = idx % g.Nx;
  const int j = (idx / g.Nx) % g.Nz;
  const int fld = idx / ((long)g.Nx * g.Nz);
  const double* c = modes + ((size_t)fld * g.Nz + j) * g.nm * 2;
  double acc = c[0];
  for (int m = 1; m < g.nm; ++m) {
    const double2 w = twn[((long)m * i) % g.Nx];     // exp(-i...) -> use conj
    const double2 cm = ld2(c + 2 * m);
    acc += 2.0 * (cm.x * w.x + cm.y * w.y);          // Re(c * conj(w))
  }
  grid[idx] = acc;
}

cudaError_t launch_get_state(const Grid& g, const Tables& t, const double* X, double* scratch, double* gT,
                             double* gu, double* gw, cudaStream_t s) {
  (void)gu;
  (void)gw;
  double* modes = scratch;
  k_state_to_modes<<<nblk((long)g.Nz * g.nm, 128), 128, 0, s>>>(g, t.Vn, t.Vn1, X, modes);
  k_modes_to_grid<<<nblk(3L * g.Nz * g.Nx, 128), 128, 0, s>>>(g, t.twn, modes, gT);
  count(2);
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Parareal transfer and correction (Eq. 20).
// ---------------------------------------------------------------------------
__global__ void k_restrict(Grid gf, Grid gc, const double* Xf, double* Xc, int B) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long per = 2L * gc.Nz * gc.nm;
  if (idx >= per * B) return;
  const int b = (int)(idx / per);
  const long r = idx - (long)b * per;
  const int m = r % gc.nm;
  const int n = (r / gc.nm) % gc.Nz;
  const int f = r / ((long)gc.nm * gc.Nz);
  st2(Xc + (size_t)b * state_doubles(gc) + soff(gc, f, n, m), ld2(Xf + (size_t)b * state_doubles(gf) + soff(gf, f, n, m)));
}

cudaError_t launch_restrict(const Grid& gf, const Grid& gc, const double* Xf, double* Xc, int B, cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  k_restrict<<<nblk(2L * gc.Nz * gc.nm * B, 128), 128, 0, s>>>(gf, gc, Xf, Xc, B);
  count();
  return cudaGetLastError();
}

__global__ void k_prolong(Grid gf, Grid gc, const double* Xc, double* Xf, int B) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long per = 2L * gf.Nz * gf.nm;
  if (idx >= per * B) return;
  const int b = (int)(idx / per);
  const long r = idx - (long)b * per;
  const int m = r % gf.nm;
  const int n = (r / gf.nm) % gf.Nz;
  const int f = r / ((long)gf.nm * gf.Nz);
  double2 v = {0.0, 0.0};
  if (m < gc.nm && n < gc.Nz) v = ld2(Xc + (size_t)b * state_doubles(gc) + soff(gc, f, n, m));
  st2(Xf + (size_t)b * state_doubles(gf) + soff(gf, f, n, m), v);
}

cudaError_t launch_prolong(const Grid& gf, const Grid& gc, const double* Xc, double* Xf, int B, cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  k_prolong<<<nblk(2L * gf.Nz * gf.nm * B, 128), 128, 0, s>>>(gf, gc, Xc, Xf, B);
  count();
  return cudaGetLastError();
}

// U = F + (prolong(Gnew) - prolong(Gold)), elementwise in that order (Eq. 20).
__global__ void k_correct(Grid gf, Grid gc, const double* Ff, const double* Gnew, const double* Gold, double* U,
                          int B) {
  const long idx = (long)blockIdx.x * blockDim.x + threadIdx.x;
  const long per = 2L * gf.Nz * gf.nm;
  if (idx >= per * B) return;
  const int b = (int)(idx / per);
  const long r = idx - (long)b * per;
  const int m = r % gf.nm;
  const int n = (r / gf.nm) % gf.Nz;
  const int f = r / ((long)gf.nm * gf.Nz);
  const size_t Sf = state_doubles(gf), Sc = state_doubles(gc);
  double2 d = {0.0, 0.0};
  if (m < gc.nm && n < gc.Nz)
    d = ld2(Gnew + (size_t)b * Sc + soff(gc, f, n, m)) - ld2(Gold + (size_t)b * Sc + soff(gc, f, n, m));
  st2(U + (size_t)b * Sf + soff(gf, f, n, m), ld2(Ff + (size_t)b * Sf + soff(gf, f, n, m)) + d);
}

cudaError_t launch_correct(const Grid& gf, const Grid& gc, const double* Ff, const double* Gnew, const double* Gold,
                           double* Uout, int B, cudaStream_t s) {
  if (B <= 0) return cudaSuccess;
  k_correct<<<nblk(2L * gf.Nz * gf.nm * B, 128), 128, 0, s>>>(gf, gc, Ff, Gnew, Gold, Uout, B);
  count();
  return cudaGetLastError();
}

// One slice of a Parareal sweep (Sec. 3.1, Eq. 20) fused with its norms (Sec. 3.7).
// mode 0 (the coarse sweep U^0):  U = prolong(Gnew).
// mode 1 (a correction):          U = F + (prolong(Gnew) - prolong(Gold)), elementwise in that order.
// Both: Gold <- Gnew (the coarse value of this iterate, which the next
// iteration subtracts); C <- restrict(U) (the next coarse step's input: the
// coarse modes of U; C may be the Gnew buffer, each element is read before
// it is written); Fnext <- U when not null (the next iteration's fine input);
// mode 1 with Uprev: norms[0] = ||T(U) - T(Uprev)||^2, norms[1] = ||T(U)||^2
// (L2 over the domain, in the order of k_l2_diff: the same bits).
// Block per tile of kCorrTile Fourier modes, all Chebyshev indices of both
// fields; the blocks' partial sums are added in block order by the last block
// to finish (partial[2 * gridDim.x], counter: left at zero).
__global__ void __launch_bounds__(kCorrThreads) k_correct_norm(
    Grid gf, Grid gc, const double* __restrict__ gram, int mode, const double* Ff, const double* Gnew, double* Gold,
    double* C, const double* __restrict__ Uprev, double* __restrict__ U, double* __restrict__ Fnext,
    double* partial, unsigned* counter, double* norms) {
  __shared__ double red[kCorrThreads];
  extern __shared__ double2 sd[];             // [kCorrTile][Nz]: T(U) - T(Uprev) of the tile's modes
  __shared__ bool last;
  const int m0 = blockIdx.x * kCorrTile;
  const int tm = min(kCorrTile, gf.nm - m0);
  const int per = 2 * gf.Nz * tm;
  const bool with_norms = mode == 1 && Uprev != nullptr;
  for (int it = threadIdx.x; it < per; it += blockDim.x) {
    const int dm = it % tm, n = (it / tm) % gf.Nz, f = it / (tm * gf.Nz);
    const int m = m0 + dm;
    const size_t o = soff(gf, f, n, m);
    const bool coarse = m < gc.nm && n < gc.Nz;
    const size_t oc = coarse ? soff(gc, f, n, m) : 0;
    double2 u;
    if (mode == 0) {
      u = coarse ? ld2(Gnew + oc) : make_double2(0.0, 0.0);
      if (coarse) st2(Gold + oc, u);
    } else {
      double2 d = {0.0, 0.0};
      if (coarse) {
        const double2 gn = ld2(Gnew + oc);
        d = gn - ld2(Gold + oc);
        st2(Gold + oc, gn);
      }
      u = ld2(Ff + o) + d;
      if (coarse) st2(C + oc, u);
    }
    st2(U + o, u);
    if (Fnext) st2(Fnext + o, u);
    if (with_norms && f == 0) sd[dm * gf.Nz + n] = u - ld2(Uprev + o);
  }
  if (!with_norms) return;
  __syncthreads();
  // sum_m w_m Re(conj(d_i) sum_j gram_ij d_j), i, j of equal parity; the same for U
  double acc_d = 0.0, acc_u = 0.0;
  for (int it = threadIdx.x; it < tm * gf.Nz; it += blockDim.x) {
    const int dm = it % tm, i = it / tm, m = m0 + dm;
    const double2 di = sd[dm * gf.Nz + i];
    const double2 ui = ld2(U + soff(gf, 0, i, m));
    double2 s = {0.0, 0.0}, t = {0.0, 0.0};
    for (int j = (i & 1); j < gf.Nz; j += 2) {
      const double gij = __ldg(gram + (size_t)i * gf.Nz + j);
      s = gram_acc(s, gij, sd[dm * gf.Nz + j]);
      t = gram_acc(t, gij, ld2(U + soff(gf, 0, j, m)));
    }
    const double w = m == 0 ? 1.0 : 2.0;
    acc_d = l2_term(acc_d, w, di, s);
    acc_u = l2_term(acc_u, w, ui, t);
  }
  acc_d = block_sum(acc_d, red);
  acc_u = block_sum(acc_u, red);
  if (threadIdx.x == 0) {
    partial[2 * blockIdx.x] = acc_d;
    partial[2 * blockIdx.x + 1] = acc_u;
    __threadfence();
    last = atomicAdd(counter, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last || threadIdx.x != 0) return;
  __threadfence();
  double sdiff = 0.0, su = 0.0;
  for (unsigned bidx = 0; bidx < gridDim.x; ++bidx) {
    sdiff += *((volatile double*)partial + 2 * bidx);
    su += *((volatile double*)partial + 2 * bidx + 1);
  }
  norms[0] = 0.5 * gf.Lx * sdiff;
  norms[1] = 0.5 * gf.Lx * su;
  *counter = 0u;
}

int correct_norm_blocks(const Grid& gf) { return (gf.nm + kCorrTile - 1) / kCorrTile; }

cudaError_t launch_correct_norm(const Grid& gf, const Grid& gc, const Tables& tf, int mode, const double* Ff,
                                const double* Gnew, double* Gold, double* C, const double* Uprev, double* U,
                                double* Fnext, double* partial, unsigned* counter, double* norms, cudaStream_t s) {
  static int allowed = 48 * 1024;
  const size_t smem = (size_t)kCorrTile * gf.Nz * sizeof(double2);
  cudaError_t e = allow_smem(k_correct_norm, (int)smem, allowed);
  if (e != cudaSuccess) return e;
  k_correct_norm<<<correct_norm_blocks(gf), kCorrThreads, smem, s>>>(gf, gc, tf.gram, mode, Ff, Gnew, Gold, C, Uprev,
                                                                     U, Fnext, partial, counter, norms);
  count();
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------
// Nusselt numbers without any allocation: the scratch of the explicit-term
// evaluation (z-inverse fields, row outputs, the <wT>_x profile and the three
// results) lives in one file-scope device array, shared by every call on a
// device.  Its device address is looked up once per device, with that device
// current, on the first call there.
// ---------------------------------------------------------------------------
static __device__ __align__(256) double g_static_scratch[kStaticScratchCapacity];
constexpr int kMaxDevices = 64;
static std::atomic<double*> g_static_ptr[kMaxDevices] = {};

// Layout: Z, Q, the <wT>_x profile (Mz rounded up to even), then 8 doubles:
// the three Nusselt numbers and, in the fifth, the int error bits of the call.
size_t static_scratch_doubles_needed(const Grid& g) {
  return z_doubles(g) + q_doubles(g) + (size_t)((g.Mz + 1) & ~1) + 8;
}

cudaError_t launch_nusselt_static(const Grid& g, const Tables& t, const double* X, double* host_out3,
                                  int* host_flags, cudaStream_t s) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= kMaxDevices) return cudaErrorInvalidDevice;
  double* base = g_static_ptr[dev].load();
  if (base == nullptr) {
    // two threads may both look it up; they store the same address
    e = cudaGetSymbolAddress((void**)&base, g_static_scratch);
    if (e != cudaSuccess) return e;
    g_static_ptr[dev].store(base);
  }
  Work w{};
  w.Z = base;
  w.Q = w.Z + z_doubles(g);
  w.wT = w.Q + q_doubles(g);
  w.small = w.wT + ((g.Mz + 1) & ~1);
  w.flags = reinterpret_cast<int*>(w.small + 4);   // the call's error bits (the tensor-core waits)
  w.err = w.flags;
  w.prof = nullptr;
  e = cudaMemsetAsync(w.flags, 0, sizeof(int), s);   // the only element read before this call writes it
  if (e != cudaSuccess) return e;
  e = launch_nusselt(g, t, w, X, w.small, s);
  if (e != cudaSuccess) return e;
  double res[5];
  e = cudaMemcpyAsync(res, w.small, sizeof(res), cudaMemcpyDeviceToHost, s);
  if (e != cudaSuccess) return e;
  e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return e;
  for (int i = 0; i < 3; ++i) host_out3[i] = res[i];
  std::memcpy(host_flags, &res[4], sizeof(int));
  return cudaSuccess;
}

}  // namespace rbc
