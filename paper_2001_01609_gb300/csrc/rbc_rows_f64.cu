// Row kernel of the FP64 mode: x inverse FFTs, advective products, x forward FFT
// (k_rows: a block per row; k_rows_cl: a cluster per row, for few rows).
//
// Bound: the FP64 pipe (2 operations per clock and SM, 84 % active at 256 x 64, 32
// states); with few rows the latency of the passes.  Measured (GB300, per launch):
// 256 x 64, 32 states 491 us, one state 41 us; 512 x 128, 3 states 207 us; 64 x 32,
// 23 states 57 us; 128 x 32, one state 20.5 us.  The same transforms in 64-bit fixed
// point on the integer pipe took 107, 16.6, 46, 16.4 and 14.4 us and are not used:
// rows with a broad spectrum lost bits (white modes, 1536 points: mean flow within
// 1e-12 of the products' x-mean, here 3e-15), and any other rounding of the FP64 mode
// moves the small defects of converging Parareal iterates by 1e-11 and more.
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include <algorithm>

#include "rbc_internal.h"

namespace rbc {

namespace {

using V = double2;

__device__ __forceinline__ V ld2(const double* p) { return *reinterpret_cast<const V*>(p); }
__device__ __forceinline__ void st2(double* p, V v) { *reinterpret_cast<V*>(p) = v; }
__device__ __forceinline__ V operator+(V a, V b) { return make_double2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ V operator-(V a, V b) { return make_double2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ V operator*(double s, V a) { return make_double2(s * a.x, s * a.y); }
// (roundings written out, so that the bits do not depend on contraction)
__device__ __forceinline__ V cmul(V a, V b) {
  return make_double2(fma(a.x, b.x, -(a.y * b.y)), fma(a.x, b.y, a.y * b.x));
}
__device__ __forceinline__ V conj2(V a) { return make_double2(a.x, -a.y); }
__device__ __forceinline__ V times_i(V a) { return make_double2(-a.y, a.x); }

__device__ __forceinline__ bool slice_active(const int* nsteps, const int* step, int b) {
  return nsteps == nullptr || *step < nsteps[b];
}

// ---------------------------------------------------------------------------
// Shared-memory mixed-radix Stockham FFT of length N = 3 * 2^p (radices
// 4, ..., 4, [2], 3) applied to na arrays of length N at once (array a at
// [a * N]).  y_q = sum_r x_r exp(sign 2 pi i q r / N), unnormalised.
// Ping-pongs between a and b; returns the buffer holding the results.
// ---------------------------------------------------------------------------
__device__ V* fft_smem(V* a, V* b, int N, int na, int sign, const V* tw) {
  int p = 0;
  for (int M = N / 3; M > 1; M >>= 1) ++p;
  const int nr = p / 2 + (p & 1) + 1;
  int Ns = 1, lns = 0;                                 // Ns = 2^lns
  V* x = a;
  V* y = b;
  const double s3 = 0.86602540378443864676 * (double)sign;   // sign * sqrt(3)/2
  const double sg = (double)sign;
  for (int pass = 0; pass < nr; ++pass) {
    const int R = (pass < p / 2) ? 4 : ((p & 1) && pass == p / 2) ? 2 : 3;
    // N = 3 2^p: N / R and N / (Ns R) by shifts (the radix-3 pass leaves 2^p)
    const int nb = R == 4 ? N >> 2 : R == 2 ? N >> 1 : 1 << p;
    const int stride = nb >> lns;
    for (int it = threadIdx.x; it < na * nb; it += blockDim.x) {
      const int arr = na == 1 ? 0 : it / nb, jj = it - arr * nb;   // one array: no division
      const V* xa = x + arr * N;
      V* ya = y + arr * N;
      const int k = jj & (Ns - 1);                  // Ns is a power of two (the radix-3 pass is last)
      V v[4];
      for (int r = 0; r < R; ++r) v[r] = xa[jj + r * nb];
      if (Ns > 1) {
        // k < Ns and r < R, so k r stride < Ns R stride = N: the index needs no reduction
        const int kstr = k * stride;
        for (int r = 1; r < R; ++r) {
          V wv = tw[kstr * r];
          if (sign > 0) wv.y = -wv.y;
          v[r] = cmul(v[r], wv);
        }
      }
      const int base = (jj - k) * R + k;            // (jj / Ns) Ns R + k
      if (R == 2) {
        ya[base] = v[0] + v[1];
        ya[base + Ns] = v[0] - v[1];
      } else if (R == 4) {
        const V a0 = v[0] + v[2], a1 = v[0] - v[2];
        const V b0 = v[1] + v[3], b1 = v[1] - v[3];
        const V ib1 = sg * times_i(b1);
        ya[base] = a0 + b0;
        ya[base + Ns] = a1 + ib1;
        ya[base + 2 * Ns] = a0 - b0;
        ya[base + 3 * Ns] = a1 - ib1;
      } else {
        const V t1 = v[1] + v[2], t2 = v[1] - v[2];
        const V m1 = v[0] - 0.5 * t1;
        // m1 +- s3 i t2 with one rounding per part (explicit fma)
        ya[base] = v[0] + t1;
        ya[base + Ns] = make_double2(fma(-s3, t2.y, m1.x), fma(s3, t2.x, m1.y));
        ya[base + 2 * Ns] = make_double2(fma(s3, t2.y, m1.x), fma(-s3, t2.x, m1.y));
      }
    }
    __syncthreads();
    V* tmp = x;
    x = y;
    y = tmp;
    Ns *= R;
    lns += R == 4 ? 2 : R == 2 ? 1 : 0;                // the radix-3 pass is the last
  }
  return x;
}

// Shared memory of k_rows: two ping-pong sets of 5 complex rows and the
// twiddles (11 Mx complex values); lean: 5 + 3 rows and the twiddles (9 Mx),
// the inverse FFTs in groups of three and two rows; or, when neither fits, two
// single rows, the twiddles and 9 real fields, with the five inverse FFTs in turn.
size_t batched_bytes(const Grid& g) { return (size_t)g.Mx * 11 * sizeof(V); }
size_t lean_bytes(const Grid& g) { return (size_t)g.Mx * 9 * sizeof(V); }
size_t serial_bytes(const Grid& g) { return (size_t)g.Mx * (3 * sizeof(V) + 9 * sizeof(double)); }

// Pair pr of real fields (2 pr, 2 pr + 1) of row j as one complex spectrum of
// length Mx: C = A + iB with the Hermitian extensions, zero beyond the kept modes.
__device__ __forceinline__ V rows_packed(const Grid& g, const double* zrow, size_t fs, int pr, int x) {
  const int fa = 2 * pr, fb = 2 * pr + 1, Mx = g.Mx, nm = g.nm;
  const double* za = zrow + fa * fs;
  const double* zb = zrow + fb * fs;
  V c = make_double2(0.0, 0.0);
  if (x < nm) {
    const V a = ld2(za + 2 * x);
    const V bb = (fb < 9) ? ld2(zb + 2 * x) : make_double2(0.0, 0.0);
    c = a + times_i(bb);
  } else if (x > Mx - nm) {
    const int m = Mx - x;
    const V a = ld2(za + 2 * m);
    const V bb = (fb < 9) ? ld2(zb + 2 * m) : make_double2(0.0, 0.0);
    c = conj2(a) + times_i(conj2(bb));
  }
  return c;
}

// Two block sums over the first 256 threads at once (the others pass nothing
// and only meet the barriers): for each value the tree of block_sum at 256
// threads, whatever blockDim is, with half the barriers of two calls.
__device__ double2 block_sum256_2(double a, double b, double2* red) {
  if (threadIdx.x < 256) red[threadIdx.x] = make_double2(a, b);
  __syncthreads();
  for (int s = 128; s >= 32; s >>= 1) {
    if ((int)threadIdx.x < s) {
      const double2 u = red[threadIdx.x], v = red[threadIdx.x + s];
      red[threadIdx.x] = make_double2(u.x + v.x, u.y + v.y);
    }
    __syncthreads();
  }
  if (threadIdx.x < 32) {
    double x = red[threadIdx.x].x, y = red[threadIdx.x].y;
#pragma unroll
    for (int s = 16; s > 0; s >>= 1) {
      x += __shfl_down_sync(0xffffffffu, x, s);
      y += __shfl_down_sync(0xffffffffu, y, s);
    }
    if (threadIdx.x == 0) red[0] = make_double2(x, y);
  }
  __syncthreads();
  const double2 r = red[0];
  __syncthreads();
  return r;
}

// ---------------------------------------------------------------------------
// Row kernel (k_rows).  Block per (slice, padded row j).  Pairs of real fields
// share one complex inverse FFT (C = A + iB with the Hermitian extensions);
// products in advective form (Eqs. 3, 5):
//   N_T = u T_x + w T_z,  N_omega = u omega_x + w omega_z,
//   <N_u>_x = <u u_x + w u_z>_x,  <w T>_x;
// one packed forward FFT (N_T + i N_omega), truncation to m < nm.
// Q[b][0][j][m] = N_T, Q[b][1][j][m] = N_omega (m >= 1), (<N_u>, 0) at m = 0.
// The x-means are summed from per-point terms staged in shared memory: thread
// t < 256 adds x = t, t + 256, ..., then a 256-wide tree, so the bits do not depend on the block size (256 to 1024
// threads, a launch shape) and equal those of k_rows_cl.
// ---------------------------------------------------------------------------
__device__ void rows_item(const Grid& g, const V* __restrict__ tw, const double* __restrict__ Z, double* __restrict__ Q,
                          double* __restrict__ wT, int B, int batched, int lean, const int* nsteps, int stepidx,
                          int blk) {
  extern __shared__ __align__(16) unsigned char rsm[];
  const int b = blk / g.Mz, j = blk - b * g.Mz;
  if (b >= B || !(nsteps == nullptr || stepidx < nsteps[b])) return;
  const int Mx = g.Mx, nm = g.nm;
  __shared__ double2 red[256];
  const size_t fs = (size_t)g.Mz * nm * 2;
  const double* zrow = Z + (size_t)b * 9 * fs + (size_t)j * nm * 2;
  const V* fld;      // field value at x: real/imag parts of the five packed rows
  const V* fld3 = nullptr;   // rows 3 and 4 (batched: fld + 3 Mx unless lean)
  V* A;
  V* Bf;
  V* tws;
  V* P = nullptr;    // free rows after the inverse FFTs: products, scratch, x-mean terms
  V* P2 = nullptr;
  double* vU = nullptr;
  double* fr = nullptr;
  if (batched) {
    // the five packed rows and the FFT scratch: five more rows, or (lean) three,
    // the inverse FFTs then running in groups of three and two rows (the same
    // arithmetic per row; less shared memory, more blocks per SM)
    A = reinterpret_cast<V*>(rsm);
    Bf = A + 5 * Mx;
    tws = Bf + (lean ? 3 : 5) * Mx;
    for (int x = threadIdx.x; x < Mx; x += blockDim.x) tws[x] = __ldg(tw + x);
    for (int pr = 0; pr < 5; ++pr)
      for (int x = threadIdx.x; x < Mx; x += blockDim.x) A[pr * Mx + x] = rows_packed(g, zrow, fs, pr, x);
    __syncthreads();
    if (!lean) {
      fld = fft_smem(A, Bf, Mx, 5, +1, tws);
      fld3 = fld + 3 * Mx;
      P = (fld == A) ? Bf : A;                 // the five rows not holding the fields
      vU = reinterpret_cast<double*>(P + Mx);
      P2 = (P == A) ? Bf : A;                  // a field row, free once the products are formed
    } else {
      fld = fft_smem(A, Bf, Mx, 3, +1, tws);
      V* fr3 = fld == A ? Bf : A;              // rows free after the first group
      fld3 = fft_smem(A + 3 * Mx, fr3, Mx, 2, +1, tws);
      // three free rows: the scratch (even pass count) or A[2..4] (odd)
      P = fld == A ? Bf : A + 2 * Mx;
      vU = reinterpret_cast<double*>(P + Mx);
      P2 = P + 2 * Mx;
    }
  } else {
    A = reinterpret_cast<V*>(rsm);
    Bf = A + Mx;
    tws = Bf + Mx;
    fr = reinterpret_cast<double*>(tws + Mx);
    for (int x = threadIdx.x; x < Mx; x += blockDim.x) tws[x] = __ldg(tw + x);
    for (int pr = 0; pr < 5; ++pr) {
      for (int x = threadIdx.x; x < Mx; x += blockDim.x) A[x] = rows_packed(g, zrow, fs, pr, x);
      __syncthreads();
      const V* res = fft_smem(A, Bf, Mx, 1, +1, tws);
      for (int x = threadIdx.x; x < Mx; x += blockDim.x) {
        fr[(2 * pr) * Mx + x] = res[x].x;
        if (pr < 4) fr[(2 * pr + 1) * Mx + x] = res[x].y;
      }
      __syncthreads();
    }
    fld = nullptr;
    P = A;
    P2 = Bf;
    vU = reinterpret_cast<double*>(P2);            // the scratch row holds the 2 Mx terms
  }
  auto field = [&](int fi, int x) -> double {
    if (fld) {
      const int k = fi >> 1;
      const V v = k < 3 ? fld[k * Mx + x] : fld3[(k - 3) * Mx + x];
      return (fi & 1) ? v.y : v.x;
    }
    return fr[fi * Mx + x];
  };
  // per-point x-mean terms
  double* vW = vU + Mx;
  for (int x = threadIdx.x; x < Mx; x += blockDim.x) {
    const double u = field(0, x), w = field(1, x);
    const double nO = fma(u, field(2, x), w * field(3, x));
    vU[x] = fma(u, field(4, x), w * field(5, x));
    const double nT = fma(u, field(7, x), w * field(8, x));
    vW[x] = w * field(6, x);
    P[x] = make_double2(nT, nO);
  }
  __syncthreads();
  double nU = 0.0, wt = 0.0;
  if (threadIdx.x < 256)
    for (int x = threadIdx.x; x < Mx; x += 256) {
      nU += vU[x];
      wt += vW[x];
    }
  const double2 sUW = block_sum256_2(nU, wt, red);
  const double sU = sUW.x, sW = sUW.y;
  const V* S = fft_smem(P, P2, Mx, 1, -1, tws);
  const double inv = 1.0 / Mx;
  const double half = 0.5 * inv;
  const size_t qs = (size_t)g.Mz * nm * 2;
  double* q0 = Q + (size_t)b * 2 * qs + (size_t)j * nm * 2;
  double* q1 = q0 + qs;
  for (int m = threadIdx.x; m < nm; m += blockDim.x) {
    const V cm = S[m];
    const V cn = conj2(S[m == 0 ? 0 : Mx - m]);
    const V s = cm + cn, d = cm - cn;
    st2(q0 + 2 * m, make_double2(half * s.x, half * s.y));
    if (m == 0)
      st2(q1, make_double2(sU / Mx, 0.0));
    else
      st2(q1 + 2 * m, make_double2(half * d.y, -half * d.x));
  }
  if (threadIdx.x == 0) wT[(size_t)b * g.Mz + j] = sW / Mx;
}

__global__ void __launch_bounds__(1024) k_rows(Grid g, const V* __restrict__ tw, const double* __restrict__ Z,
                                              double* __restrict__ Q, double* __restrict__ wT, int B, int batched,
                                              int lean, const int* nsteps, const int* step) {
  pdl_wait();
  rows_item(g, tw, Z, Q, wT, B, batched, lean, nsteps, nsteps ? *step : 0, blockIdx.x);
}

// ---------------------------------------------------------------------------
// Row kernel for small batches (k_rows_cl): the same arithmetic as k_rows,
// spread over a cluster of five CTAs per row so that a single slice uses five
// times as many SMs' FP64 pipes.  CTA c runs the inverse FFT of field pair c
// (fields 2c, 2c+1) in its shared memory; after a cluster barrier every CTA
// forms the products for its share of the x points, reading the nine fields
// from the five CTAs through distributed shared memory, and writes them, with
// the per-point terms of the two x-means, into CTA 0.  After a second barrier
// CTA 0 sums the x-means with exactly the per-thread order and tree of k_rows
// (256 threads) and runs the forward FFT, so the results are bit for bit
// those of k_rows.
// ---------------------------------------------------------------------------
constexpr int kRowsCluster = 5;
constexpr int kRowsThreads = 256;

__global__ void __cluster_dims__(kRowsCluster, 1, 1) __launch_bounds__(kRowsThreads)
    k_rows_cl(Grid g, const V* __restrict__ tw, const double* __restrict__ Z, double* __restrict__ Q,
              double* __restrict__ wT, int B, const int* nsteps, const int* step) {
  namespace cg = cooperative_groups;
  extern __shared__ __align__(16) unsigned char csm[];
  __shared__ double2 red[kRowsThreads];
  pdl_wait();
  cg::cluster_group cl = cg::this_cluster();
  const int c = (int)cl.block_rank();
  const int row = blockIdx.x / kRowsCluster;
  const int b = row / g.Mz, j = row - b * g.Mz;
  // uniform over the cluster (same b and step): no CTA reaches a cluster barrier alone
  if (b >= B || !slice_active(nsteps, step, b)) return;
  const int Mx = g.Mx, nm = g.nm;
  V* A = reinterpret_cast<V*>(csm);
  V* Bf = A + Mx;
  V* tws = Bf + Mx;
  V* P = tws + Mx;
  V* P2 = P + Mx;
  double* vU = reinterpret_cast<double*>(P2 + Mx);
  double* vW = vU + Mx;
  const size_t fs = (size_t)g.Mz * nm * 2;
  const double* zrow = Z + (size_t)b * 9 * fs + (size_t)j * nm * 2;
  for (int x = threadIdx.x; x < Mx; x += blockDim.x) {
    tws[x] = __ldg(tw + x);
    A[x] = rows_packed(g, zrow, fs, c, x);
  }
  __syncthreads();
  const V* res = fft_smem(A, Bf, Mx, 1, +1, tws);   // same buffer in every CTA
  cl.sync();
  const V* fr[kRowsCluster];
#pragma unroll
  for (int r = 0; r < kRowsCluster; ++r) fr[r] = cl.map_shared_rank(res, r);
  V* P0 = cl.map_shared_rank(P, 0);
  double* vU0 = cl.map_shared_rank(vU, 0);
  double* vW0 = cl.map_shared_rank(vW, 0);
  auto field = [&](int fi, int x) -> double {
    const V v = fr[fi >> 1][x];
    return (fi & 1) ? v.y : v.x;
  };
  const int per = (Mx + kRowsCluster - 1) / kRowsCluster;
  const int x0 = c * per, x1 = min(Mx, x0 + per);
  for (int x = x0 + threadIdx.x; x < x1; x += blockDim.x) {
    const double u = field(0, x), w = field(1, x);
    const double nO = fma(u, field(2, x), w * field(3, x));
    vU0[x] = fma(u, field(4, x), w * field(5, x));
    const double nT = fma(u, field(7, x), w * field(8, x));
    vW0[x] = w * field(6, x);
    P0[x] = make_double2(nT, nO);
  }
  cl.sync();
  if (c != 0) return;
  // x-means: thread t adds x = t, t + 256, ... from 0, then the tree of k_rows
  double nU = 0.0, wt = 0.0;
  for (int x = threadIdx.x; x < Mx; x += blockDim.x) {
    nU += vU[x];
    wt += vW[x];
  }
  const double2 sUW = block_sum256_2(nU, wt, red);   // kRowsThreads = 256: the same tree
  const double sU = sUW.x, sW = sUW.y;
  const V* S = fft_smem(P, P2, Mx, 1, -1, tws);
  const double inv = 1.0 / Mx;
  const double half = 0.5 * inv;
  const size_t qs = (size_t)g.Mz * nm * 2;
  double* q0 = Q + (size_t)b * 2 * qs + (size_t)j * nm * 2;
  double* q1 = q0 + qs;
  for (int m = threadIdx.x; m < nm; m += blockDim.x) {
    const V cm = S[m];
    const V cn = conj2(S[m == 0 ? 0 : Mx - m]);
    const V s2 = cm + cn, d = cm - cn;
    st2(q0 + 2 * m, make_double2(half * s2.x, half * s2.y));
    if (m == 0)
      st2(q1, make_double2(sU / Mx, 0.0));
    else
      st2(q1 + 2 * m, make_double2(half * d.y, -half * d.x));
  }
  if (threadIdx.x == 0) wT[(size_t)b * g.Mz + j] = sW / Mx;
}

}  // namespace

bool rows_f64_batched(const Grid& g) { return batched_bytes(g) <= 200 * 1024; }
size_t rows_f64_bytes(const Grid& g, bool lean) {
  return rows_f64_batched(g) ? (lean ? lean_bytes(g) : batched_bytes(g)) : serial_bytes(g);
}
size_t rows_f64_cl_bytes(const Grid& g) {
  // A, Bf, twiddles, P, P2 (complex) and two real per-point arrays
  return (size_t)g.Mx * (5 * sizeof(V) + 2 * sizeof(double));
}

namespace {
// The lean layout by default where the full one leaves room for a single block per SM
// and the lean one for two (512 x 128: one state 107 us, 115 in the full layout; 16
// states 1057 and 1194).
bool lean_default(const Grid& g) {
  return rows_f64_batched(g) && batched_bytes(g) > 113 * 1024 && lean_bytes(g) <= 113 * 1024;
}
// A cluster per row up to two rows per SM, where a block per row leaves SMs idle: a
// first choice, of which the autotuner times the other side (64 x 32, one state 18.2
// us, 19.5 with a block per row; 512 x 128, one state 105 and 107; but 256 x 64, one
// state 41.4 and 36.5, three states 72 and 56).
bool use_cluster(const Grid& g, int B) { return (long)B * g.Mz <= 2L * 152 && rows_f64_cl_bytes(g) <= 200 * 1024; }

// The dynamic shared-memory allowances only ever grow, so that a later handle
// on a smaller grid does not shrink them below an earlier one's need.
template <typename F> cudaError_t allow_smem(F* fn, int need, int& allowed) {
  if (need <= allowed) return cudaSuccess;
  cudaError_t e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, need);
  if (e == cudaSuccess) allowed = need;
  return e;
}
}  // namespace

cudaError_t configure_rows_f64(const Grid& g) {
  static int a_rows = 48 * 1024, a_cl = 48 * 1024;
  cudaError_t e = allow_smem(k_rows, (int)rows_f64_bytes(g, false), a_rows);
  if (e == cudaSuccess && rows_f64_cl_bytes(g) <= 200 * 1024) e = allow_smem(k_rows_cl, (int)rows_f64_cl_bytes(g), a_cl);
  return e;
}

void rows_f64_form(const Grid& g, const Shapes& sh, int B, int* cl, int* threads, int* lean) {
  *cl = sh.rows_cl >= 0 ? sh.rows_cl : use_cluster(g, B);
  *threads = 0;
  *lean = -1;
  if (*cl) return;
  *threads = sh.rows_threads > 0 ? sh.rows_threads : kRowsThreads;
  if (rows_f64_batched(g)) *lean = sh.rows_lean >= 0 ? sh.rows_lean : lean_default(g);
}

cudaError_t launch_rows_f64(const Grid& g, const Tables& t, const Work& w, int B, const int* ns, cudaStream_t s) {
  int cl, threads, lean;
  rows_f64_form(g, w.shapes ? *w.shapes : Shapes{}, B, &cl, &threads, &lean);
  if (cl)
    return launch_pdl(w.pdl != 0, k_rows_cl, (unsigned)(B * g.Mz * kRowsCluster), kRowsThreads, rows_f64_cl_bytes(g), s,
                      g, t.tw, w.Z, w.Q, w.wT, B, ns, w.step);
  return launch_pdl(w.pdl != 0, k_rows, (unsigned)(B * g.Mz), threads, rows_f64_bytes(g, lean == 1), s, g, t.tw, w.Z,
                    w.Q, w.wT, B, rows_f64_batched(g) ? 1 : 0, lean == 1 ? 1 : 0, ns, w.step);
}

}  // namespace rbc
