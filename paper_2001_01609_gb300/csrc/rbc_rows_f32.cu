// Row kernel of the mixed mode: x inverse FFTs, advective products, x forward
// FFT in FP32.
//
// Z holds nine fields per padded row j (complex modes m < nm): u, w, d_x omega,
// d_z omega, d_x u, d_z u, T, d_x T, d_z T.  Pairs of real fields share one
// complex inverse FFT of length N = Mx = 3 2^p (C = A + iB with the Hermitian
// extensions); products in advective form (Eqs. 3, 5),
//   N_T = u T_x + w T_z,  N_omega = u omega_x + w omega_z,
//   <N_u>_x = <u u_x + w u_z>_x,  <w T>_x;
// one packed forward FFT (N_T + i N_omega), truncation to m < nm.
// Q[b][0][j][m] = N_T, Q[b][1][j][m] = N_omega (m >= 1), (<N_u>, 0) at m = 0.
//
// The FFT is the decimation-in-time sequence of radices 4, .., 4, [2], 3 (the
// roundings of each butterfly written out); up to two of its steps run in
// registers at a time: N = RA RB RC, RA = 16 or 4 (two or one radix-4 steps,
// the inputs straight from global memory), RB = 16, 4 or 1, RC = 6 or 3.  Each
// pass works in place: a butterfly's outputs take the places of its inputs, an
// odd leading dimension keeps consecutive threads in different banks.
//   A  modes -> packed spectrum, RA-point butterflies (five FFTs)
//   B  RB-point butterflies
//   C  RC-point butterflies of all five FFTs at the thread's points, products
//   D, E, F  the same three passes for the forward FFT;  G  unpacking, store
// Block: NR rows, one thread per C item (N / RC per row); items of the other
// passes are flattened over the block's rows.  SPLIT (one row per block, launches
// of at most two blocks per SM): the last inverse pass is spread over all five
// FFTs' items too, and the row's activity is checked while its values arrive.
//
// The x-means' terms are summed in unevaluated triples of FP32 (error-free
// additions: at least the 53 bits of an FP64 sum), thread by thread in x order,
// by a fixed shuffle tree and over the warps in order: the bits do not depend on
// the launch shape.  FP64 conversions and additions, two per point, took longer
// than the FFTs (an FP64 warp instruction holds its sub-partition for 64 clocks).
//
// Bound: issue slots, about 350 instructions per point, of them 220 FP32
// arithmetic; with few rows the chain of passes.  Measured (GB300, per launch; one
// radix-4 step per pass with twiddles and operands in shared memory, 18 barriers,
// before; the bits are the same): 1024 x 256, 32 states 1560 -> 568 us; 512 x 128,
// 64 states 568 -> 263 us; 256 x 64, 8 states 32.9 -> 16.4 us, one state 16.7 ->
// 12.4 us; 128 x 32, one state 12.3 -> 12.2 us, six 20.8 -> 12.4 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <type_traits>

#include "rbc_internal.h"

namespace rbc {

namespace {

using C = float2;

__device__ __forceinline__ C operator+(C a, C b) { return make_float2(a.x + b.x, a.y + b.y); }
__device__ __forceinline__ C operator-(C a, C b) { return make_float2(a.x - b.x, a.y - b.y); }
__device__ __forceinline__ C cmul(C a, C b) {
  return make_float2(fmaf(a.x, b.x, -(a.y * b.y)), fmaf(a.x, b.y, a.y * b.x));
}
template <int S> __device__ __forceinline__ C addi(C a, C d) {   // a + S i d
  return S > 0 ? make_float2(a.x - d.y, a.y + d.x) : make_float2(a.x + d.y, a.y - d.x);
}
// twiddle exp(S 2 pi i k / N) from the table of exp(-2 pi i k / N)
template <int S> __device__ __forceinline__ C tw(const C* __restrict__ t, int k) {
  C w = __ldg(t + k);
  if (S > 0) w.y = -w.y;
  return w;
}

template <int S> __device__ __forceinline__ void radix4(C& a, C& b, C& c, C& d) {
  const C a0 = a + c, a1 = a - c, b0 = b + d, b1 = b - d;
  a = a0 + b0;
  b = addi<S>(a1, b1);
  c = a0 - b0;
  d = addi<-S>(a1, b1);
}
template <int S> __device__ __forceinline__ void radix3(C& a, C& b, C& c) {
  const float s3 = 0.86602540378443864676f * (float)S;
  const C t1 = b + c, t2 = b - c;
  const C m1 = make_float2(fmaf(-0.5f, t1.x, a.x), fmaf(-0.5f, t1.y, a.y));
  a = a + t1;
  b = make_float2(fmaf(-s3, t2.y, m1.x), fmaf(s3, t2.x, m1.y));
  c = make_float2(fmaf(s3, t2.y, m1.x), fmaf(-s3, t2.x, m1.y));
}

// R = 16 or 4 points of one butterfly at stride Ns, position k < Ns: one or two
// radix-4 steps (first at Ns, then at 4 Ns); x[t] in, outputs b' in x[b'].
template <int S, int R, int N, int Ns>
__device__ __forceinline__ void step4(C* x, const C* __restrict__ t, int k) {
  if constexpr (R >= 4) {
    if constexpr (Ns > 1) {
#pragma unroll
      for (int r1 = 1; r1 < 4; ++r1) {
        const C w = tw<S>(t, k * r1 * (N / (4 * Ns)));
#pragma unroll
        for (int r2 = 0; r2 < R / 4; ++r2) x[r2 + r1 * (R / 4)] = cmul(x[r2 + r1 * (R / 4)], w);
      }
    }
#pragma unroll
    for (int r2 = 0; r2 < R / 4; ++r2) radix4<S>(x[r2], x[r2 + R / 4], x[r2 + R / 2], x[r2 + 3 * (R / 4)]);
  }
  if constexpr (R == 16) {
    // x[r2 + 4 r1']: the second step over r2 at position k + r1' Ns
#pragma unroll
    for (int r1 = 0; r1 < 4; ++r1) {
#pragma unroll
      for (int r2 = 1; r2 < 4; ++r2)
        if (Ns > 1 || r1 > 0) x[r2 + 4 * r1] = cmul(x[r2 + 4 * r1], tw<S>(t, (k + r1 * Ns) * r2 * (N / (16 * Ns))));
      radix4<S>(x[4 * r1], x[4 * r1 + 1], x[4 * r1 + 2], x[4 * r1 + 3]);
    }
    // x[4 r1' + r2'] -> position b' = r1' + 4 r2'
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = i + 1; j < 4; ++j) {
        const C v = x[4 * i + j];
        x[4 * i + j] = x[4 * j + i];
        x[4 * j + i] = v;
      }
  }
}

// the last step(s): R = 6 (radix 2 at Ns = N / 6, radix 3) or 3; x[r] at k + r Ns in,
// outputs at k + i Ns in x[i]
template <int S, int R, int N>
__device__ __forceinline__ void step_last(C* x, const C* __restrict__ t, int k) {
  constexpr int Ns = N / R;
  if constexpr (R == 6) {
    const C w = tw<S>(t, 3 * k);
    C y[6];   // y[2 q + r']
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      const C v = Ns > 1 ? cmul(x[q + 3], w) : x[q + 3];
      y[2 * q] = x[q] + v;
      y[2 * q + 1] = x[q] - v;
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int k2 = k + r * Ns;
      C a = y[r], b = cmul(y[2 + r], tw<S>(t, k2)), c = cmul(y[4 + r], tw<S>(t, 2 * k2));
      radix3<S>(a, b, c);
      x[r] = a;
      x[r + 2] = b;
      x[r + 4] = c;
    }
  } else {
    x[1] = cmul(x[1], tw<S>(t, k));
    x[2] = cmul(x[2], tw<S>(t, 2 * k));
    radix3<S>(x[0], x[1], x[2]);
  }
}

// Unevaluated sum a + b + c of FP32 numbers, built by error-free additions.
struct Sum3 {
  float a, b, c;
};
__device__ __forceinline__ float two_sum(float x, float y, float& e) {
  const float s = __fadd_rn(x, y), t = __fsub_rn(s, x);
  e = __fadd_rn(__fsub_rn(x, __fsub_rn(s, t)), __fsub_rn(y, t));
  return s;
}
__device__ __forceinline__ void acc(Sum3& s, float x) {
  float e, f;
  s.a = two_sum(s.a, x, e);
  s.b = two_sum(s.b, e, f);
  s.c = __fadd_rn(s.c, f);
}
__device__ __forceinline__ Sum3 plus(Sum3 p, Sum3 q) {
  float e, f, h;
  Sum3 r;
  r.a = two_sum(p.a, q.a, e);
  r.b = two_sum(p.b, q.b, f);
  r.b = two_sum(r.b, e, h);
  r.c = __fadd_rn(__fadd_rn(p.c, q.c), __fadd_rn(f, h));
  return r;
}
__device__ __forceinline__ double value(Sum3 s) { return ((double)s.c + (double)s.b) + (double)s.a; }

template <int P> struct Plan32 {
  static constexpr int L = 1 << P, N = 3 * L;
  static constexpr int RA = P >= 4 ? 16 : P >= 2 ? 4 : 1;
  static constexpr int left = L / RA;
  static constexpr int RB = left >= 16 ? 16 : left >= 4 ? 4 : 1;
  static constexpr int RC = N / (RA * RB);          // 6 or 3
  static constexpr int NK = RA * RB;                // C items per row, a power of two
  static constexpr int GA = N / RA;                 // A items per FFT
  static constexpr int LD = (RB * RC) | 1;          // slot (j0, a): a LD + j0, odd
  static constexpr int FS = RA * LD;
  static constexpr size_t row_bytes = (size_t)(5 * FS + N) * sizeof(C);
  static_assert(RC == 6 || RC == 3, "radices");
};

constexpr int kMaxRows = 16;
constexpr int kSplitThreads = 640;   // SPLIT: the five FFTs' C items of 128 points

template <int P, bool SPLIT>
__global__ void __launch_bounds__(SPLIT ? kSplitThreads : 512) k_rows_f32(Grid g, const C* __restrict__ TW, const float* __restrict__ Z,
                                                  float* __restrict__ Q, double* __restrict__ wT, int nrows, int NR,
                                                  const int* nsteps, const int* step) {
  using PL = Plan32<P>;
  constexpr int N = PL::N, L = PL::L, RA = PL::RA, RB = PL::RB, RC = PL::RC, NK = PL::NK, GA = PL::GA, LD = PL::LD,
                FS = PL::FS;
  extern __shared__ __align__(16) unsigned char rsm[];
  __shared__ int act[kMaxRows];
  __shared__ Sum3 part[kMaxRows][8][2];   // warps' sums of the x-means of each row
  const int tid = threadIdx.x, T = blockDim.x;
  const int row0 = blockIdx.x * NR;
  if constexpr (SPLIT) {
    // twiddles into L1 while the launch before this one finishes: the passes'
    // first uses, one after another, would each wait for L2
    for (int i = tid * 16; i < N; i += T * 16) {
      float x, y;
      asm volatile("ld.global.nc.v2.f32 {%0, %1}, [%2];" : "=f"(x), "=f"(y) : "l"(TW + i));
    }
  }
  pdl_wait();
  int now = 0, last = 1;
  if constexpr (SPLIT) {   // one row, which exists: checked after its values are on their way
    if (nsteps != nullptr) {
      now = *step;
      last = nsteps[row0 / g.Mz];
    }
  } else {
    if (tid < NR) {
      const int row = row0 + tid;
      act[tid] = row < nrows && (nsteps == nullptr || *step < nsteps[row / g.Mz]);
    }
    __syncthreads();
  }
  const size_t fs = (size_t)g.Mz * L * 2;
  auto H = [&](int r) { return reinterpret_cast<C*>(rsm + (size_t)r * PL::row_bytes); };   // [5][FS]
  auto Pb = [&](int r) { return H(r) + 5 * FS; };                                          // [N], natural order

  // ---- A
  for (int i = tid; i < NR * 5 * GA; i += T) {
    const int r = i / (5 * GA), i1 = i - r * 5 * GA;
    const int pr = i1 / GA, j0 = i1 - pr * GA;
    if (!SPLIT && !act[r]) continue;
    const int row = row0 + r, b = row / g.Mz;
    const float* za = Z + (size_t)b * 9 * fs + 2 * pr * fs + (size_t)(row - b * g.Mz) * L * 2;
    const float* zb = za + fs;
    C x[RA];
#pragma unroll
    for (int t = 0; t < RA; ++t) {
      const int xx = j0 + t * GA;
      C v = make_float2(0.f, 0.f);
      if (xx < L || xx > 2 * L) {
        const int m = xx < L ? xx : N - xx;
        const C a = __ldcg(reinterpret_cast<const C*>(za) + m);
        const C d = pr < 4 ? __ldcg(reinterpret_cast<const C*>(zb) + m) : make_float2(0.f, 0.f);
        v = xx < L ? make_float2(a.x - d.y, a.y + d.x) : make_float2(a.x + d.y, d.x - a.y);
      }
      x[t] = v;
    }
    step4<1, RA, N, 1>(x, TW, 0);
    C* h = H(r) + pr * FS + j0;
#pragma unroll
    for (int a = 0; a < RA; ++a) h[a * LD] = x[a];
  }
  if (SPLIT && now >= last) return;   // uniform
  __syncthreads();

  // ---- B (in place)
  auto pass_b = [&](auto sign, int ffts) {
    constexpr int S = decltype(sign)::value;
    for (int i = tid; i < NR * ffts * RA * RC; i += T) {
      const int r = i / (ffts * RA * RC), i1 = i - r * ffts * RA * RC;
      const int ff = i1 / (RA * RC), i2 = i1 - ff * RA * RC;
      const int q2 = i2 / RA, k = i2 - q2 * RA;
      if (!SPLIT && !act[r]) continue;
      C* h = H(r) + ff * FS + k * LD + q2;
      C x[RB];
#pragma unroll
      for (int t = 0; t < RB; ++t) x[t] = h[RC * t];
      step4<S, RB, N, RA>(x, TW, k);
#pragma unroll
      for (int t = 0; t < RB; ++t) h[RC * t] = x[t];
    }
    __syncthreads();
  };
  if constexpr (RB > 1) pass_b(std::integral_constant<int, 1>(), 5);

  // ---- SPLIT: the last pass of each inverse FFT by its own item, in place
  if constexpr (SPLIT) {
    for (int i = tid; i < NR * 5 * NK; i += T) {
      const int r = i / (5 * NK), i1 = i - r * 5 * NK, pr = i1 / NK, k = i1 - pr * NK;
      C* h = H(r) + pr * FS + (k & (RA - 1)) * LD + RC * (k / RA);
      C x[RC];
#pragma unroll
      for (int q = 0; q < RC; ++q) x[q] = h[q];
      step_last<1, RC, N>(x, TW, k);
#pragma unroll
      for (int q = 0; q < RC; ++q) h[q] = x[q];
    }
    __syncthreads();
  }

  // ---- C: item (row, k') per thread, points k' + i NK
  const int cr = tid / NK, ck = tid - cr * NK;
  const bool con = tid < NR * NK && (SPLIT || act[min(cr, NR - 1)]);
  const int cslot = (ck & (RA - 1)) * LD + RC * (ck / RA);
  {
    Sum3 sU = {0.f, 0.f, 0.f}, sW = {0.f, 0.f, 0.f};
    if (con) {
      const C* h = H(cr) + cslot;
      C x[RC];
      float u[RC], w[RC], no[RC], dt[RC];
      auto inverse = [&](int pr) {
#pragma unroll
        for (int r = 0; r < RC; ++r) x[r] = h[pr * FS + r];
        if constexpr (!SPLIT) step_last<1, RC, N>(x, TW, ck);
      };
      inverse(0);
#pragma unroll
      for (int i = 0; i < RC; ++i) {
        u[i] = x[i].x;
        w[i] = x[i].y;
      }
      inverse(1);
#pragma unroll
      for (int i = 0; i < RC; ++i) no[i] = fmaf(u[i], x[i].x, w[i] * x[i].y);
      inverse(2);
#pragma unroll
      for (int i = 0; i < RC; ++i) acc(sU, fmaf(u[i], x[i].x, w[i] * x[i].y));
      inverse(3);
#pragma unroll
      for (int i = 0; i < RC; ++i) {
        acc(sW, w[i] * x[i].x);
        dt[i] = x[i].y;
      }
      inverse(4);
      C* p = Pb(cr) + ck;
#pragma unroll
      for (int i = 0; i < RC; ++i) p[i * NK] = make_float2(fmaf(u[i], dt[i], w[i] * x[i].x), no[i]);
    }
    // x-means: a fixed tree over the lanes of a row (rows of fewer than 32 items share a warp)
#pragma unroll
    for (int s = 1; s < 32 && s < NK; s *= 2) {
      Sum3 o;
      o.a = __shfl_xor_sync(0xffffffffu, sU.a, s);
      o.b = __shfl_xor_sync(0xffffffffu, sU.b, s);
      o.c = __shfl_xor_sync(0xffffffffu, sU.c, s);
      sU = plus(sU, o);
      o.a = __shfl_xor_sync(0xffffffffu, sW.a, s);
      o.b = __shfl_xor_sync(0xffffffffu, sW.b, s);
      o.c = __shfl_xor_sync(0xffffffffu, sW.c, s);
      sW = plus(sW, o);
    }
    if (con && (ck & 31) == 0) {
      part[cr][ck >> 5][0] = sU;
      part[cr][ck >> 5][1] = sW;
    }
  }
  __syncthreads();

  // ---- D, E, F: the forward FFT, in the first FFT's place
  for (int i = tid; i < NR * GA; i += T) {
    const int r = i / GA, j0 = i - r * GA;
    if (!SPLIT && !act[r]) continue;
    const C* p = Pb(r) + j0;
    C x[RA];
#pragma unroll
    for (int t = 0; t < RA; ++t) x[t] = p[t * GA];
    step4<-1, RA, N, 1>(x, TW, 0);
    C* h = H(r) + j0;
#pragma unroll
    for (int a = 0; a < RA; ++a) h[a * LD] = x[a];
  }
  __syncthreads();
  if constexpr (RB > 1) pass_b(std::integral_constant<int, -1>(), 1);
  if (con) {
    const C* h = H(cr) + cslot;
    C x[RC];
#pragma unroll
    for (int r = 0; r < RC; ++r) x[r] = h[r];
    step_last<-1, RC, N>(x, TW, ck);
    C* p = Pb(cr) + ck;
#pragma unroll
    for (int i = 0; i < RC; ++i) p[i * NK] = x[i];
  }
  __syncthreads();

  // ---- G
  const float inv = 1.0f / (float)N, half = 0.5f * inv;
  const size_t qs = (size_t)g.Mz * L * 2;
  for (int i = tid; i < NR * L; i += T) {
    const int r = i / L, m = i - r * L;
    if (!SPLIT && !act[r]) continue;
    const int row = row0 + r, b = row / g.Mz, j = row - b * g.Mz;
    const C* p = Pb(r);
    const C cm = p[m], c2 = p[m == 0 ? 0 : N - m];
    const C s = make_float2(cm.x + c2.x, cm.y - c2.y), d = make_float2(cm.x - c2.x, cm.y + c2.y);
    C n1 = make_float2(half * d.y, -half * d.x);
    if (m == 0) {
      Sum3 sU = part[r][0][0], sW = part[r][0][1];
      for (int w = 1; w < NK / 32; ++w) {
        sU = plus(sU, part[r][w][0]);
        sW = plus(sW, part[r][w][1]);
      }
      n1 = make_float2((float)(value(sU) / N), 0.f);
      wT[(size_t)b * g.Mz + j] = value(sW) / N;
    }
    float* q0 = Q + (size_t)b * 2 * qs + (size_t)j * L * 2 + 2 * m;
    *reinterpret_cast<C*>(q0) = make_float2(half * s.x, half * s.y);
    *reinterpret_cast<C*>(q0 + qs) = n1;
  }
}

// SPLIT up to two rows per SM: a stage of 128 x 32, one state takes 25.2 us with it,
// 26.1 without; beyond, blocks of 640 threads crowd each other out.
constexpr int kSplitRows = 2 * 152;

// Rows per block: up to 256 C items and 48 KB, fewer while the launch would not
// give every SM two blocks; a row alone takes threads for the A items too.
template <int P> int per_block(const Shapes& sh, int nrows) {
  using PL = Plan32<P>;
  int nr = 1;
  while (nr < kMaxRows && 2 * nr * PL::NK <= 256 && 2 * nr * PL::row_bytes <= 48 * 1024) nr *= 2;
  if (sh.rows_cl == 1) return 1;
  if (sh.rows_cl < 0)
    while (nr > 1 && (long)nrows < 2L * 152 * nr) nr /= 2;
  return nr;
}

template <int P>
cudaError_t launch_rows_P(const Grid& g, const Tables& t, const Work& w, int B, const int* ns, cudaStream_t s) {
  using PL = Plan32<P>;
  const int nrows = B * g.Mz, nr = per_block<P>(w.shapes ? *w.shapes : Shapes{}, nrows);
  const unsigned blocks = (unsigned)((nrows + nr - 1) / nr);
  const float* Z = reinterpret_cast<const float*>(w.Z);
  float* Q = reinterpret_cast<float*>(w.Q);
  if (nr == 1 && nrows <= kSplitRows) {
    const int th = std::min(kSplitThreads, (std::max(5 * PL::NK, 5 * PL::GA) + 31) / 32 * 32);
    return launch_pdl(w.pdl != 0, k_rows_f32<P, true>, blocks, th, PL::row_bytes, s, g, t.tw32, Z, Q, w.wT, nrows, nr,
                      ns, w.step);
  }
  // 1024 x 256, 32 states: 568 us with a thread per item of passes A and B (480 per
  // row), 722 with 256; shorter rows, several to a block, are slower beyond 256
  const int th = P == 9 ? 512 : std::max((nr * PL::NK + 31) / 32 * 32, std::min(256, (nr * 5 * PL::GA + 31) / 32 * 32));
  return launch_pdl(w.pdl != 0, k_rows_f32<P, false>, blocks, th, nr * PL::row_bytes, s, g, t.tw32, Z, Q, w.wT, nrows,
                    nr, ns, w.step);
}

}  // namespace

template <int P>
cudaError_t configure_P() {
  constexpr cudaFuncAttribute smem = cudaFuncAttributeMaxDynamicSharedMemorySize;
  const cudaError_t e = cudaFuncSetAttribute(k_rows_f32<P, false>, smem, 100 * 1024);
  return e == cudaSuccess ? cudaFuncSetAttribute(k_rows_f32<P, true>, smem, 100 * 1024) : e;
}

#define RBC_ROWS_CASES(X) X(1) X(2) X(3) X(4) X(5) X(6) X(7) X(8) X(9)

cudaError_t configure_rows_f32(const Grid& g) {
  switch (g.nm) {
#define X(P) case 1 << P: return configure_P<P>();
    RBC_ROWS_CASES(X)
#undef X
  }
  return cudaErrorInvalidValue;
}

int rows_f32_per_block(const Grid& g, const Shapes& sh, int B) {
  switch (g.nm) {
#define X(P) case 1 << P: return per_block<P>(sh, B * g.Mz);
    RBC_ROWS_CASES(X)
#undef X
  }
  return 0;
}

cudaError_t launch_rows_f32(const Grid& g, const Tables& t, const Work& w, int B, const int* ns, cudaStream_t s) {
  switch (g.nm) {
#define X(P) case 1 << P: return launch_rows_P<P>(g, t, w, B, ns, s);
    RBC_ROWS_CASES(X)
#undef X
  }
  return cudaErrorInvalidValue;
}

}  // namespace rbc
