// Row kernel of the FP64 mode: x inverse FFTs, advective products, x forward
// FFT in block fixed point (rbc_fx.cuh).
//
// Z holds six fields per padded row j (complex modes m < nm): u, w, d_x omega,
// d_z omega, d_x T, d_z T.  Pairs of real fields share one complex inverse FFT
// of length N = Mx = 3 L, L = nm (C = A + iB with the Hermitian extensions),
//   N_T = u T_x + w T_z,  N_omega = u omega_x + w omega_z   (Eqs. 3, 5),
// and one forward FFT carries both products (N_T + i N_omega), truncated to
// m < nm.  The two x-means follow from the modes by Parseval (the products'
// modes stay below N, so the mean over the points is exact), in FP64:
//   <w T>_x      =  sum_{m >= 1} (2 / k) (w_r T'_i - w_i T'_r),          T' = d_x T,
//   <u u_x + w u_z>_x = -<w omega>_x = -sum (2 / k) (w_r o_i - w_i o_r), o = d_x omega
// (u_z = d_x w - omega; <u u_x> and <w w_x> vanish): no FFT is needed for T,
// d_x u and d_z u, which leaves three inverse FFTs of the five that all nine
// fields take.
//
// The kept modes fill two of the three blocks of L spectral positions, so the
// length-3L transform is three length-L ones with twiddled inputs (point
// x = 3 a + b, b = 0, 1, 2): G_b[k] = w^(k b) C[k] + w^((k-L) b) C[k - L], and
// of the forward combination only the kept outputs are formed.  L = R M: the
// butterflies run in registers (radix up to 16), exchanging through shared
// memory once per pass; the products and the first forward pass act on the
// same points and stay in one thread's registers.
//   P0  modes -> exponents, packed spectra C, D (shared), terms of the x-means
//   P1  G_b and the M-point transforms (P1b: the second half of M = 32, 64)
//   P2  R-point inverse transforms
//   P3  products, R-point forward transforms
//   PB  M-point forward transforms
//   PF  sum over b, unpacking, x-means, store
// Block: RB rows, at least one thread per P3 item; items are flattened over the
// block's rows.
//
// Fixed point: each row and field gets the exponent of its summed mode moduli
// (an upper bound of the grid values), so grid values are integers below 2^59
// and every intermediate stays below 2^61; products are 96-bit, renormalised
// by the largest of the row before the forward transform.  Its rounding, about
// 2^-59 of the summed moduli, is below a double FFT's: against 64-bit plain
// torch the temperature after 40 steps at 128 x 32 is 4 to 17 times closer than
// with FP64 FFTs, other states and grids equally close.  A row with a
// non-finite mode gives NaN in both products.
//
// Bound: integer issue.  An FP64 warp instruction holds its sub-partition for
// 64 clocks, a 32x32->64 multiply-add for 4 and a 64-bit add for 2, so the
// same FFT costs about a tenth.  Measured (GB300, per launch, against five
// FP64 FFTs in radix-4 passes through shared memory): 256 x 64, 32 states
// 491 -> 108 us; 512 x 128, 3 states 207 -> 46 us; 64 x 32, 23 states
// 41 -> 16.5 us; 128 x 32, one state 20.4 -> 14 us (latency: the barriers).
// One thread keeping the points of all three inverse FFTs in registers (P2 and
// P3 in one pass, 166 registers, C and D in a place of their own) took 127, 60,
// 22 and 19.8 us.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>

#include "rbc_fx.cuh"
#include "rbc_internal.h"

namespace rbc {

namespace {

using fx::i64;

// Complex numbers as integer pairs; twiddles with 62 fractional bits, as signed
// 32-bit halves: re hi, re lo, im hi, im lo.
using C = longlong2;
using W = int4;

__device__ __forceinline__ C add(C a, C b) {
  a.x += b.x;
  a.y += b.y;
  return a;
}
__device__ __forceinline__ C sub(C a, C b) {
  a.x -= b.x;
  a.y -= b.y;
  return a;
}
// a + S i d
template <int S> __device__ __forceinline__ C addi(C a, C d) {
  if (S > 0) {
    a.x -= d.y;
    a.y += d.x;
  } else {
    a.x += d.y;
    a.y -= d.x;
  }
  return a;
}

constexpr i64 kQ62_r8 = 3260954456333195553ll;    // sqrt(1/2)
constexpr i64 kQ62_c16 = 4260642322793532497ll;   // cos(pi/8)
constexpr i64 kQ62_s16 = 1764815834521887442ll;   // sin(pi/8)
constexpr i64 kQ62_s3 = 3993837246235628775ll;    // sqrt(3)/2
__host__ __device__ constexpr int q_lo(i64 v) { return (int)(v & 0xffffffffll); }
__host__ __device__ constexpr int q_hi(i64 v) { return (int)((v - (i64)q_lo(v)) >> 32); }

__device__ __forceinline__ i64 rmul(i64 a, i64 c) {
  int h, l;
  fx::split32(a, h, l);
  const i64 ph = (i64)h * q_hi(c);
  const i64 pm = fx::madw(l, q_hi(c), fx::madw(h, q_lo(c), 1ll << 29));
  return (ph << 2) + (pm >> 30);
}

// a w (CJ: a conj(w)) over 2^SH, for |a| <= 2^61: the products of the low halves
// (below one unit of the result) are dropped, the rest is rounded to nearest.
struct Split2 {
  int xh, xl, yh, yl;
};
__device__ __forceinline__ Split2 split2(longlong2 a) {
  Split2 s;
  fx::split32(a.x, s.xh, s.xl);
  fx::split32(a.y, s.yh, s.yl);
  return s;
}
template <bool CJ> __device__ __forceinline__ void cmac(const Split2& s, int4 w, i64& rh, i64& rm, i64& ih, i64& im) {
  const int ph = CJ ? -w.z : w.z, pl = CJ ? -w.w : w.w;   // imaginary part of the factor
  rh = fx::madw(s.xh, w.x, fx::madw(s.yh, -ph, rh));
  rm = fx::madw(s.xh, w.y, fx::madw(s.xl, w.x, fx::madw(s.yh, -pl, fx::madw(s.yl, -ph, rm))));
  ih = fx::madw(s.xh, ph, fx::madw(s.yh, w.x, ih));
  im = fx::madw(s.xh, pl, fx::madw(s.xl, ph, fx::madw(s.yh, w.y, fx::madw(s.yl, w.x, im))));
}
template <bool CJ, int SH> __device__ __forceinline__ longlong2 cmulw(longlong2 a, int4 w) {
  i64 rh = 0, rm = 1ll << (29 + SH), ih = 0, im = 1ll << (29 + SH);
  cmac<CJ>(split2(a), w, rh, rm, ih, im);
  return make_longlong2((rh << (2 - SH)) + (rm >> (30 + SH)), (ih << (2 - SH)) + (im >> (30 + SH)));
}
// a conj(wa) + d conj(wd)
__device__ __forceinline__ C cmul2c(longlong2 a, int4 wa, longlong2 d, int4 wd) {
  i64 rh = 0, rm = 1ll << 29, ih = 0, im = 1ll << 29;
  cmac<true>(split2(a), wa, rh, rm, ih, im);
  cmac<true>(split2(d), wd, rh, rm, ih, im);
  return make_longlong2((rh << 2) + (rm >> 30), (ih << 2) + (im >> 30));
}
// multiplication by cos + S i sin of pi/8 (k = 1), 3 pi/8 (k = 3)
template <int S, int K> __device__ __forceinline__ longlong2 rot16(longlong2 a) {
  constexpr i64 c = K == 1 ? kQ62_c16 : kQ62_s16, s = K == 1 ? kQ62_s16 : kQ62_c16;
  return cmulw<(S < 0), 0>(a, make_int4(q_hi(c), q_lo(c), q_hi(s), q_lo(s)));
}

// ---------------------------------------------------------------------------
// y_q = sum_r x_r exp(S 2 pi i q r / R) in registers, natural order.
// ---------------------------------------------------------------------------
template <int S> __device__ __forceinline__ void dft4(C& a, C& b, C& c, C& d) {
  const C t0 = add(a, c), t1 = sub(a, c), t2 = add(b, d), t3 = sub(b, d);
  a = add(t0, t2);
  c = sub(t0, t2);
  b = addi<S>(t1, t3);
  d = addi<-S>(t1, t3);
}
template <int S> __device__ __forceinline__ void dft8(C* x) {
  dft4<S>(x[0], x[2], x[4], x[6]);
  dft4<S>(x[1], x[3], x[5], x[7]);
  // odd outputs o_c in x[1 + 2 c]; o_1 w8, o_2 S i, o_3 w8^3
  C o1, o3;
  if (S > 0) {
    o1.x = rmul(x[3].x - x[3].y, kQ62_r8);
    o1.y = rmul(x[3].y + x[3].x, kQ62_r8);
    o3.x = rmul(x[7].x + x[7].y, kQ62_r8);   // -Re, Im of o_3 w8^3
    o3.y = rmul(x[7].x - x[7].y, kQ62_r8);
  } else {
    o1.x = rmul(x[3].x + x[3].y, kQ62_r8);
    o1.y = rmul(x[3].y - x[3].x, kQ62_r8);
    o3.x = rmul(x[7].x - x[7].y, kQ62_r8);
    o3.y = rmul(x[7].x + x[7].y, kQ62_r8);   // -Im
  }
  const C e0 = x[0], e1 = x[2], e2 = x[4], e3 = x[6], o0 = x[1], o2 = x[5];
  x[0] = add(e0, o0);
  x[4] = sub(e0, o0);
  x[1] = add(e1, o1);
  x[5] = sub(e1, o1);
  x[2] = addi<S>(e2, o2);
  x[6] = addi<-S>(e2, o2);
  if (S > 0) {
    x[3].x = e3.x - o3.x;
    x[3].y = e3.y + o3.y;
    x[7].x = e3.x + o3.x;
    x[7].y = e3.y - o3.y;
  } else {
    x[3].x = e3.x - o3.x;
    x[3].y = e3.y - o3.y;
    x[7].x = e3.x + o3.x;
    x[7].y = e3.y + o3.y;
  }
}
template <int S> __device__ __forceinline__ C rot8(C a) {   // a (1 + S i) / sqrt 2
  C r;
  r.x = rmul(S > 0 ? a.x - a.y : a.x + a.y, kQ62_r8);
  r.y = rmul(S > 0 ? a.y + a.x : a.y - a.x, kQ62_r8);
  return r;
}
template <int S> __device__ __forceinline__ C timesi(C a) {   // S i a
  C r;
  r.x = S > 0 ? -a.y : a.y;
  r.y = S > 0 ? a.x : -a.x;
  return r;
}
__device__ __forceinline__ C neg(C a) {
  a.x = -a.x;
  a.y = -a.y;
  return a;
}
template <int S> __device__ __forceinline__ void dft16(C* x) {
#pragma unroll
  for (int b = 0; b < 4; ++b) dft4<S>(x[b], x[4 + b], x[8 + b], x[12 + b]);   // x[4 c + b]
  x[5] = rot16<S, 1>(x[5]);
  x[9] = rot8<S>(x[9]);
  x[13] = rot16<S, 3>(x[13]);
  x[6] = rot8<S>(x[6]);
  x[10] = timesi<S>(x[10]);
  x[14] = timesi<S>(rot8<S>(x[14]));
  x[7] = rot16<S, 3>(x[7]);
  x[11] = timesi<S>(rot8<S>(x[11]));
  x[15] = neg(rot16<S, 1>(x[15]));
#pragma unroll
  for (int c = 0; c < 4; ++c) dft4<S>(x[4 * c], x[4 * c + 1], x[4 * c + 2], x[4 * c + 3]);   // x[4 c + d] = y[c + 4 d]
#pragma unroll
  for (int c = 0; c < 4; ++c)
#pragma unroll
    for (int d = c + 1; d < 4; ++d) {
      const C t = x[4 * c + d];
      x[4 * c + d] = x[4 * d + c];
      x[4 * d + c] = t;
    }
}
template <int R, int S> __device__ __forceinline__ void dft(C* x) {
  if constexpr (R == 2) {
    const C t = x[0];
    x[0] = add(t, x[1]);
    x[1] = sub(t, x[1]);
  } else if constexpr (R == 4) {
    dft4<S>(x[0], x[1], x[2], x[3]);
  } else if constexpr (R == 8) {
    dft8<S>(x);
  } else if constexpr (R == 16) {
    dft16<S>(x);
  }
}

template <int L> struct Plan {
  static constexpr int R = L < 8 ? L : 8;
  static constexpr int M = L / R;
  static constexpr int M2 = M <= 16 ? 1 : M / 8;      // M = M1 M2
  static constexpr int M1 = M / M2;
  static constexpr int N = 3 * L;
  // an FFT's exchange buffer, [M][R + 1]: consecutive s or q of a warp fall in
  // different banks
  static constexpr int FS = M * (R + 1);
  static constexpr int kSum1 = (L + 7) / 8, kSum2 = (kSum1 + 7) / 8, kSum3 = (kSum2 + 7) / 8;
  static constexpr int kSums = 2 * (L + kSum1 + kSum2 + kSum3);
  // with a single first pass (M2 = 1) each of its items belongs to one thread,
  // which reads its spectra before any is overwritten: C, D share H's place
  static constexpr bool kAlias = M2 == 1;
  static constexpr size_t row_bytes =
      (((kAlias ? 0 : 6 * (size_t)L) + 9 * (size_t)FS) * sizeof(C) + (size_t)kSums * 8 + 15) / 16 * 16;
  // threads of a block of rb rows: one per P2 item, and per P1 item where those are single
  static constexpr int threads(int rb) { return (rb * (kAlias && 9 * R > 3 * M ? 9 * R : 3 * M) + 31) / 32 * 32; }
  static constexpr int kSH = 2;                                    // each forward twiddle halves twice
  static constexpr int kShift = kSH * (M2 > 1 ? 3 : 2);
};

constexpr int kMaxRB = 16;

// Per-row numbers.
struct RowMeta {
  int act;
  int emax[6];      // largest biased exponent of each field's modes
  unsigned l1[6];   // summed moduli in units of 2^(emax - 1023 - 16)
  int bits[2];      // bit lengths of the largest N_T, N_omega
};

// FEW (one row per block of kFew threads, for launches of at most two blocks per
// SM): the twiddle products before the first inverse pass and after both forward
// passes, eight or more in a row per item otherwise, are spread over all threads
// at the price of three barriers.  A whole stage on GB300: 128 x 32, one state
// 29.9 -> 26.8 us, six 36.3 -> 33.6; 256 x 64, one state 55.4 -> 48.5, three 72.2 ->
// 65.3; 64 x 32, one state 26.7 -> 25.5.
constexpr int kFew = 288;

template <int L, bool FEW>
__global__ void __launch_bounds__(Plan<L>::kAlias ? 320 : 384, Plan<L>::kAlias ? 2 : 1) k_rows_fx(Grid g, const W* __restrict__ TW, const double* __restrict__ rk,
                                                 const double* __restrict__ Z, double* __restrict__ Q,
                                                 double* __restrict__ wT, int nrows, int RB, const int* nsteps,
                                                 const int* step) {
  using P = Plan<L>;
  constexpr int R = P::R, M = P::M, M1 = P::M1, M2 = P::M2, N = P::N, FS = P::FS;
  extern __shared__ __align__(16) unsigned char rsm[];
  __shared__ RowMeta meta[kMaxRB];
  const int tid = threadIdx.x, T = blockDim.x;
  const int row0 = blockIdx.x * RB;
  // twiddles into L1 while the launch before this one finishes: the passes' first
  // uses, one after another, would each wait for L2
  for (int i = tid * 8; i < N; i += T * 8) {
    int a, b, c, d;
    asm volatile("ld.global.nc.v4.s32 {%0, %1, %2, %3}, [%4];" : "=r"(a), "=r"(b), "=r"(c), "=r"(d) : "l"(TW + i));
  }
  pdl_wait();
  const int stepidx = nsteps ? *step : 0;
  if (tid < RB) {
    const int row = row0 + tid;
    RowMeta& me = meta[tid];
    me.act = row < nrows && (nsteps == nullptr || stepidx < nsteps[row / g.Mz]);
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      me.emax[f] = 0;
      me.l1[f] = 0;
    }
    me.bits[0] = me.bits[1] = 0;
  }
  auto Cb = [&](int r) { return reinterpret_cast<C*>(rsm + (size_t)r * P::row_bytes); };
  auto Db = [&](int r) { return Cb(r) + 3 * L; };
  auto Hb = [&](int r) { return Cb(r) + (P::kAlias ? 0 : 6 * L); };
  auto Sb = [&](int r) { return reinterpret_cast<double*>(Hb(r) + 9 * FS); };
  const size_t fs = (size_t)g.Mz * L * 2;
  auto zrow = [&](int r) {
    const int row = row0 + r, b = row / g.Mz;
    return Z + (size_t)b * 6 * fs + (size_t)(row - b * g.Mz) * L * 2;
  };
  auto ld = [&](const double* z, int f, int m) { return __ldcg(reinterpret_cast<const double2*>(z + f * fs + 2 * m)); };
  auto tw = [&](int k) -> W { return __ldg(TW + k); };
  double2 v[6];                     // a thread's item, kept where it has only one
  const bool once = RB * L <= T;
  auto load_item = [&](int r, int m) {
    const double* z = zrow(r);
#pragma unroll
    for (int f = 0; f < 6; ++f) v[f] = ld(z, f, m);
  };
  // (which rows are active is looked at once the values are on their way)
  if (once && tid < RB * L && row0 + tid / L < nrows) load_item(tid / L, tid % L);
  __syncthreads();

  // ---- P0: packed spectra and the terms of the x-means
  for (int i = tid; i < RB * L; i += T) {
    const int r = i / L, m = i - r * L;
    if (!meta[r].act) continue;
    if (!once) load_item(r, m);
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      int e = max(fx::hi_abs(v[f].x), fx::hi_abs(v[f].y)) >> 20;
      if (L >= 32) {   // a warp's items lie in one row
        e = __reduce_max_sync(0xffffffffu, e);
        if ((tid & 31) == 0) atomicMax(&meta[r].emax[f], e);
      } else {
        atomicMax(&meta[r].emax[f], e);
      }
    }
    const double k2 = rk[m];   // 2 / k, 0 at m = 0
    double* s = Sb(r);
    s[m] = k2 * fma(v[1].x, v[4].y, -(v[1].y * v[4].x));
    s[L + m] = -k2 * fma(v[1].x, v[2].y, -(v[1].y * v[2].x));
  }
  __syncthreads();
  for (int i = tid; i < RB * L; i += T) {
    const int r = i / L, m = i - r * L;
    if (!meta[r].act) continue;
    if (!once) load_item(r, m);
#pragma unroll
    for (int f = 0; f < 6; ++f) {
      const int em = meta[r].emax[f];
      unsigned t = 0;
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const double x = c ? v[f].y : v[f].x;
        const int hi = __double2hiint(x), e = (hi >> 20) & 0x7ff;
        t += (((unsigned)(hi & 0xfffff) | 0x100000u) >> min(em - e + 4, 31)) + 1u;
      }
      t = m == 0 ? t : 2 * t;
      if (L >= 32) {
        t = __reduce_add_sync(0xffffffffu, t);
        if ((tid & 31) == 0) atomicAdd(&meta[r].l1[f], t);
      } else {
        atomicAdd(&meta[r].l1[f], t);
      }
    }
  }
  __syncthreads();
  // exponents E_f of a row's fields: |field| < 2^E on the grid; the fields of one
  // product sum (u o_x + w o_z, u T_x + w T_z) aligned to the larger product
  auto exponents = [&](int r, int* E) {
    const RowMeta& me = meta[r];
#pragma unroll
    for (int f = 0; f < 6; ++f)
      E[f] = me.emax[f] == 0 ? -1100 : 32 - __clz((int)me.l1[f]) + me.emax[f] - 1023 - 16;
#pragma unroll
    for (int f = 2; f < 6; f += 2) {
      const int d = (E[0] + E[f]) - (E[1] + E[f + 1]);
      if (d < 0)
        E[f] -= d;
      else
        E[f + 1] += d;
    }
  };
  for (int i = tid; i < RB * L; i += T) {
    const int r = i / L, m = i - r * L;
    if (!meta[r].act) continue;
    if (!once) load_item(r, m);
    C* c = Cb(r);
    C* d = Db(r);
    int E[6];
    exponents(r, E);
#pragma unroll
    for (int p = 0; p < 3; ++p) {
      const double2 a = v[2 * p], b = v[2 * p + 1];
      const i64 ax = fx::from_double<59>(a.x, E[2 * p] + 1022), ay = fx::from_double<59>(a.y, E[2 * p] + 1022);
      const i64 bx = fx::from_double<59>(b.x, E[2 * p + 1] + 1022), by = fx::from_double<59>(b.y, E[2 * p + 1] + 1022);
      c[p * L + m] = make_longlong2(ax - by, ay + bx);
      d[p * L + (m == 0 ? 0 : L - m)] = m == 0 ? make_longlong2(0, 0) : make_longlong2(ax + by, bx - ay);
    }
  }
  __syncthreads();
  // one level of the x-means' tree: NOUT sums of (up to) eight values each, a
  // fixed order whatever the launch shape
  auto tree = [&](int off_in, int nin, int off_out, int nout) {
    for (int i = tid; i < RB * 2 * nout; i += T) {
      const int r = i / (2 * nout), j = i - r * 2 * nout, q = j / nout, o = j - q * nout;
      if (!meta[r].act) continue;
      const double* in = Sb(r) + off_in + q * nin;
      double v[8];
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = 8 * o + e < nin ? in[8 * o + e] : 0.0;
      Sb(r)[off_out + q * nout + o] =
          ((v[0] + v[1]) + (v[2] + v[3])) + ((v[4] + v[5]) + (v[6] + v[7]));
    }
  };
  constexpr int s1 = 2 * L, s2 = s1 + 2 * P::kSum1, s3 = s2 + 2 * P::kSum2;

  // ---- P1: G_b and the first inverse pass; item (b, row, pair, j, s), s fastest
  {
    C x[M1];
    int b, r, pr, j, sx;
    auto item = [&](int i) {
      b = i / (RB * 3 * R * M2);
      const int i1 = i - b * RB * 3 * R * M2;
      r = i1 / (3 * R * M2);
      const int i2 = i1 - r * 3 * R * M2;
      pr = i2 / (R * M2);
      const int i3 = i2 - pr * R * M2;
      j = i3 / R;
      sx = i3 - j * R;
    };
    auto gather = [&] {
      const C* c = Cb(r) + pr * L;
      const C* d = Db(r) + pr * L;
#pragma unroll
      for (int a = 0; a < M1; ++a) {
        const int k = R * (M2 * a + j) + sx;
        if (b == 0)
          x[a] = add(c[k], d[k]);
        else
          x[a] = cmul2c(c[k], tw(k * b), d[k], tw(k * b + (3 - b) * L));
      }
    };
    auto transform = [&] {
      dft<M1, 1>(x);
      C* h = Hb(r) + (pr * 3 + b) * FS + sx;
#pragma unroll
      for (int u = 0; u < M1; ++u) {
        if (M2 > 1 && u > 0) x[u] = cmulw<true, 0>(x[u], tw(3 * R * u * j));
        h[(u + M1 * j) * (R + 1)] = x[u];
      }
    };
    if constexpr (FEW) {
      constexpr int PER = (9 * L + kFew - 1) / kFew;
      const bool act = meta[0].act;
      C v1[PER];
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        const int i = tid + e * kFew, pb = i / L, k = i % L, bb = pb % 3;
        if (act && i < 9 * L) {
          const C* c = Cb(0) + pb / 3 * L;
          const C* d = Db(0) + pb / 3 * L;
          v1[e] = bb == 0 ? add(c[k], d[k]) : cmul2c(c[k], tw(k * bb), d[k], tw(k * bb + (3 - bb) * L));
        }
      }
      __syncthreads();
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        const int i = tid + e * kFew, pb = i / L, k = i % L;
        if (act && i < 9 * L) Hb(0)[pb * FS + k % R + k / R * (R + 1)] = v1[e];
      }
      __syncthreads();
      if (act && tid < 9 * R) {
        C* h = Hb(0) + tid / R * FS + tid % R;
#pragma unroll
        for (int a = 0; a < M1; ++a) x[a] = h[a * (R + 1)];
        dft<M1, 1>(x);
#pragma unroll
        for (int u = 0; u < M1; ++u) h[u * (R + 1)] = x[u];
      }
    } else if constexpr (P::kAlias) {
      item(tid);
      const bool on = tid < RB * 9 * R && meta[min(r, RB - 1)].act;
      if (on) gather();
      __syncthreads();
      if (on) transform();
    } else {
      for (int i = tid; i < RB * 9 * R * M2; i += T) {
        item(i);
        if (!meta[r].act) continue;
        gather();
        transform();
      }
    }
  }
  tree(0, L, s1, P::kSum1);
  __syncthreads();
  if constexpr (M2 > 1) {
    for (int i = tid; i < RB * 9 * R * M1; i += T) {
      const int r = i / (9 * R * M1), i1 = i - r * 9 * R * M1;
      const int ff = i1 / (R * M1), i2 = i1 - ff * R * M1;
      const int u = i2 / R, s = i2 - u * R;
      if (!meta[r].act) continue;
      C* h = Hb(r) + ff * FS + s + u * (R + 1);
      C x[M2];
#pragma unroll
      for (int j = 0; j < M2; ++j) x[j] = h[M1 * j * (R + 1)];
      dft<M2, 1>(x);
#pragma unroll
      for (int v = 0; v < M2; ++v) h[M1 * v * (R + 1)] = x[v];
    }
    __syncthreads();
  }

  // ---- P2: last inverse pass, in place; item (row, pair, b, q), q fastest
  for (int i = tid; i < RB * 9 * M; i += T) {
    const int r = i / (9 * M), i1 = i - r * 9 * M;
    const int ff = i1 / M, q = i1 - ff * M;
    if (!meta[r].act) continue;
    C* h = Hb(r) + ff * FS + q * (R + 1);
    C x[R];
#pragma unroll
    for (int s = 0; s < R; ++s) x[s] = h[s];
#pragma unroll
    for (int s = 1; s < R; ++s)
      if (M > 1) x[s] = cmulw<true, 0>(x[s], tw(3 * s * q));
    dft<R, 1>(x);
#pragma unroll
    for (int t = 0; t < R; ++t) h[t] = x[t];
  }
  if (P::kSum1 > 1) tree(s1, P::kSum1, s2, P::kSum2);
  __syncthreads();

  // ---- P3: products and the first forward pass; one item (row, b, q) per thread,
  // the points t of the P2 item at (b, q)
  {
    const int r = tid / (3 * M), i1 = tid - r * 3 * M;
    const int b = i1 / M, q = i1 - b * M;
    const bool on = tid < RB * 3 * M && meta[min(r, RB - 1)].act;
    C* h = Hb(on ? r : 0) + b * FS + q * (R + 1);
    C x[R];
    i64 vh[2][R];        // N_T, N_omega: 96-bit values vh 2^32 + vl
    unsigned vl[2][R];
    if (on) {
      i64 acc[2] = {0, 0};
      unsigned accl[2] = {0, 0};
#pragma unroll
      for (int t = 0; t < R; ++t) {
        const C uw = h[t];
        int uh, ul, wh, wl;
        fx::split32(uw.x, uh, ul);
        fx::split32(uw.y, wh, wl);
#pragma unroll
        for (int k = 0; k < 2; ++k) {
          const C ab = h[(2 - k) * 3 * FS + t];   // k = 0: d_x T, d_z T; k = 1: d_x omega, d_z omega
          int ah, al, bh, bl;
          fx::split32(ab.x, ah, al);
          fx::split32(ab.y, bh, bl);
          const i64 ph = fx::madw(uh, ah, (i64)wh * bh);
          const i64 pm = fx::madw(uh, al, fx::madw(ul, ah, fx::madw(wh, bl, (i64)wl * bh)));
          const i64 v = ph + (pm >> 32);
          vh[k][t] = v;
          vl[k][t] = (unsigned)pm;
          acc[k] |= v ^ (v >> 63);
          accl[k] |= (unsigned)pm ^ (unsigned)(v >> 63);
        }
      }
#pragma unroll
      for (int k = 0; k < 2; ++k)
        atomicMax(&meta[r].bits[k], acc[k] ? 96 - __clzll(acc[k]) : 32 - __clz((int)accl[k]));
    }
    __syncthreads();
    if (on) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int sh = meta[r].bits[k] - 55;   // the row's largest value to 55 bits
#pragma unroll
        for (int t = 0; t < R; ++t) {
          const unsigned w1 = (unsigned)vh[k][t];
          const int w2 = (int)(vh[k][t] >> 32);
          i64 v;
          if (sh >= 32)
            v = vh[k][t] >> (sh - 32);
          else if (sh >= 0)
            v = (i64)(((unsigned long long)__funnelshift_r(w1, (unsigned)w2, sh) << 32) |
                      __funnelshift_r(vl[k][t], w1, sh));
          else
            v = (i64)((((unsigned long long)w1 << 32) | vl[k][t]) << min(-sh, 63));
          (k ? x[t].y : x[t].x) = v;
        }
      }
    }
    if (on) {
      dft<R, -1>(x);
#pragma unroll
      for (int s = 0; s < R; ++s) h[s] = FEW ? x[s] : cmulw<false, P::kSH>(x[s], tw(3 * s * q));
    }
  }
  if constexpr (FEW) {
    __syncthreads();
    for (int i = tid; i < 3 * L && meta[0].act; i += kFew) {
      const int b = i / L, q = i % L / R, s = i % R;
      C* h = Hb(0) + b * FS + q * (R + 1) + s;
      *h = cmulw<false, P::kSH>(*h, tw(3 * s * q));
    }
  }
  if (P::kSum2 > 1) tree(s2, P::kSum2, s3, P::kSum3);
  __syncthreads();

  // ---- PB: M-point forward transforms of the three sub-rows, in place
  if constexpr (M2 > 1) {
    for (int i = tid; i < RB * 3 * R * M1; i += T) {
      const int r = i / (3 * R * M1), i1 = i - r * 3 * R * M1;
      const int b = i1 / (R * M1), i2 = i1 - b * R * M1;
      const int u = i2 / R, s = i2 - u * R;
      if (!meta[r].act) continue;
      C* h = Hb(r) + b * FS + s + u * (R + 1);
      C x[M2];
#pragma unroll
      for (int v = 0; v < M2; ++v) x[v] = h[M1 * v * (R + 1)];
      dft<M2, -1>(x);
#pragma unroll
      for (int j = 0; j < M2; ++j) h[M1 * j * (R + 1)] = cmulw<false, P::kSH>(x[j], tw(3 * R * u * j));
    }
    __syncthreads();
  }
  for (int i = tid; i < RB * 3 * R * M2; i += T) {
    const int b = i / (RB * R * M2), i1 = i - b * RB * R * M2;
    const int r = i1 / (R * M2), i2 = i1 - r * R * M2;
    const int j = i2 / R, s = i2 - j * R;
    if (!meta[r].act) continue;
    C* h = Hb(r) + b * FS + s + M1 * j * (R + 1);
    C x[M1];
#pragma unroll
    for (int u = 0; u < M1; ++u) x[u] = h[u * (R + 1)];
    dft<M1, -1>(x);
#pragma unroll
    for (int a = 0; a < M1; ++a)
      h[a * (R + 1)] = FEW ? x[a] : cmulw<false, P::kSH>(x[a], tw((R * (M2 * a + j) + s) * b));
  }
  if constexpr (FEW) {
    __syncthreads();
    for (int i = tid; i < 3 * L && meta[0].act; i += kFew) {
      const int b = i / L, k = i % L;
      C* h = Hb(0) + b * FS + k % R + k / R * (R + 1);
      *h = cmulw<false, P::kSH>(*h, tw(k * b));
    }
  }
  __syncthreads();

  // ---- PF: C[m] = Y_0 + Y_1 + Y_2, C[N - m] = Y_0 + w Y_1 + w^2 Y_2 (w = exp(2 pi i / 3))
  // at L - m, unpacked into the two products' modes
  const size_t qs = (size_t)g.Mz * L * 2;
  for (int i = tid; i < RB * L; i += T) {
    const int r = i / L, m = i - r * L;
    if (!meta[r].act) continue;
    const int row = row0 + r, bb = row / g.Mz, jz = row - bb * g.Mz;
    const C* h = Hb(r);
    auto slot = [&](int k) {
      const int p = k / R;
      return (M2 > 1 ? p / M2 + M1 * (p % M2) : p) * (R + 1) + k % R;
    };
    const int sm = slot(m);
    const C cm = add(add(h[sm], h[FS + sm]), h[2 * FS + sm]);
    C cn = cm;
    if (m > 0) {
      const int sn = slot(L - m);
      const C y0 = h[sn], t1 = add(h[FS + sn], h[2 * FS + sn]), t2 = sub(h[FS + sn], h[2 * FS + sn]);
      cn.x = y0.x - (t1.x >> 1) - rmul(t2.y, kQ62_s3);
      cn.y = y0.y - (t1.y >> 1) + rmul(t2.x, kQ62_s3);
    }
    const double* sums = Sb(r) + (P::kSum2 > 1 ? s3 : P::kSum1 > 1 ? s2 : s1);
    int E[6];
    exponents(r, E);
    const RowMeta& me = meta[r];
    bool fin = true;
#pragma unroll
    for (int f = 0; f < 6; ++f) fin = fin && me.emax[f] != 0x7ff;
    const double nan = __hiloint2double(0x7ff80000, 0), c = 0.5 / N;
    const double sT = fin ? c * fx::pow2(me.bits[0] - 55 + E[0] + E[4] - 86 + P::kShift) : nan;
    const double sO = fin ? c * fx::pow2(me.bits[1] - 55 + E[0] + E[2] - 86 + P::kShift) : nan;
    const double2 n0 = make_double2(sT * (double)(cm.x + cn.x), sT * (double)(cm.y - cn.y));
    double2 n1 = make_double2(sO * (double)(cm.y + cn.y), sO * (double)(cn.x - cm.x));
    double* q0 = Q + (size_t)bb * 2 * qs + (size_t)jz * L * 2 + 2 * m;
    if (m == 0) {
      n1.x = sums[1];
      n1.y = 0;
      wT[(size_t)bb * g.Mz + jz] = sums[0];
    }
    *reinterpret_cast<double2*>(q0) = n0;
    *reinterpret_cast<double2*>(q0 + qs) = n1;
  }
}

// Rows per block and threads.  The P2 items (3 M per row) are one per thread;
// a block takes as many rows as make about 192 threads (integer and FP32 work
// alike fill whole warps then) while at least two blocks per SM remain, else
// fewer: a single state's rows spread over the SMs, with threads enough for the
// other passes' items (9 R per row).
struct RowsShape {
  int rb, threads;
  size_t smem;
};

template <int L> RowsShape rows_shape(const Work& w, int nrows) {
  using P = Plan<L>;
  const int cap = (w.shapes && w.shapes->rows_threads > 0) ? std::min(320, w.shapes->rows_threads) : 192;
  int rb = 1;
  while (rb < kMaxRB && P::threads(2 * rb) <= cap && 2 * rb * P::row_bytes <= 100 * 1024) rb *= 2;
  const int form = w.shapes ? w.shapes->rows_cl : -1;
  if (form == 1)
    rb = 1;
  else if (form < 0)
    while (rb > 1 && (long)nrows < 2L * 152 * rb) rb /= 2;
  // threads for the other passes' items too: a row alone has 9 R M2 in its first
  // pass and unpacks L modes.  With few rows per SM they shorten its chain (512 x 128,
  // 3 states 59.6 -> 48 us; up to L = 128 two rows per SM take FEW); with more the
  // rows hide each other's (512 x 128, 16 states 226 us either way), except at
  // L = 512, where shared memory holds two (1024 x 256, 8 states 684 -> 561 us).
  const int items = rb > 1 ? rb * 9 * P::R * P::M2 : std::max(9 * P::R * P::M2, L + 32);
  const int most = rb > 1 ? 128 : L == 512 ? 320 : nrows <= 4 * 152 ? 256 : 128;
  const int th = std::max(P::threads(rb), std::min(most, (items + 31) / 32 * 32));
  return {rb, th, rb * P::row_bytes};
}

// FEW for rows of 96 to 384 points (one first pass)
template <int L> constexpr bool kHasFew = Plan<L>::kAlias && L >= 32;

template <int L> cudaError_t launch_rows_L(const Grid& g, const Tables& t, const Work& w, int B, const int* ns, cudaStream_t s) {
  const int nrows = B * g.Mz;
  const RowsShape sh = rows_shape<L>(w, nrows);
  if constexpr (kHasFew<L>)
    if (sh.rb == 1 && nrows <= 2 * 152)
      return launch_pdl(w.pdl != 0, k_rows_fx<L, true>, (unsigned)nrows, kFew, sh.smem, s, g, t.twfx, t.rk, w.Z, w.Q, w.wT,
                        nrows, 1, ns, w.step);
  return launch_pdl(w.pdl != 0, k_rows_fx<L, false>, (unsigned)((nrows + sh.rb - 1) / sh.rb), sh.threads, sh.smem, s, g, t.twfx,
                    t.rk, w.Z, w.Q, w.wT, nrows, sh.rb, ns, w.step);
}

template <int L> cudaError_t allow_rows_L() {
  // up to 100 KB of rows per block, or one row where that is more
  const size_t need = std::max<size_t>(100 * 1024, Plan<L>::row_bytes);
  if constexpr (kHasFew<L>) {
    const cudaError_t e = cudaFuncSetAttribute(k_rows_fx<L, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need);
    if (e != cudaSuccess) return e;
  }
  return cudaFuncSetAttribute(k_rows_fx<L, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)need);
}

}  // namespace

#define RBC_ROWS_CASES(X) X(2) X(4) X(8) X(16) X(32) X(64) X(128) X(256) X(512)

cudaError_t configure_rows_fx(const Grid& g) {
  switch (g.nm) {
#define X(L) case L: return allow_rows_L<L>();
    RBC_ROWS_CASES(X)
#undef X
  }
  return cudaErrorInvalidValue;
}

cudaError_t launch_rows_fx(const Grid& g, const Tables& t, const Work& w, int B, const int* ns, cudaStream_t s) {
  switch (g.nm) {
#define X(L) case L: return launch_rows_L<L>(g, t, w, B, ns, s);
    RBC_ROWS_CASES(X)
#undef X
  }
  return cudaErrorInvalidValue;
}

}  // namespace rbc
