// z transforms of the FP64 mode in block fixed point (rbc_fx.cuh).
//
// Both are products with small dense tables, sum_n A[r][n] x[n], one real
// column (Fourier mode, real or imaginary part) per lane.  Table rows and data
// columns are integers of up to 60 bits with an exponent per row and per
// column, each split into halves of 30 bits, v = h 2^30 + l; a term is three
// 32x32->64-bit multiply-adds,
//   h_A h_x into the sum of high parts, h_A l_x + l_A h_x into the middle one
// (l_A l_x, below 2^-60 of the bound, is dropped), and the middle sum joins the
// high one, rounded, after every eight terms.  The groups of eight are fixed by
// the grid, and integer sums do not depend on their order: the split of a sum
// over warps and the row tiling never change a bit.
//
// Bound: integer issue, 13 clocks of a sub-partition per term and warp (12 of
// them the multiply-adds) against 64 for an FP64 multiply-add.
// Measured (GB300, per launch, FP64 sums before): inverse, 256 x 64, 32 states
// 301 -> 116 us, 8 states 82 -> 39 us, one state 40 -> 14 us; 512 x 128, 3 states
// 215 -> 89 us; 64 x 32, 23 states 26.5 -> 16.5 us.  Forward: 100 -> 38 us,
// 30 -> 16.4 us, 12.4 -> 10.1 us, 83 -> 33 us, 10.8 -> 9.9 us.  (128 x 32, one
// state: 13.3 -> 10.3 and 9.3 -> 8.3 us, of which about 7 are the launch as timed.)
// Against 64-bit plain torch the temperature after a few steps is 2 to 3 times
// closer than with FP64 sums, psi equally close (its solve dominates).
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdint>
#include <vector>

#include "rbc_fx.cuh"
#include "rbc_internal.h"

namespace rbc {

namespace {

using fx::i64;

constexpr int kGroup = 8;       // terms per rounding of the middle sum: 8 (2^30 2^29) + 2^59 < 2^63
constexpr int kCols = 32;       // real columns per block: 16 modes x re/im
constexpr int kWarps = 8;
constexpr int kNaN = 0x7fff;    // column exponent of a non-finite column

__host__ __device__ constexpr int pad_group(int k) { return (k + kGroup - 1) / kGroup * kGroup; }

__device__ __forceinline__ int2 halves30(i64 v) {
  const int l = ((int)((unsigned)v << 2)) >> 2;       // low 30 bits, signed
  return make_int2((int)((v - l) >> 30), l);
}
__device__ __forceinline__ void mac30(int2 a, int2 x, i64& hi, i64& mid) {
  hi = fx::madw(a.x, x.x, hi);
  mid = fx::madw(a.x, x.y, fx::madw(a.y, x.x, mid));
}
constexpr i64 kHalf = 1ll << 29;
// 2^e v for a column exponent that may mark a non-finite column; INT: on the integer
// pipe.  The inverse, whose blocks alternate between sums on the integer pipe and
// fields on the FP64 pipe, gains (128 -> 121 us at 256 x 64, 32 states); the
// forward sums, two instructions of 64 clocks against 20, do not (37.7 -> 38.9 us).
template <bool INT>
__device__ __forceinline__ double scaled(i64 v, int ecol, int e) {
  if (ecol >= kNaN) return __hiloint2double(0x7ff80000, 0);
  return INT ? fx::to_double(v, ecol - 1022 + e) : (double)v * fx::pow2(ecol - 1022 + e);
}

}  // namespace

// ---------------------------------------------------------------------------
// z inverse transform (k_zinv_fx): fields of the padded rows from the state.
// Even/odd split: at the points s_j and s_{Mz-1-j} = -s_j the sums E, O over
// even and odd n of V^(q)[j][n] x[n] give f^(q) = E + O and (-1)^q (E - O).
// Operators q = 0..3 for psi and q = 0, 1 for T.  The q-th derivative's rows
// grow like n^(2q) at the walls and n^q inside; both tables and columns are
// scaled by 2^-G_q(n), 2^G_q(n), G_q = 1.5 q log2(n), so that neither spans
// more than n^(q/2) and 60 bits keep the relative accuracy of FP64 sums.
// Block: one field (psi: four operators, T: two), 16 modes (32 real columns, one
// per lane), eight warps.  A warp sums two row pairs, so that every column value
// read from shared memory serves two of them, or KS warps share one row pair
// where a launch would otherwise leave SMs idle.  The block converts the columns
// (one scaled version per operator) into shared memory once, or in chunks of 64
// coefficients; a warp's table rows come 32 entries at a time through registers
// into shared memory of its own, where all lanes read the same entry (read
// straight from L2, group by group, they left the warps waiting two thirds of
// the time: 138 -> 129 us at 256 x 64, 32 states, 137 -> 99 us at 512 x 128, 3).
// ---------------------------------------------------------------------------
namespace {

constexpr int kSub = 32;        // table entries per row pair on their way at a time

template <int NQ, int KS>
__device__ __forceinline__ void zinv_block(const Grid& g, const int2* __restrict__ A, const int* __restrict__ Ea,
                                           const int4* __restrict__ gexp, const double* __restrict__ Xb,
                                           double* __restrict__ Zb, int ct, int jb, int jblocks, int chunk, int diag,
                                           unsigned char* zsm, size_t asm_off, int (*ecol)[kCols], const int* nsteps,
                                           const int* step) {
  const int Kp = pad_group(g.nq), LN = 2 * Kp, Mh = (g.Mz + 1) / 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int m = ct * 16 + (lane >> 1), c = lane & 1;
  const bool valid = m < g.nm;
  const size_t xs = (size_t)g.nm * 2;                                       // coefficient stride
  const double* x0 = Xb + (NQ == 4 ? g.Nz * xs : 0) + (size_t)2 * (valid ? m : 0) + c;
  constexpr int JW = KS == 1 ? 2 : 1;                                       // row pairs per warp
  int4* XS = reinterpret_cast<int4*>(zsm);                                  // [chunk][NQ / 2][32], two operators each
  i64* part = reinterpret_cast<i64*>(zsm + (size_t)chunk * NQ * kCols * sizeof(int2));   // [8][NQ][32], KS > 1
  // Table rows of the warp's JW row pairs, up to kSub entries at a time, on
  // their way through registers while the entries before them are summed.
  int4* arow = reinterpret_cast<int4*>(zsm + asm_off) + warp * (JW * kSub * (NQ / 2));   // [JW][kSub][NQ / 2]
  int4 ahead[JW][NQ / 2];
  auto fetch = [&](int jp, int i) {   // lane: entry i + lane of each row pair
#pragma unroll
    for (int r = 0; r < JW; ++r) {
      const int row = min(jp + r, Mh - 1), e = min(i + lane, LN - 1);
      const int4* a = reinterpret_cast<const int4*>(A + ((size_t)row * LN + e) * 4);
#pragma unroll
      for (int h = 0; h < NQ / 2; ++h) ahead[r][h] = __ldg(a + h);
    }
  };
  auto place = [&] {
    __syncwarp();
#pragma unroll
    for (int r = 0; r < JW; ++r)
#pragma unroll
      for (int h = 0; h < NQ / 2; ++h) arow[(r * kSub + lane) * (NQ / 2) + h] = ahead[r][h];
    __syncwarp();
  };
  constexpr int JB = kWarps / KS * JW;                          // row pairs per round
  const int js = (KS == 1 ? warp : warp / KS) * JW, ks = KS == 1 ? 0 : warp % KS;
  // KS > 1: warps ks = 0, 2, .. share the groups of the even coefficients, 1, 3, ..
  // those of the odd ones; lanes 8 i .. 8 i + 7 fetch the warp's i-th group
  constexpr int every = (KS > 1 ? KS / 2 : 1) * kGroup;
  const int first = (ks >> 1) * kGroup;
  auto share = [&](int i) { return (ks & 1) * Kp + min(i + (lane / kGroup) * every + lane % kGroup, Kp - 1) - lane; };
  fetch(jb * JB + js, KS == 1 ? 0 : share(first));
  pdl_wait();
  // (whether the state is active is looked at once its values are on their way)
  const int now = nsteps ? *step : 0, last = nsteps ? *nsteps : 1;
  for (int i = threadIdx.x; i < NQ * kCols; i += blockDim.x) (&ecol[0][0])[i] = 0;
  __syncthreads();
  {
    int em[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) em[q] = 0;
#pragma unroll 4
    for (int n = warp; n < g.Nz; n += kWarps) {
      const int4 gq = __ldg(gexp + n);
      const int gs[4] = {gq.x, gq.y, gq.z, gq.w};
      const int e = fx::biased_exp(valid ? __ldg(x0 + n * xs) : 0.0);
      const int v = e == 0x7ff ? kNaN : e;
#pragma unroll
      for (int q = 0; q < NQ; ++q) em[q] = max(em[q], e > 0 ? v + gs[q] : 0);
    }
    if (now >= last) return;   // uniform per block
#pragma unroll
    for (int q = 0; q < NQ; ++q) atomicMax(&ecol[q][lane], em[q]);
  }
  __syncthreads();
  int ec[NQ];
#pragma unroll
  for (int q = 0; q < NQ; ++q) ec[q] = ecol[q][lane];
  auto stage = [&](int i0, int i1) {   // list entries [i0, i1): parity i / Kp, coefficient 2 (i % Kp) + parity
#pragma unroll 2
    for (int i = i0 + warp; i < i1; i += kWarps) {
      const int p = i / Kp, n = 2 * (i - p * Kp) + p;
      int4* dst = XS + (size_t)(i - i0) * (NQ / 2) * kCols + lane;
      const double v = valid && n < g.Nz ? __ldg(x0 + n * xs) : 0.0;
      const int4 gq = __ldg(gexp + (n < g.Nz ? n : 0));
      const int gs[4] = {gq.x, gq.y, gq.z, gq.w};
#pragma unroll
      for (int h = 0; h < NQ / 2; ++h) {
        const int2 a = halves30(fx::from_double<60>(v, ec[2 * h] - gs[2 * h]));
        const int2 b = halves30(fx::from_double<60>(v, ec[2 * h + 1] - gs[2 * h + 1]));
        dst[h * kCols] = make_int4(a.x, a.y, b.x, b.y);
      }
    }
  };
  // one group of eight terms, entries e0 .. e0 + 7 of arow against staged columns x0s ..
  auto group = [&](int e0, int x0s, i64 (*hi)[NQ]) {
    const int4* x = XS + (size_t)x0s * (NQ / 2) * kCols + lane;
    i64 mid[JW][NQ];
#pragma unroll
    for (int r = 0; r < JW; ++r)
#pragma unroll
      for (int q = 0; q < NQ; ++q) mid[r][q] = kHalf;
#pragma unroll
    for (int e = 0; e < kGroup; ++e) {
      int4 xv[NQ / 2];
#pragma unroll
      for (int h = 0; h < NQ / 2; ++h) xv[h] = x[(e * (NQ / 2) + h) * kCols];
#pragma unroll
      for (int r = 0; r < JW; ++r)
#pragma unroll
        for (int h = 0; h < NQ / 2; ++h) {
          const int4 v = arow[(r * kSub + e0 + e) * (NQ / 2) + h], w = xv[h];
          mac30(make_int2(v.x, v.y), make_int2(w.x, w.y), hi[r][2 * h], mid[r][2 * h]);
          mac30(make_int2(v.z, v.w), make_int2(w.z, w.w), hi[r][2 * h + 1], mid[r][2 * h + 1]);
        }
    }
#pragma unroll
    for (int r = 0; r < JW; ++r)
#pragma unroll
      for (int q = 0; q < NQ; ++q) hi[r][q] += mid[r][q] >> 30;
  };
  const double k = g.kfac * m, kk = k * k;
  const size_t fs = (size_t)g.Mz * g.nm * 2;
  double* Zc = Zb + (NQ == 4 ? 0 : 4 * fs) + (size_t)2 * (valid ? m : 0) + c;
  // fields of padded row j from the sums of its row pair jp (sg = -1: the mirrored row)
  auto emit = [&](int jp, int j, int sg, const i64* E, const i64* O) {
    // 2^q times the q-th sum: the factors of two of the fields below (exact)
    double P[NQ];
#pragma unroll
    for (int q = 0; q < NQ; ++q) {
      const i64 v = sg > 0 ? E[q] + O[q] : (q & 1) ? O[q] - E[q] : E[q] - O[q];
      P[q] = scaled<true>(v, ec[q], __ldg(Ea + q * Mh + jp) - 60 + q);
    }
    // i z of a complex value: the partner lane's part, negated in the real lane
    auto timesi = [&](double v) {
      const double o = __shfl_xor_sync(0xffffffffu, v, 1);
      return c == 0 ? -o : o;
    };
    const bool m0 = m == 0;
    double* z = Zc + (size_t)j * g.nm * 2;
    if constexpr (NQ == 4) {
      const double ip = timesi(P[0]);
      const double om = fma(kk, P[0], -P[2]);                   // omega = k^2 psi - 4 d2(psi)
      const double io = timesi(om);
      if (!valid) return;
      z[0] = m0 ? (c == 0 ? P[0] : 0.0) : P[1];                 // u = d_z psi (m = 0: U)
      z[fs] = m0 ? 0.0 : -k * ip;                               // w = -ik psi
      z[2 * fs] = m0 ? 0.0 : k * io;                            // d_x omega
      z[3 * fs] = m0 ? (c == 0 ? -P[2] : 0.0) : fma(kk, P[1], -P[3]);   // d_z omega = 2 k^2 d1 - 8 d3
    } else {
      const double it = timesi(P[0]);
      if (!valid) return;
      z[0] = diag ? P[0] : m0 ? 0.0 : k * it;                   // d_x T (the averages of Sec. 2.2: T)
      z[fs] = P[1];                                             // d_z T
    }
  };
  const int rounds = (Mh + jblocks * JB - 1) / (jblocks * JB);
  if (chunk >= LN) {
    stage(0, LN);
    __syncthreads();
  }
  for (int r = 0; r < rounds; ++r) {
    const int jp = (r * jblocks + jb) * JB + js;
    const bool on = jp < Mh;
    i64 E[JW][NQ], O[JW][NQ];
    if (KS == 1) {
#pragma unroll 1
      for (int p = 0; p < 2; ++p) {
        i64 sum[JW][NQ];
#pragma unroll
        for (int w = 0; w < JW; ++w)
#pragma unroll
          for (int q = 0; q < NQ; ++q) sum[w][q] = 0;
        for (int i0 = 0; i0 < Kp; i0 += chunk) {
          const int i1 = min(Kp, i0 + chunk);
          if (chunk < LN) {
            __syncthreads();
            stage(p * Kp + i0, p * Kp + i1);
            __syncthreads();
          }
          for (int i = i0; i < i1; i += kSub) {
            place();
            // the next entries: of this row pair, of the other parity, of the next round
            int nj = jp, ni = p * Kp + i + kSub;
            if (i + kSub >= Kp) {
              ni = p == 0 ? Kp : 0;
              nj = p == 0 ? jp : jp + jblocks * JB;
            }
            fetch(nj, ni);
            if (on)
              for (int e = 0; e < min(kSub, i1 - i); e += kGroup) group(e, (chunk < LN ? -i0 : p * Kp) + i + e, sum);
          }
        }
#pragma unroll
        for (int w = 0; w < JW; ++w)
#pragma unroll
          for (int q = 0; q < NQ; ++q) {
            E[w][q] = p ? E[w][q] : sum[w][q];
            O[w][q] = sum[w][q];
          }
      }
#pragma unroll
      for (int w = 0; w < JW; ++w)
        if (jp + w < Mh) {
          emit(jp + w, jp + w, 1, E[w], O[w]);
          if (g.Mz - 1 - (jp + w) != jp + w) emit(jp + w, g.Mz - 1 - (jp + w), -1, E[w], O[w]);
        }
    } else {
#pragma unroll
      for (int q = 0; q < NQ; ++q) E[0][q] = 0;
      for (int i = first; i < Kp; i += (kSub / kGroup) * every) {
        place();
        const int next = i + (kSub / kGroup) * every;
        fetch(next < Kp ? jp : jp + jblocks * JB, share(next < Kp ? next : first));
        if (on)
          for (int s = 0; s < kSub / kGroup && i + s * every < Kp; ++s)
            group(s * kGroup, (ks & 1) * Kp + i + s * every, E);
      }
#pragma unroll
      for (int q = 0; q < NQ; ++q) part[(warp * NQ + q) * kCols + lane] = E[0][q];
      __syncthreads();
      if (on && ks < 2) {
#pragma unroll
        for (int q = 0; q < NQ; ++q) {
          i64 e = 0, o = 0;
#pragma unroll
          for (int s = 0; s < KS; s += 2) {
            e += part[((js * KS + s) * NQ + q) * kCols + lane];
            o += part[((js * KS + s + 1) * NQ + q) * kCols + lane];
          }
          E[0][q] = e;
          O[0][q] = o;
        }
        if (ks == 0)
          emit(jp, jp, 1, E[0], O[0]);
        else if (g.Mz - 1 - jp != jp)
          emit(jp, g.Mz - 1 - jp, -1, E[0], O[0]);
      }
      __syncthreads();
    }
  }
}

}  // namespace

template <int KS>
__global__ void __launch_bounds__(32 * kWarps, 2) k_zinv_fx(Grid g, const int2* __restrict__ A, const int* __restrict__ Ea,
                                                            const int4* __restrict__ gexp, const double* __restrict__ X,
                                                            size_t S, double* __restrict__ Z, int B, int jblocks,
                                                            int chunk, const int* nsteps, const int* step, int diag) {
  extern __shared__ __align__(16) unsigned char zsm[];
  __shared__ int ecol[4][kCols];
  const int ctiles = (g.nm + 15) / 16;
  int rem = blockIdx.x;
  const int jb = rem % jblocks;
  rem /= jblocks;
  const int ct = rem % ctiles;
  rem /= ctiles;
  const int f = rem & 1, b = rem >> 1;
  const int* ns = nsteps == nullptr ? nullptr : nsteps + b;   // the grid is exact: b < B
  const double* Xb = X + (size_t)b * S;
  double* Zb = Z + (size_t)b * 6 * ((size_t)g.Mz * g.nm * 2);
  // table rows behind the staged columns and the partial sums
  const size_t asm_off = (size_t)chunk * 4 * kCols * sizeof(int2) + (KS > 1 ? (size_t)kWarps * 4 * kCols * sizeof(i64) : 0);
  if (f == 0)
    zinv_block<4, KS>(g, A, Ea, gexp, Xb, Zb, ct, jb, jblocks, chunk, diag, zsm, asm_off, ecol, ns, step);
  else
    zinv_block<2, KS>(g, A, Ea, gexp, Xb, Zb, ct, jb, jblocks, chunk, diag, zsm, asm_off, ecol, ns, step);
}

// Warps per row pair (KS) and blocks per column tile, from a sweep of both over
// 18 grids and batches (time of a whole stage).  One warp per two row pairs and a
// block per 16 of them (every block converts its columns again, which costs less
// than a second round: 256 x 64, 32 states 349 us in one round, 360 in two) from
// 4864 row pairs on (152 SMs x 32), or 2432 where 128 coefficients leave room for
// one block per SM only; below, two warps share a row pair (256 x 64, 4 states 90 us
// against 95 with one) and below 608 row pairs four (128 x 32, one state 33.8 us
// against 34.6).  Shared row pairs take rounds in blocks of two per SM (64 x 32,
// 23 states: 50.0 us in two rounds, 52.3 in one).
namespace {
struct ZinvShape {
  int ks, jblocks, chunk;
  size_t smem;
};
ZinvShape zinv_shape(const Grid& g, int B) {
  const int Kp = pad_group(g.nq), LN = 2 * Kp, Mh = (g.Mz + 1) / 2, ctiles = (g.nm + 15) / 16;
  const long cols = 2L * B * ctiles;   // (state, field, column tile)
  int ks = 1;
  if (LN <= 128)
    while (ks < 4 && ks < 2 * (Kp / kGroup) && cols * Mh * ks < (ks > 1 ? 1216 : LN <= 64 ? 4864 : 2432)) ks *= 2;
  const int jb = ks == 1 ? 2 * kWarps : kWarps / ks, most = (Mh + jb - 1) / jb;
  const int rounds = ks == 1 ? 1 : (int)std::min<long>(most, (cols * most + 303) / 304);
  const int jblocks = (most + rounds - 1) / rounds;
  const int chunk = ks > 1 ? LN : std::min(LN, 64);
  const size_t smem = (size_t)chunk * 4 * kCols * sizeof(int2) + (ks > 1 ? (size_t)kWarps * 4 * kCols * sizeof(i64) : 0) +
                      (size_t)kWarps * (ks > 1 ? 1 : 2) * kSub * 2 * sizeof(int4);
  return {ks, jblocks, chunk, smem};
}
constexpr int kZinvSmem =
    128 * 4 * kCols * (int)sizeof(int2) + kWarps * 4 * kCols * (int)sizeof(i64) + kWarps * 2 * kSub * 2 * (int)sizeof(int4);

template <int KS>
cudaError_t launch_zinv_ks(const Grid& g, const Tables& t, const Work& w, const double* X, double* Z, int B,
                           const ZinvShape& sh, const int* ns, bool diag, cudaStream_t s) {
  const int ctiles = (g.nm + 15) / 16;
  return launch_pdl(w.pdl != 0 && !diag, k_zinv_fx<KS>, (unsigned)(2 * B * ctiles * sh.jblocks), 32 * kWarps, sh.smem, s,
                    g, t.zfxA, t.zfxAe, t.zfxG, X, state_doubles(g), Z, B, sh.jblocks, sh.chunk, ns, w.step, diag ? 1 : 0);
}
}  // namespace

cudaError_t launch_zinv_fx(const Grid& g, const Tables& t, const Work& w, const double* X, int B, const int* ns,
                           bool diag, cudaStream_t s) {
  const ZinvShape sh = zinv_shape(g, B);
  switch (sh.ks) {
    case 1: return launch_zinv_ks<1>(g, t, w, X, w.Z, B, sh, ns, diag, s);
    case 2: return launch_zinv_ks<2>(g, t, w, X, w.Z, B, sh, ns, diag, s);
    default: return launch_zinv_ks<4>(g, t, w, X, w.Z, B, sh, ns, diag, s);
  }
}

// ---------------------------------------------------------------------------
// z forward transform (k_zfwd_fx): F_n = sum_{jh < ceil(Mz/2)} W[n][jh] fold_p[jh],
// p = n mod 2, fold_p = Q_j +- Q_{Mz-1-j} (the middle row of an odd Mz once, for
// p = 0).  Block: one state, field, parity, 16 modes (32 real columns, one per
// lane) and a share of the coefficients; the folds are formed as integers in
// shared memory (one exponent per column), each warp sums NI coefficients at a
// time.
// ---------------------------------------------------------------------------
template <int NI>
__global__ void __launch_bounds__(32 * kWarps) k_zfwd_fx(Grid g, const int2* __restrict__ Wt, const int* __restrict__ We,
                                                         const double* __restrict__ Q, double* __restrict__ F, size_t S,
                                                         int B, int nblocks, const int* nsteps, const int* step) {
  extern __shared__ __align__(16) unsigned char fsm[];
  __shared__ int ecol[kCols];
  __shared__ __align__(16) int2 wsm[kWarps][NI * kSub];
  const int Mh = (g.Mz + 1) / 2, Kh = pad_group(Mh), ctiles = (g.nm + 15) / 16;
  int rem = blockIdx.x;
  const int nb = rem % nblocks;
  rem /= nblocks;
  const int ct = rem % ctiles;
  rem /= ctiles;
  const int p = rem & 1, f = (rem >> 1) & 1, b = rem >> 2;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int first = (nb * kWarps + warp) * NI;
  // table rows of the warp's coefficients, kSub entries at a time, on their way
  // through registers while the entries before them are summed
  int2* wrow = wsm[warp];
  int2 ahead[NI];
  auto fetch = [&](int r0, int i0) {
#pragma unroll
    for (int i = 0; i < NI; ++i)
      ahead[i] = __ldg(Wt + (size_t)(2 * min(r0 + i, g.nq - 1) + p) * Kh + min(i0 + lane, Kh - 1));
  };
  auto place = [&] {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < NI; ++i) wrow[i * kSub + lane] = ahead[i];
    __syncwarp();
  };
  fetch(first, 0);
  pdl_wait();
  const int now = nsteps ? *step : 0, last = nsteps ? nsteps[b] : 1;   // (the grid is exact: b < B)
  const int m = ct * 16 + (lane >> 1), c = lane & 1;
  const bool valid = m < g.nm;
  const size_t rs = (size_t)g.nm * 2;
  const double* q = Q + (size_t)(b * 2 + f) * g.Mz * rs + (size_t)2 * (valid ? m : 0) + c;
  int2* FS = reinterpret_cast<int2*>(fsm);   // [Kh][32]
  if (threadIdx.x < kCols) ecol[threadIdx.x] = 0;
  __syncthreads();
  int em = 0;
  for (int j = warp; j < g.Mz; j += kWarps) {
    const int e = fx::biased_exp(valid ? __ldg(q + j * rs) : 0.0);
    em = max(em, e == 0x7ff ? kNaN : e);
  }
  if (now >= last) return;   // uniform per block
  atomicMax(&ecol[lane], em);
  __syncthreads();
  em = ecol[lane];
  for (int jh = warp; jh < Kh; jh += kWarps) {
    i64 v = 0;
    if (valid && jh < Mh) {
      const int jr = g.Mz - 1 - jh;
      const i64 a = fx::from_double<59>(__ldg(q + jh * rs), em);
      if (jr != jh) {
        const i64 d = fx::from_double<59>(__ldg(q + jr * rs), em);
        v = p == 0 ? a + d : a - d;
      } else {
        v = p == 0 ? a : 0;
      }
    }
    FS[jh * kCols + lane] = halves30(v);
  }
  __syncthreads();
  double* Fb = F + (size_t)b * S + (size_t)f * g.Nz * rs + (size_t)2 * (valid ? m : 0) + c;
  for (int r0 = first; r0 < g.nq; r0 += nblocks * kWarps * NI) {
    i64 hi[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) hi[i] = 0;
    for (int i0 = 0; i0 < Kh; i0 += kSub) {
      place();
      const bool more = i0 + kSub < Kh;
      fetch(more ? r0 : r0 + nblocks * kWarps * NI, more ? i0 + kSub : 0);
      for (int j0 = 0; j0 < min(kSub, Kh - i0); j0 += kGroup) {
        i64 mid[NI];
#pragma unroll
        for (int i = 0; i < NI; ++i) mid[i] = kHalf;
#pragma unroll
        for (int e = 0; e < kGroup; e += 2) {
          const int2 x0 = FS[(i0 + j0 + e) * kCols + lane], x1 = FS[(i0 + j0 + e + 1) * kCols + lane];
#pragma unroll
          for (int i = 0; i < NI; ++i) {
            const int4 a = *reinterpret_cast<const int4*>(wrow + i * kSub + j0 + e);
            mac30(make_int2(a.x, a.y), x0, hi[i], mid[i]);
            mac30(make_int2(a.z, a.w), x1, hi[i], mid[i]);
          }
        }
#pragma unroll
        for (int i = 0; i < NI; ++i) hi[i] += mid[i] >> 30;
      }
    }
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if (valid && r0 + i < g.nq) {
        const int n = 2 * (r0 + i) + p;
        Fb[n * rs] = scaled<false>(hi[i], em, __ldg(We + n) - 59);
      }
  }
}

namespace {
size_t zfwd_fx_smem(const Grid& g) { return (size_t)pad_group((g.Mz + 1) / 2) * kCols * sizeof(int2); }

template <int NI>
cudaError_t launch_zfwd_ni(const Grid& g, const Tables& t, const Work& w, int B, cudaStream_t s) {
  const int ctiles = (g.nm + 15) / 16;
  const long base = 4L * B * ctiles;
  const int most = (g.nq + kWarps * NI - 1) / (kWarps * NI);
  const int rounds = (int)std::min<long>((most + 1) / 2, (base * most + 455) / 456);
  const int nblocks = (most + rounds - 1) / rounds;
  return launch_pdl(w.pdl != 0, k_zfwd_fx<NI>, (unsigned)(base * nblocks), 32 * kWarps, zfwd_fx_smem(g), s, g, t.zfxW,
                    t.zfxWe, w.Q, w.F, state_doubles(g), B, nblocks, w.nsteps, w.step);
}
}  // namespace

// Coefficients per warp: four share each fold read from shared memory (a stage of
// 256 x 64, 8 states takes 112.3 us with four, 112.6 with two, 114 with one); fewer
// where four would leave SMs without a block (one state: 61.2 with one, 63.8 with
// four).  Two rounds or more per block where one would make more than three blocks
// per SM (1024 x 256, one state: 425 us, 432 in one round).
cudaError_t launch_zfwd_fx(const Grid& g, const Tables& t, const Work& w, int B, cudaStream_t s) {
  const long warps = 4L * B * ((g.nm + 15) / 16) * g.nq;   // one coefficient each
  if (warps >= 4096) return launch_zfwd_ni<4>(g, t, w, B, s);
  if (warps > 2048) return launch_zfwd_ni<2>(g, t, w, B, s);
  return launch_zfwd_ni<1>(g, t, w, B, s);
}

// the largest row of folds that rbc_create accepts (Nz = 512)
constexpr int kZfwdSmem = 384 * kCols * (int)sizeof(int2);

cudaError_t configure_zfx(const Grid& g) {
  cudaError_t e = cudaSuccess;
  auto allow = [&](auto* fn, int need) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, need);
  };
  allow(k_zinv_fx<1>, kZinvSmem);
  allow(k_zinv_fx<2>, kZinvSmem);
  allow(k_zinv_fx<4>, kZinvSmem);
  if (!g.mixed) {
    allow(k_zfwd_fx<1>, kZfwdSmem);
    allow(k_zfwd_fx<2>, kZfwdSmem);
    allow(k_zfwd_fx<4>, kZfwdSmem);
  }
  return e;
}

// ---------------------------------------------------------------------------
// Tables (host).
// ---------------------------------------------------------------------------
namespace {
// halves of v = round(a), |a| < 2^60: v = h 2^30 + l, -2^29 <= l < 2^29
void store30(double a, int* out) {
  const long long v = std::llrint(a);
  long long l = v & ((1ll << 30) - 1);
  if (l >= (1ll << 29)) l -= 1ll << 30;
  out[0] = (int)((v - l) >> 30);
  out[1] = (int)l;
}
int bound_exp(double l1) {   // smallest e with l1 (1 + 2^-20) <= 2^e
  if (!(l1 > 0)) return 0;
  int e;
  std::frexp(l1 * (1.0 + 1.0 / (1 << 20)), &e);
  return e;
}
}  // namespace

void zfx_build(const Grid& g, const double* zinv, const double* zfwd, std::vector<int>& A, std::vector<int>& Ae,
               std::vector<int>& G, std::vector<int>& W, std::vector<int>& We) {
  const int Kp = pad_group(g.nq), LN = 2 * Kp, Mh = (g.Mz + 1) / 2, Kh = pad_group(Mh);
  G.assign((size_t)4 * g.Nz, 0);
  for (int n = 2; n < g.Nz; ++n)
    for (int q = 0; q < 4; ++q) G[(size_t)4 * n + q] = (int)std::lround(1.5 * q * std::log2((double)n));
  A.assign((size_t)Mh * LN * 4 * 2, 0);
  Ae.assign((size_t)4 * Mh, 0);
  std::vector<double> sc(g.Nz);   // 2^-G_q(n); products with powers of two are exact
  for (int q = 0; q < 4; ++q) {
    for (int n = 0; n < g.Nz; ++n) sc[n] = std::ldexp(1.0, -G[(size_t)4 * n + q]);
    for (int j = 0; j < Mh; ++j) {
      const double* row = zinv + ((size_t)q * g.Mz + j) * g.Nz;
      double l1 = 0.0;
      for (int n = 0; n < g.Nz; ++n) l1 += std::fabs(row[n] * sc[n]);
      const int e = bound_exp(l1);
      const double up = std::ldexp(1.0, 60 - e);
      Ae[(size_t)q * Mh + j] = e;
      for (int n = 0; n < g.Nz; ++n)
        store30((row[n] * sc[n]) * up, &A[(((size_t)j * LN + (n & 1) * Kp + n / 2) * 4 + q) * 2]);
    }
  }
  W.assign((size_t)g.Nz * Kh * 2, 0);
  We.assign(g.Nz, 0);
  for (int n = 0; n < g.Nz; ++n) {
    double l1 = 0.0;
    for (int j = 0; j < Mh; ++j) l1 += std::fabs(zfwd[(size_t)n * g.Mz + j]);
    const int e = bound_exp(l1);
    We[n] = e;
    const double up = std::ldexp(1.0, 60 - e);
    for (int j = 0; j < Mh; ++j) store30(zfwd[(size_t)n * g.Mz + j] * up, &W[((size_t)n * Kh + j) * 2]);
  }
}

}  // namespace rbc
