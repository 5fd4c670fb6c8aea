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
// 301 -> 135 us, one state 40 -> 21 us; 512 x 128, 3 states 215 -> 136 us;
// 128 x 32, one state 13.3 -> 11.4 us.  Forward: 100 -> 40 us, 12.4 -> 10.7 us,
// 83 -> 36 us, 9.3 -> 8.4 us.  Against 64-bit plain torch the temperature after
// a few steps is 2 to 3 times closer than with FP64 sums, psi equally close
// (its solve dominates).
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
// 2^e v for a column exponent that may mark a non-finite column
__device__ __forceinline__ double scaled(i64 v, int ecol, int e) {
  return ecol >= kNaN ? __hiloint2double(0x7ff80000, 0) : (double)v * fx::pow2(ecol - 1022 + e);
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
// Block: 16 modes (32 real columns, one per lane), eight warps; warp = (row
// pair, share of the groups of eight coefficients): KS warps share a row pair
// where a launch would otherwise leave SMs idle.  The block converts the
// columns (six scaled versions) into shared memory once, or in chunks of 64
// coefficients, and every row pair reads them there.
// ---------------------------------------------------------------------------
template <int KS>
__global__ void __launch_bounds__(32 * kWarps) k_zinv_fx(Grid g, const int2* __restrict__ A, const int* __restrict__ Ea,
                                                         const int4* __restrict__ gexp, const double* __restrict__ X,
                                                         size_t S, double* __restrict__ Z, int B, int jblocks,
                                                         int chunk, const int* nsteps, const int* step, int diag) {
  extern __shared__ __align__(16) unsigned char zsm[];
  __shared__ int ecol[6][kCols];
  pdl_wait();
  const int Kp = pad_group(g.nq), LN = 2 * Kp, Mh = (g.Mz + 1) / 2;
  const int ctiles = (g.nm + 15) / 16;
  const int b = blockIdx.x / (ctiles * jblocks), rem = blockIdx.x - b * ctiles * jblocks;
  const int ct = rem / jblocks, jb = rem - ct * jblocks;
  if (b >= B || !(nsteps == nullptr || *step < nsteps[b])) return;   // uniform per block
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int m = ct * 16 + (lane >> 1), c = lane & 1;
  const bool valid = m < g.nm;
  const double* xt = X + (size_t)b * S + (size_t)2 * (valid ? m : 0) + c;   // T; psi follows Nz * nm modes later
  const double* xp = xt + (size_t)g.Nz * g.nm * 2;
  const size_t xs = (size_t)g.nm * 2;                                       // coefficient stride
  int2* XS = reinterpret_cast<int2*>(zsm);                                  // [chunk][6][32]
  i64* part = reinterpret_cast<i64*>(zsm + (size_t)chunk * 6 * kCols * sizeof(int2));   // [8][6][32], KS > 1
  for (int i = threadIdx.x; i < 6 * kCols; i += blockDim.x) (&ecol[0][0])[i] = 0;
  __syncthreads();
  {
    int em[6] = {0, 0, 0, 0, 0, 0};
    for (int n = warp; n < g.Nz; n += kWarps) {
      const int4 gq = __ldg(gexp + n);
      const int ep = fx::biased_exp(valid ? __ldg(xp + n * xs) : 0.0), et = fx::biased_exp(valid ? __ldg(xt + n * xs) : 0.0);
      if (ep > 0) {
        const int q = ep == 0x7ff ? kNaN : ep;
        em[0] = max(em[0], q + gq.x);
        em[1] = max(em[1], q + gq.y);
        em[2] = max(em[2], q + gq.z);
        em[3] = max(em[3], q + gq.w);
      }
      if (et > 0) {
        const int q = et == 0x7ff ? kNaN : et;
        em[4] = max(em[4], q + gq.x);
        em[5] = max(em[5], q + gq.y);
      }
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) atomicMax(&ecol[q][lane], em[q]);
  }
  __syncthreads();
  int ec[6];
#pragma unroll
  for (int q = 0; q < 6; ++q) ec[q] = ecol[q][lane];
  auto stage = [&](int i0, int i1) {   // list entries [i0, i1): parity i / Kp, coefficient 2 (i % Kp) + parity
    for (int i = i0 + warp; i < i1; i += kWarps) {
      const int p = i / Kp, n = 2 * (i - p * Kp) + p;
      int2* dst = XS + (size_t)(i - i0) * 6 * kCols + lane;
      const bool in = valid && n < g.Nz;
      const double vp = in ? __ldg(xp + n * xs) : 0.0, vt = in ? __ldg(xt + n * xs) : 0.0;
      const int4 gq = __ldg(gexp + (n < g.Nz ? n : 0));
      const int gs[4] = {gq.x, gq.y, gq.z, gq.w};
#pragma unroll
      for (int q = 0; q < 6; ++q)
        dst[q * kCols] = halves30(fx::from_double<60>(q < 4 ? vp : vt, ec[q] - gs[q < 4 ? q : q - 4]));
    }
  };
  // one group of eight terms of row pair jp into the six sums
  auto group = [&](int jp, int i, int i0, i64* hi) {
    const int4* a = reinterpret_cast<const int4*>(A + ((size_t)jp * LN + i) * 4);
    const int2* x = XS + (size_t)(i - i0) * 6 * kCols + lane;
    i64 mid[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) mid[q] = kHalf;
#pragma unroll 4
    for (int e = 0; e < kGroup; ++e) {
      const int4 a01 = __ldg(a + 2 * e), a23 = __ldg(a + 2 * e + 1);
      const int2 a0 = make_int2(a01.x, a01.y), a1 = make_int2(a01.z, a01.w);
      const int2 a2 = make_int2(a23.x, a23.y), a3 = make_int2(a23.z, a23.w);
      mac30(a0, x[(e * 6 + 0) * kCols], hi[0], mid[0]);
      mac30(a1, x[(e * 6 + 1) * kCols], hi[1], mid[1]);
      mac30(a2, x[(e * 6 + 2) * kCols], hi[2], mid[2]);
      mac30(a3, x[(e * 6 + 3) * kCols], hi[3], mid[3]);
      mac30(a0, x[(e * 6 + 4) * kCols], hi[4], mid[4]);
      mac30(a1, x[(e * 6 + 5) * kCols], hi[5], mid[5]);
    }
#pragma unroll
    for (int q = 0; q < 6; ++q) hi[q] += mid[q] >> 30;
  };
  const double k = g.kfac * m;
  const size_t fs = (size_t)g.Mz * g.nm * 2;
  double* Zb = Z + (size_t)b * 6 * fs + (size_t)2 * (valid ? m : 0) + c;
  // fields of padded row j from the sums of its row pair jp (sg = -1: the mirrored row)
  auto emit = [&](int jp, int j, int sg, const i64* E, const i64* O) {
    double P[6];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
      const int o = q < 4 ? q : q - 4;   // operator
      const i64 v = sg > 0 ? E[q] + O[q] : (o & 1) ? O[q] - E[q] : E[q] - O[q];
      P[q] = scaled(v, ec[q], __ldg(Ea + o * Mh + jp) - 60);
    }
    // i z of a complex value: the partner lane's part, negated in the real lane
    auto timesi = [&](double v) {
      const double o = __shfl_xor_sync(0xffffffffu, v, 1);
      return c == 0 ? -o : o;
    };
    const double ip = timesi(P[0]);
    const double om = fma(k * k, P[0], -4.0 * P[2]);            // omega = k^2 psi - 4 d2(psi)
    const double io = timesi(om), it = timesi(P[4]);
    if (!valid) return;
    double* z = Zb + (size_t)j * g.nm * 2;
    const bool m0 = m == 0;
    z[0] = m0 ? (c == 0 ? P[0] : 0.0) : 2.0 * P[1];             // u = d_z psi (m = 0: U)
    z[fs] = m0 ? 0.0 : -k * ip;                                 // w = -ik psi
    z[2 * fs] = m0 ? 0.0 : k * io;                              // d_x omega
    z[3 * fs] = m0 ? (c == 0 ? -4.0 * P[2] : 0.0) : fma((2.0 * k) * k, P[1], -8.0 * P[3]);   // d_z omega
    z[4 * fs] = diag ? P[4] : m0 ? 0.0 : k * it;                // d_x T (the averages of Sec. 2.2: T)
    z[5 * fs] = 2.0 * P[5];                                     // d_z T
  };
  constexpr int JB = kWarps / KS;                               // row pairs per round
  const int js = KS == 1 ? warp : warp / KS, ks = KS == 1 ? 0 : warp % KS;
  const int rounds = (Mh + jblocks * JB - 1) / (jblocks * JB);
  if (chunk >= LN) {
    stage(0, LN);
    __syncthreads();
  }
  for (int r = 0; r < rounds; ++r) {
    const int jp = (r * jblocks + jb) * JB + js;
    const bool on = jp < Mh;
    i64 E[6] = {0, 0, 0, 0, 0, 0}, O[6] = {0, 0, 0, 0, 0, 0};
    if (KS == 1) {
#pragma unroll 1
      for (int p = 0; p < 2; ++p) {
        i64 acc[6] = {0, 0, 0, 0, 0, 0};
        for (int i0 = 0; i0 < Kp; i0 += chunk) {
          const int i1 = min(Kp, i0 + chunk);
          if (chunk < LN) {
            __syncthreads();
            stage(p * Kp + i0, p * Kp + i1);
            __syncthreads();
          }
          if (on)
            for (int i = i0; i < i1; i += kGroup) group(jp, p * Kp + i, chunk < LN ? p * Kp + i0 : 0, acc);
        }
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          E[q] = p ? E[q] : acc[q];
          O[q] = acc[q];
        }
      }
      if (on) {
        emit(jp, jp, 1, E, O);
        if (g.Mz - 1 - jp != jp) emit(jp, g.Mz - 1 - jp, -1, E, O);
      }
    } else {
      // warps ks = 0, 2, .. share the even coefficients, 1, 3, .. the odd ones
      const int p = ks & 1;
      if (on)
        for (int i = (ks >> 1) * kGroup; i < Kp; i += (KS / 2) * kGroup) group(jp, p * Kp + i, 0, E);
#pragma unroll
      for (int q = 0; q < 6; ++q) part[(warp * 6 + q) * kCols + lane] = E[q];
      __syncthreads();
      if (on && ks < 2) {
#pragma unroll
        for (int q = 0; q < 6; ++q) {
          i64 e = 0, o = 0;
#pragma unroll
          for (int s = 0; s < KS; s += 2) {
            e += part[((js * KS + s) * 6 + q) * kCols + lane];
            o += part[((js * KS + s + 1) * 6 + q) * kCols + lane];
          }
          E[q] = e;
          O[q] = o;
        }
        if (ks == 0)
          emit(jp, jp, 1, E, O);
        else if (g.Mz - 1 - jp != jp)
          emit(jp, g.Mz - 1 - jp, -1, E, O);
      }
      __syncthreads();
    }
  }
}

// Warps per row pair and blocks per column tile.  Enough warps to fill the SMs
// (152 x 16) come from the row pairs of larger batches: one warp per row pair
// then, and as few blocks per column tile as still make two per SM (each block
// converts the columns again).  Below that a row pair's groups are shared by up
// to eight warps.  Grids with more than 64 padded coefficients stage them in
// chunks of 64 (98 KB of shared memory), except where warps share them.
namespace {
struct ZinvShape {
  int ks, jblocks, chunk;
  size_t smem;
};
ZinvShape zinv_shape(const Grid& g, int B) {
  const int Kp = pad_group(g.nq), LN = 2 * Kp, Mh = (g.Mz + 1) / 2, ctiles = (g.nm + 15) / 16;
  const long tasks = (long)B * ctiles * Mh;
  int ks = 1;
  if (LN <= 128)
    while (ks < 8 && ks < 2 * (Kp / kGroup) && tasks * ks < 152L * 16) ks *= 2;
  const int jb = kWarps / ks, most = (Mh + jb - 1) / jb;
  const int jblocks = (int)std::min<long>(most, std::max<long>(1, (304 + (long)B * ctiles - 1) / ((long)B * ctiles)));
  const int chunk = ks > 1 ? LN : std::min(LN, 64);
  const size_t smem = (size_t)chunk * 6 * kCols * sizeof(int2) + (ks > 1 ? (size_t)kWarps * 6 * kCols * sizeof(i64) : 0);
  return {ks, jblocks, chunk, smem};
}
constexpr int kZinvSmem = 128 * 6 * kCols * (int)sizeof(int2) + kWarps * 6 * kCols * (int)sizeof(i64);

template <int KS>
cudaError_t launch_zinv_ks(const Grid& g, const Tables& t, const Work& w, const double* X, double* Z, int B,
                           const ZinvShape& sh, const int* ns, bool diag, cudaStream_t s) {
  const int ctiles = (g.nm + 15) / 16;
  return launch_pdl(w.pdl != 0 && !diag, k_zinv_fx<KS>, (unsigned)(B * ctiles * sh.jblocks), 32 * kWarps, sh.smem, s, g,
                    t.zfxA, t.zfxAe, t.zfxG, X, state_doubles(g), Z, B, sh.jblocks, sh.chunk, ns, w.step, diag ? 1 : 0);
}
}  // namespace

cudaError_t launch_zinv_fx(const Grid& g, const Tables& t, const Work& w, const double* X, int B, const int* ns,
                           bool diag, cudaStream_t s) {
  const ZinvShape sh = zinv_shape(g, B);
  switch (sh.ks) {
    case 1: return launch_zinv_ks<1>(g, t, w, X, w.Z, B, sh, ns, diag, s);
    case 2: return launch_zinv_ks<2>(g, t, w, X, w.Z, B, sh, ns, diag, s);
    case 4: return launch_zinv_ks<4>(g, t, w, X, w.Z, B, sh, ns, diag, s);
    default: return launch_zinv_ks<8>(g, t, w, X, w.Z, B, sh, ns, diag, s);
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
  pdl_wait();
  const int Mh = (g.Mz + 1) / 2, Kh = pad_group(Mh), ctiles = (g.nm + 15) / 16;
  int rem = blockIdx.x;
  const int nb = rem % nblocks;
  rem /= nblocks;
  const int ct = rem % ctiles;
  rem /= ctiles;
  const int p = rem & 1, f = (rem >> 1) & 1, b = rem >> 2;
  if (b >= B || !(nsteps == nullptr || *step < nsteps[b])) return;   // uniform per block
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
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
  for (int r0 = (nb * kWarps + warp) * NI; r0 < g.nq; r0 += nblocks * kWarps * NI) {
    i64 hi[NI];
#pragma unroll
    for (int i = 0; i < NI; ++i) hi[i] = 0;
    for (int j0 = 0; j0 < Kh; j0 += kGroup) {
      i64 mid[NI];
#pragma unroll
      for (int i = 0; i < NI; ++i) mid[i] = kHalf;
#pragma unroll
      for (int e = 0; e < kGroup; e += 2) {
        const int2 x0 = FS[(j0 + e) * kCols + lane], x1 = FS[(j0 + e + 1) * kCols + lane];
#pragma unroll
        for (int i = 0; i < NI; ++i) {
          const int r = min(r0 + i, g.nq - 1);
          const int4 a = __ldg(reinterpret_cast<const int4*>(Wt + (size_t)(2 * r + p) * Kh + j0 + e));
          mac30(make_int2(a.x, a.y), x0, hi[i], mid[i]);
          mac30(make_int2(a.z, a.w), x1, hi[i], mid[i]);
        }
      }
#pragma unroll
      for (int i = 0; i < NI; ++i) hi[i] += mid[i] >> 30;
    }
#pragma unroll
    for (int i = 0; i < NI; ++i)
      if (valid && r0 + i < g.nq) {
        const int n = 2 * (r0 + i) + p;
        Fb[n * rs] = scaled(hi[i], em, __ldg(We + n) - 59);
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
  const int nblocks = (int)std::min<long>(most, std::max<long>(1, (456 + base - 1) / base));
  return launch_pdl(w.pdl != 0, k_zfwd_fx<NI>, (unsigned)(base * nblocks), 32 * kWarps, zfwd_fx_smem(g), s, g, t.zfxW,
                    t.zfxWe, w.Q, w.F, state_doubles(g), B, nblocks, w.nsteps, w.step);
}
}  // namespace

// Coefficients per warp: four share each fold read from shared memory; fewer
// where four would leave SMs without a block.
cudaError_t launch_zfwd_fx(const Grid& g, const Tables& t, const Work& w, int B, cudaStream_t s) {
  const long warps = 4L * B * ((g.nm + 15) / 16) * g.nq;   // one coefficient each
  if (warps >= 4L * 152 * 16) return launch_zfwd_ni<4>(g, t, w, B, s);
  if (warps >= 2L * 152 * 16) return launch_zfwd_ni<2>(g, t, w, B, s);
  return launch_zfwd_ni<1>(g, t, w, B, s);
}

cudaError_t configure_zfx(const Grid& g) {
  static int a_fwd = 48 * 1024;
  cudaError_t e = cudaSuccess;
  auto allow = [&](auto* fn, int need) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, need);
  };
  allow(k_zinv_fx<1>, kZinvSmem);
  allow(k_zinv_fx<2>, kZinvSmem);
  allow(k_zinv_fx<4>, kZinvSmem);
  allow(k_zinv_fx<8>, kZinvSmem);
  if ((int)zfwd_fx_smem(g) > a_fwd) {   // only grows: earlier handles keep theirs
    a_fwd = (int)zfwd_fx_smem(g);
  }
  allow(k_zfwd_fx<1>, a_fwd);
  allow(k_zfwd_fx<2>, a_fwd);
  allow(k_zfwd_fx<4>, a_fwd);
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
