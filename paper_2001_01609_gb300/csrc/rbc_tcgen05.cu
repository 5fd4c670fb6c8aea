// Tensor-core (tcgen05) z inverse transform for the mixed-precision path.
//
// The z inverse transform of one slice and one field is a dense contraction:
// C[(j, op)][col] = sum_n A[(j, op)][n] X[n][col], with A the values of
// d^q T_n / ds^q at the padded Lobatto points (rows interleaved as j * nops + op,
// nops = 4 for psi: V, VD, VD^2, VD^3; nops = 2 for T: V, VD) and X the state's
// Chebyshev coefficients (columns = Fourier mode x real/imaginary part).  It runs
// on the 5th-generation tensor cores with TF32 operands and split compensation:
// a = a_hi + a_lo, x = x_hi + x_lo (each a TF32 value), and
// A X ~ A_hi X_hi + A_hi X_lo + A_lo X_hi, accumulated in FP32 in tensor memory,
// which keeps about FP32 accuracy (the mixed mode computes the transforms and
// products in FP32).
//
// CTA per (slice, tile of 64 columns, row tiles of one field's operators): the X
// tile (all K) becomes hi/lo operands in shared memory, the operator images'
// K-chunks (pre-swizzled on the host, 16 KB each, hi and lo) stream in by bulk
// (TMA) copies, and the fields of the z-inverse output are formed from the
// 128 x 64 FP32 accumulators with the ik factors (the epilogue of k_zinv).
// Operands are K-major with the 128-byte swizzle; every mbarrier wait is bounded
// and reports through the slice's error flag, and nothing (MMA or copy) is in
// flight when a kernel frees its tensor memory.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdint>
#include <cstring>

#include "rbc_internal.h"

namespace rbc {

namespace {

constexpr int kTileN = 64;       // columns per CTA (32 Fourier modes x re/im)
constexpr int kTileM = 128;      // rows per MMA tile
constexpr int kChunkFloats = kTileM * 32;   // one 128-row image chunk of 128-byte rows: 16 KB
// threads of a tensor-core CTA: kTcGroups groups of four warps; in the
// epilogue warp w reads the accumulator's lane quarter w % 4 (the quarter a
// warp may access) and the column range w / 4 of kTileN / kTcGroups columns,
// so that kTcGroups times as many stores are in flight as with four warps
constexpr int kTcGroups = 2;
constexpr int kTcThreads = 128 * kTcGroups;
constexpr int kWsThreads = kTcThreads + 64;   // and the copying and the issuing warp
// columns and row stride (floats) of the staged accumulator in k_zinv_tc's
// epilogue (16-byte rows whose 128-bit accesses meet no bank twice)
constexpr int kEpiCols = 32, kEpiStride = kEpiCols + 4;
constexpr int kEpiBytes = kTileM * kEpiStride * 4;
constexpr long long kWaitLimit = 1LL << 24;   // default spin limit of a bounded wait

__device__ __forceinline__ uint32_t saddr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// K-elements per 128-byte swizzle row: 32 TF32 or 64 BF16 values
__host__ __device__ inline int tc_ke(const Grid& g) { return g.tcbf16 ? 64 : 32; }

// byte offset of the element at byte `kb` (< 128) of row r in a K-major, 128B-swizzled tile
__host__ __device__ inline uint32_t swz_b(int r, int kb) {
  return (uint32_t)(r * 128 + (((kb >> 4) ^ (r & 7)) << 4) + (kb & 15));
}

// shared-memory matrix descriptor: K-major, 128B swizzle, 8-row groups 1024 B apart
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  const uint64_t lbo = 16, sbo = 1024;
  return (uint64_t)((addr & 0x3FFFF) >> 4) | ((lbo >> 4) << 16) | ((sbo >> 4) << 32) | (1ull << 46) |
         (2ull << 61);
}

// instruction descriptor: kind::tf32, FP32 accumulator, K-major A and B, M x N
__device__ __forceinline__ uint32_t instr_desc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// instruction descriptor: kind::f16 with BF16 A and B, FP32 accumulator, K-major, M x N
__device__ __forceinline__ uint32_t instr_desc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ uint32_t to_tf32(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ void mma_tf32(uint32_t tmem, uint64_t ad, uint64_t bd, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(ad), "l"(bd), "r"(idesc), "r"(acc));
}

__device__ __forceinline__ void commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(saddr(mbar)));
}

// arrive on an mbarrier, announcing `bytes` of bulk-copy transactions for the phase
__device__ __forceinline__ void arrive_expect_tx(uint64_t* mbar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(saddr(mbar)), "r"(bytes) : "memory");
}

// bulk (TMA) copy of `bytes` contiguous bytes, global -> shared, completing on mbar
// (both addresses 16-byte aligned, bytes a multiple of 16)
__device__ __forceinline__ void bulk_g2s(void* dst, const void* src, uint32_t bytes, uint64_t* mbar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(saddr(dst)),
      "l"(src), "r"(bytes), "r"(saddr(mbar))
      : "memory");
}

// bounded wait for the completion of phase `parity` of an mbarrier: at most
// `limit` polls (limit 0: gives up at once)
__device__ __forceinline__ bool wait_parity(uint64_t* mbar, uint32_t parity, long long limit) {
  uint32_t done = 0;
  for (long long it = 0; it < limit; ++it) {
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(saddr(mbar)), "r"(parity));
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void tmem_ld16(uint32_t ta, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(ta));
  asm volatile("tcgen05.wait::ld.sync.aligned;");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ size_t soff2(const Grid& g, int f, int n, int m) {
  return ((size_t)(f * g.Nz + n) * g.nm + m) * 2;
}

__device__ __forceinline__ void store_c(float* Zb, const Grid& g, int field, int j, int m, float re, float im) {
  const size_t fs = (size_t)g.Mz * g.nm * 2;
  *reinterpret_cast<float2*>(Zb + field * fs + ((size_t)j * g.nm + m) * 2) = make_float2(re, im);
}

// Spin limit of the waits that wait for MMAs to complete before the kernel goes
// on (set by tc_set_wait_limit; tests lower it to make the waits give up).
__device__ long long g_wait_limit = kWaitLimit;

// 4 K-steps x 3 MMAs (hi*hi, hi*lo, lo*hi) of one chunk: descriptors of the hi
// operands; the lo ones lie a fixed distance behind (addresses / 16 below 2^14,
// so sums stay in the descriptors' address field)
template <bool BF>
__device__ __forceinline__ void mma_chunk(uint32_t tmem, uint64_t a, uint64_t x, uint64_t xlo, uint32_t idesc, bool more) {
  constexpr uint64_t alo = kTileM * 128 >> 4;
#pragma unroll
  for (int ks = 0; ks < 4; ++ks) {            // four 32-byte K-steps per 128-byte row
    const uint64_t o = 2 * ks;
    const uint32_t acc0 = (more || ks > 0) ? 1u : 0u;
    if (BF) {
      mma_bf16(tmem, a + o, x + o, idesc, acc0);
      mma_bf16(tmem, a + o, x + xlo + o, idesc, 1u);
      mma_bf16(tmem, a + alo + o, x + o, idesc, 1u);
    } else {
      mma_tf32(tmem, a + o, x + o, idesc, acc0);
      mma_tf32(tmem, a + o, x + xlo + o, idesc, 1u);
      mma_tf32(tmem, a + alo + o, x + o, idesc, 1u);
    }
  }
}

// barriers of the eight converting warps
__device__ __forceinline__ void group_sync() { asm volatile("bar.sync 1, %0;" ::"n"(kTcThreads) : "memory"); }
__device__ __forceinline__ bool group_and(bool v) {
  uint32_t r;
  asm volatile(
      "{\n .reg .pred p, q;\n setp.ne.u32 p, %1, 0;\n barrier.cta.red.and.pred q, 1, %2, p;\n selp.u32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(kTcThreads)
      : "memory");
  return r != 0;
}

// FP32 -> FP64 on the integer pipe (a conversion instruction holds its
// sub-partition's FP64 pipe for 64 clocks); denormals, infinities and NaN take the
// instruction.
__device__ __forceinline__ double widen(float v) {
  const uint32_t u = __float_as_uint(v), a = u & 0x7fffffffu;
  if (a - 0x00800000u < 0x7f000000u) return __hiloint2double((int)((u & 0x80000000u) | ((a >> 3) + 0x38000000u)), (int)(u << 29));
  if (a == 0) return __hiloint2double((int)u, 0);
  return (double)v;
}

// Values val(raw(k)), k < kc K-chunks, of column tid % 64 of the tile as hi/lo
// operands, K-major (row = column of the tile): 16 bytes of consecutive k per
// item.  raw() loads without a branch, and the loads of several items are in flight
// together (item by item, a tile of 1024 x 256 took three times as long to convert
// as to multiply).
template <bool BF, int ITEMS, typename Raw, typename Load, typename Val>
__device__ __forceinline__ void convert_tile(Load&& raw, Val&& val, int kc, int tid, unsigned char* hi, unsigned char* lo) {
  constexpr int PER = BF ? 8 : 4, KE = BF ? 64 : 32;   // operands per 16 bytes, per 128-byte row
  constexpr int U = BF ? ITEMS / 2 : ITEMS, STEP = kTcThreads / kTileN;
  const int col = tid & (kTileN - 1);
  for (int kb = tid / kTileN; kb < kc * 8; kb += U * STEP) {
    Raw in[U][PER];
#pragma unroll
    for (int u = 0; u < U; ++u)
#pragma unroll
      for (int e = 0; e < PER; ++e) in[u][e] = raw((kb + u * STEP) * PER + e);
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int k0 = (kb + u * STEP) * PER;
      if (k0 >= kc * KE) break;
      float v[PER];
#pragma unroll
      for (int e = 0; e < PER; ++e) v[e] = val(in[u][e], k0 + e);
      const uint32_t o = (uint32_t)(k0 / KE) * kTileN * 128 + swz_b(col, (k0 % KE) * (16 / PER));
      uint32_t h[4], l[4];
      if (BF) {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const __nv_bfloat16 h0 = __float2bfloat16_rn(v[2 * e]), h1 = __float2bfloat16_rn(v[2 * e + 1]);
          const __nv_bfloat16 l0 = __float2bfloat16_rn(v[2 * e] - __bfloat162float(h0));
          const __nv_bfloat16 l1 = __float2bfloat16_rn(v[2 * e + 1] - __bfloat162float(h1));
          h[e] = (uint32_t)__bfloat16_as_ushort(h0) | ((uint32_t)__bfloat16_as_ushort(h1) << 16);
          l[e] = (uint32_t)__bfloat16_as_ushort(l0) | ((uint32_t)__bfloat16_as_ushort(l1) << 16);
        }
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          h[e] = to_tf32(v[e]);
          l[e] = to_tf32(v[e] - __uint_as_float(h[e]));
        }
      }
      *reinterpret_cast<uint4*>(hi + o) = make_uint4(h[0], h[1], h[2], h[3]);
      *reinterpret_cast<uint4*>(lo + o) = make_uint4(l[0], l[1], l[2], l[3]);
    }
  }
}

// K-chunk c of the images (hi, lo) into stage buf
__device__ __forceinline__ void fetch_chunk(unsigned char* sA, const float* Ahi, const float* Alo, int c, int buf,
                                            uint64_t* full) {
  constexpr uint32_t bytes = kChunkFloats * 4;   // 16 KB
  unsigned char* ah = sA + (size_t)buf * 2 * bytes;
  arrive_expect_tx(full, 2 * bytes);
  bulk_g2s(ah, Ahi + (size_t)c * kChunkFloats, bytes, full);
  bulk_g2s(ah + bytes, Alo + (size_t)c * kChunkFloats, bytes, full);
}

// The loader: chunks NB .. n - 1, each once its stage is free; false if a wait gave
// up.  A stage has one copy or one chunk's MMAs in flight at a time, so the
// parities below name the only phase that can be pending.  Returns with no copy
// in flight.
__device__ __forceinline__ bool stream_chunks(unsigned char* sA, const float* Ahi, const float* Alo, int n, int NB,
                                              uint64_t* full, uint64_t* empty, long long limit) {
  bool ok = true;
  int c = min(NB, n), buf = 0;
  uint32_t par = 0;                           // of the stages' next phase
  for (; c < n; ++c) {
    ok = wait_parity(&empty[buf], par, limit);   // chunk c - NB has been used
    if (!ok) break;
    fetch_chunk(sA, Ahi, Alo, c, buf, &full[buf]);
    if (++buf == NB) {
      buf = 0;
      par ^= 1;
    }
  }
  for (int i = max(0, c - NB); i < c; ++i) wait_parity(&full[i % NB], (i / NB) & 1, kWaitLimit);
  return ok;
}

// The issuer's place in the ring, chunks issued so far.
struct Ring {
  int buf;
  uint32_t par;
  int used;
};

// The MMAs of one row tile (kc chunks) as they land; false if a wait gave up.
__device__ __forceinline__ bool issue_tile(bool bf, uint32_t tmem, unsigned char* sA, unsigned char* sXhi, int kc, int NB,
                                           Ring& ring, uint64_t* full, uint64_t* empty, uint32_t idesc, long long limit) {
  const uint64_t da = smem_desc(saddr(sA)), dx = smem_desc(saddr(sXhi)), xlo = (uint64_t)(kc * kTileN * 128) >> 4;
  for (int c = 0; c < kc; ++c) {
    if (!wait_parity(&full[ring.buf], ring.par, limit)) return false;
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint64_t a = da + (uint64_t)ring.buf * (2 * kTileM * 128 >> 4), x = dx + (uint64_t)c * (kTileN * 128 >> 4);
    if (bf)
      mma_chunk<true>(tmem, a, x, xlo, idesc, c > 0);
    else
      mma_chunk<false>(tmem, a, x, xlo, idesc, c > 0);
    commit(&empty[ring.buf]);
    ++ring.used;
    if (++ring.buf == NB) {
      ring.buf = 0;
      ring.par ^= 1;
    }
  }
  return true;
}
// waits for the MMAs of the last chunks issued
__device__ __forceinline__ void drain_ring(int used, int NB, uint64_t* empty) {
  for (int i = max(0, used - NB); i < used; ++i) wait_parity(&empty[i % NB], (i / NB) & 1, kWaitLimit);
}

// kEpiCols columns of the accumulator, from column cb on, to shared memory
__device__ __forceinline__ void stage_rows(uint32_t tmem, float* epi, int cb, int warp, int lane) {
  const int r = (warp & 3) * 32 + lane;       // tile row = TMEM lane
  const int cw = (warp >> 2) * (kEpiCols / kTcGroups);   // this warp's 16 of them
  float v[16];
  tmem_ld16(tmem + ((uint32_t)((warp & 3) * 32) << 16) + cb + cw, v);
  float4* dst = reinterpret_cast<float4*>(epi + r * kEpiStride + cw);
#pragma unroll
  for (int i = 0; i < 4; ++i) dst[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
}

// Fields of row tile t, columns c0 .. c0 + 63, from the accumulator at tmem,
// kEpiCols columns at a time: its rows go to shared memory, and each half-warp
// forms the fields of one j at 16 modes, so that every store is one 128-byte
// segment.  All eight warps.
__device__ __forceinline__ void zinv_fields(const Grid& g, uint32_t tmem, float* epi, const float* kf, float* Zb,
                                            int nops, int t, int c0, int warp, int lane) {
  const int lj = nops == 4 ? 2 : 1, jper = kTileM >> lj;
  for (int cb = 0; cb < kTileN; cb += kEpiCols) {
    stage_rows(tmem, epi, cb, warp, lane);
    group_sync();
    const int ml = lane & 15, m = ((c0 + cb) >> 1) + ml;
    if (m < g.nm) {
      const float k = kf[cb / 2 + ml];
      for (int jl = warp * 2 + (lane >> 4); jl < jper; jl += 2 * (kTcThreads / 32)) {
        const int j = t * jper + jl;
        if (j >= g.Mz) break;
        const float* e = epi + (jl << lj) * kEpiStride + 2 * ml;
        const float2 P0 = *reinterpret_cast<const float2*>(e), P1 = *reinterpret_cast<const float2*>(e + kEpiStride);
        if (nops == 4) {
          // P[q] = (re, im) of d^q psi/ds^q (m = 0: of U)
          const float2 P2 = *reinterpret_cast<const float2*>(e + 2 * kEpiStride);
          const float2 P3 = *reinterpret_cast<const float2*>(e + 3 * kEpiStride);
          if (m == 0) {
            store_c(Zb, g, 0, j, 0, P0.x, 0.f);            // u = U
            store_c(Zb, g, 1, j, 0, 0.f, 0.f);             // w
            store_c(Zb, g, 2, j, 0, 0.f, 0.f);             // d_x omega
            store_c(Zb, g, 3, j, 0, -4.f * P2.x, 0.f);     // d_z omega = -U_zz
            store_c(Zb, g, 4, j, 0, 0.f, 0.f);             // d_x u
            store_c(Zb, g, 5, j, 0, 2.f * P1.x, 0.f);      // d_z u = U_z
          } else {
            const float omr = k * k * P0.x - 4.f * P2.x, omi = k * k * P0.y - 4.f * P2.y;
            store_c(Zb, g, 0, j, m, 2.f * P1.x, 2.f * P1.y);   // u = d_z psi
            store_c(Zb, g, 1, j, m, k * P0.y, -k * P0.x);      // w = -ik psi
            store_c(Zb, g, 2, j, m, -k * omi, k * omr);        // d_x omega = ik omega
            store_c(Zb, g, 3, j, m, 2.f * k * k * P1.x - 8.f * P3.x, 2.f * k * k * P1.y - 8.f * P3.y);
            store_c(Zb, g, 4, j, m, -k * 2.f * P1.y, k * 2.f * P1.x);   // d_x u = ik u
            store_c(Zb, g, 5, j, m, 4.f * P2.x, 4.f * P2.y);            // d_z u
          }
        } else {
          store_c(Zb, g, 6, j, m, P0.x, P0.y);                          // T
          store_c(Zb, g, 7, j, m, m == 0 ? 0.f : -k * P0.y, m == 0 ? 0.f : k * P0.x);   // d_x T
          store_c(Zb, g, 8, j, m, 2.f * P1.x, 2.f * P1.y);              // d_z T
        }
      }
    }
    if (cb + kEpiCols < kTileN) group_sync();   // read before the next columns overwrite it
  }
}

// Error bits of a state and of its handle (kFlagTimeout when a wait gave up).
__device__ __forceinline__ void flag_timeout(int* flags, int* err, int b) {
  atomicOr(flags + b, kFlagTimeout);
  if (err) atomicOr(err, kFlagTimeout);
}

}  // namespace

cudaError_t tc_set_wait_limit(long long limit) {
  const long long v = limit < 0 ? kWaitLimit : limit;
  return cudaMemcpyToSymbol(g_wait_limit, &v, sizeof(v));
}

// Number of 128-row tiles and K-chunks of the operator images (host and device agree).
__host__ __device__ int tc_zinv_mtiles(const Grid& g, int nops) { return (nops * g.Mz + kTileM - 1) / kTileM; }
__host__ __device__ int tc_zinv_kchunks(const Grid& g) { return (g.Nz + tc_ke(g) - 1) / tc_ke(g); }
size_t tc_zinv_image_floats(const Grid& g, int nops) {
  return (size_t)tc_zinv_mtiles(g, nops) * tc_zinv_kchunks(g) * kChunkFloats;
}

// hi/lo split of v into the operand type of the grid, written at byte offset
// `off` of the hi and lo chunks: TF32 (hi = v rounded to 10 mantissa bits, lo
// = the rest, rounded alike) or BF16 (hi = v rounded to nearest even on 7
// mantissa bits, lo = the rest, rounded alike).
static void split_store(const Grid& g, double v, float* hi, float* lo, int off) {
  if (g.tcbf16) {
    auto bf = [](float x) {
      uint32_t u;
      memcpy(&u, &x, 4);
      u += 0x7FFFu + ((u >> 16) & 1u);          // round to nearest, ties to even
      return (uint16_t)(u >> 16);
    };
    auto fl = [](uint16_t b) {
      const uint32_t u = (uint32_t)b << 16;
      float x;
      memcpy(&x, &u, 4);
      return x;
    };
    const uint16_t h = bf((float)v);
    const uint16_t l = bf((float)(v - (double)fl(h)));
    memcpy(reinterpret_cast<unsigned char*>(hi) + off, &h, 2);
    memcpy(reinterpret_cast<unsigned char*>(lo) + off, &l, 2);
    return;
  }
  float f = (float)v;
  uint32_t u;
  memcpy(&u, &f, 4);
  u = (u + 0x1000u) & 0xFFFFE000u;
  float h;
  memcpy(&h, &u, 4);
  float l = (float)(v - (double)h);
  memcpy(&u, &l, 4);
  u = (u + 0x1000u) & 0xFFFFE000u;
  memcpy(&l, &u, 4);
  memcpy(reinterpret_cast<unsigned char*>(hi) + off, &h, 4);
  memcpy(reinterpret_cast<unsigned char*>(lo) + off, &l, 4);
}

// Pre-swizzled hi/lo operator images for field f (nops operators per row j),
// [mtile][kchunk][128 x 32 swizzled].  d[q][j][n] = d^q T_n / ds^q at s_j.
void tc_zinv_build_images(const Grid& g, const double* zinv, int nops, float* hi, float* lo) {
  const int mt = tc_zinv_mtiles(g, nops), kc = tc_zinv_kchunks(g), ke = tc_ke(g), es = 128 / ke;
  for (int t = 0; t < mt; ++t)
    for (int c = 0; c < kc; ++c) {
      float* bh = hi + ((size_t)t * kc + c) * kChunkFloats;
      float* bl = lo + ((size_t)t * kc + c) * kChunkFloats;
      for (int r = 0; r < kTileM; ++r)
        for (int k = 0; k < ke; ++k) {
          const int row = t * kTileM + r, j = row / nops, q = row % nops, n = c * ke + k;
          double v = 0.0;
          if (j < g.Mz && n < g.Nz) v = zinv[((size_t)q * g.Mz + j) * g.Nz + n];
          split_store(g, v, bh, bl, (int)swz_b(r, k * es));
        }
    }
}

// Grid-only choice (so a state gives the same bits in any batch): the tensor
// cores take grids with at least 64 Chebyshev coefficients whose X tile and
// first image stages fit in 200 KB of shared memory.
bool tc_zinv_supported(const Grid& g) {
  const size_t x = (size_t)tc_zinv_kchunks(g) * kTileN * 128 * 2, stage = 2 * kTileM * 128;
  return g.Nz >= 64 && x + stage + 1024 <= 200 * 1024;
}

// Shape of a k_zinv_tc launch: row tiles per CTA, image stages (16 KB hi + 16 KB
// lo per K-chunk) and shared memory: X tile hi/lo (all K), stages, the epilogue's
// rows, alignment slack.  The fewest row tiles that make no more CTAs than SMs
// (1024 x 256, one state: 26 us with two, 35 with one, 72 with all twelve), else
// all of a field's, so that its X tile is converted once (512 x 128, 64 states in
// BF16: 142 us, 207 with one).
struct ZinvTcShape {
  int tiles, stages;
  size_t smem;
};
static ZinvTcShape tc_zinv_shape(const Grid& g, int B) {
  const int kc = tc_zinv_kchunks(g), ntile = (2 * g.nm + kTileN - 1) / kTileN;
  const size_t x = (size_t)kc * kTileN * 128 * 2, stage = 2 * kTileM * 128;
  const int m4 = tc_zinv_mtiles(g, 4), m2 = tc_zinv_mtiles(g, 2);
  int tiles = 1;
  while (tiles < m4 && (long)B * ntile * ((m4 + tiles - 1) / tiles + (m2 + tiles - 1) / tiles) > 152) ++tiles;
  const size_t rest = (tiles == 1 ? 0 : kEpiBytes) + 1024;   // (one tile: the epilogue's rows replace the operands)
  int nb = std::min(4, kc * tiles);
  while (nb > 1 && x + nb * stage + rest > 222 * 1024) --nb;
  return {tiles, nb, x + nb * stage + rest};
}

// Output fields: psi (nops = 4): u, w, d_x omega, d_z omega, d_x u, d_z u (0..5);
// T (nops = 2): T, d_x T, d_z T (6..8).
// CTA per (slice, 64-column tile, field, `tiles` consecutive 128-row tiles of the
// field's operator rows).  Eight warps convert the X tile to hi/lo operands and
// then form the fields, tile after tile.  One lane of a ninth streams the K-chunks
// of the operator images into a ring of NB shared-memory stages with bulk (TMA)
// copies, one of a tenth issues 3 x 4 MMAs per chunk as it lands, one tile ahead:
// the accumulators of two tiles alternate in tensor memory.
// Bound: the images' way from L2 into shared memory (1024 x 256: 256 KB per
// row tile, two stages of 32 KB in flight) and the conversion of X.  Measured
// (GB300, per launch; before, one thread issued, refilled and waited in turn,
// all threads polled, fields were stored in scattered 8-byte pieces and wave
// numbers converted from FP64 at every store; same bits): 1024 x 256, 32 states
// 1067 -> 439 us, one state 195 -> 26 us; 512 x 128, 64 states 472 -> 159 us, in
// BF16 342 -> 142 us; 256 x 64, 8 states 24.7 -> 14 us, one state 19 -> 12 us.
__global__ void __launch_bounds__(kWsThreads) k_zinv_tc(Grid g, const float* __restrict__ Ahi_psi,
                                                 const float* __restrict__ Alo_psi, const float* __restrict__ Ahi_T,
                                                 const float* __restrict__ Alo_T, const double* __restrict__ X,
                                                 size_t S, float* __restrict__ Z, int B, const int* nsteps,
                                                 const int* step, int* flags, int* err, int tiles, int NB) {
  pdl_wait();
  extern __shared__ __align__(1024) unsigned char tc_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)tc_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[4], empty[4], accb[2], accfree[2];
  __shared__ uint32_t tmem_base;
  __shared__ float kf[kTileN / 2];            // wave numbers of the tile's modes
  const int ntile = (2 * g.nm + kTileN - 1) / kTileN;
  const int mt4 = tc_zinv_mtiles(g, 4), mt2 = tc_zinv_mtiles(g, 2);
  const int u4 = (mt4 + tiles - 1) / tiles, units = u4 + (mt2 + tiles - 1) / tiles;   // CTAs per (slice, column tile)
  const int per_b = ntile * units;
  const int b = blockIdx.x / per_b;
  int rem = blockIdx.x - b * per_b;
  const int ct = rem / units;
  const int q = rem - ct * units;
  const int fsel = q < u4 ? 0 : 1;            // 0: psi (nops 4), 1: T (nops 2)
  const int t0 = (fsel == 0 ? q : q - u4) * tiles;
  const int t1 = min(t0 + tiles, fsel == 0 ? mt4 : mt2);
  const int c0 = ct * kTileN;
  if (b >= B || !(nsteps == nullptr || *step < nsteps[b])) return;   // uniform per block
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int nops = fsel == 0 ? 4 : 2;
  const int f = fsel == 0 ? 1 : 0;            // state field: psi slot 1, T slot 0
  const int kc = tc_zinv_kchunks(g);
  const int nchunks = (t1 - t0) * kc;         // the chunks this CTA streams, tile after tile
  const bool bf = g.tcbf16 != 0;
  unsigned char* sXhi = base;
  unsigned char* sXlo = sXhi + (size_t)kc * kTileN * 128;
  unsigned char* sA = sXlo + (size_t)kc * kTileN * 128;   // [stage][hi, lo][128 x 128 B]
  // the epilogue's rows, [128][kEpiStride]: where one tile is all, in the operands' place
  float* epi = reinterpret_cast<float*>(tiles == 1 ? base : sA + (size_t)NB * 2 * kTileM * 128);
  const long long limit = g_wait_limit;
  const bool loader = tid == kTcThreads, issuer = tid == kTcThreads + 32;

  const float* Ahi = (fsel == 0 ? Ahi_psi : Ahi_T) + (size_t)t0 * kc * kChunkFloats;
  const float* Alo = (fsel == 0 ? Alo_psi : Alo_T) + (size_t)t0 * kc * kChunkFloats;
  if (loader) {
    for (int i = 0; i < NB; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&empty[i])));
    }
    for (int i = 0; i < 2; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&accb[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&accfree[i])));
    }
    asm volatile("fence.mbarrier_init.release.cluster;");
    // the first NB chunks of the operator images start streaming in at once
    for (int c = 0; c < NB && c < nchunks; ++c) fetch_chunk(sA, Ahi, Alo, c, c, &full[c]);
  }
  if (warp == kTcThreads / 32) {
    __syncwarp();                             // the warp converged again after the loader's set-up
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 128;" ::"r"(saddr(&tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  } else if (warp < kTcThreads / 32) {
    if (tid < kTileN / 2) kf[tid] = (float)(g.kfac * (c0 / 2 + tid));
    // X tile -> hi/lo operands, K-major (row = column of the tile, k = n)
    const int w = 2 * g.nm, gc = c0 + (tid & (kTileN - 1));
    const double* x = X + (size_t)b * S + soff2(g, f, 0, 0) + min(gc, w - 1);
    auto coef = [&](int n) { return __ldg(x + (size_t)min(n, g.Nz - 1) * w); };
    auto real = [&](double v, int n) { return gc < w && n < g.Nz ? (float)v : 0.f; };
    if (bf)
      convert_tile<true, 8, double>(coef, real, kc, tid, sXhi, sXlo);
    else
      convert_tile<false, 8, double>(coef, real, kc, tid, sXhi, sXlo);
  }
  asm volatile("fence.proxy.async.shared::cta;");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  // Nothing may be in flight when the kernel frees tensor memory and exits: the
  // loader waits for its last copies, the issuer for its last commits, with the
  // default limit.  An accumulator has one tile's MMAs in flight at a time.
  if (loader) {
    const bool ok = stream_chunks(sA, Ahi, Alo, nchunks, NB, full, empty, limit);
    if (!ok) flag_timeout(flags, err, b);     // a bounded wait gave up
  } else if (issuer) {
    const uint32_t idesc = bf ? instr_desc_bf16(kTileM, kTileN) : instr_desc_tf32(kTileM, kTileN);
    bool ok = true;
    Ring ring = {0, 0, 0};
    int done = 0;                             // tiles committed
    for (int t = t0; t < t1; ++t) {
      const int ab = done & 1;
      if (done >= 2) {                        // the fields of tile t - 2 have been formed
        ok = wait_parity(&accfree[ab], (done / 2 - 1) & 1, limit);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;");
      }
      ok = issue_tile(bf, tmem + ab * kTileN, sA, sXhi, kc, NB, ring, full, empty, idesc, limit);
      if (!ok) break;
      commit(&accb[ab]);
      ++done;
    }
    drain_ring(ring.used, NB, empty);
    for (int i = max(0, done - 2); i < done; ++i) wait_parity(&accb[i & 1], (i >> 1) & 1, kWaitLimit);
    if (!ok) flag_timeout(flags, err, b);
  } else if (warp < kTcThreads / 32) {
    float* Zb = Z + (size_t)b * 9 * g.Mz * g.nm * 2;
    bool ok = true;
    for (int t = t0; t < t1 && ok; ++t) {
      const int ab = (t - t0) & 1;
      ok = group_and(tid != 0 || wait_parity(&accb[ab], ((t - t0) >> 1) & 1, limit));
      asm volatile("tcgen05.fence::after_thread_sync;");
      if (!ok) break;
      zinv_fields(g, tmem + ab * kTileN, epi, kf, Zb, nops, t, c0, warp, lane);
      asm volatile("tcgen05.fence::before_thread_sync;");
      group_sync();                           // accumulator and staged rows read
      if (tid == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(saddr(&accfree[ab])) : "memory");
    }
    if (!ok && tid == 0) flag_timeout(flags, err, b);
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == kTcThreads / 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 128;" ::"r"(tmem));
}

// ---------------------------------------------------------------------------
// Tensor-core z forward transform for the mixed-precision path.
//
// For one slice, one field and one Chebyshev parity p the z-forward transform
// is F[n][col] = sum_{jh < ceil(Mz/2)} W[n][jh] fold_p[jh][col], n = 2r + p,
// with fold_0 = Q_j + Q_{Mz-1-j} and fold_1 = Q_j - Q_{Mz-1-j} (the middle row
// of an odd Mz once in fold_0) and col = (Fourier mode, real/imaginary part).
// CTA per (slice, field, parity, 64-column tile): the folds are formed in FP32
// from the row kernel's output, split into hi/lo TF32 operands in shared memory
// (K-major, 128-byte swizzle); the rows of W of parity p are pre-split images
// [mtile][kchunk][128 x 32]; three MMAs per 8-wide K step (hi*hi, hi*lo, lo*hi)
// accumulate in tensor memory; the epilogue writes F in FP64 for the solve.
// The waits, the drain and the tensor-memory release follow k_zinv_tc.
// ---------------------------------------------------------------------------
__host__ __device__ int tc_zfwd_mtiles(const Grid& g) { return (g.Nz / 2 + kTileM - 1) / kTileM; }
__host__ __device__ int tc_zfwd_kchunks(const Grid& g) { return ((g.Mz + 1) / 2 + tc_ke(g) - 1) / tc_ke(g); }
size_t tc_zfwd_image_floats(const Grid& g) { return (size_t)tc_zfwd_mtiles(g) * tc_zfwd_kchunks(g) * kChunkFloats; }

void tc_zfwd_build_images(const Grid& g, const double* zfwd, int p, float* hi, float* lo) {
  const int mt = tc_zfwd_mtiles(g), kc = tc_zfwd_kchunks(g), Mh = (g.Mz + 1) / 2, ke = tc_ke(g), es = 128 / ke;
  for (int t = 0; t < mt; ++t)
    for (int c = 0; c < kc; ++c) {
      float* bh = hi + ((size_t)t * kc + c) * kChunkFloats;
      float* bl = lo + ((size_t)t * kc + c) * kChunkFloats;
      for (int r = 0; r < kTileM; ++r)
        for (int k = 0; k < ke; ++k) {
          const int n = 2 * (t * kTileM + r) + p, jh = c * ke + k;
          const double v = (n < g.Nz && jh < Mh) ? zfwd[(size_t)n * g.Mz + jh] : 0.0;
          split_store(g, v, bh, bl, (int)swz_b(r, k * es));
        }
    }
}

// Image stages of k_zfwd_tc, as for k_zinv_tc.
static int tc_zfwd_stages(const Grid& g) {
  const int kc = tc_zfwd_kchunks(g);
  for (int nb = std::min(kc, 4); nb > 1; --nb)
    if ((size_t)kc * kTileN * 128 * 2 + (size_t)nb * 2 * kTileM * 128 + 1024 <= 200 * 1024) return nb;
  return 1;
}

size_t tc_zfwd_smem_bytes(const Grid& g) {
  return (size_t)tc_zfwd_kchunks(g) * kTileN * 128 * 2 + (size_t)tc_zfwd_stages(g) * 2 * kTileM * 128 + 1024;
}
// Grid-only choices (so a state gives the same bits in any batch): the tensor
// cores take grids with at least 64 Chebyshev coefficients whose operands fit
// in 200 KB of shared memory.  Below Nz = 64 a transform is one or two 32-wide
// K-chunks, and the FP32 CUDA-core kernels finish sooner (measured on a
// single 128 x 32 slice: 0.123 ms per RK443 step against 0.187 ms).
bool tc_zfwd_supported(const Grid& g) { return g.Nz >= 64 && tc_zfwd_smem_bytes(g) <= 200 * 1024; }

// CTA per (slice, field, parity, 64-column tile, 128-row tile of W's rows of
// that parity); the images stream in through the bulk-copy ring of k_zinv_tc.
// Roles as in k_zinv_tc.
// Bound: latency of a CTA's chain (folds, images, MMAs, stores), one or two CTAs
// per SM.  Measured (GB300, per launch; one thread issuing, copying and waiting,
// loads item by item and scattered 16-byte stores before; same bits): 1024 x 256,
// 32 states 319 -> 232 us, in BF16 262 -> 168 us; 512 x 128, 64 states 170 -> 136
// us, in BF16 104 -> 66 us; 256 x 64, 8 states 14.4 -> 10.8 us.
// ITEMS (K-major 16-byte items per thread in flight): 8 where shared memory leaves
// one CTA per SM, 4 (fewer registers) where two fit.
template <int ITEMS>
__global__ void __launch_bounds__(kWsThreads, ITEMS == 4 ? 2 : 1) k_zfwd_tc(Grid g, const float* __restrict__ Whi0, const float* __restrict__ Wlo0,
                                                 const float* __restrict__ Whi1, const float* __restrict__ Wlo1,
                                                 const float* __restrict__ Q, double* __restrict__ F, size_t S, int B,
                                                 const int* nsteps, const int* step, int* flags, int* err, int NB) {
  pdl_wait();
  extern __shared__ __align__(1024) unsigned char tc_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)tc_raw + 1023) & ~(uintptr_t)1023);
  __shared__ __align__(8) uint64_t full[4], empty[4], accb[1];
  __shared__ uint32_t tmem_base;
  const int ntile = (2 * g.nm + kTileN - 1) / kTileN;
  const int mtiles = tc_zfwd_mtiles(g);
  const int per_b = 2 * 2 * ntile * mtiles;
  const int b = blockIdx.x / per_b;
  int rem = blockIdx.x - b * per_b;
  const int f = rem / (2 * ntile * mtiles);
  rem -= f * 2 * ntile * mtiles;
  const int p = rem / (ntile * mtiles);
  rem -= p * ntile * mtiles;
  const int ct = rem / mtiles, t = rem - ct * mtiles;
  const int c0 = ct * kTileN;
  if (b >= B || !(nsteps == nullptr || *step < nsteps[b])) return;   // uniform per block
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int kc = tc_zfwd_kchunks(g);
  const bool bf = g.tcbf16 != 0;
  unsigned char* sXhi = base;
  unsigned char* sXlo = sXhi + (size_t)kc * kTileN * 128;
  unsigned char* sA = sXlo + (size_t)kc * kTileN * 128;   // [stage][hi, lo][128 x 128 B]
  float* epi = reinterpret_cast<float*>(base);            // the epilogue's rows replace the operands
  const long long limit = g_wait_limit;
  const bool loader = tid == kTcThreads, issuer = tid == kTcThreads + 32;
  const float* Ahi = (p == 0 ? Whi0 : Whi1) + (size_t)t * kc * kChunkFloats;
  const float* Alo = (p == 0 ? Wlo0 : Wlo1) + (size_t)t * kc * kChunkFloats;
  if (loader) {
    for (int i = 0; i < NB; ++i) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&full[i])));
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&empty[i])));
    }
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(saddr(&accb[0])));
    asm volatile("fence.mbarrier_init.release.cluster;");
    for (int c = 0; c < NB && c < kc; ++c) fetch_chunk(sA, Ahi, Alo, c, c, &full[c]);
  }
  if (warp == kTcThreads / 32) {
    __syncwarp();                             // the warp converged again after the loader's set-up
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], 64;" ::"r"(saddr(&tmem_base)));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
  } else if (warp < kTcThreads / 32) {
    // folds of parity p -> hi/lo operands, K-major (row = column of the tile, k = jh)
    const float* q = Q + (size_t)(b * 2 + f) * g.Mz * g.nm * 2;
    const int w = 2 * g.nm, Mh = (g.Mz + 1) / 2, gc = c0 + (tid & (kTileN - 1));
    const float* qc = q + min(gc, w - 1);
    auto pair = [&](int jh) {
      const int j = min(jh, Mh - 1);
      return make_float2(__ldg(qc + (size_t)j * w), __ldg(qc + (size_t)(g.Mz - 1 - j) * w));
    };
    auto fold = [&](float2 v, int jh) {
      const bool twice = g.Mz - 1 - jh != jh;
      const float x = p == 0 ? (twice ? v.x + v.y : v.x) : (twice ? v.x - v.y : 0.f);
      return gc < w && jh < Mh ? x : 0.f;
    };
    if (bf)
      convert_tile<true, ITEMS, float2>(pair, fold, kc, tid, sXhi, sXlo);
    else
      convert_tile<false, ITEMS, float2>(pair, fold, kc, tid, sXhi, sXlo);
  }
  asm volatile("fence.proxy.async.shared::cta;");
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  const uint32_t tmem = tmem_base;
  // (one phase per stage and pass over the ring, one of the accumulator: see k_zinv_tc)
  if (loader) {
    const bool ok = stream_chunks(sA, Ahi, Alo, kc, NB, full, empty, limit);
    if (!ok) flag_timeout(flags, err, b);     // a bounded wait gave up
  } else if (issuer) {
    const uint32_t idesc = bf ? instr_desc_bf16(kTileM, kTileN) : instr_desc_tf32(kTileM, kTileN);
    Ring ring = {0, 0, 0};
    const bool ok = issue_tile(bf, tmem, sA, sXhi, kc, NB, ring, full, empty, idesc, limit);
    if (ok) commit(&accb[0]);
    drain_ring(ring.used, NB, empty);
    if (ok)
      wait_parity(&accb[0], 0, kWaitLimit);
    else
      flag_timeout(flags, err, b);
  } else if (warp < kTcThreads / 32) {
    const bool ok = group_and(tid != 0 || wait_parity(&accb[0], 0, limit));
    asm volatile("tcgen05.fence::after_thread_sync;");
    if (ok) {
      // kEpiCols columns at a time through shared memory: each half-warp widens
      // and stores 32 of them, 256 bytes, of one row
      double* Fb = F + (size_t)b * S;
      for (int cb = 0; cb < kTileN; cb += kEpiCols) {
        stage_rows(tmem, epi, cb, warp, lane);
        group_sync();
        const int m = ((c0 + cb) >> 1) + (lane & 15);
        if (m < g.nm)
          for (int r = warp * 2 + (lane >> 4); r < kTileM; r += 2 * (kTcThreads / 32)) {
            const int n = 2 * (t * kTileM + r) + p;
            if (n >= g.Nz) break;
            const float2 v = *reinterpret_cast<const float2*>(epi + r * kEpiStride + 2 * (lane & 15));
            *reinterpret_cast<double2*>(Fb + soff2(g, f, n, m)) = make_double2(widen(v.x), widen(v.y));
          }
        if (cb + kEpiCols < kTileN) group_sync();
      }
    } else if (tid == 0) {
      flag_timeout(flags, err, b);
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;");
  if (warp == kTcThreads / 32) asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, 64;" ::"r"(tmem));
}

cudaError_t launch_zfwd_tc(const Grid& g, const Tables& t, const Work& w, int B, cudaStream_t s) {
  const size_t smem = tc_zfwd_smem_bytes(g);
  auto* kernel = smem > 112 * 1024 ? k_zfwd_tc<8> : k_zfwd_tc<4>;
  static const cudaError_t e8 = cudaFuncSetAttribute(k_zfwd_tc<8>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  static const cudaError_t e4 = cudaFuncSetAttribute(k_zfwd_tc<4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 200 * 1024);
  if (e8 != cudaSuccess || e4 != cudaSuccess) return e8 != cudaSuccess ? e8 : e4;
  const int ntile = (2 * g.nm + kTileN - 1) / kTileN;
  return launch_pdl(w.pdl != 0, kernel, (unsigned)(B * 2 * 2 * ntile * tc_zfwd_mtiles(g)), kWsThreads, smem, s, g,
                    t.tcW_hi[0], t.tcW_lo[0], t.tcW_hi[1], t.tcW_lo[1], reinterpret_cast<const float*>(w.Q), w.F,
                    state_doubles(g), B, w.nsteps, w.step, w.flags, w.err, tc_zfwd_stages(g));
}

cudaError_t launch_zinv_tc(const Grid& g, const Tables& t, const Work& w, const double* X, int B, const int* ns,
                           cudaStream_t s) {
  const ZinvTcShape sh = tc_zinv_shape(g, B);
  static const cudaError_t e = cudaFuncSetAttribute(k_zinv_tc, cudaFuncAttributeMaxDynamicSharedMemorySize, 222 * 1024);
  if (e != cudaSuccess) return e;
  const int ntile = (2 * g.nm + kTileN - 1) / kTileN;
  const int units = (tc_zinv_mtiles(g, 4) + sh.tiles - 1) / sh.tiles + (tc_zinv_mtiles(g, 2) + sh.tiles - 1) / sh.tiles;
  return launch_pdl(w.pdl != 0, k_zinv_tc, (unsigned)(B * ntile * units), kWsThreads, sh.smem, s, g, t.tcA_psi_hi,
                    t.tcA_psi_lo, t.tcA_T_hi, t.tcA_T_lo, X, state_doubles(g), reinterpret_cast<float*>(w.Z), B, ns,
                    w.step, w.flags, w.err, sh.tiles, sh.stages);
}

}  // namespace rbc
