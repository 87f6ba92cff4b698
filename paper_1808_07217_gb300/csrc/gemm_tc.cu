// Grouped bf16 GEMM on the 5th-generation tensor cores (tcgen05 / TMEM / TMA), sm_103a.
//
// The per-replica dense-layer products of Eq. 2's local gradient: forward act x W^T, data
// gradient dZ x W and weight gradient dZ^T x act, for K replicas at once.  Operands live in the
// replica-major buffers; each is described by one rank-3 TMA map whose outermost coordinate is the
// replica, so the CTA for (n-tile, m-tile, replica g) loads its tiles at coordinate z = g.
//
// One CTA computes a 128 x BN fp32 tile in TMEM:
//   warps 0, 3         TMA producers of A and of B: k-blocks of 64 bf16 (one 128-byte swizzle row)
//                      into a ring of shared-memory stages, completion signalled on the stage's
//                      mbarrier;
//   warp 1             MMA issuer: 4 x tcgen05.mma (M=128, N=BN, K=16) per stage, accumulate in
//                      TMEM; tcgen05.commit frees the stage and finally signals the epilogue;
//   warp 2             allocates / frees the TMEM columns;
//   warps 0-3          epilogue: tcgen05.ld of their 32 TMEM lanes (= tile rows), bias / ReLU /
//                      ReLU-mask, store to global.
// K-major operands use the canonical SWIZZLE_128B K-major layout (8-row atoms of 128 B; SBO =
// 1024 B; the k-th 16-element slice starts 32 B further); MN-major operands are loaded as
// 64-element-wide boxes stacked along MN (LBO = box stride, SBO = 1024 B; the k-th slice starts
// 16 rows = 2048 B further).  Every mbarrier wait is bounded: on expiry the kernel records an error
// flag, stops issuing, and still frees its TMEM.
//
// wgrad_update_kernel (further down) is the weight gradient fused with the local update: a
// persistent variant of the same pipeline whose epilogue streams the parameters through shared
// memory by TMA.
#include <cudaTypedefs.h>

#include <algorithm>
#include <cstdlib>
#include <mutex>
#include <type_traits>

#include "common.cuh"
#include "lsgd_internal.h"

namespace lsgd {

__device__ int g_tc_timeout = 0;

namespace {

constexpr int BM = 128;
constexpr int BK = 64;
constexpr long long kWaitCycles = 4000000000LL;  // ~2 s at 2 GHz

__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ void mbar_init(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_expect_tx(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_u32(bar)),
               "r"(bytes)
               : "memory");
}

__device__ __forceinline__ bool mbar_try_wait(uint64_t* bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(smem_u32(bar)), "r"(parity)
      : "memory");
  return ok != 0;
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_u32(bar)) : "memory");
}

// Bounded wait on an mbarrier phase; false (and the global error flag set) on expiry.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity,
                                          long long limit_cycles = kWaitCycles) {
  if (mbar_try_wait(bar, parity)) return true;
  const long long t0 = clock64();
  while (!mbar_try_wait(bar, parity)) {
    if (clock64() - t0 > limit_cycles) {
      atomicExch(&g_tc_timeout, 1);
      return false;
    }
  }
  return true;
}

// The TMA and MMA instructions take their operands from uniform registers.  Their issue loops are run
// by a whole warp (the warp index broadcast, so that the compiler knows the control flow to be
// uniform and keeps descriptors, addresses and counters in uniform registers) and one elected lane
// issues.  A loop under "lane == 0" instead moves every operand across for every instruction: at
// least 46 cycles per tcgen05.mma, and 90 to 150 with the descriptor arithmetic of these kernels,
// where the tensor core takes 23 (M = 64, N = 16), 39 (M = 128, N = 16), 48 (N = 64) or 128 (N = 256).
__device__ __forceinline__ int uniform_warp() { return __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0); }

__device__ __forceinline__ bool elect_one() {
  uint32_t ok;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(ok));
  return ok != 0;
}

// mbar_wait by every lane; true if all saw the phase (one that ran out cannot split the warp).
__device__ __forceinline__ bool mbar_wait_warp(uint64_t* bar, uint32_t parity) {
  return __all_sync(0xffffffffu, mbar_wait(bar, parity) ? 1 : 0) != 0;
}

// A tensor map into the descriptor cache (maps are kernel parameters: no dependency on other kernels).
__device__ __forceinline__ void prefetch_map(const CUtensorMap* map) {
  asm volatile("prefetch.tensormap [%0];" ::"l"(reinterpret_cast<uint64_t>(map)) : "memory");
}

__device__ __forceinline__ void tma_load_3d(void* dst, const CUtensorMap* map, uint64_t* bar, int x,
                                            int y, int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(x), "r"(y), "r"(z)
      : "memory");
}

__device__ __forceinline__ void tma_load_5d(void* dst, const CUtensorMap* map, uint64_t* bar, int c0,
                                            int c1, int c2, int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%3, %4, %5, %6, %7}], [%2];" ::"r"(smem_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(smem_u32(bar)), "r"(c0), "r"(c1), "r"(c2), "r"(c3),
      "r"(c4)
      : "memory");
}

// Shared-memory descriptor of a K-major operand whose rows are `swz` bytes (32, 64 or 128) with the
// matching swizzle: core matrices of 8 rows, SBO = 8 rows, layout code 6 / 4 / 2.
__device__ __forceinline__ uint64_t smem_desc_kmajor(uint32_t addr, uint32_t swz) {
  const uint64_t layout = swz == 128 ? 2ull : (swz == 64 ? 4ull : 6ull);
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)1u << 16;  // LBO (unused by swizzled K-major layouts)
  d |= (uint64_t)(((8u * swz) >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;
  d |= layout << 61;
  return d;
}

// An MN-major (or any) descriptor with the 32-, 64- or 128-byte swizzle given in bytes.
__device__ __forceinline__ uint64_t smem_desc_swz(uint32_t addr, uint32_t lbo, uint32_t sbo,
                                                  uint32_t swz) {
  const uint64_t layout = swz == 128 ? 2ull : (swz == 64 ? 4ull : 6ull);
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;  // descriptor version (tcgen05)
  d |= layout << 61;
  return d;
}

__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr >> 4) & 0x3FFFu);
  d |= (uint64_t)((lbo >> 4) & 0x3FFFu) << 16;
  d |= (uint64_t)((sbo >> 4) & 0x3FFFu) << 32;
  d |= 1ull << 46;  // descriptor version (tcgen05)
  d |= 2ull << 61;  // SWIZZLE_128B
  return d;
}

// kind::f16 instruction descriptor: fp32 accumulator, bf16 A and B, majors, N >> 3, M >> 4.
__host__ __device__ constexpr uint32_t make_idesc(int M, int N, bool a_mn, bool b_mn) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16) |
         ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
          smem_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15},"
      " [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

__device__ __forceinline__ void tmem_ld16_nowait(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15},"
      " [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
}

// Three groups of 16 columns, all loads in flight before the one wait (which the registers pass
// through, so that no use of them moves above it).
__device__ __forceinline__ void tmem_ld16x3(uint32_t t0, uint32_t t1, uint32_t t2, float (&v0)[16],
                                            float (&v1)[16], float (&v2)[16]) {
  uint32_t r0[16], r1[16], r2[16];
  tmem_ld16_nowait(t0, r0);
  tmem_ld16_nowait(t1, r1);
  tmem_ld16_nowait(t2, r2);
  asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    asm volatile("" : "+r"(r0[i]), "+r"(r1[i]), "+r"(r2[i]));
    v0[i] = __uint_as_float(r0[i]);
    v1[i] = __uint_as_float(r1[i]);
    v2[i] = __uint_as_float(r2[i]);
  }
}

// Sums 16 values per lane over the 32 lanes of a warp in four halving exchanges and one final
// exchange: afterwards lane l holds the warp's sum of value l / 2 (lanes 2 j and 2 j + 1 agree).
__device__ __forceinline__ float warp_colsum16(float (&v)[16], int lane) {
#pragma unroll
  for (int w = 8; w >= 1; w >>= 1) {
    const bool up = (lane & (2 * w)) != 0;
#pragma unroll
    for (int i = 0; i < w; ++i) {
      const float send = up ? v[i] : v[i + w];
      const float keep = up ? v[i + w] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 2 * w);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

constexpr int kTcMaxStages = 16;
// Barriers of the one-tile kernel, behind its ring: `stages` A tiles (a_bytes each), then as many B
// tiles, all 1024-byte aligned for the 128-byte swizzle.
struct TcSync {
  uint64_t full[kTcMaxStages], empty[kTcMaxStages];
  uint64_t accum;
  uint32_t tmem_base;
};

// ---- GEMM epilogue (one-tile and persistent kernels) ----
// Sixteen consecutive outputs of one row: 32-byte stores where the row is aligned and whole, 16-byte
// ones where it is aligned to that (a bf16 row of an odd multiple of 8 elements), else element by
// element up to the matrix edge.  The 16-byte form took four EF-sign steps of MLP 776-520-264-17, K =
// 5, B = 50, from 408 to 394 us.
__device__ __forceinline__ void store_row16(void* C, bool c_bf16, int64_t off, int n, int N,
                                            const float (&x)[16]) {
  if (c_bf16) {
    uint16_t* out = reinterpret_cast<uint16_t*>(C) + off;
    if (n + 16 <= N && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
      uint32_t w[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) w[j] = (uint32_t)f2bf(x[2 * j]) | ((uint32_t)f2bf(x[2 * j + 1]) << 16);
      if ((reinterpret_cast<uintptr_t>(out) & 31) == 0) {
        asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out), "r"(w[0]),
                     "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
                     : "memory");
      } else {
        reinterpret_cast<uint4*>(out)[0] = make_uint4(w[0], w[1], w[2], w[3]);
        reinterpret_cast<uint4*>(out)[1] = make_uint4(w[4], w[5], w[6], w[7]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (n + i < N) out[i] = f2bf(x[i]);
    }
  } else {
    float* out = reinterpret_cast<float*>(C) + off;
    if (n + 16 <= N && (reinterpret_cast<uintptr_t>(out) & 15) == 0) {
      if ((reinterpret_cast<uintptr_t>(out) & 31) == 0) {
#pragma unroll
        for (int j = 0; j < 2; ++j)
          asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(out + 8 * j),
                       "f"(x[8 * j]), "f"(x[8 * j + 1]), "f"(x[8 * j + 2]), "f"(x[8 * j + 3]),
                       "f"(x[8 * j + 4]), "f"(x[8 * j + 5]), "f"(x[8 * j + 6]), "f"(x[8 * j + 7])
                       : "memory");
      } else {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          reinterpret_cast<float4*>(out)[j] = make_float4(x[4 * j], x[4 * j + 1], x[4 * j + 2], x[4 * j + 3]);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 16; ++i)
        if (n + i < N) out[i] = x[i];
    }
  }
}

// The GEMM epilogue of one 128 x BN tile for one epilogue thread: tile row et (TMEM lane et)
// leaves TMEM 16 columns at a time and is written straight from registers: C(m, n) at
// C + c_base + m c_rs + n, with bias (+ ReLU) or the ReLU mask of the stored activation applied (the
// next 16 mask values requested while these are used).  With hs_warp (bias_colsum) the stored values
// -- rounded to bf16 when C is bf16 -- are also summed over the warp's 32 rows, per column, by a fixed
// butterfly (rows past M add nothing); hs_warp[c] gets column c's partial.
// One loop of one 16-column body: the one-tile kernel's CTAs run it once, and unrolled over a tile its
// instructions came from memory (column sums of 128 columns: 22,000 cycles for 50 x 264, K = 5;
// 64 columns of MLP 3072-512-512-10: 10,000; the persistent data gradients of MLP-4096 77 -> 58 us).
template <int BN>
__device__ __forceinline__ void epilogue_rows(const TcGemmArgs& args, int et, int lane,
                                              uint32_t tmem_acc, int g, int m0, int n0,
                                              int64_t c_base, float* hs_warp) {
  const int m = m0 + et;
  const bool row_ok = m < args.M;
  const int epi = args.epi;
  const bool has_bias = epi == EPI_BIAS || epi == EPI_BIAS_RELU;
  const float* bias = has_bias ? args.bias + (int64_t)g * args.bias_gs : nullptr;
  const bool bias_al = has_bias && (reinterpret_cast<uintptr_t>(bias + n0) & 15) == 0;
  const int64_t coff = c_base + (int64_t)m * args.c_rs;
  const int64_t moff = (int64_t)g * args.mask_gs + (int64_t)m * args.mask_rs;
  const uint16_t* mrow = epi == EPI_MASK && args.mask_bf16
                             ? reinterpret_cast<const uint16_t*>(args.mask) + moff + n0
                             : nullptr;
  const bool mal = mrow && row_ok && (reinterpret_cast<uintptr_t>(mrow) & 15) == 0;
  const uint32_t tl = tmem_acc + ((uint32_t)(et & ~31) << 16);
  // the mask values of 16 columns (two per word) where they are whole and aligned
  auto load_mask = [&](int cc, uint4 (&mk)[2]) {
    if (mal && cc < BN && n0 + cc + 16 <= args.N) {
      mk[0] = __ldg(reinterpret_cast<const uint4*>(mrow + cc));
      mk[1] = __ldg(reinterpret_cast<const uint4*>(mrow + cc) + 1);
    }
  };
  uint4 mk[2] = {};
  load_mask(0, mk);
#pragma unroll 1
  for (int cc = 0; cc < BN; cc += 16) {
    const int nb = n0 + cc;
    if (nb >= args.N) break;  // uniform over the CTA
    const bool whole = nb + 16 <= args.N;
    float4 bv[4];
    if (bias_al && whole) {
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = __ldg(reinterpret_cast<const float4*>(bias + nb) + j);
    }
    const uint32_t mw[8] = {mk[0].x, mk[0].y, mk[0].z, mk[0].w, mk[1].x, mk[1].y, mk[1].z, mk[1].w};
    load_mask(cc + 16, mk);
    float x[16];
    tmem_ld16(tl + (uint32_t)cc, x);
    if (has_bias) {
      if (bias_al && whole) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          x[4 * j] += bv[j].x;
          x[4 * j + 1] += bv[j].y;
          x[4 * j + 2] += bv[j].z;
          x[4 * j + 3] += bv[j].w;
        }
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] += nb + i < args.N ? __ldg(bias + nb + i) : 0.f;
      }
      if (epi == EPI_BIAS_RELU) {
#pragma unroll
        for (int i = 0; i < 16; ++i) x[i] = fmaxf(x[i], 0.f);
      }
    } else if (epi == EPI_MASK) {
      if (mal && whole) {
#pragma unroll
        for (int i = 0; i < 16; ++i)
          x[i] = bf2f((uint16_t)((i & 1) ? (mw[i >> 1] >> 16) : (mw[i >> 1] & 0xffffu))) > 0.f ? x[i] : 0.f;
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const int n = nb + i;
          const float mv = !(row_ok && n < args.N) ? 0.f
                           : args.mask_bf16 ? bf2f(reinterpret_cast<const uint16_t*>(args.mask)[moff + n])
                                            : reinterpret_cast<const float*>(args.mask)[moff + n];
          x[i] = mv > 0.f ? x[i] : 0.f;
        }
      }
    }
    if (row_ok) store_row16(args.C, args.c_bf16, coff + nb, nb, args.N, x);
    if (hs_warp) {
      float t[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) t[i] = !row_ok ? 0.f : (args.c_bf16 ? bf2f(f2bf(x[i])) : x[i]);
      const float sum = warp_colsum16(t, lane);
      if (!(lane & 1)) hs_warp[cc + (lane >> 1)] = sum;
    }
  }
}

// The bias of the layer below, for the column-sum mode: each of the 128 epilogue threads takes
// columns et + 128 i of the tile; their parameters are requested before the accumulator wait.
template <int BN>
constexpr int kBiasCols = (BN + 127) / 128;  // columns per epilogue thread

template <int BN>
__device__ __forceinline__ void bias_prefetch(const TcGemmArgs& args, int et, int g, int n0,
                                              float (&bsw)[kBiasCols<BN>],
                                              float (&bsu)[kBiasCols<BN>]) {
#pragma unroll
  for (int i = 0; i < kBiasCols<BN>; ++i) {
    const int c = 128 * i + et, n = n0 + c;
    const bool v = args.bias_colsum && args.bsgd.w && c < BN && n < args.N;
    const int64_t k = (int64_t)g * args.bias_gs + n;
    bsw[i] = v ? args.bsgd.w[k] : 0.f;
    bsu[i] = v && args.bsgd.u ? args.bsgd.u[k] : 0.f;
  }
}

// After the four warps' partials are in hs (this tile's buffer): the bias gradient of each of
// this thread's columns, (warp 0 + warp 1) + (warp 2 + warp 3), and its local update (or the
// gradient itself without bsgd.w).
template <int BN>
__device__ __forceinline__ void bias_update(const TcGemmArgs& args, int et, int g, int n0,
                                            const float (*hs)[BN], const float (&bsw)[kBiasCols<BN>],
                                            const float (&bsu)[kBiasCols<BN>]) {
#pragma unroll
  for (int i = 0; i < kBiasCols<BN>; ++i) {
    const int c = 128 * i + et, n = n0 + c;
    if (c >= BN || n >= args.N) continue;
    const float gb = __fadd_rn(__fadd_rn(hs[0][c], hs[1][c]), __fadd_rn(hs[2][c], hs[3][c]));
    const int64_t k = (int64_t)g * args.bias_gs + n;
    if (!args.bsgd.w) {
      args.bias_grad[k] = gb;
      continue;
    }
    const SgdParams& sp = args.bsgd;
    float w = bsw[i], u = bsu[i];
    const bool sg = sp.sign != 0;
    if (sp.mom == 0.f)
      sgd_elem<false, false>(w, u, gb, sp.lr, 0.f, sp.wd, sg);
    else if (sp.nesterov)
      sgd_elem<true, true>(w, u, gb, sp.lr, sp.mom, sp.wd, sg);
    else
      sgd_elem<true, false>(w, u, gb, sp.lr, sp.mom, sp.wd, sg);
    sp.w[k] = w;
    if (sp.u) sp.u[k] = u;
    if (sp.wb) sp.wb[k] = f2bf(w);
  }
}

// The ring is as deep as the reduction and the shared memory of the CTAs that share an SM allow
// (launch_one_tile): a TMA load takes 500 (L2) to 2,400 cycles to land, so a k-block costs 2,400 / stages
// of them.
template <int BN>
__global__ void __launch_bounds__(128, 1) gemm_tc_kernel(const __grid_constant__ TcGemmArgs args) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int STAGES = args.stages;
  // K-major A: the box's rows (a mini-batch of fewer than 128); the product reads on into what
  // follows for the tile's other rows, which are not stored
  const uint32_t a_bytes = args.A.mn_major ? (uint32_t)BM * BK * 2 : (uint32_t)args.A.box_rows * BK * 2;
  constexpr uint32_t kBytesB = BN * BK * 2;
  uint8_t* ring_b = ring + STAGES * a_bytes;
  TcSync& sm = *reinterpret_cast<TcSync*>(ring_b + STAGES * kBytesB);
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const int splits = args.splits > 1 ? args.splits : 1;
  const int n0 = blockIdx.x * BN, m0 = blockIdx.y * BM, g = blockIdx.z / splits;
  // implicit convolution: the tile's 128 output pixels are rows of whole images (TW = Wout) from
  // pixel m0 on, i.e. output row oy0 of image b0
  const int cv_b0 = args.conv ? m0 / (args.cv_hout * args.cv_wout) : 0;
  const int cv_oy0 = args.conv ? (m0 / args.cv_wout) % args.cv_hout : 0;
  const int split = blockIdx.z % splits;
  const int nk_all = args.conv ? (9 + 64 / args.cv_ck - 1) / (64 / args.cv_ck) : (args.Kd + BK - 1) / BK;
  const int per_split = (nk_all + splits - 1) / splits;
  const int kb_first = split * per_split;
  const int nk = min(nk_all - kb_first, per_split);  // >= 1 (the host makes every split nonempty)
  const int64_t c_base = (int64_t)g * args.c_gs + (int64_t)split * args.c_split_stride;
  const bool a_mn = args.A.mn_major, b_mn = args.B.mn_major;

  if (threadIdx.x == 0) {
    prefetch_map(&args.A.map);
    prefetch_map(&args.B.map);
    for (int s = 0; s < STAGES; ++s) {
      mbar_init(&sm.full[s], args.conv ? 1 : 2);  // both producers
      mbar_init(&sm.empty[s], 1);
    }
    mbar_init(&sm.accum, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sm.tmem_base)),
                 "r"((uint32_t)BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sm.tmem_base;
  pdl_begin();  // everything above touched only shared memory and TMEM

  bool ok = true;
  if (warp == 0 || (warp == 3 && !args.conv)) {
    // ---------------- TMA producers: warp 0 A (of a convolution both), warp 3 B ----------------
    // Issuing a load takes its warp about 100 cycles and a wait 150, so the operands have a warp each
    // (with one, a k-block took 380 cycles, twice the products), and the ring's first lap no waits.
    const bool el = elect_one();
    int issued = 0, s = 0;
    uint32_t ph = 1;  // of the lap before: the second lap waits for phase 0
    const int gb = args.b_shared ? 0 : g;  // identical replicas: group 0's copy for all
    for (int kb = 0; kb < nk; ++kb) {
      if (kb >= STAGES && !mbar_wait_warp(&sm.empty[s], ph)) {
        ok = false;
        break;
      }
      if (args.conv) {
        // 64 / Ck taps per stage; tap t: the input shifted by (kh - 1, kw - 1) (zero outside the
        // image, stride by the map's element strides) and the weights' tap-t slice [N][Ck]
        const int ck = args.cv_ck, tps = 64 / ck;
        const int t0 = (kb_first + kb) * tps, t1 = min(9, t0 + tps);
        if (el) {
          mbar_expect_tx(&sm.full[s], (uint32_t)(t1 - t0) * (BM + BN) * ck * 2);
          for (int t = t0; t < t1; ++t) {
            const int kh = t / 3, kw = t % 3, j = t - t0;
            tma_load_5d(ring + s * a_bytes + j * BM * ck * 2, &args.A.map, &sm.full[s], 0, kw - 1,
                        cv_oy0 * args.cv_stride + kh - 1, cv_b0, g);
            tma_load_3d(ring_b + s * kBytesB + j * BN * ck * 2, &args.B.map, &sm.full[s], t * ck, n0, g);
          }
        }
      } else if (el) {
        const int k0 = (kb_first + kb) * BK;
        if (warp == 0) {
          mbar_expect_tx(&sm.full[s], a_bytes);
          if (!a_mn) {
            tma_load_3d(ring + s * a_bytes, &args.A.map, &sm.full[s], k0, m0, g);
          } else {
#pragma unroll
            for (int i = 0; i < BM / 64; ++i)
              tma_load_3d(ring + s * a_bytes + i * 64 * BK * 2, &args.A.map, &sm.full[s], m0 + 64 * i, k0, g);
          }
        } else {
          mbar_expect_tx(&sm.full[s], kBytesB);
          if (!b_mn && args.B.box_rows == BN) {
            tma_load_3d(ring_b + s * kBytesB, &args.B.map, &sm.full[s], k0, n0, gb);
          } else {
            // 64-row boxes stacked along N (K-major) or 64-wide ones (MN-major)
#pragma unroll
            for (int i = 0; i < BN / 64; ++i)
              tma_load_3d(ring_b + s * kBytesB + i * 64 * BK * 2, &args.B.map, &sm.full[s],
                          b_mn ? n0 + 64 * i : k0, b_mn ? k0 : n0 + 64 * i, gb);
          }
        }
      }
      issued = kb + 1;
      if (++s == STAGES) {
        s = 0;
        ph ^= 1;
      }
    }
    if (!ok) {
      // let copies already in flight land before the CTA can exit
      for (int kb = (issued > STAGES ? issued - STAGES : 0); kb < issued; ++kb)
        mbar_wait(&sm.full[kb % STAGES], (kb / STAGES) & 1);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const bool el = elect_one();
    constexpr uint32_t idesc_kk = make_idesc(BM, BN, false, false);
    const uint32_t idesc = idesc_kk | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16);
    // descriptors of stage 0; a stage and a 16-deep slice add their byte offsets / 16
    const uint64_t a_desc0 = a_mn ? smem_desc(smem_u32(ring), 64 * BK * 2, 1024) : smem_desc(smem_u32(ring), 16, 1024);
    const uint64_t b_desc0 = b_mn ? smem_desc(smem_u32(ring_b), 64 * BK * 2, 1024) : smem_desc(smem_u32(ring_b), 16, 1024);
    const uint32_t a_step = a_mn ? 2048 >> 4 : 32 >> 4, b_step = b_mn ? 2048 >> 4 : 32 >> 4;
    int s = 0;
    uint32_t ph = 0;
    for (int kb = 0; kb < nk; ++kb) {
      if (!mbar_wait_warp(&sm.full[s], ph)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      if (args.conv) {
        // each tap's sub-tiles: rows of Ck bf16 = swz bytes; K = 16 per MMA, 32 bytes further
        const uint32_t a_base = smem_u32(ring + s * a_bytes), b_base = smem_u32(ring_b + s * kBytesB);
        const int ck = args.cv_ck, tps = 64 / ck;
        const int nt = min(9, (kb_first + kb + 1) * tps) - (kb_first + kb) * tps;
        const uint32_t swz = (uint32_t)ck * 2;
        if (el)
          for (int j = 0; j < nt; ++j)
            for (int kk = 0; kk < ck / 16; ++kk)
              mma_bf16(tmem, smem_desc_kmajor(a_base + j * BM * ck * 2 + kk * 32, swz),
                       smem_desc_kmajor(b_base + j * BN * ck * 2 + kk * 32, swz), idesc,
                       (kb > 0 || j > 0 || kk > 0) ? 1u : 0u);
      } else {
        const uint64_t ad = a_desc0 + (uint32_t)s * (a_bytes >> 4), bd = b_desc0 + (uint32_t)s * (kBytesB >> 4);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
          if (el) mma_bf16(tmem, ad + kk * a_step, bd + kk * b_step, idesc, (kb > 0 || kk > 0) ? 1u : 0u);
      }
      if (el) mma_commit(&sm.empty[s]);  // stage reusable once these MMAs have read it
      if (++s == STAGES) {
        s = 0;
        ph ^= 1;
      }
    }
    if (ok && el) mma_commit(&sm.accum);  // accumulator complete
  } else if (warp == 2 && args.epi == EPI_MASK && args.mask) {
    // warp 2 idles through the mainloop: it brings the tile's ReLU-mask rows (the stored
    // activation) into L1, so that the epilogue's mask loads hit L1 instead of waiting on DRAM
    // (the TMA operand loads bypass L1).  Every line prefetched starts inside the tile.
    const int esz = args.mask_bf16 ? 2 : 4;
    const int ncols = min(BN, args.N - n0);
    const int lines = (ncols * esz + 127) / 128;
    const int rows = min(BM, args.M - m0);
    const char* base = reinterpret_cast<const char*>(args.mask) +
                       ((int64_t)g * args.mask_gs + (int64_t)m0 * args.mask_rs + n0) * esz;
    for (int t = lane; t < rows * lines; t += 32) {
      const int r = t / lines, l = t % lines;
      asm volatile("prefetch.global.L1 [%0];" ::"l"(base + (int64_t)r * args.mask_rs * esz + l * 128));
    }
  }
  __syncwarp();

  // ---------------- epilogue (all 4 warps) ----------------
  // Thread t writes tile row t from registers (epilogue_rows).  For the bias column sums the
  // stage buffers, free once the accumulator is complete (every MMA has read its operands), hold
  // the four warps' partials.
  float bsw[kBiasCols<BN>], bsu[kBiasCols<BN>];
  bias_prefetch<BN>(args, (int)threadIdx.x, g, n0, bsw, bsu);
  const bool have_acc = mbar_wait(&sm.accum, 0);
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  float(*hs)[BN] = reinterpret_cast<float(*)[BN]>(ring);
  if (have_acc)
    epilogue_rows<BN>(args, (int)threadIdx.x, lane, tmem, g, m0, n0, c_base,
                          args.bias_colsum ? hs[warp] : nullptr);
  if (args.bias_colsum) {
    __syncthreads();  // every thread passes it, so a wait that ran out cannot split the CTA
    if (have_acc) bias_update<BN>(args, (int)threadIdx.x, g, n0, hs, bsw, bsu);
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"((uint32_t)BN)
                 : "memory");
  }
}

// =============================================================================================
// Persistent grouped GEMM for the long products (forward and data gradient of the dense
// layers): C[g] = epilogue(A[g] B[gb]^T) over 128 x PBN output tiles.  One CTA per SM walks the
// tiles blockIdx.x, blockIdx.x + gridDim.x, ... with the replica innermost (so the CTAs that
// share a weight tile when every replica reads replica 0's, b_shared, run together and L2 serves
// it), and two TMEM accumulators let one tile's epilogue overlap the next tile's products:
//   warps 0, 3  TMA producers: A (128 x 64) and 64 of B's columns, and the rest of B's PBN, of each
//               k-block into a PST-stage ring
//   warp 1      MMA issuer: tcgen05.mma (M = 128, N = PBN, K = 16), accumulator (tile & 1)
//   warp 2      TMEM allocation (2 PBN columns)
//   warps 4-7   epilogue (epilogue_rows: bias / ReLU / ReLU mask; column sums + bias
//               update): each thread writes its tile row straight from registers, each warp
//               waits for the accumulator and hands it back by itself
// 128 x 256 tiles halve the shared-memory operand bytes per MMA of the 64-wide one-tile kernel
// (whose N = 64 MMAs read as many operand bytes as they compute).
namespace pt {
constexpr int PBN = 256;
constexpr int PST = 4;  // 192 KB of operands in flight: the epilogue needs no staging tile
constexpr int THREADS = 256;
}  // namespace pt

struct PtSmem {
  uint8_t a[pt::PST][BM * BK * 2];       // 16 KB each (1024-aligned)
  uint8_t b[pt::PST][pt::PBN * BK * 2];  // 32 KB each
  float hs[2][4][pt::PBN];  // bias column sums: per tile parity, per epilogue warp
  uint64_t full[pt::PST], empty[pt::PST];
  uint64_t acc_full[2], acc_empty[2];
  uint32_t tmem_base;
  int fail;  // an epilogue warp's accumulator wait ran out (column-sum mode)
};

__global__ void __launch_bounds__(pt::THREADS, 1) gemm_pt_kernel(const __grid_constant__ TcGemmArgs args) {
  extern __shared__ uint8_t smem_raw[];
  PtSmem& sm = *reinterpret_cast<PtSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                          ~uintptr_t(1023));
  constexpr int PBN = pt::PBN, PST = pt::PST;
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const int tiles_n = (args.N + PBN - 1) / PBN, tiles_m = (args.M + BM - 1) / BM;
  const int tiles = tiles_n * tiles_m * args.G;
  const int nk = (args.Kd + BK - 1) / BK;
  const bool a_mn = args.A.mn_major, b_mn = args.B.mn_major;
  constexpr uint32_t kBytesA = BM * BK * 2, kBytesB = PBN * BK * 2;
  // tile t: replica fastest, then m-tile, then n-tile
  auto coords = [&](int t, int& g, int& m0, int& n0) {
    g = t % args.G;
    const int r = t / args.G;
    m0 = (r % tiles_m) * BM;
    n0 = (r / tiles_m) * PBN;
  };

  if (threadIdx.x == 0) {
    for (int s = 0; s < PST; ++s) {
      mbar_init(&sm.full[s], 2);  // both producers
      mbar_init(&sm.empty[s], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sm.acc_full[i], 1);
      mbar_init(&sm.acc_empty[i], 4);  // one arrival per epilogue warp
    }
    sm.fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sm.tmem_base)),
                 "r"(2u * PBN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sm.tmem_base;
  pdl_begin();  // everything above touched only shared memory and TMEM

  if (warp == 0 || warp == 3) {
    // ---------------- TMA producers: warp 0 A and the first 64 of B's columns, warp 3 the others ----------------
    const bool el = elect_one();
    int it = 0, s = 0;
    uint32_t ph = 1;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x) {
      int g, m0, n0;
      coords(t, g, m0, n0);
      const int gb = args.b_shared ? 0 : g;  // identical replicas: replica 0's copy for all
      for (int kb = 0; kb < nk; ++kb, ++it) {
        if (!mbar_wait_warp(&sm.empty[s], ph)) {
          ok = false;
          break;
        }
        if (el) {
          const int k0 = kb * BK;
          if (warp == 0) {
            mbar_expect_tx(&sm.full[s], kBytesA + kBytesB / 4);
            if (!a_mn) {
              tma_load_3d(sm.a[s], &args.A.map, &sm.full[s], k0, m0, g);
            } else {
#pragma unroll
              for (int i = 0; i < BM / 64; ++i)
                tma_load_3d(sm.a[s] + i * 64 * BK * 2, &args.A.map, &sm.full[s], m0 + 64 * i, k0, g);
            }
          } else {
            mbar_expect_tx(&sm.full[s], kBytesB / 4 * 3);
          }
          // 64-row boxes stacked along N (K-major) or 64-wide ones (MN-major)
          for (int i = warp == 0 ? 0 : 1; i < (warp == 0 ? 1 : PBN / 64); ++i)
            tma_load_3d(sm.b[s] + i * 64 * BK * 2, &args.B.map, &sm.full[s], b_mn ? n0 + 64 * i : k0,
                        b_mn ? k0 : n0 + 64 * i, gb);
        }
        if (++s == PST) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    if (!ok) {
      for (int j = (it > PST ? it - PST : 0); j < it; ++j)
        mbar_wait(&sm.full[j % PST], (j / PST) & 1);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const bool el = elect_one();
    constexpr uint32_t idesc_kk = make_idesc(BM, PBN, false, false);
    const uint32_t idesc = idesc_kk | ((a_mn ? 1u : 0u) << 15) | ((b_mn ? 1u : 0u) << 16);
    // descriptors of stage 0; a stage and a 16-deep slice add their byte offsets / 16
    const uint64_t a_desc0 = a_mn ? smem_desc(smem_u32(sm.a[0]), 64 * BK * 2, 1024) : smem_desc(smem_u32(sm.a[0]), 16, 1024);
    const uint64_t b_desc0 = b_mn ? smem_desc(smem_u32(sm.b[0]), 64 * BK * 2, 1024) : smem_desc(smem_u32(sm.b[0]), 16, 1024);
    const uint32_t a_step = a_mn ? 2048 >> 4 : 32 >> 4, b_step = b_mn ? 2048 >> 4 : 32 >> 4;
    int i = 0, s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (int t = blockIdx.x; t < tiles && ok; t += gridDim.x, ++i) {
      const int ab = i & 1;
      if (!mbar_wait_warp(&sm.acc_empty[ab], ((i >> 1) & 1) ^ 1)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t acc = tmem + (uint32_t)(ab * PBN);
      for (int kb = 0; kb < nk; ++kb) {
        if (!mbar_wait_warp(&sm.full[s], ph)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t ad = a_desc0 + (uint32_t)s * (kBytesA >> 4), bd = b_desc0 + (uint32_t)s * (kBytesB >> 4);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
          if (el) mma_bf16(acc, ad + kk * a_step, bd + kk * b_step, idesc, (kb > 0 || kk > 0) ? 1u : 0u);
        if (el) mma_commit(&sm.empty[s]);
        if (++s == PST) {
          s = 0;
          ph ^= 1;
        }
      }
      if (ok && el) mma_commit(&sm.acc_full[ab]);
    }
  } else if (warp >= 4) {
    // ---------------- epilogue ----------------
    // Each warp waits for the accumulator by itself (every lane polls; the warp goes on only if
    // all lanes saw the phase) and gives it back with one arrival.  Only the column-sum mode
    // brings the four warps together, once per tile; there a wait that ran out is shared through
    // sm.fail before that barrier, so all four leave together.
    const int et = threadIdx.x - 128, quarter = warp & 3;
    const bool colsum = args.bias_colsum;
    auto warp_wait = [&](uint64_t* bar, uint32_t parity) -> bool {
      const bool okl = mbar_wait(bar, parity);
      return __all_sync(0xffffffffu, okl);
    };
    int i = 0;
    for (int t = blockIdx.x; t < tiles; t += gridDim.x, ++i) {
      int g, m0, n0;
      coords(t, g, m0, n0);
      const int ab = i & 1;
      float bsw[kBiasCols<PBN>], bsu[kBiasCols<PBN>];
      bias_prefetch<PBN>(args, et, g, n0, bsw, bsu);
      if (args.epi == EPI_MASK && args.mask && m0 + et < args.M) {
        // this thread's row of the tile's ReLU mask (the stored activation) into L2 while the
        // tile's products run, so that the copy-out's mask loads do not each wait on DRAM
        const int esz = args.mask_bf16 ? 2 : 4;
        const int ncols = min(PBN, args.N - n0);
        const char* rowp = reinterpret_cast<const char*>(args.mask) +
                           ((int64_t)g * args.mask_gs + (int64_t)(m0 + et) * args.mask_rs + n0) * esz;
        for (int b = 0; b < ncols * esz; b += 128) asm volatile("prefetch.global.L2 [%0];" ::"l"(rowp + b));
      }
      const bool okw = warp_wait(&sm.acc_full[ab], (i >> 1) & 1);
      const uint32_t acc = tmem + (uint32_t)(ab * PBN);
      if (!colsum) {
        if (!okw) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        epilogue_rows<PBN>(args, et, lane, acc, g, m0, n0, (int64_t)g * args.c_gs, nullptr);
      } else {
        if (okw) {
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          epilogue_rows<PBN>(args, et, lane, acc, g, m0, n0, (int64_t)g * args.c_gs,
                                 sm.hs[ab][quarter]);
        } else if (lane == 0) {
          sm.fail = 1;
        }
        asm volatile("bar.sync 1, 128;" ::: "memory");
        if (*reinterpret_cast<volatile int*>(&sm.fail)) break;
        // hs[ab] is written again two tiles on, after every warp has passed the next barrier
        bias_update<PBN>(args, et, g, n0, sm.hs[ab], bsw, bsu);
      }
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&sm.acc_empty[ab]);  // this warp's rows have left the accumulator
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(2u * pt::PBN)
                 : "memory");
  }
}

// =============================================================================================
// Weight gradient fused with the local update: persistent, every parameter byte moved by TMA.
//
// For replica g and a 128 x 128 tile (rows m = output units, columns n = inputs) of a layer's
// weight matrix, the gradient dZ[g]^T act[g] (k = B_loc) accumulates in one of two TMEM
// accumulators while the previous tile's update runs.  The tile's parameters and momentum stream
// through a ring of shared-memory slots in 32-column chunks (128 rows x 128 B, SWIZZLE_128B), are
// updated in place, and go back to HBM by TMA stores (clipped at the matrix edge), together with
// the bf16 shadow staged in a 64-byte-swizzled buffer.  The tiles of up to two layers form one
// list (the first layer's, then the second's), so a layer's last partial wave and the launch's
// ramp are paid once for both.  One CTA per SM:
//   warp 0      operand producer: dZ / act k-blocks into a two-stage ring
//   warp 1      MMA issuer: tcgen05.mma (M = N = 128, K = 16) into accumulator (tile & 1)
//   warp 2      TMEM allocation (256 columns, 512 in averaging mode); w / u chunk producer
//   warp 3      TMA store issuer: stores each finished chunk and hands its slot back
//   warps 4-19  epilogue, four threads per tile row (TMEM lane quarter = warp % 4; warps
//               4 + 4 p .. 7 + 4 p take columns 8 p .. 8 p + 7 of each chunk): per chunk,
//               tcgen05.ld of the gradient columns, the local momentum-SGD update (weight decay,
//               heavy-ball or Nesterov momentum, Sec. A.4) on w, u in shared memory, bf16 w
//               into the slot's staging buffer.
// Each epilogue warp waits on the accumulator and chunk barriers by itself and releases the chunk
// (to the store issuer) and the accumulator (to the MMA issuer) with one arrival per warp, so the
// warps overlap one another's latencies; a wait that runs out ends that warp's loop only.
//
// Averaging mode (args.avg): the step ends with the K-way average of Eq. 2 (right), so a CTA takes
// one weight tile through all G replicas in turn (replica innermost in its tile sequence).  Each
// replica's tile gets its own gradient and local update exactly as above (u written back), and the
// updated values are summed over the replicas with the average's TwoSum in two further TMEM
// regions (s, c: columns 256-511); after the last replica the mean, divided as the average does,
// goes to replica 0's parameters and bf16 shadow -- the other replicas equal it, and the runtime
// writes their copies only when something reads them (every kernel of the next step reads
// replica 0).  Neither the per-replica updated parameters nor their shadow reach HBM.  With
// args.w_rep0 (the replicas are identical at the step's start, in either mode) each tile's
// parameters are read from replica 0.  The results equal those of this kernel in plain mode
// followed by the K-way average kernel, bit for bit.
namespace wu {
constexpr int TN = 128;                     // tile columns (= rows: BM)
constexpr int CW = 32;                      // chunk columns (fp32: one 128-byte row)
constexpr int ST = 2;                       // operand stages
constexpr int NS = 4;                       // w / u chunk slots
constexpr int SD = 2;                       // chunks whose TMA stores may be in flight (<= NS)
constexpr int EPI_WARPS = 16;               // four per TMEM lane quarter
constexpr int THREADS = 128 + 32 * EPI_WARPS;
constexpr int CPT = CW / (EPI_WARPS / 4);   // chunk columns per epilogue thread (8)
constexpr uint32_t kChunkF32 = BM * CW * 4;  // 16 KB
constexpr uint32_t kChunkB16 = BM * CW * 2;  // 8 KB
}  // namespace wu

struct WuSmem {
  uint8_t a[wu::ST][BM * BK * 2];         // 16 KB each
  uint8_t b[wu::ST][wu::TN * BK * 2];     // 16 KB each
  uint8_t w[wu::NS][wu::kChunkF32];       // 1024-aligned (SWIZZLE_128B)
  uint8_t u[wu::NS][wu::kChunkF32];
  uint8_t wb[wu::NS][wu::kChunkB16];      // bf16 staging, one per slot; 512-aligned (SWIZZLE_64B)
  uint64_t op_full[wu::ST], op_empty[wu::ST];
  uint64_t acc_full[2], acc_empty[2];
  uint64_t wu_full[wu::NS], wu_empty[wu::NS];
  uint64_t st_full[wu::NS];  // every epilogue warp has finished the slot's chunk: store it
  uint32_t tmem_base;
};

__device__ __forceinline__ void tmem_ld8(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}

// One epilogue thread's share of a chunk: 8 gradient columns at tg and its 16-column pair region
// at tsc (s then c, 8 each), both loads in flight before one wait.
__device__ __forceinline__ void tmem_ld_g8_sc16(uint32_t tg, uint32_t tsc, float (&g)[8],
                                                float (&sc)[16]) {
  uint32_t a[8], b[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%24];\n"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,"
      "%20,%21,%22,%23}, [%25];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(a[0]), "=r"(a[1]), "=r"(a[2]), "=r"(a[3]), "=r"(a[4]), "=r"(a[5]), "=r"(a[6]),
        "=r"(a[7]), "=r"(b[0]), "=r"(b[1]), "=r"(b[2]), "=r"(b[3]), "=r"(b[4]), "=r"(b[5]),
        "=r"(b[6]), "=r"(b[7]), "=r"(b[8]), "=r"(b[9]), "=r"(b[10]), "=r"(b[11]), "=r"(b[12]),
        "=r"(b[13]), "=r"(b[14]), "=r"(b[15])
      : "r"(tg), "r"(tsc)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) g[i] = __uint_as_float(a[i]);
#pragma unroll
  for (int i = 0; i < 16; ++i) sc[i] = __uint_as_float(b[i]);
}

__device__ __forceinline__ void tmem_st16_nowait(uint32_t taddr, const float (&v)[16]) {
  asm volatile(
      "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
      "%14,%15,%16};" ::"r"(taddr),
      "r"(__float_as_uint(v[0])), "r"(__float_as_uint(v[1])), "r"(__float_as_uint(v[2])),
      "r"(__float_as_uint(v[3])), "r"(__float_as_uint(v[4])), "r"(__float_as_uint(v[5])),
      "r"(__float_as_uint(v[6])), "r"(__float_as_uint(v[7])), "r"(__float_as_uint(v[8])),
      "r"(__float_as_uint(v[9])), "r"(__float_as_uint(v[10])), "r"(__float_as_uint(v[11])),
      "r"(__float_as_uint(v[12])), "r"(__float_as_uint(v[13])), "r"(__float_as_uint(v[14])),
      "r"(__float_as_uint(v[15]))
      : "memory");
}

// tcgen05.st has no wait of its own: tmem_wait_st before reading the columns back or freeing them.
__device__ __forceinline__ void tmem_wait_st() {
  asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory");
}

__device__ __forceinline__ void tma_store_3d(const CUtensorMap* map, const void* src, int x, int y,
                                             int z) {
  asm volatile(
      "cp.async.bulk.tensor.3d.global.shared::cta.bulk_group [%0, {%2, %3, %4}], [%1];" ::"l"(
          reinterpret_cast<uint64_t>(map)),
      "r"(smem_u32(src)), "r"(x), "r"(y), "r"(z)
      : "memory");
}

__device__ __forceinline__ int wu_chunks(int N, int n0) {
  const int left = N - n0;
  return left >= wu::TN ? wu::TN / wu::CW : (left + wu::CW - 1) / wu::CW;
}

namespace wu {
// What the epilogue does with a chunk, fixed at compile time so that the per-element code has no
// branches: PLAIN writes the updated parameters; AVG folds them into the running pair (FIRST
// starts it, LAST turns it into the mean and writes that).
enum : int { kPlain = 0, kFirst = 1, kLast = 2, kAvg = 4 };
}  // namespace wu

// The local update of four consecutive parameters under one update rule (0: no momentum,
// 1: heavy ball, 2: Nesterov) through sgd_elem, the arithmetic of every update kernel.
template <bool SG, int RULE>
__device__ __forceinline__ void sgd4_rule(float4& w, float4& u, const float4 g, const SgdParams& sp) {
  constexpr bool MOM = RULE != 0, NEST = RULE == 2;
  const float m = MOM ? sp.mom : 0.f;
  sgd_elem<MOM, NEST>(w.x, u.x, g.x, sp.lr, m, sp.wd, SG);
  sgd_elem<MOM, NEST>(w.y, u.y, g.y, sp.lr, m, sp.wd, SG);
  sgd_elem<MOM, NEST>(w.z, u.z, g.z, sp.lr, m, sp.wd, SG);
  sgd_elem<MOM, NEST>(w.w, u.w, g.w, sp.lr, m, sp.wd, SG);
}

// One epilogue thread's CPT columns of a 32-column chunk of its tile row r: the update of CPT
// parameters (w, u in the swizzled shared-memory slot rows wrow / urow), in averaging mode folded
// into the running pair (s, c) = (sc[0, CPT), sc[CPT, 2 CPT)) and, at the unit's last replica,
// replaced by the mean; wherever the parameters leave for HBM their bf16 shadow goes to brow.
// Without momentum u is neither read nor changed (its slot goes back to HBM as loaded).
template <bool SG, int RULE, int MODE>
__device__ __forceinline__ void wu_part_chunk(const float (&gv)[wu::CPT], float (&sc)[2 * wu::CPT],
                                              uint8_t* wrow, uint8_t* urow, uint8_t* brow, int part,
                                              int r, const SgdParams& sp, float Gf, float invG,
                                              bool pow2) {
  constexpr bool AVG = (MODE & wu::kAvg) != 0, FIRST = (MODE & wu::kFirst) != 0,
                 LAST = (MODE & wu::kLast) != 0;
  constexpr bool WRITE_W = !AVG || LAST;
  uint32_t packed[wu::CPT / 2];
#pragma unroll
  for (int jj = 0; jj < wu::CPT / 4; ++jj) {
    const int j = (wu::CPT / 4) * part + jj;  // float4 column group within the chunk
    const int phys = (j ^ (r & 7)) << 4;
    float4 wv = *reinterpret_cast<const float4*>(wrow + phys);
    float4 uv = RULE != 0 ? *reinterpret_cast<const float4*>(urow + phys)
                          : make_float4(0.f, 0.f, 0.f, 0.f);
    sgd4_rule<SG, RULE>(wv, uv, make_float4(gv[4 * jj], gv[4 * jj + 1], gv[4 * jj + 2], gv[4 * jj + 3]),
                        sp);
    if (RULE != 0) *reinterpret_cast<float4*>(urow + phys) = uv;
    if (AVG) {
      float* sv = sc + 4 * jj;            // s of these four columns
      float* cv = sc + wu::CPT + 4 * jj;  // c of these four columns
      const float wn[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        if (FIRST) {
          sv[e] = wn[e];
          cv[e] = 0.f;
        } else {
          two_sum_add(sv[e], cv[e], wn[e]);
        }
      }
      if (LAST) {
        float m[4];
        if (pow2) {
#pragma unroll
          for (int e = 0; e < 4; ++e) m[e] = mean_of_pow2(sv[e], cv[e], Gf, invG);
        } else {
#pragma unroll
          for (int e = 0; e < 4; ++e) m[e] = mean_of(sv[e], cv[e], Gf);
        }
        wv = make_float4(m[0], m[1], m[2], m[3]);
      }
    }
    if (WRITE_W) {
      *reinterpret_cast<float4*>(wrow + phys) = wv;
      packed[2 * jj] = (uint32_t)f2bf(wv.x) | ((uint32_t)f2bf(wv.y) << 16);
      packed[2 * jj + 1] = (uint32_t)f2bf(wv.z) | ((uint32_t)f2bf(wv.w) << 16);
    }
  }
  if (WRITE_W) {
#pragma unroll
    for (int hh = 0; hh < wu::CPT / 8; ++hh) {
      const int h = (wu::CPT / 8) * part + hh;  // 16-byte unit of the 64-byte bf16 row
      *reinterpret_cast<uint4*>(brow + ((h ^ ((r >> 1) & 3)) << 4)) =
          make_uint4(packed[4 * hh], packed[4 * hh + 1], packed[4 * hh + 2], packed[4 * hh + 3]);
    }
  }
}

__global__ void __launch_bounds__(wu::THREADS, 1) wgrad_update_kernel(
    const __grid_constant__ WgradUpdateArgs args) {
  extern __shared__ uint8_t smem_raw[];
  WuSmem& sm = *reinterpret_cast<WuSmem*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                          ~uintptr_t(1023));
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  // the layers' tiles one layer after another (operand layouts are the same in all): layer l's
  // tiles follow uc_l tile positions (uc_l G tiles) of the layers before it (scalars, so that
  // nothing needs local memory)
  static_assert(kWgradMaxLayers == 3, "the bookkeeping below names three layers");
  const int tn0 = (args.L[0].N + wu::TN - 1) / wu::TN;
  const int tn1 = args.nl > 1 ? (args.L[1].N + wu::TN - 1) / wu::TN : 0;
  const int tn2 = args.nl > 2 ? (args.L[2].N + wu::TN - 1) / wu::TN : 0;
  const int uc1 = tn0 * ((args.L[0].M + BM - 1) / BM);
  const int uc2 = uc1 + (args.nl > 1 ? tn1 * ((args.L[1].M + BM - 1) / BM) : 0);
  const int uc3 = uc2 + (args.nl > 2 ? tn2 * ((args.L[2].M + BM - 1) / BM) : 0);
  const int tiles = uc3 * args.G;
  const int nk = (args.Kd + BK - 1) / BK;
  const bool a_mn = args.L[0].A.mn_major, b_mn = args.L[0].B.mn_major;
  const bool has_u = args.sgd.u != nullptr;
  const bool avg = args.avg != 0;
  constexpr uint32_t kBytesA = BM * BK * 2, kBytesB = wu::TN * BK * 2;
  // This CTA's tile sequence: units blockIdx.x, blockIdx.x + gridDim.x, ...; a unit is one tile,
  // or one tile position of a layer taken through all G replicas -- in averaging mode, and
  // whenever every replica reads replica 0's parameters (w_rep0): then replica 0's tile comes
  // last, so that no replica reads it after it has been updated.
  const bool by_unit = avg || args.w_rep0;
  const int units = by_unit ? uc3 : tiles;
  const int per_unit = by_unit ? args.G : 1;
  const int my_count =
      (int)blockIdx.x < units ? ((units - 1 - (int)blockIdx.x) / (int)gridDim.x + 1) * per_unit : 0;
  const uint32_t tmem_cols = avg ? 4u * wu::TN : 2u * wu::TN;

  if (threadIdx.x == 0) {
    for (int i = 0; i < wu::ST; ++i) {
      mbar_init(&sm.op_full[i], 1);
      mbar_init(&sm.op_empty[i], 1);
    }
    // the epilogue warps release the accumulator and the chunk slots one arrival per warp
    for (int i = 0; i < 2; ++i) {
      mbar_init(&sm.acc_full[i], 1);
      mbar_init(&sm.acc_empty[i], wu::EPI_WARPS);
    }
    for (int i = 0; i < wu::NS; ++i) {
      mbar_init(&sm.wu_full[i], 1);
      mbar_init(&sm.wu_empty[i], 1);
      mbar_init(&sm.st_full[i], wu::EPI_WARPS);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&sm.tmem_base)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = sm.tmem_base;
  pdl_begin();  // everything above touched only shared memory and TMEM

  // tile position x (< uc3) -> its layer l, the position within the layer and the layer's
  // column-tile count
  auto locate = [&](int x, int& l, int& r, int& tnl) {
    l = (x >= uc1 ? 1 : 0) + (x >= uc2 ? 1 : 0);
    r = x - (l == 0 ? 0 : (l == 1 ? uc1 : uc2));
    tnl = l == 0 ? tn0 : (l == 1 ? tn1 : tn2);
  };
  auto tile_coords = [&](int t, const WgradUpdateLayer*& ly, int& g, int& m0, int& n0) {
    // layer by layer, each layer's tiles replica by replica
    const int l0 = (t >= uc1 * args.G ? 1 : 0) + (t >= uc2 * args.G ? 1 : 0);
    const int base = l0 == 0 ? 0 : (l0 == 1 ? uc1 : uc2);
    const int per_g = (l0 == 0 ? uc1 : (l0 == 1 ? uc2 : uc3)) - base;
    t -= base * args.G;
    g = t / per_g;
    int l, r, tnl;
    locate(base + t % per_g, l, r, tnl);
    ly = &args.L[l];
    m0 = (r / tnl) * BM;
    n0 = (r % tnl) * wu::TN;
  };
  // the j-th tile of this CTA's sequence; gi = its replica's position within the unit
  auto tile_at = [&](int j, const WgradUpdateLayer*& ly, int& g, int& m0, int& n0, int& gi) {
    const int u = (int)blockIdx.x + (j / per_unit) * (int)gridDim.x;
    gi = j % per_unit;
    if (!by_unit) {
      tile_coords(u, ly, g, m0, n0);
      return;
    }
    int l, r, tnl;
    locate(u, l, r, tnl);
    ly = &args.L[l];
    m0 = (r / tnl) * BM;
    n0 = (r % tnl) * wu::TN;
    // averaging: replicas in order (the average's summation order); else replica 0 last
    g = avg ? gi : (gi + 1) % args.G;
  };

  if (warp == 0) {
    // ---------------- operand producer ----------------
    const bool el = elect_one();
    int it = 0, s = 0;
    uint32_t ph = 1;
    bool ok = true;
    for (int j = 0; j < my_count && ok; ++j) {
      const WgradUpdateLayer* ly;
      int g, m0, n0, gi;
      tile_at(j, ly, g, m0, n0, gi);
      for (int kb = 0; kb < nk; ++kb, ++it) {
        if (!mbar_wait_warp(&sm.op_empty[s], ph)) {
          ok = false;
          break;
        }
        if (el) {
          mbar_expect_tx(&sm.op_full[s], kBytesA + kBytesB);
          const int k0 = kb * BK;
          if (!a_mn) {
            tma_load_3d(sm.a[s], &ly->A.map, &sm.op_full[s], k0, m0, g);
          } else {
#pragma unroll
            for (int i = 0; i < BM / 64; ++i)
              tma_load_3d(sm.a[s] + i * 64 * BK * 2, &ly->A.map, &sm.op_full[s], m0 + 64 * i, k0, g);
          }
          if (!b_mn) {
            tma_load_3d(sm.b[s], &ly->B.map, &sm.op_full[s], k0, n0, g);
          } else {
#pragma unroll
            for (int i = 0; i < wu::TN / 64; ++i)
              tma_load_3d(sm.b[s] + i * 64 * BK * 2, &ly->B.map, &sm.op_full[s], n0 + 64 * i, k0, g);
          }
        }
        if (++s == wu::ST) {
          s = 0;
          ph ^= 1;
        }
      }
    }
    if (!ok) {
      // let copies in flight land before the CTA can exit
      for (int j = (it > wu::ST ? it - wu::ST : 0); j < it; ++j)
        mbar_wait(&sm.op_full[j % wu::ST], (j / wu::ST) & 1);
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const bool el = elect_one();
    const uint32_t idesc = make_idesc(BM, wu::TN, a_mn, b_mn);
    // descriptors of stage 0; a stage and a 16-deep slice add their byte offsets / 16
    const uint64_t a_desc0 = a_mn ? smem_desc(smem_u32(sm.a[0]), 64 * BK * 2, 1024) : smem_desc(smem_u32(sm.a[0]), 16, 1024);
    const uint64_t b_desc0 = b_mn ? smem_desc(smem_u32(sm.b[0]), 64 * BK * 2, 1024) : smem_desc(smem_u32(sm.b[0]), 16, 1024);
    const uint32_t a_step = a_mn ? 2048 >> 4 : 32 >> 4, b_step = b_mn ? 2048 >> 4 : 32 >> 4;
    int i = 0, s = 0;
    uint32_t ph = 0;
    bool ok = true;
    for (; i < my_count && ok; ++i) {
      const int ab = i & 1;
      if (!mbar_wait_warp(&sm.acc_empty[ab], ((i >> 1) & 1) ^ 1)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t acc = tmem + (uint32_t)(ab * wu::TN);
      for (int kb = 0; kb < nk; ++kb) {
        if (!mbar_wait_warp(&sm.op_full[s], ph)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t ad = a_desc0 + (uint32_t)s * (kBytesA >> 4), bd = b_desc0 + (uint32_t)s * (kBytesB >> 4);
#pragma unroll
        for (int kk = 0; kk < BK / 16; ++kk)
          if (el) mma_bf16(acc, ad + kk * a_step, bd + kk * b_step, idesc, (kb > 0 || kk > 0) ? 1u : 0u);
        if (el) mma_commit(&sm.op_empty[s]);
        if (++s == wu::ST) {
          s = 0;
          ph ^= 1;
        }
      }
      if (ok && el) mma_commit(&sm.acc_full[ab]);
    }
  } else if (warp == 2) {
    // ---------------- w / u chunk producer ----------------
    const bool el = elect_one();
    int q = 0, sl = 0;
    uint32_t ph = 1;
    bool ok = true;
    const uint32_t bytes = wu::kChunkF32 * (has_u ? 2u : 1u);
    for (int j = 0; j < my_count && ok; ++j) {
      const WgradUpdateLayer* ly;
      int g, m0, n0, gi;
      tile_at(j, ly, g, m0, n0, gi);
      const int gw = args.w_rep0 ? 0 : g;  // identical replicas: read replica 0's
      const int nc = wu_chunks(ly->N, n0);
      for (int c = 0; c < nc; ++c, ++q) {
        if (!mbar_wait_warp(&sm.wu_empty[sl], ph)) {
          ok = false;
          break;
        }
        if (el) {
          mbar_expect_tx(&sm.wu_full[sl], bytes);
          tma_load_3d(sm.w[sl], &ly->wmap, &sm.wu_full[sl], n0 + c * wu::CW, m0, gw);
          if (has_u) tma_load_3d(sm.u[sl], &ly->umap, &sm.wu_full[sl], n0 + c * wu::CW, m0, g);
        }
        if (++sl == wu::NS) {
          sl = 0;
          ph ^= 1;
        }
      }
    }
    if (!ok) {
      for (int j = (q > wu::NS ? q - wu::NS : 0); j < q; ++j)
        mbar_wait(&sm.wu_full[j % wu::NS], (j / wu::NS) & 1);
    }
  } else if (warp == 3) {
    // ---------------- store issuer ----------------
    // Each finished chunk leaves by TMA stores (u; the updated w and its bf16 shadow, or in
    // averaging mode at the unit's last replica the mean to replica 0); once they have read the
    // slot it goes back to the w / u producer.  Issuing stores here keeps their cost (a few
    // hundred cycles each) off the epilogue threads.  One and the same elected lane issues, commits
    // and waits for the store groups (they are a thread's own).
    const bool el = elect_one();
    int q = 0, sl = 0, back = 0;  // chunks stored; their slot; the slot to hand back next
    uint32_t ph = 0;
    bool ok = true;
    for (int j = 0; j < my_count && ok; ++j) {
      const WgradUpdateLayer* ly;
      int g, m0, n0, gi;
      tile_at(j, ly, g, m0, n0, gi);
      const bool last = gi == per_unit - 1;
      const int nc = wu_chunks(ly->N, n0);
      for (int c = 0; c < nc; ++c, ++q) {
        if (!mbar_wait_warp(&sm.st_full[sl], ph)) {
          ok = false;
          break;
        }
        if (el) {
          const int x = n0 + c * wu::CW;
          if (has_u) tma_store_3d(&ly->umap, sm.u[sl], x, m0, g);
          if (!avg) {
            tma_store_3d(&ly->wmap, sm.w[sl], x, m0, g);
            if (args.sgd.wb) tma_store_3d(&ly->wbmap, sm.wb[sl], x, m0, g);
          } else if (last) {
            // the mean goes to replica 0 only; the runtime copies it to the other replicas when
            // something needs them (every consumer of the next step reads replica 0)
            tma_store_3d(&ly->wmap, sm.w[sl], x, m0, 0);
            if (args.sgd.wb) tma_store_3d(&ly->wbmap, sm.wb[sl], x, m0, 0);
          }
          asm volatile("cp.async.bulk.commit_group;" ::: "memory");
          // SD chunks' store groups in flight: once at most SD - 1 are still reading shared
          // memory, the oldest one's slot goes back to the w / u producer
          asm volatile("cp.async.bulk.wait_group.read %0;" ::"n"(wu::SD - 1) : "memory");
          if (q >= wu::SD - 1) mbar_arrive(&sm.wu_empty[back]);
        }
        if (q >= wu::SD - 1 && ++back == wu::NS) back = 0;
        if (++sl == wu::NS) {
          sl = 0;
          ph ^= 1;
        }
      }
    }
    if (el) {
      asm volatile("cp.async.bulk.wait_group 0;" ::: "memory");
      // the last SD - 1 chunks' slots (their stores have now completed)
      for (int j = (q > wu::SD - 1 ? q - (wu::SD - 1) : 0); j < q; ++j) mbar_arrive(&sm.wu_empty[j % wu::NS]);
    }
  } else if (warp >= 4) {
    // ---------------- epilogue ----------------
    // The epilogue warps do not wait for one another: each waits for the accumulator and for
    // each chunk itself and hands the chunk on (and, after a tile's last chunk, the accumulator
    // back) with one mbarrier arrival per warp, so warps at different points of the chunk
    // sequence overlap their latencies.  No warp can get a ring's length ahead: a slot comes
    // back only after all of them have arrived.
    const int quarter = warp & 3;
    const int part = (warp - 4) >> 2;   // which CPT columns of each chunk
    const int r = quarter * 32 + lane;  // tile row of this thread
    const SgdParams& sp = args.sgd;
    // Every lane polls (acquiring what the barrier guards); the warp goes on only if all lanes
    // saw the phase, so a wait that runs out never splits the warp-wide tensor-memory
    // instructions that follow.
    auto warp_wait = [&](uint64_t* bar, uint32_t parity) -> bool {
      const bool okl = mbar_wait(bar, parity);
      return __all_sync(0xffffffffu, okl);
    };
    const float Gf = (float)args.G;
    const bool pow2 = (args.G & (args.G - 1)) == 0;
    const float invG = 1.0f / Gf;  // exact when G is a power of two
    // the update rule (0: no momentum, 1: heavy ball, 2: Nesterov); momentum implies u
    const int rule = sp.mom == 0.f ? 0 : (sp.nesterov ? 2 : 1);
    // This thread's CPT columns of a chunk, through the variant of wu_part_chunk for this launch's
    // rule and sign option and this tile's place in its unit: one branch per chunk, none per
    // element.
    auto part_chunk = [&](const float (&gv)[wu::CPT], float (&sc)[2 * wu::CPT], uint8_t* wrow,
                          uint8_t* urow, uint8_t* brow, bool first, bool last) {
      auto by_mode = [&](auto sg_tag, auto rule_tag) {
        constexpr bool SG = decltype(sg_tag)::value;
        constexpr int R = decltype(rule_tag)::value;
        if (!avg)
          wu_part_chunk<SG, R, wu::kPlain>(gv, sc, wrow, urow, brow, part, r, sp, Gf, invG, pow2);
        else if (first && last)
          wu_part_chunk<SG, R, wu::kAvg | wu::kFirst | wu::kLast>(gv, sc, wrow, urow, brow, part, r,
                                                                  sp, Gf, invG, pow2);
        else if (first)
          wu_part_chunk<SG, R, wu::kAvg | wu::kFirst>(gv, sc, wrow, urow, brow, part, r, sp, Gf,
                                                      invG, pow2);
        else if (last)
          wu_part_chunk<SG, R, wu::kAvg | wu::kLast>(gv, sc, wrow, urow, brow, part, r, sp, Gf,
                                                     invG, pow2);
        else
          wu_part_chunk<SG, R, wu::kAvg>(gv, sc, wrow, urow, brow, part, r, sp, Gf, invG, pow2);
      };
      auto by_rule = [&](auto sg_tag) {
        if (rule == 0)
          by_mode(sg_tag, std::integral_constant<int, 0>{});
        else if (rule == 1)
          by_mode(sg_tag, std::integral_constant<int, 1>{});
        else
          by_mode(sg_tag, std::integral_constant<int, 2>{});
      };
      if (sp.sign)
        by_rule(std::true_type{});
      else
        by_rule(std::false_type{});
    };
    int q = 0, i = 0;
    bool ok = true;
    for (; i < my_count && ok; ++i) {
      const WgradUpdateLayer* ly;
      int g, m0, n0, gi;
      tile_at(i, ly, g, m0, n0, gi);
      const bool first = gi == 0, last = gi == per_unit - 1;
      const int ab = i & 1;
      const int nc = wu_chunks(ly->N, n0);
      if (!warp_wait(&sm.acc_full[ab], (i >> 1) & 1)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      for (int c = 0; c < nc; ++c, ++q) {
        const int sl = q % wu::NS;
        if (!warp_wait(&sm.wu_full[sl], (q / wu::NS) & 1)) {
          ok = false;
          break;
        }
        const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
        const uint32_t g_col = (uint32_t)(ab * wu::TN + c * wu::CW + wu::CPT * part);
        // averaging mode: this thread's running pair of the chunk over the replicas so far,
        // 2 CPT columns from 256 + 64 chunk + 2 CPT part (s in sc[0 .. CPT), c after it)
        const uint32_t sc_col = 2u * wu::TN + (uint32_t)(c * 2 * wu::CW + 2 * wu::CPT * part);
        float gv[wu::CPT], sc[2 * wu::CPT];
        if (avg && !first) {
          tmem_wait_st();  // this chunk's pair, stored at the previous replica
          tmem_ld_g8_sc16(tmem + lane_base + g_col, tmem + lane_base + sc_col, gv, sc);
        } else {
          tmem_ld8(tmem + lane_base + g_col, gv);
        }
        uint8_t* wrow = sm.w[sl] + r * 128;
        uint8_t* urow = sm.u[sl] + r * 128;
        uint8_t* brow = sm.wb[sl] + r * 64;
        part_chunk(gv, sc, wrow, urow, brow, first, last);
        if (avg && !last) tmem_st16_nowait(tmem + lane_base + sc_col, sc);
        // this warp's shared-memory writes reach the TMA stores, its accumulator reads are done
        asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) {
          mbar_arrive(&sm.st_full[sl]);  // the store issuer takes the chunk once all warps have
          if (c == nc - 1) mbar_arrive(&sm.acc_empty[ab]);  // ... and the MMA the accumulator
        }
      }
    }
    tmem_wait_st();  // no tensor-memory store outstanding when the columns are freed
    (void)ok;
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem),
                 "r"(tmem_cols)
                 : "memory");
  }
}

// =============================================================================================
// Implicit-GEMM 3x3 convolution, persistent: out[g][p][n] = sum over taps t and k < ck of
// in[g][shift_t(p)][k] w[g][n][t][k] (zero padding 1, stride 1 or 2), fp32 out.
//
// A CTA owns one replica and every cpr-th 128-pixel tile of it.  The replica's weights (all nine
// taps, N rows of ck channels) are loaded once; the input streams through a ring of shared-memory
// stages by TMA (rank-5 boxes of the NHWC input, out-of-bounds fill = the zero padding, element
// strides = the convolution stride); two TMEM accumulators let a tile's MMAs overlap the previous
// tile's epilogue.  Two stage forms:
//   strip (stride 1, a tile = whole rows of one image): one stage per tile holds, for each kw, the
//     tile's rows plus one halo row above and below, shifted by kw - 1 columns; tap (kh, kw) is
//     that box from row kh on (a whole number of swizzle atoms further), so 3 boxes serve 9 taps;
//   per kernel row: three stages per tile, stage kh holds the three kw-shifted boxes of the
//     tile's rows under kernel row kh (stride 2, and tiles that span several images).
//   warp 0      TMA producer (weights once, then one stage per tap)
//   warp 1      MMA issuer (the whole warp, one lane issuing: 72 -> 65 us for a first-stage forward
//               of 16 workers x 128 images): per tap ck / 16 tcgen05.mma (M = 128, N = NP, K = 16),
//               descriptors from precomputed bases; with nsplit = 3 the taps of column kw
//               accumulate into partial kw
//   warp 2      TMEM allocation
//   warps 4-7   epilogue: tcgen05.ld of the tile row's NP columns (the partials' sum), fp32
//               stores
// nacc accumulator buffers (each nsplit x NP columns) let the MMAs of the next tiles run while
// the epilogue drains this one.
namespace cv {
constexpr int THREADS = 256;
constexpr int RING_BYTES = 96 * 1024;
constexpr int MAX_STAGES = 24;  // 4 KB stages (ck = 16)
constexpr int EPI0 = 128;
constexpr size_t SMEM_MAX = 227 * 1024;  // dynamic shared memory of one CTA
constexpr int MAX_ACC = 4;  // accumulator buffers in TMEM
// barriers, TMEM slot (16 bytes), and the BatchNorm-backward epilogue's mean / rstd (64 each)
constexpr size_t AUX_BYTES = (2 * MAX_STAGES + 2 * MAX_ACC + 1) * 8 + 16 + 2 * 64 * 4;
}  // namespace cv


__global__ void __launch_bounds__(cv::THREADS, 2) conv_tc_kernel(const __grid_constant__ ConvArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const int ck = a.ck, np = a.np;
  // per-kernel-row form: a stage holds the three taps of one kernel row (three TMA boxes, one
  // handshake); strip form: a stage holds the three kw boxes of (rows + 2) image rows
  const uint32_t tap_bytes = (uint32_t)BM * ck * 2;
  const uint32_t row_bytes = (uint32_t)a.wout * ck * 2;  // one image row of the input box
  const uint32_t box_bytes = a.strip ? tap_bytes + 2 * row_bytes : tap_bytes;
  const uint32_t stage_bytes = 3 * box_bytes;
  const int spt = a.strip ? 1 : 3;  // stages per tile
  const int nst = min(cv::MAX_STAGES, a.ring_bytes / (int)stage_bytes);
  uint8_t* ring = base;
  uint8_t* wsm = base + a.ring_bytes;
  const uint32_t wtap = (uint32_t)np * ck * 2;  // bytes of one tap's weights
  uint64_t* bars = reinterpret_cast<uint64_t*>(wsm + 9 * wtap);
  uint64_t* full = bars;
  uint64_t* empty = bars + cv::MAX_STAGES;
  uint64_t* acc_full = bars + 2 * cv::MAX_STAGES;
  uint64_t* acc_empty = acc_full + cv::MAX_ACC;
  uint64_t* w_full = acc_empty + cv::MAX_ACC;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w_full + 1);
  float* bw_mu = reinterpret_cast<float*>(tmem_slot + 4);  // [64]
  float* bw_rs = bw_mu + 64;                                // [64]

  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const int g = blockIdx.y, cpr = gridDim.x;
  const int tiles = a.P / BM;  // per replica
  const int per_img = a.hout * a.wout;
  const int nacc = a.nacc, nsplit = a.nsplit;
  const uint32_t acc_cols = (uint32_t)(nsplit * np);  // one accumulator buffer
  const uint32_t tmem_cols = conv_tmem_cols(nacc * nsplit, np);

  if (threadIdx.x == 0) {
    for (int i = 0; i < nst; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < nacc; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], 4);  // one arrival per epilogue warp
    }
    mbar_init(w_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  pdl_begin();  // everything above touched only shared memory and TMEM

  if (warp == 0) {
    // ---------------- producer ----------------
    const bool el = elect_one();
    if (el) {
      mbar_expect_tx(w_full, 9 * wtap);
      for (int t = 0; t < 9; ++t) tma_load_3d(wsm + t * wtap, &a.w_map, w_full, t * ck, 0, g);
    }
    // a tile's first image and row; the next one is cpr tiles on: step_b images and step_y rows (walked
    // image by image that is 512 steps for a single replica of 512 images of 16 x 16 pixels, 32 -> 64
    // channels at stride 2: forward 10.0 us against 7.2)
    const int rows_img = a.hout, row_step = cpr * (BM / a.wout);
    const int step_b = row_step / rows_img, step_y = row_step - step_b * rows_img;
    int b0 = (int)blockIdx.x * BM / per_img, y = (int)blockIdx.x * BM % per_img / a.wout;
    int q = 0, sl = 0;
    uint32_t ph = 1;
    bool ok = true;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += cpr) {
      for (int sp = 0; sp < spt; ++sp, ++q) {
        if (!mbar_wait_warp(&empty[sl], ph)) {
          ok = false;
          break;
        }
        // strip: rows y - 1 .. y + rows (the halo rows out of the image read as zeros);
        // per kernel row sp: the rows under kernel row sp
        const int y0 = a.strip ? y - 1 : y * a.stride + sp - 1;
        if (el) {
          mbar_expect_tx(&full[sl], stage_bytes);
          uint8_t* st = ring + sl * stage_bytes;
          tma_load_5d(st, &a.in_map, &full[sl], 0, -1, y0, b0, g);
          tma_load_5d(st + box_bytes, &a.in_map, &full[sl], 0, 0, y0, b0, g);
          tma_load_5d(st + 2 * box_bytes, &a.in_map, &full[sl], 0, 1, y0, b0, g);
        }
        if (++sl == nst) {
          sl = 0;
          ph ^= 1;
        }
      }
      y += step_y;
      b0 += step_b;
      if (y >= rows_img) {
        y -= rows_img;
        ++b0;
      }
    }
    // copies in flight land before the CTA can exit
    mbar_wait(w_full, 0);
    for (int j = (q > nst ? q - nst : 0); j < q; ++j) mbar_wait(&full[j % nst], (j / nst) & 1);
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const bool el = elect_one();
    const uint32_t idesc = make_idesc(BM, np, false, false);
    const uint32_t swz = (uint32_t)ck * 2;
    // descriptors of the ring's start and of tap 0's weights: the address field is in 16-byte
    // units, so the descriptor of a tap / stage / K-step is the base plus its byte offset / 16
    const uint64_t a_desc0 = smem_desc_kmajor(smem_u32(ring), swz);
    const uint64_t b_desc0 = smem_desc_kmajor(smem_u32(wsm), swz);
    const uint32_t kw_step = box_bytes >> 4, kh_step = (a.strip ? row_bytes : 0u) >> 4;
    const uint32_t tap_step = wtap >> 4;
    const bool split3 = nsplit == 3;
    const uint32_t acc_kw = split3 ? (uint32_t)np : 0u;
    bool ok = mbar_wait_warp(w_full, 0);
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    int sl = 0, ab = 0;
    uint32_t ph = 0, ph_acc = 1;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += cpr) {
      if (!mbar_wait_warp(&acc_empty[ab], ph_acc)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint32_t acc = tmem + (uint32_t)ab * acc_cols;
      for (int sp = 0; sp < spt; ++sp) {
        if (!mbar_wait_warp(&full[sl], ph)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const uint64_t st_desc = a_desc0 + ((uint32_t)sl * stage_bytes >> 4);
#pragma unroll
        for (int kh = 0; kh < 3; ++kh) {
          if (!a.strip && kh != sp) continue;
          const uint64_t row_desc = st_desc + (uint32_t)kh * kh_step;
          const uint64_t tap_desc = b_desc0 + (uint32_t)(3 * kh) * tap_step;
#pragma unroll
          for (int kk = 0; kk < 4; ++kk) {
            if (16 * kk >= ck) break;
#pragma unroll
            for (int kw = 0; kw < 3; ++kw) {
              // partial kw (nsplit = 3) starts at its first kernel row; a single accumulator at
              // the first tap
              const bool first = kk == 0 && kh == 0 && (kw == 0 || split3);
              if (el)
                mma_bf16(acc + kw * acc_kw, row_desc + (uint32_t)kw * kw_step + (uint32_t)(2 * kk),
                         tap_desc + (uint32_t)kw * tap_step + (uint32_t)(2 * kk), idesc,
                         first ? 0u : 1u);
            }
          }
        }
        // strip form: the epilogue releases the stage once it sees the tile's accumulator (one
        // commit per tile); per kernel row: the stage is released as soon as its MMAs complete
        if (!a.strip && el) mma_commit(&empty[sl]);
        if (++sl == nst) {
          sl = 0;
          ph ^= 1;
        }
      }
      if (ok && el) mma_commit(&acc_full[ab]);
      if (++ab == nacc) {
        ab = 0;
        ph_acc ^= 1;
      }
    }
  } else if (warp >= 4) {
    // ---------------- epilogue ----------------
    // The four epilogue warps do not wait for one another: each waits for a tile's accumulator
    // itself (every lane polls; the warp goes on only if all lanes saw the phase, so a wait that
    // runs out never splits a warp-wide tensor-memory load) and gives it back with one arrival.
    const int quarter = warp & 3, r = quarter * 32 + lane;
    // per-channel BatchNorm statistics of the output pixels (forward convolutions), per
    // epilogue warp: lanes 2 j, 2 j + 1 keep channel 16 ci + j's running count, mean and M2 over
    // the warp's 32 rows of every tile
    const bool with_stats = a.stats != nullptr;
    float run_n = 0.f, run_mu[4] = {0.f, 0.f, 0.f, 0.f}, run_m2[4] = {0.f, 0.f, 0.f, 0.f};
    // the data gradient's BatchNorm-backward epilogue (a.bwd): that layer's mean and rstd in
    // shared memory; lanes 2 j, 2 j + 1 keep channel 16 ci + j's running sums of g and g xhat
    const ConvBwdFuse& bw = a.bwd;
    const bool with_bwd = bw.y != nullptr;
    const int dx_h = a.dst_h > 0 ? a.dst_h : a.hout, dx_w = a.dst_w > 0 ? a.dst_w : a.wout;
    float run_g[4] = {0.f, 0.f, 0.f, 0.f}, run_gx[4] = {0.f, 0.f, 0.f, 0.f};
    if (with_bwd) {
      const int et = threadIdx.x - cv::EPI0;
      if (et < a.N) {
        bw_mu[et] = bw.mean[g * a.N + et];
        bw_rs[et] = bw.rstd[g * a.N + et];
      }
      asm volatile("bar.sync 1, 128;" ::: "memory");
    }
    int ab = 0, sl = 0;  // the tile's accumulator and (strip form) input stage
    uint32_t ph = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += cpr) {
      if (!mbar_wait_warp(&acc_full[ab], ph)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      // strip form: this tile's MMAs (and so its reads of its input stage) are complete
      if (a.strip && quarter == 0 && lane == 0) mbar_arrive(&empty[sl]);
      if (++sl == nst) sl = 0;
      int64_t dst = (int64_t)tile * BM + r;
      if (a.dst_h > 0) {
        const int pp = tile * BM + r, img = pp / per_img, rem = pp - img * per_img;
        const int oy = rem / a.wout, ox = rem - oy * a.wout;
        dst = ((int64_t)img * a.dst_h + 2 * oy + a.ph_y) * a.dst_w + 2 * ox + a.ph_x;
      }
      float* orow = a.out + (int64_t)g * a.out_gs + dst * a.N;
      // the shortcut's source pixel in the block output (stride 1: the same pixel; stride 2: the
      // pixels on the stride grid), or -1
      auto sc_pixel = [&](int64_t d) -> int64_t {
        if (!bw.sc_dout) return -1;
        const int img = (int)(d / ((int64_t)dx_h * dx_w)), rem = (int)(d % ((int64_t)dx_h * dx_w));
        const int iy = rem / dx_w, ix = rem - iy * dx_w;
        if (bw.sc_stride == 1) return d;
        if ((iy & 1) || (ix & 1)) return -1;
        return ((int64_t)img * (dx_h / 2) + iy / 2) * (dx_w / 2) + ix / 2;
      };
      int64_t sc_px = with_bwd ? sc_pixel(dst) : -1;
      if (with_bwd && tile + cpr < tiles) {
        // this thread's row of the next tile into L1 while this tile is processed: the loads
        // below would otherwise each wait on DRAM
        const int nt = tile + cpr;
        int64_t nd = (int64_t)nt * BM + r;
        if (a.dst_h > 0) {
          const int pp = nt * BM + r, img = pp / per_img, rem = pp - img * per_img;
          const int oy = rem / a.wout, ox = rem - oy * a.wout;
          nd = ((int64_t)img * a.dst_h + 2 * oy + a.ph_y) * a.dst_w + 2 * ox + a.ph_x;
        }
        const int64_t ne = (int64_t)g * a.out_gs + nd * a.N;
        for (int b = 0; b < a.N * 2; b += 128)
          asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(bw.mask + ne) + b));
        for (int b = 0; b < a.N * 4; b += 128)
          asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(bw.y + ne) + b));
        const int64_t ns = sc_pixel(nd);
        if (ns >= 0) {
          const int64_t se = (int64_t)g * bw.sc_gs + ns * bw.sc_C;
          for (int b = 0; b < a.N * 4; b += 128)
            asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(bw.sc_dout + se) + b));
          for (int b = 0; b < a.N * 2; b += 128)
            asm volatile("prefetch.global.L1 [%0];" ::"l"(reinterpret_cast<const char*>(bw.sc_out + se) + b));
        }
      }
#pragma unroll
      for (int ci = 0; ci < 4; ++ci) {
        const int c0 = 16 * ci;
        if (c0 >= a.N) break;
        float v[16];
        const uint32_t tl = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)ab * acc_cols + c0;
        if (nsplit == 3) {
          // the three column partials, added in column order
          float u1[16], u2[16];
          tmem_ld16x3(tl, tl + (uint32_t)np, tl + (uint32_t)(2 * np), v, u1, u2);
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = (v[j] + u1[j]) + u2[j];
        } else {
          tmem_ld16(tl, v);
        }
        if (with_bwd) {
          // dx (+ the shortcut's share) masked by the layer below's ReLU, and that layer's
          // BatchNorm-backward sums over this warp's rows
          if (sc_px >= 0) {
            const float4* sd = reinterpret_cast<const float4*>(
                bw.sc_dout + (int64_t)g * bw.sc_gs + sc_px * bw.sc_C + c0);
            const uint4* so = reinterpret_cast<const uint4*>(
                bw.sc_out + (int64_t)g * bw.sc_gs + sc_px * bw.sc_C + c0);
#pragma unroll
            for (int h = 0; h < 2; ++h) {
              const uint4 o8 = __ldg(so + h);
              const float4 d0 = __ldg(sd + 2 * h), d1 = __ldg(sd + 2 * h + 1);
              const uint32_t ow[4] = {o8.x, o8.y, o8.z, o8.w};
              const float dd[8] = {d0.x, d0.y, d0.z, d0.w, d1.x, d1.y, d1.z, d1.w};
#pragma unroll
              for (int k = 0; k < 8; ++k) {
                const float o = bf2f((uint16_t)(k & 1 ? ow[k >> 1] >> 16 : ow[k >> 1] & 0xffffu));
                v[8 * h + k] += o > 0.f ? dd[k] : 0.f;
              }
            }
          }
          const uint4* mk = reinterpret_cast<const uint4*>(bw.mask + (int64_t)g * a.out_gs + dst * a.N + c0);
          const float4* yv = reinterpret_cast<const float4*>(bw.y + (int64_t)g * a.out_gs + dst * a.N + c0);
          float gx[16];
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const uint4 m8 = __ldg(mk + h);
            const float4 y0 = __ldg(yv + 2 * h), y1 = __ldg(yv + 2 * h + 1);
            const uint32_t mw[4] = {m8.x, m8.y, m8.z, m8.w};
            const float yy[8] = {y0.x, y0.y, y0.z, y0.w, y1.x, y1.y, y1.z, y1.w};
#pragma unroll
            for (int k = 0; k < 8; ++k) {
              const int j = 8 * h + k;
              const float m = bf2f((uint16_t)(k & 1 ? mw[k >> 1] >> 16 : mw[k >> 1] & 0xffffu));
              v[j] = m > 0.f ? v[j] : 0.f;
              gx[j] = v[j] * ((yy[k] - bw_mu[c0 + j]) * bw_rs[c0 + j]);
            }
          }
          float t[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) t[j] = v[j];
          run_g[ci] += warp_colsum16(t, lane);
          run_gx[ci] += warp_colsum16(gx, lane);
        }
        if (a.st32) {
          // whole 32-byte sectors per lane and instruction
#pragma unroll
          for (int j = 0; j < 2; ++j)
            asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(
                             orow + c0 + 8 * j),
                         "f"(v[8 * j]), "f"(v[8 * j + 1]), "f"(v[8 * j + 2]), "f"(v[8 * j + 3]),
                         "f"(v[8 * j + 4]), "f"(v[8 * j + 5]), "f"(v[8 * j + 6]), "f"(v[8 * j + 7])
                         : "memory");
        } else {
#pragma unroll
          for (int j = 0; j < 4; ++j)
            *reinterpret_cast<float4*>(orow + c0 + 4 * j) =
                make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
        }
        if (with_stats) {
          // this warp's 32 pixels of the tile: mean, then the sum of squared deviations from
          // it (two passes over the registers), each summed over the warp's lanes
          float t[16];
#pragma unroll
          for (int j = 0; j < 16; ++j) t[j] = v[j];
          const float mt = warp_colsum16(t, lane) * (1.f / 32);
#pragma unroll
          for (int j = 0; j < 16; ++j) {
            const float e = v[j] - __shfl_sync(0xffffffffu, mt, 2 * j);
            t[j] = e * e;
          }
          const float m2t = warp_colsum16(t, lane);
          // Chan et al.'s combination of the running (n, mean, M2) with these 32 pixels'
          const float nt = run_n + 32.f, f = 32.f / nt, delta = mt - run_mu[ci];
          run_mu[ci] = fmaf(delta, f, run_mu[ci]);
          run_m2[ci] = run_m2[ci] + m2t + delta * delta * run_n * f;
        }
      }
      if (with_stats) run_n += 32.f;
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&acc_empty[ab]);
      if (++ab == nacc) {
        ab = 0;
        ph ^= 1;
      }
    }
    if (with_bwd && !(lane & 1)) {
#pragma unroll
      for (int ci = 0; ci < 4; ++ci) {
        if (16 * ci >= a.N) break;
        bw.part[((int64_t)g * bw.part_gs + bw.part_off + 4 * blockIdx.x + quarter) * a.N + 16 * ci +
                (lane >> 1)] = make_float2(run_g[ci], run_gx[ci]);
      }
    }
    if (with_stats && !(lane & 1)) {
      // one partial per epilogue warp: stats[g][4 q + quarter]
#pragma unroll
      for (int ci = 0; ci < 4; ++ci) {
        if (16 * ci >= a.N) break;
        a.stats[((int64_t)g * cpr * 4 + 4 * blockIdx.x + quarter) * a.N + 16 * ci + (lane >> 1)] =
            make_float4(run_n, run_mu[ci], run_m2[ci], 0.f);
      }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols)
                 : "memory");
  }
}


// =============================================================================================
// The 3x3 convolutions of images whose rows are 512 channel values (32 x 16, 16 x 32 or 8 x 64
// channels: every ResNet-20 stage), persistent, 64 / ck neighbouring pixels as one 64-channel
// "super-pixel": an image row is then eight 128-byte rows -- one row group of a K-major operand --
// and the next image row the next group.  A tile is TR = 16 or 8 image rows (M = 128 or 64 rows of
// super-pixels) and its whole input, halo included, is ONE box of (TR - 1) S + 3 rows of ten
// super-pixels: tap rows are a row further, and the 16-channel slices from the pixel left of the
// super-pixel to the one right of it follow one another in memory, so a product's operand is the
// box read from a shifted start (the hardware swizzles address bits).  The weights are laid out per
// slice as [output pixel, output channel][16] with zeros where the slice is not under the tap (a
// block Toeplitz matrix), by every CTA from the packed weights.
// What it buys at 16 channels over one pixel per row (conv_tc_kernel): a product has N = 64 columns
// (48 cycles) for four pixels instead of N = 16 (39) for one; the box has 180 128-byte rows per 512
// pixels instead of 2,304 32-byte ones, whose TMA rate bound that kernel; a thread owns four
// pixels (256 contiguous bytes), so the statistics' warp sums run once per four.
// A stride-2 data gradient's four parity phases are one such product: output row parity = 64-column
// segment, column parity = alternate pixels, taps of kernel rows 1 and 2 of the phase weights.
//   warp 0      TMA producer           warp 1      MMA issuer
//   warp 2      TMEM allocation        warps 1-7   weight layout at the start
//   warps 4-7   epilogue
// The epilogue reads TMEM in the 16 x 256-bit shape, which gives a row to four lanes, and the weight
// rows (= columns) are laid out so that each of them gets two runs of eight consecutive outputs: the
// four write (and read, for the BatchNorm backward) whole 128-byte lines.  With a row per lane every
// 32-byte access of a warp touched 32 lines, and the L1's line rate bound the BatchNorm-backward
// epilogue at 107 us (141 with the shortcut) for a first-stage layer of 16 workers x 128 images.
// A lane then also holds few channels (8, or 16 of 64), so running moments and sums stay in its
// registers until the end of the kernel: no exchange per tile.
// Measured there: forward with statistics 41 us (201 MB: 4.9 TB/s), data gradient with the
// BatchNorm-backward epilogue 66 (402 MB: 6.1 TB/s), 104 with the shortcut, where conv_tc_kernel took
// 65, 102 and 135.
// 16 outputs or 64 inputs to a pixel: each kernel row has partial columns of its own (npart), added by the
// epilogue, which hands them back as soon as they are in registers.  A tensor-core sum rounds with every
// product added: one chain over the kernel rows was off by 8.5e-8 and 3.0e-7 (relative, 16 and 64
// channels, forward; 4.8e-7 the 64-channel data gradient) where three are off by 4.9e-8, 1.1e-7 and
// 1.7e-7, as conv_tc_kernel is.  It cost 7.41 -> 7.79 ms for two ResNet-20 steps: fewer tiles in TMEM.  The
// partials are read eight registers at a time (sixteen spilled: 8.05 ms).
// The BatchNorm-backward epilogue reads up to 192 bytes for every 64 it writes, and four warps that
// went through a tile's rows one after another were bound by the latency of those reads (102 us, 158
// with the shortcut): its sixteen warps (eight of an M = 64 tile) take 16 rows x 32 columns each, on
// one CTA per SM, and request all they read of a tile before they wait for its accumulator.
namespace sp {
template <int M, int MODE>
constexpr int kEpq = MODE == 2 ? M / 32 : 1;  // epilogue warps per TMEM lane quarter
template <int M, int MODE>
constexpr int kThreads = 128 + 128 * kEpq<M, MODE>;
constexpr int MAX_ST = 6;
constexpr size_t kTwoPerSm = 113 * 1024, kOnePerSm = 224 * 1024;
constexpr int BOX_W = 10;                    // super-pixels of a box row
constexpr uint32_t ROWB = BOX_W * 128;       // bytes of a box row
constexpr size_t AUX = (2 * MAX_ST + 2 * cv::MAX_ACC + 1) * 8 + 16;
}  // namespace sp

// Eight consecutive values (32-byte aligned) in one access.
__device__ __forceinline__ void ld8(const float* p, float* v) {
  asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]),
                 "=f"(v[7])
               : "l"(p));
}
__device__ __forceinline__ void st8(float* p, const float* v) {
  asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "f"(v[0]), "f"(v[1]),
               "f"(v[2]), "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}
// Sixteen TMEM lanes x 64 columns: lane l of the warp gets, of rows l / 4 and l / 4 + 8, columns
// 8 k + 2 (l mod 4) and the next for k < 8: v[4 k .. 4 k + 3] = row l / 4's two, then row l / 4 + 8's.
__device__ __forceinline__ void tmem_ld_16x256_x8(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x8.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}
// The same for 32 columns.
__device__ __forceinline__ void tmem_ld_16x256_x4(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x4.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}
// And for 16.
__device__ __forceinline__ void tmem_ld_16x256_x2(uint32_t taddr, float (&v)[8]) {
  uint32_t r[8];
  asm volatile(
      "tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
      : "r"(taddr)
      : "memory");
#pragma unroll
  for (int i = 0; i < 8; ++i) v[i] = __uint_as_float(r[i]);
}
// The partial accumulators np columns apart beyond the first, added in order.
template <int NV>
__device__ __forceinline__ void tmem_add_16x256(uint32_t at, int npart, int np, float (&v)[NV]) {
#pragma unroll 1
  for (int p = 1; p < npart; ++p) {
#pragma unroll
    for (int i = 0; i < NV / 8; ++i) {
      float q[8];
      tmem_ld_16x256_x2(at + (uint32_t)(p * np + 16 * i), q);
#pragma unroll
      for (int k = 0; k < 8; ++k) v[8 * i + k] += q[k];
    }
  }
}
__device__ __forceinline__ bool bf_positive(const uint32_t (&w)[4], int k) {
  return bf2f((uint16_t)(k & 1 ? w[k >> 1] >> 16 : w[k >> 1] & 0xffffu)) > 0.f;
}

// MODE 0: plain, 1: BatchNorm statistics, 2: BatchNorm-backward epilogue.  A32: the output is 32-byte
// aligned; at 16 bytes (a caller's view) the same products and sums, and so the same bits, leave in 128-bit
// stores.  A branch around each store instead took conv3x3 forward + data gradient + weight gradient of 16
// workers x 128 first-stage images from 137 to 141 us.
template <int M, int MODE, bool A32 = true>
__global__ void __launch_bounds__(sp::kThreads<M, MODE>, MODE == 2 ? 1 : 2) conv_sp_kernel(
    const __grid_constant__ ConvSpArgs a) {
  constexpr int EPQ = sp::kEpq<M, MODE>, THREADS = sp::kThreads<M, MODE>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const int ck = a.ck, ks = ck / 16, nst = a.nst, nacc = a.nacc;
  const int np = 64 * a.nseg, npart = a.npart;       // a partial accumulator's columns; partials of a tile
  const int per_row = a.nj * ks, nmma = a.nkh * per_row;
  const uint32_t box_bytes = (uint32_t)a.box_rows * sp::ROWB, pitch = (box_bytes + 1023u) & ~1023u;
  const uint32_t slice_bytes = (uint32_t)np * 32u;   // one slice's weights
  uint8_t* wsm = base + nst * pitch;
  uint64_t* full = reinterpret_cast<uint64_t*>(wsm + nmma * slice_bytes);
  uint64_t* empty = full + sp::MAX_ST;
  uint64_t* acc_full = empty + sp::MAX_ST;
  uint64_t* acc_empty = acc_full + cv::MAX_ACC;
  uint64_t* w_full = acc_empty + cv::MAX_ACC;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(w_full + 1);
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const int g = blockIdx.y, cpr = gridDim.x;
  const int tpi = a.hg / a.tr, tiles = a.B * tpi;  // tiles per image, per replica
  const uint32_t tmem_cols = conv_tmem_cols(nacc * npart, np);

  if (threadIdx.x == 0) {
    for (int i = 0; i < nst; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    for (int i = 0; i < nacc; ++i) {
      mbar_init(&acc_full[i], 1);
      mbar_init(&acc_empty[i], 4 * EPQ);
    }
    mbar_init(w_full, THREADS / 32 - 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  pdl_begin();  // everything above touched only shared memory and TMEM

  // from tile t of image b to the CTA's next one, cpr tiles on (walked image by image, a single replica's
  // 304 CTAs are as many steps per tile of 8 x 8 pixels: 512 images of 64 channels, forward 18.1 us against
  // 11.2)
  const int step_b = cpr / tpi, step_t = cpr - step_b * tpi;
  auto next_tile = [&](int& b, int& t) {
    t += step_t;
    b += step_b;
    if (t >= tpi) {
      t -= tpi;
      ++b;
    }
  };
  // an epilogue warp has read all that it reads of a tile's accumulators
  auto give_back = [&](int ab) {
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(&acc_empty[ab]);
  };
  if (warp > 0) {
    // the weights: 16-byte chunk e = (slice, column n, half of its 16 channels), kWU of a thread's chunks
    // requested together; sizes are powers of two and slices few, so nothing is divided.  (One load at a
    // time with four divisions: 11.7 us for 8 images of 8 x 8 pixels, 64 channels, against 5.7.)
    constexpr int kWU = 8;
    const uint16_t* w = a.w + (int64_t)g * a.w_gs;
    const int total = nmma * np * 2, np_log2 = 5 + a.nseg, ks_log2 = ks >> 1, n_log2 = 31 - __clz(a.N);
    const uint32_t inv_row = 65536u / (uint32_t)per_row + 1u;  // sl / per_row = sl inv_row / 65536: sl < 64
    for (int e0 = threadIdx.x - 32; e0 < total; e0 += kWU * (THREADS - 32)) {
      uint4 v[kWU];
      uint32_t dst[kWU];
#pragma unroll
      for (int i = 0; i < kWU; ++i) {
        const int e = e0 + i * (THREADS - 32);
        const int h = e & 1, n = (e >> 1) & (np - 1), sl = e >> (1 + np_log2);
        const int khi = (int)((uint32_t)sl * inv_row >> 16), r = sl - khi * per_row;
        const int jj = r >> ks_log2, kq = r & (ks - 1);
        // column n of a segment is output o of its 64: lane m = (n mod 8) / 2 of a row's four holds
        // columns 8 k + 2 m, + 1, which are to be outputs 32 i + 8 m + r, r = 2 (k mod 4) + n mod 2
        const int seg = n >> 6, o = (n & 32) + ((n & 6) << 2) + ((n >> 2) & 6) + (n & 1);
        const int px = o >> n_log2, ch = o & (a.N - 1);
        // segment and pixel of a column -> source pixel p and (phases) which phase's weights
        const int p = a.nseg == 2 ? px >> 1 : px, phase = a.nseg == 2 ? 2 * seg + (px & 1) : 0;
        const int d = a.j0 + jj - p * a.S;  // kernel column
        v[i] = make_uint4(0u, 0u, 0u, 0u);
        if (e < total && d >= 0 && d <= 2)
          v[i] = __ldg(reinterpret_cast<const uint4*>(
              w + phase * a.w_ps + (ch * 9 + (a.kh0 + khi) * 3 + d) * ck + kq * 16 + h * 8));
        dst[i] = (uint32_t)sl * slice_bytes + (uint32_t)(n * 32 + ((h ^ ((n >> 2) & 1)) << 4));
      }
#pragma unroll
      for (int i = 0; i < kWU; ++i)
        if (e0 + i * (THREADS - 32) < total) *reinterpret_cast<uint4*>(wsm + dst[i]) = v[i];
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    __syncwarp();
    if (lane == 0) mbar_arrive(w_full);
  }

  if (warp == 0) {
    // ---------------- producer ----------------
    const bool el = elect_one();
    int b = (int)blockIdx.x / tpi, t = (int)blockIdx.x % tpi;
    int q = 0, sl = 0;
    uint32_t ph = 1;
    for (int tile = blockIdx.x; tile < tiles; tile += cpr, ++q) {
      if (!mbar_wait_warp(&empty[sl], ph)) break;
      if (el) {
        mbar_expect_tx(&full[sl], box_bytes);
        tma_load_5d(base + sl * pitch, &a.in_map, &full[sl], 0, -1, t * a.tr * a.S + a.kh0 - 1, b, g);
      }
      if (++sl == nst) {
        sl = 0;
        ph ^= 1;
      }
      next_tile(b, t);
    }
    // copies in flight land before the CTA can exit
    for (int j = (q > nst ? q - nst : 0); j < q; ++j) mbar_wait(&full[j % nst], (j / nst) & 1);
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const bool el = elect_one();
    const uint32_t idesc = make_idesc(M, np, false, false);
    // slice j0 of box row 0: the pixels before it in the super-pixel left of the tile's first
    const uint64_t a_desc0 =
        smem_desc_swz(smem_u32(base) + 128 - 2 * ck + a.j0 * 2 * ck, 16, (uint32_t)a.S * sp::ROWB, 128);
    const uint64_t b_desc0 = smem_desc_kmajor(smem_u32(wsm), 32);
    const uint32_t b_step = slice_bytes >> 4;
    bool ok = mbar_wait_warp(w_full, 0);
    int sl = 0, ab = 0;
    uint32_t ph = 0, ph_acc = 1;
    for (int tile = blockIdx.x; tile < tiles && ok; tile += cpr) {
      if (!mbar_wait_warp(&acc_empty[ab], ph_acc) || !mbar_wait_warp(&full[sl], ph)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      uint32_t acc = tmem + (uint32_t)(ab * npart * np);
      const uint64_t st = a_desc0 + ((uint32_t)sl * pitch >> 4);
      uint64_t bd = b_desc0;
      uint32_t on = 0;
      for (int kh = 0; kh < a.nkh; ++kh) {
        if (kh > 0 && npart > 1) {
          acc += (uint32_t)np;
          on = 0;
        }
        uint64_t ad = st + (uint32_t)kh * (sp::ROWB >> 4);
#pragma unroll 4
        for (int r = 0; r < per_row; ++r) {
          if (el) mma_bf16(acc, ad, bd, idesc, on);
          on = 1;
          ad += 2;
          bd += b_step;
        }
      }
      if (el) {
        mma_commit(&empty[sl]);
        mma_commit(&acc_full[ab]);
      }
      if (++sl == nst) {
        sl = 0;
        ph ^= 1;
      }
      if (++ab == nacc) {
        ab = 0;
        ph_acc ^= 1;
      }
    }
  } else if (MODE == 2 && warp >= 4) {
    // ---------------- BatchNorm-backward epilogue ----------------
    // Warp (h, i) of a quarter: rows 16 h .. 16 h + 15 (two image rows) and outputs 32 i .. 32 i + 31 of
    // a segment; lane = (super-pixel sx, part m) with outputs 32 i + 8 m + r of both image rows.
    const int quarter = warp & 3, hi = (warp - 4) >> 2, h = hi >> 1, i = hi & 1;
    const int sx = lane >> 2, m = lane & 3;
    const int N = a.N, ps = 64 / N;  // pixels of a segment
    const ConvBwdFuse& bw = a.bwd;
    const int o = 32 * i + 8 * m, px = o / N, ch = o & (N - 1);  // this lane's pixel and first channel
    float sg[8], sgx[8], mu[8];  // sums of g and g (y - mean); the mean
#pragma unroll
    for (int r = 0; r < 8; ++r) {
      sg[r] = sgx[r] = 0.f;
      mu[r] = bw.mean[g * N + ch + r];
    }
    int b = (int)blockIdx.x / tpi, t = (int)blockIdx.x % tpi;
    int ab = 0;
    uint32_t ph = 0;
    // this lane's first output of image row `row` (0, 1) and segment seg of tile (b, t), in pixels
    auto pixel = [&](int bb, int tt, int row, int seg) -> int64_t {
      return ((int64_t)bb * a.ho + (tt * a.tr + quarter * (M / 32) + 2 * h + row) * a.rs + seg) * a.wo +
             sx * ps;
    };
    for (int tile = blockIdx.x; tile < tiles; tile += cpr) {
      const int img = b, tt = t;
      next_tile(b, t);
      bool ok = true;
      for (int seg = 0; seg < a.nseg; ++seg) {
        uint4 mk[2], so[2];
        float yv[2][8], sd[2][8];
        bool has = false;
#pragma unroll
        for (int row = 0; row < 2; ++row) {
          const int64_t pix = pixel(img, tt, row, seg);
          const int64_t e = (int64_t)g * a.out_gs + pix * N + o;
          mk[row] = *reinterpret_cast<const uint4*>(bw.mask + e);
          ld8(bw.y + e, yv[row]);
          if (bw.sc_dout) {
            // the shortcut's source pixel: the same one (stride 1) or, in even rows, every other
            // pixel's (stride 2: segment 0 is the even row)
            int64_t src = pix + px;
            has = true;
            if (bw.sc_stride == 2) {
              has = seg == 0 && !(px & 1);
              src = ((int64_t)img * (a.ho / 2) + tt * a.tr + quarter * (M / 32) + 2 * h + row) * (a.wo / 2) +
                    (sx * ps + px) / 2;
            }
            if (has) {
              const int64_t se = (int64_t)g * bw.sc_gs + src * bw.sc_C + ch;
              so[row] = *reinterpret_cast<const uint4*>(bw.sc_out + se);
              ld8(bw.sc_dout + se, sd[row]);
            }
          }
        }
        if (tile + cpr < tiles) {
          // the next tile's into L2
#pragma unroll
          for (int row = 0; row < 2; ++row) {
            const int64_t pix = pixel(b, t, row, seg);
            const int64_t e = (int64_t)g * a.out_gs + pix * N + o;
            if (m == 0) {
              asm volatile("prefetch.global.L2 [%0];" ::"l"(bw.y + e));
              if (i == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(bw.mask + e));
              if (bw.sc_dout && bw.sc_stride == 1) {
                const int64_t se = (int64_t)g * bw.sc_gs + (pix + px) * bw.sc_C + ch;
                asm volatile("prefetch.global.L2 [%0];" ::"l"(bw.sc_dout + se));
                if (i == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(bw.sc_out + se));
              }
            }
          }
        }
        if (seg == 0) {
          ok = mbar_wait_warp(&acc_full[ab], ph);
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        }
        float v[16];  // v[4 k + 2 row + b]: column 32 i + 8 k + 2 m + b
        const uint32_t at = tmem + ((uint32_t)(quarter * 32 + 16 * h) << 16) +
                            (uint32_t)(ab * npart * np + 64 * seg + 32 * i);
        tmem_ld_16x256_x4(at, v);
        tmem_add_16x256(at, npart, np, v);
        if (seg == a.nseg - 1) give_back(ab);
#pragma unroll
        for (int row = 0; row < 2; ++row) {
          // dx (+ the shortcut's share) masked by the layer below's ReLU, and that layer's sums
          const uint32_t mw[4] = {mk[row].x, mk[row].y, mk[row].z, mk[row].w};
          const uint32_t ow[4] = {so[row].x, so[row].y, so[row].z, so[row].w};
          float x[8];
#pragma unroll
          for (int r = 0; r < 8; ++r) {
            x[r] = v[4 * (r >> 1) + 2 * row + (r & 1)];
            if (has) x[r] += bf_positive(ow, r) ? sd[row][r] : 0.f;
            x[r] = bf_positive(mw, r) ? x[r] : 0.f;
            sg[r] += x[r];
            sgx[r] = fmaf(x[r], yv[row][r] - mu[r], sgx[r]);
          }
          st8(a.out + (int64_t)g * a.out_gs + pixel(img, tt, row, seg) * N + o, x);
        }
      }
      if (!ok) break;
      if (++ab == nacc) {
        ab = 0;
        ph ^= 1;
      }
    }
    // one partial per warp: the lanes of a channel added in a fixed order (zeros for the channels
    // of the other i)
#pragma unroll
    for (int r = 0; r < 8; ++r) {
#pragma unroll
      for (int d = 4; d <= 16; d <<= 1) {
        sg[r] += __shfl_xor_sync(0xffffffffu, sg[r], d);
        sgx[r] += __shfl_xor_sync(0xffffffffu, sgx[r], d);
      }
      if (N == 16) {
        sg[r] += __shfl_xor_sync(0xffffffffu, sg[r], 2);
        sgx[r] += __shfl_xor_sync(0xffffffffu, sgx[r], 2);
      }
    }
    float2* out = bw.part + ((int64_t)g * bw.part_gs + (int64_t)4 * EPQ * blockIdx.x + (warp - 4)) * N;
    if (sx == 0 && 8 * m < N) {
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        out[ch + r] = make_float2(sg[r], sgx[r] * bw.rstd[g * N + ch + r]);
        if (N == 64) out[(ch ^ 32) + r] = make_float2(0.f, 0.f);
      }
    }
  } else if (MODE != 2 && warp >= 4) {
    // ---------------- epilogue ----------------
    // A warp reads 16 rows of its TMEM lane quarter at a time: two image rows of eight super-pixels
    // each; lane = (super-pixel sx, part m), and m's outputs of a 64-output segment are 32 i + 8 m + r,
    // i < 2, r < 8.  The warps wait for accumulators and return them by themselves.
    const int quarter = warp & 3, sx = lane >> 2, m = lane & 3;
    const int N = a.N, ps = 64 / N;  // pixels of a segment
    // statistics: running mean and sum of squared deviations of the lane's outputs (i, r)
    float mean[2][8], m2[2][8];
    float run_n = 0.f;
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int r = 0; r < 8; ++r) mean[i][r] = m2[i][r] = 0.f;
    int b = (int)blockIdx.x / tpi, t = (int)blockIdx.x % tpi;
    int ab = 0;
    uint32_t ph = 0;
    for (int tile = blockIdx.x; tile < tiles; tile += cpr) {
      const int img = b, y_first = t * a.tr + quarter * (M / 32);  // this warp's first group row
      next_tile(b, t);
      if (!mbar_wait_warp(&acc_full[ab], ph)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll 1
      for (int hs = 0; hs < (M / 64) * a.nseg; ++hs) {
        const int h = a.nseg == 2 ? hs >> 1 : hs, seg = a.nseg == 2 ? hs & 1 : 0;
        float v[32];  // v[4 k + 2 row + b]: column 8 k + 2 m + b of image row `row`
        const uint32_t at =
            tmem + ((uint32_t)(quarter * 32 + 16 * h) << 16) + (uint32_t)(ab * npart * np + 64 * seg);
        tmem_ld_16x256_x8(at, v);
        tmem_add_16x256(at, npart, np, v);
        if (hs == (M / 64) * a.nseg - 1) give_back(ab);
        const int64_t pix0 = ((int64_t)img * a.ho + (y_first + 2 * h) * a.rs + seg) * a.wo + sx * ps;
#pragma unroll
        for (int row = 0; row < 2; ++row) {
          float* orow = a.out + (int64_t)g * a.out_gs + (pix0 + (int64_t)row * a.rs * a.wo) * N + 8 * m;
          float f = 0.f;
          if (MODE == 1) {
            run_n += 1.f;
            f = 1.f / run_n;
          }
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            float x[8];
#pragma unroll
            for (int r = 0; r < 8; ++r) x[r] = v[4 * (4 * i + (r >> 1)) + 2 * row + (r & 1)];
            if constexpr (A32) {
              st8(orow + 32 * i, x);
            } else {
              reinterpret_cast<float4*>(orow + 32 * i)[0] = make_float4(x[0], x[1], x[2], x[3]);
              reinterpret_cast<float4*>(orow + 32 * i)[1] = make_float4(x[4], x[5], x[6], x[7]);
            }
            if (MODE == 1) {
              // Welford's update of the running moments
#pragma unroll
              for (int r = 0; r < 8; ++r) {
                const float d = x[r] - mean[i][r];
                mean[i][r] = fmaf(d, f, mean[i][r]);
                m2[i][r] = fmaf(d, x[r] - mean[i][r], m2[i][r]);
              }
            }
          }
        }
      }
      if (++ab == nacc) {
        ab = 0;
        ph ^= 1;
      }
    }
    if (MODE == 1) {
      // one partial per warp: the lanes that hold the same channel combined in a fixed order, all of
      // them with the same count
      float cnt = run_n;
      auto merge = [&](float& ma, float& sa, float mb, float sb) {
        const float d = ma - mb;
        ma = 0.5f * (ma + mb);
        sa = (sa + sb) + d * d * (0.5f * cnt);
      };
      for (int o = 4; o <= 16; o <<= 1) {
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
          for (int r = 0; r < 8; ++r)
            merge(mean[i][r], m2[i][r], __shfl_xor_sync(0xffffffffu, mean[i][r], o),
                  __shfl_xor_sync(0xffffffffu, m2[i][r], o));
        cnt *= 2.f;
      }
      if (N <= 32) {
#pragma unroll
        for (int r = 0; r < 8; ++r) merge(mean[0][r], m2[0][r], mean[1][r], m2[1][r]);
        cnt *= 2.f;
      }
      if (N == 16) {
#pragma unroll
        for (int r = 0; r < 8; ++r)
          merge(mean[0][r], m2[0][r], __shfl_xor_sync(0xffffffffu, mean[0][r], 2),
                __shfl_xor_sync(0xffffffffu, m2[0][r], 2));
        cnt *= 2.f;
      }
      if (sx == 0 && 8 * m < N)
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          if (32 * i + 8 * m >= N) break;
#pragma unroll
          for (int r = 0; r < 8; ++r)
            a.stats[((int64_t)g * cpr * 4 + 4 * blockIdx.x + quarter) * N + 32 * i + 8 * m + r] =
                make_float4(cnt, mean[i][r], m2[i][r], 0.f);
        }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(tmem_cols)
                 : "memory");
  }
}

// =============================================================================================
// Weight gradient of a 3x3 convolution on the tensor cores, straight from the NHWC operands:
//   dW[g][co][t][ci] = sum over output pixels p of dy[g][p][co] x[g][src_t(p)][ci].
// As D[m][n] = sum_k A[m][k] B[n][k] with k = output pixels, n = co and, for each kernel column kw,
// m = (kh, ci).  Both operands lie in shared memory as TMA writes them, one pixel's channels per
// swizzled row (32, 64 or 128 bytes), i.e. pixel-major = MN-major.  A's three row groups (kh) are
// the same strip of input rows read one image row further each: the descriptor's stride between
// swizzle atoms along m is one strip row.  The kernel column shifts the strip by pixels: the
// hardware swizzles address bits, so a descriptor may start at any pixel of the strip, and one
// strip with its halo serves all nine taps -- no column matrix is ever built.  (A builder that gathered
// it in shared memory, with single-lane issue loops, took 114 us for a first-stage layer of 16
// workers x 128 images (134 MB, 9.7 GFLOP); the strips with such loops 111; with whole-warp loops
// 42: 17 cycles over the tensor core's 23 per M = 64, N = 16 product.)
//
// Per tile of kp (128 or 64) output pixels -- whole rows of one image -- the strip holds the
// (R - 1) S + 3 input rows under it, Wp pixels wide from column -1 on (zeros outside the image by
// TMA's fill).  At stride 2 pixels of one parity are neighbours for the MMA, so two strips hold the
// odd (kw = 0, 2) and the even (kw = 1) columns.  A CTA owns one replica and a contiguous range of
// tiles and keeps the accumulators (per kw: 64 rows of 3 x 16, 128 of 3 x 32, or 128 + 64 of
// 3 x 64 channels) in TMEM; it writes its partial dW, and a second kernel adds the CTAs' partials
// in order.  Rows m beyond the third kernel row multiply whatever lies behind the strip and are
// never read.
//
// Outputs narrower than 8 pixels have no 16 pixels in a row or two, so their tiles run down the image
// columns instead (ConvWgradGeom::cols): a strip row is one column of the input under the tile's
// kp / Wout rows, a box of its own (columns start at whole swizzle atoms: `pitch`), the output-gradient
// tile is Wout columns likewise, and kernel rows and columns change places.  On the fp32 cores, which
// staged 8-pixel rows and left tensor cores idle, 16 workers x 128 images of 64 x 1 pixels and 64 x 64
// channels took 4,332 us, of 16 x 4 pixels 1,094 (a gathered column matrix 31 and 33); so 20 and 23.
//   warp 0      TMA producer (strip(s) + output-gradient tile per stage)
//   warp 1      MMA issuer: per 16 pixels and kernel column one tcgen05.mma (two for 64 channels)
//   warp 2      TMEM allocation
//   warps 0-3   at the end, tcgen05.ld of the accumulators and the partial's stores
namespace cw {
constexpr int THREADS = 128;
constexpr int MAX_ST = 8;            // stages
constexpr uint32_t kTwoPerSm = 113 * 1024;  // shared memory that still fits two CTAs on an SM
constexpr uint32_t kOnePerSm = 224 * 1024;
}  // namespace cw

namespace {
__host__ __device__ inline uint32_t up1k(uint32_t v) { return (v + 1023u) & ~1023u; }
}  // namespace

__global__ void __launch_bounds__(cw::THREADS, 1) conv_wgrad_tc_kernel(
    const __grid_constant__ ConvWgradArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* base = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~uintptr_t(1023));
  const ConvWgradGeom& gm = a.geom;
  const int cin = a.cin, nst = gm.stages;
  const uint32_t rowb = (uint32_t)cin * 2;               // bytes of one pixel
  const uint32_t row_bytes = (uint32_t)gm.pitch * rowb;  // one strip row
  const uint32_t strip_pitch = up1k(gm.rows * row_bytes);
  const uint32_t tile_b = (uint32_t)gm.kp * a.nb * 2;
  const uint32_t stage_pitch = gm.strips * strip_pitch + up1k(tile_b);
  uint64_t* full = reinterpret_cast<uint64_t*>(base + nst * stage_pitch + gm.pad);
  uint64_t* empty = full + cw::MAX_ST;
  uint64_t* acc_full = empty + cw::MAX_ST;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
  const int warp = uniform_warp(), lane = threadIdx.x & 31;
  const int g = blockIdx.y, q = blockIdx.x, cpr = gridDim.x;
  const int ntiles = a.P / gm.kp, per_img = a.hout * a.wout;
  const int t0 = (int)((int64_t)q * ntiles / cpr), nt = (int)((int64_t)(q + 1) * ntiles / cpr) - t0;
  const int mt_n = cin == 64 ? 2 : 1;

  if (threadIdx.x == 0) {
    for (int i = 0; i < nst; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], 1);
    }
    mbar_init(acc_full, 1);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(tmem_slot)),
                 "r"(gm.tmem_cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  pdl_begin();  // everything above touched only shared memory and TMEM

  if (warp == 0) {
    // ---------------- producer ----------------
    const bool el = elect_one();
    int j = 0, s = 0;
    uint32_t ph = 1;
    int p0 = t0 * gm.kp, b = p0 / per_img, y = p0 % per_img / a.wout;  // the tile's image and row
    const int R = gm.kp / a.wout;
    for (; j < nt; ++j) {
      if (!mbar_wait_warp(&empty[s], ph)) break;
      uint8_t* st = base + s * stage_pitch;
      if (el) {
        mbar_expect_tx(&full[s], (uint32_t)(gm.strips * gm.rows * gm.wp) * rowb + tile_b);
        uint8_t* tile = st + gm.strips * strip_pitch;
        if (!gm.cols) {
          tma_load_5d(st, &a.x_map, &full[s], 0, -1, y * a.stride - 1, b, g);
          if (gm.strips == 2) tma_load_5d(st + strip_pitch, &a.x_map, &full[s], 0, 0, y * a.stride - 1, b, g);
          tma_load_3d(tile, &a.dy_map, &full[s], 0, p0, g);
        } else {
          for (int r = 0; r < gm.rows; ++r)
            for (int i = 0; i < gm.strips; ++i)
              tma_load_5d(st + i * strip_pitch + r * row_bytes, &a.x_map, &full[s], 0, r - 1,
                          y * a.stride - 1 + i, b, g);
          for (int x = 0; x < a.wout; ++x)
            tma_load_5d(tile + (uint32_t)(x * gm.inner * a.nb) * 2, &a.dy_map, &full[s], 0, x, y, b, g);
        }
      }
      p0 += gm.kp;
      y += R;
      if (y == a.hout) {
        y = 0;
        ++b;
      }
      if (++s == nst) {
        s = 0;
        ph ^= 1;
      }
    }
    // copies in flight land before the CTA can exit
    for (int i = (j > nst ? j - nst : 0); i < j; ++i) mbar_wait(&full[i % nst], (i / nst) & 1);
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    const bool el = elect_one();
    const int m0 = cin == 16 ? 64 : 128;
    const uint32_t idesc0 = make_idesc(m0, a.nb, true, true), idesc1 = make_idesc(64, a.nb, true, true);
    const uint32_t ux = rowb >> 4;  // one strip pixel in the descriptors' 16-byte units
    // along k: eight pixels to the next core group (a whole output row where rows are 8 wide);
    // along m: one strip row to the next kernel row (columns: kernel column)
    const uint32_t row_px = (uint32_t)gm.pitch * a.stride;  // strip pixels from one output row to the next
    const uint64_t a_desc0 =
        smem_desc_swz(smem_u32(base), row_bytes, (gm.inner == 8 ? row_px : 8u) * rowb, rowb);
    const uint64_t b_desc0 = smem_desc_swz(smem_u32(base) + gm.strips * strip_pitch, 16u * a.nb,
                                           16u * a.nb, 2u * a.nb);
    // kernel column kw (columns: kernel row): which strip and how many pixels into it
    const uint32_t col1 = a.stride == 1 ? ux : strip_pitch >> 4, col2 = a.stride == 1 ? 2 * ux : ux;
    const uint32_t mt_off = 2u * gm.pitch * ux;  // the third row group of 64 channels
    const uint32_t acc_kw = (uint32_t)(mt_n * a.nb);
    const int lw = 31 - __clz(gm.inner);
    bool ok = true;
    int s = 0;
    uint32_t ph = 0, acc = 0;
    for (int j = 0; j < nt; ++j) {
      if (!mbar_wait_warp(&full[s], ph)) {
        ok = false;
        break;
      }
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const uint64_t ad0 = a_desc0 + ((uint32_t)s * stage_pitch >> 4);
      const uint64_t bd0 = b_desc0 + ((uint32_t)s * stage_pitch >> 4);
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if (16 * k >= gm.kp) break;
        // the 16 pixels from 16 k on: their output row and the column in it
        const uint64_t ad = ad0 + (((16u * k) >> lw) * row_px + ((16u * k) & (gm.inner - 1))) * ux;
        const uint64_t bd = bd0 + (uint32_t)(2 * a.nb * k);
        if (el) {
          mma_bf16(tmem, ad, bd, idesc0, acc);
          mma_bf16(tmem + acc_kw, ad + col1, bd, idesc0, acc);
          mma_bf16(tmem + 2 * acc_kw, ad + col2, bd, idesc0, acc);
          if (mt_n == 2) {
            mma_bf16(tmem + a.nb, ad + mt_off, bd, idesc1, acc);
            mma_bf16(tmem + acc_kw + a.nb, ad + col1 + mt_off, bd, idesc1, acc);
            mma_bf16(tmem + 2 * acc_kw + a.nb, ad + col2 + mt_off, bd, idesc1, acc);
          }
        }
        acc = 1;
      }
      if (el) mma_commit(&empty[s]);
      if (++s == nst) {
        s = 0;
        ph ^= 1;
      }
    }
    if (ok && nt > 0 && el) mma_commit(acc_full);
  }
  __syncwarp();

  // ---------------- epilogue ----------------
  if (nt > 0 && __all_sync(0xffffffffu, mbar_wait(acc_full, 0) ? 1 : 0)) {
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    float* out = a.part + ((int64_t)g * cpr + q) * a.cout * 9 * cin;
    for (int t = 0; t < 3; ++t)  // the tap along the strip's rows; th across them
      for (int mt = 0; mt < mt_n; ++mt) {
        // TMEM lane -> row m: all 128 lanes of an M = 128 accumulator, the first 16 of each warp's
        // 32 of an M = 64 one
        const bool half = cin == 16 || mt == 1;
        const int m = half ? warp * 16 + lane : warp * 32 + lane;
        const int th = 2 * mt + m / cin, ci = m % cin, tap = gm.cols ? t * 3 + th : th * 3 + t;
        const bool row_ok = th < 3 && (!half || lane < 16);
        for (int c0 = 0; c0 < a.cout; c0 += 16) {
          float v[16];
          tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)((t * mt_n + mt) * a.nb + c0), v);
          if (row_ok) {
#pragma unroll
            for (int i = 0; i < 16; ++i) out[((int64_t)(c0 + i) * 9 + tap) * cin + ci] = v[i];
          }
        }
      }
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 2) {
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(gm.tmem_cols)
                 : "memory");
  }
}

PFN_cuTensorMapEncodeTiled_v12000 g_encode = nullptr;
std::once_flag g_encode_once;

void load_encode() {
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult q;
  if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &q) ==
          cudaSuccess &&
      q == cudaDriverEntryPointSuccess)
    g_encode = reinterpret_cast<PFN_cuTensorMapEncodeTiled_v12000>(fn);
  else
    cudaGetLastError();
}

int device_sms(int* sms) {
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev);
  return e == cudaSuccess ? dev : -1;
}

template <int BN>
cudaError_t launch_one_tile(const TcGemmArgs& a, dim3 grid, int nk, cudaStream_t stream) {
  int sms = 0;
  const int dev = device_sms(&sms);
  if (dev < 0) return cudaErrorInvalidDevice;
  static std::atomic<int> attr_dev{-1};  // several threads may launch
  if (attr_dev != dev) {
    cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize, 224 * 1024);
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  // shared memory for one, two or three CTAs per SM, by what the grid gives an SM; the ring takes
  // what it needs of it, two to sixteen stages.  (Two CTAs of four 24 KB stages whatever the grid:
  // 64 CTAs, one per SM, took 27,700 cycles for 48 k-blocks.)
  const int64_t ctas = (int64_t)grid.x * grid.y * grid.z;
  const size_t budget = ctas <= sms ? 220 * 1024 : ctas <= 2 * (int64_t)sms || nk > 2 ? 112 * 1024 : 72 * 1024;
  const size_t stage = (a.A.mn_major ? (size_t)BM : (size_t)a.A.box_rows) * BK * 2 + (size_t)BN * BK * 2;
  const size_t fixed = 1024 + sizeof(TcSync);
  TcGemmArgs la = a;
  la.stages = (int)std::min<size_t>({(budget - fixed) / stage, (size_t)std::max(2, nk), (size_t)kTcMaxStages});
  // the product's reads past a short A box stay inside the ring: B tiles follow (two at least)
  static_assert(2 * BN * BK * 2 >= BM * BK * 2, "reads past the last A box end inside the B tiles");
  return launch_pdl(gemm_tc_kernel<BN>, grid, dim3(128), fixed + la.stages * stage, stream, la);
}

}  // namespace

bool tc_available() {
  int dev = 0;
  cudaDeviceProp p;
  if (cudaGetDevice(&dev) != cudaSuccess || cudaGetDeviceProperties(&p, dev) != cudaSuccess) {
    cudaGetLastError();
    return false;
  }
  std::call_once(g_encode_once, load_encode);
  return p.major == 10 && g_encode != nullptr;
}

bool make_tma_map_f32(CUtensorMap* map, const void* base, uint64_t dim0, uint64_t dim1,
                      uint64_t dim2, uint64_t s1, uint64_t s2, uint32_t box0, uint32_t box1) {
  std::call_once(g_encode_once, load_encode);
  if (!g_encode) return false;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || ((s1 * 4) & 15) || ((s2 * 4) & 15)) return false;
  cuuint64_t dims[3] = {dim0, dim1, dim2};
  cuuint64_t strides[2] = {s1 * 4, s2 * 4};
  cuuint32_t box[3] = {box0, box1, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_FLOAT32, 3, const_cast<void*>(base), dims,
                        strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

namespace {
// The expiry path of the GEMM's bounded waits, on its own: one thread waits on an mbarrier phase
// that completes only if `arrive` is set, through the same mbar_wait (limit in SM cycles).
// out = 1 if the phase completed, 0 if the wait ran out (g_tc_timeout is then set).
__global__ void bounded_wait_selftest_kernel(long long limit_cycles, int arrive, int* out) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  if (arrive) mbar_arrive(&bar);
  *out = mbar_wait(&bar, 0, limit_cycles) ? 1 : 0;
}
}  // namespace

cudaError_t launch_bounded_wait_selftest(long long limit_cycles, int arrive, int* out,
                                         cudaStream_t stream) {
  if (limit_cycles < 0 || limit_cycles > kWaitCycles || !out) return cudaErrorInvalidValue;
  bounded_wait_selftest_kernel<<<1, 32, 0, stream>>>(limit_cycles, arrive, out);
  return cudaGetLastError();
}

int tc_take_timeout_flag() {
  int h = 0;
  if (cudaMemcpyFromSymbol(&h, g_tc_timeout, sizeof(int)) != cudaSuccess) {
    cudaGetLastError();
    return 0;
  }
  if (h) {
    const int zero = 0;
    cudaMemcpyToSymbol(g_tc_timeout, &zero, sizeof(int));
  }
  return h;
}

bool make_tma_map_bf16(CUtensorMap* map, const void* base, uint64_t dim0, uint64_t dim1,
                       uint64_t dim2, uint64_t s1, uint64_t s2, uint32_t box0, uint32_t box1) {
  std::call_once(g_encode_once, load_encode);
  if (!g_encode) return false;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || ((s1 * 2) & 15) || ((s2 * 2) & 15)) return false;
  cuuint64_t dims[3] = {dim0, dim1, dim2};
  cuuint64_t strides[2] = {s1 * 2, s2 * 2};
  cuuint32_t box[3] = {box0, box1, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims,
                        strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
                        CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool make_tma_map(CUtensorMap* map, const void* base, bool bf16, uint64_t dim0, uint64_t dim1,
                  uint64_t dim2, uint64_t s1, uint64_t s2, uint32_t box0, uint32_t box1,
                  int swizzle_bytes) {
  std::call_once(g_encode_once, load_encode);
  if (!g_encode) return false;
  const uint64_t esz = bf16 ? 2 : 4;
  if ((reinterpret_cast<uintptr_t>(base) & 15) || ((s1 * esz) & 15) || ((s2 * esz) & 15)) return false;
  CUtensorMapSwizzle sw;
  switch (swizzle_bytes) {
    case 0: sw = CU_TENSOR_MAP_SWIZZLE_NONE; break;
    case 32: sw = CU_TENSOR_MAP_SWIZZLE_32B; break;
    case 64: sw = CU_TENSOR_MAP_SWIZZLE_64B; break;
    case 128: sw = CU_TENSOR_MAP_SWIZZLE_128B; break;
    default: return false;
  }
  if (swizzle_bytes && box0 * esz > (uint64_t)swizzle_bytes) return false;
  cuuint64_t dims[3] = {dim0, dim1, dim2};
  cuuint64_t strides[2] = {s1 * esz, s2 * esz};
  cuuint32_t box[3] = {box0, box1, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = g_encode(map, bf16 ? CU_TENSOR_MAP_DATA_TYPE_BFLOAT16 : CU_TENSOR_MAP_DATA_TYPE_FLOAT32,
                        3, const_cast<void*>(base), dims, strides, box, estr,
                        CU_TENSOR_MAP_INTERLEAVE_NONE, sw, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                        CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

namespace {
// The launch shape of conv_tc_kernel: false if the arguments are not taken.
bool conv_tc_plan(const ConvArgs& a, int sms, int* per_sm, size_t* ring, size_t* smem, int* cpr) {
  if (a.stats && a.dst_h > 0) return false;
  if (a.bwd.y && (!a.bwd.mask || !a.bwd.mean || !a.bwd.rstd || !a.bwd.part ||
                  (a.bwd.sc_dout && (!a.bwd.sc_out || a.bwd.sc_C < a.N ||
                                     (a.bwd.sc_stride != 1 && a.bwd.sc_stride != 2)))))
    return false;
  int rows = 0, images = 0;
  if ((a.ck != 16 && a.ck != 32 && a.ck != 64) || (a.stride != 1 && a.stride != 2) ||
      (a.N != 16 && a.N != 32 && a.N != 64) || a.np != a.N || !a.out || a.G > 65535 ||
      !conv_tile_shape(a.hout, a.wout, &rows, &images) || a.P % (a.hout * a.wout) || a.P % BM ||
      (a.dst_h > 0 && (a.dst_h < 2 * a.hout || a.dst_w < 2 * a.wout || a.ph_y < 0 || a.ph_y > 1 ||
                       a.ph_x < 0 || a.ph_x > 1)))
    return false;
  const size_t fixed = 1024 + 9 * (size_t)a.np * a.ck * 2 + cv::AUX_BYTES;
  const bool strip = a.strip != 0;
  if (strip && !conv_strip_ok(a.hout, a.wout, a.stride)) return false;
  const size_t stage_bytes = 3 * ((size_t)BM + (strip ? 2 * a.wout : 0)) * a.ck * 2;
  const size_t two_budget = 113 * 1024;
  *ring = cv::RING_BYTES;
  *per_sm = 1;
  if (two_budget > fixed && (two_budget - fixed) / stage_bytes >= 3) {
    *ring = std::min<size_t>(cv::RING_BYTES, ((two_budget - fixed) / 1024) * 1024);
    *per_sm = 2;
  }
  if (*per_sm == 1) {
    // one CTA per SM: the ring takes what the weights leave of the 227 KB (at most 24 stages)
    *ring = std::min<size_t>((size_t)cv::MAX_STAGES * stage_bytes,
                             ((cv::SMEM_MAX - fixed) / stage_bytes) * stage_bytes);
  }
  *smem = fixed + *ring;
  // CTAs per replica: as many as fit on the SMs at once over all replicas (one wave), at most one
  // per tile
  *cpr = std::max(1, std::min(a.P / BM, *per_sm * sms / a.G));
  return true;
}

}  // namespace

int conv_tc_ctas(const ConvArgs& a) {
  int sms = 0, per_sm = 1, cpr = 0;
  size_t ring = 0, smem = 0;
  if (a.P <= 0 || a.G <= 0 || device_sms(&sms) < 0) return 0;
  return conv_tc_plan(a, sms, &per_sm, &ring, &smem, &cpr) ? cpr : 0;
}

cudaError_t launch_conv_tc(const ConvArgs& a, cudaStream_t stream, int* ctas_per_replica) {
  if (a.P <= 0 || a.G <= 0) return cudaSuccess;
  int rows = 0, images = 0;
  if ((a.ck != 16 && a.ck != 32 && a.ck != 64) || (a.stride != 1 && a.stride != 2) ||
      (a.N != 16 && a.N != 32 && a.N != 64) || a.np != a.N || !a.out || a.G > 65535 ||
      !conv_tile_shape(a.hout, a.wout, &rows, &images) || a.P % (a.hout * a.wout) || a.P % BM ||
      (a.dst_h > 0 && (a.dst_h < 2 * a.hout || a.dst_w < 2 * a.wout || a.ph_y < 0 || a.ph_y > 1 ||
                       a.ph_x < 0 || a.ph_x > 1)))
    return cudaErrorInvalidValue;
  (void)rows;
  (void)images;
  // Two CTAs per SM where the weights leave room for a ring of at least three stages (a CTA's
  // tiles pass through a chain of handshakes one after another; two CTAs overlap their chains),
  // else one CTA with the full ring (conv_tc_plan).
  int sms = 0, per_sm = 1, cpr = 0;
  size_t ring = 0, smem = 0;
  const int dev = device_sms(&sms);
  if (dev < 0) return cudaErrorInvalidDevice;
  if (!conv_tc_plan(a, sms, &per_sm, &ring, &smem, &cpr)) return cudaErrorInvalidValue;
  cudaError_t e = cudaSuccess;
  ConvArgs la = a;
  la.ring_bytes = (int)ring;
  la.st32 = (reinterpret_cast<uintptr_t>(a.out) & 31) == 0 && a.out_gs % 8 == 0 ? 1 : 0;
  static std::atomic<int> attr_dev{-1};  // several threads may launch
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(conv_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)cv::SMEM_MAX);
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  // accumulators (measured in the ResNet-20 step): four buffers of three column partials where
  // the CTAs on one SM fit in its 512 TMEM columns (16 channels); else four single buffers where
  // they fit (32 channels, two CTAs per SM), else two buffers of three partials (64 channels)
  if (conv_tmem_cols(12, a.np) * per_sm <= 512) {
    la.nacc = 4;
    la.nsplit = 3;
  } else if (conv_tmem_cols(4, a.np) * per_sm <= 512 && per_sm > 1) {
    la.nacc = 4;
    la.nsplit = 1;
  } else {
    la.nacc = 2;
    la.nsplit = conv_tmem_cols(6, a.np) * per_sm <= 512 ? 3 : 1;
  }
  if (ctas_per_replica) *ctas_per_replica = 4 * cpr;  // statistics partials: one per epilogue warp
  return launch_pdl(conv_tc_kernel, dim3(cpr, a.G), dim3(cv::THREADS), smem, stream, la);
}

// The launch shape of conv_sp_kernel; false if it does not take the convolution.
namespace {
bool conv_sp_plan(ConvSpArgs& a, int sms, int* cpr, size_t* smem) {
  if ((a.ck != 16 && a.ck != 32 && a.ck != 64) || (a.N != 16 && a.N != 32 && a.N != 64) || a.wi * a.ck != 512 ||
      (a.stride != 1 && a.stride != 2) || a.B < 1 || a.G < 1 || a.G > 65535)
    return false;
  const int s = 64 / a.ck;  // pixels per super-pixel
  if (a.phases) {
    if (2 * s * a.N != 64 || a.stride != 1) return false;
    a.nseg = 2, a.rs = 2, a.S = 1, a.kh0 = 1, a.nkh = 2, a.j0 = 1, a.nj = s + 1;
    a.hg = a.hi, a.ho = 2 * a.hi, a.wo = 2 * a.wi;
  } else {
    if (a.hi % a.stride || s % a.stride || (s / a.stride) * a.N != 64) return false;
    a.nseg = 1, a.rs = 1, a.S = a.stride, a.kh0 = 0, a.nkh = 3, a.j0 = 0, a.nj = s + 3 - a.stride;
    a.hg = a.ho = a.hi / a.stride, a.wo = a.wi / a.stride;
  }
  if (a.hg % 8) return false;
  // 16 image rows a tile (one M = 128 product costs 1.5 of M = 64) where every SM still gets two
  a.tr = a.hg % 16 == 0 && a.S == 1 && (int64_t)a.G * a.B * (a.hg / 16) >= 2 * sms ? 16 : 8;
  a.box_rows = (a.tr - 1) * a.S + a.nkh;
  const size_t pitch = ((size_t)a.box_rows * sp::ROWB + 1023) / 1024 * 1024;
  const size_t fixed = 1024 + (size_t)a.nkh * a.nj * (a.ck / 16) * 64 * a.nseg * 32 + sp::AUX;
  // Two CTAs per SM, where each still has two stages, overlap one's products with the other's epilogue; but
  // both lay out the weights (up to 73 KB), and alone a CTA has two accumulator sets for that.  So one where
  // it gets at most eight tiles: forward of 1 x 512 images of 32 x 32 pixels, 16 channels, 11.7 -> 10.2 us,
  // data gradient of 16 x 16 pixels, 32 -> 64 at stride 2, 14.2 -> 11.0; forward of 16 x 128 images of that (13
  // tiles) would be 11.4 -> 12.7.  Not with statistics: their partials, one per CTA and warp, stay as they are.
  const bool few = (int64_t)a.G * a.B * (a.hg / a.tr) <= 8LL * sms && !a.stats;
  int per_sm = 2;
  size_t st = sp::kTwoPerSm > fixed ? (sp::kTwoPerSm - fixed) / pitch : 0;
  if (st < 2 || a.bwd.y || few) {
    per_sm = 1;
    st = (sp::kOnePerSm - fixed) / pitch;
  }
  if (st < 2) return false;
  a.nst = (int)std::min<size_t>(st, sp::MAX_ST);
  a.npart = a.N == 16 || a.ck == 64 ? a.nkh : 1;
  a.nacc = std::min(4, 512 / per_sm / (64 * a.nseg * a.npart));
  *smem = fixed + a.nst * pitch;
  *cpr = std::max(1, std::min(a.B * (a.hg / a.tr), per_sm * sms / a.G));
  return true;
}
}  // namespace

int conv_sp_parts(const ConvSpArgs& a) {
  int sms = 0, cpr = 0;
  size_t smem = 0;
  ConvSpArgs t = a;
  if (device_sms(&sms) < 0) return 0;
  if (!conv_sp_plan(t, sms, &cpr, &smem)) return 0;
  // one per epilogue warp
  return 4 * (!a.bwd.y ? 1 : t.tr == 16 ? sp::kEpq<128, 2> : sp::kEpq<64, 2>) * cpr;
}

cudaError_t launch_conv_sp(const ConvSpArgs& a, const void* in, cudaStream_t stream) {
  int sms = 0, cpr = 0;
  size_t smem = 0;
  ConvSpArgs la = a;
  const int dev = device_sms(&sms);
  if (dev < 0) return cudaErrorInvalidDevice;
  const uintptr_t out = reinterpret_cast<uintptr_t>(la.out);
  if (!conv_sp_plan(la, sms, &cpr, &smem) || !la.out || !la.w || (out & (la.bwd.y ? 31 : 15)) ||
      la.out_gs % 8 || (reinterpret_cast<uintptr_t>(la.w) & 15) || la.w_gs % 8 || la.w_ps % 8 ||
      (la.stats && la.bwd.y))
    return cudaErrorInvalidValue;
  std::call_once(g_encode_once, load_encode);
  if (!g_encode || (reinterpret_cast<uintptr_t>(in) & 15)) return cudaErrorInvalidValue;
  // the NHWC input with 64 channel values (64 / ck pixels) innermost
  const cuuint64_t H = la.hi, B = la.B, G = la.G;
  cuuint64_t dims[5] = {64, 8, H, B, G};
  cuuint64_t strides[4] = {128, 1024, 1024 * H, 1024 * H * B};
  cuuint32_t box[5] = {64, (cuuint32_t)sp::BOX_W, (cuuint32_t)la.box_rows, 1, 1};
  cuuint32_t estr[5] = {1, 1, 1, 1, 1};
  if (g_encode(&la.in_map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(in), dims, strides, box,
               estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
               CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) != CUDA_SUCCESS)
    return cudaErrorInvalidValue;
  const int mode = la.stats ? 1 : (la.bwd.y ? 2 : 0);
  const bool a32 = (out & 31) == 0;
  static std::atomic<int> attr_dev[2][5];  // device + 1; several threads may launch
  auto run = [&](auto kernel, int threads) -> cudaError_t {
    std::atomic<int>& ad = attr_dev[la.tr == 16][a32 ? mode : 3 + mode];
    if (ad != dev + 1) {
      const cudaError_t e =
          cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sp::kOnePerSm);
      if (e != cudaSuccess) return e;
      ad = dev + 1;
    }
    return launch_pdl(kernel, dim3(cpr, la.G), dim3(threads), smem, stream, la);
  };
  if (!a32) {
    if (la.tr == 16)
      return mode == 1 ? run(conv_sp_kernel<128, 1, false>, sp::kThreads<128, 1>)
                       : run(conv_sp_kernel<128, 0, false>, sp::kThreads<128, 0>);
    return mode == 1 ? run(conv_sp_kernel<64, 1, false>, sp::kThreads<64, 1>)
                     : run(conv_sp_kernel<64, 0, false>, sp::kThreads<64, 0>);
  }
  if (la.tr == 16)
    return mode == 1   ? run(conv_sp_kernel<128, 1>, sp::kThreads<128, 1>)
           : mode == 2 ? run(conv_sp_kernel<128, 2>, sp::kThreads<128, 2>)
                       : run(conv_sp_kernel<128, 0>, sp::kThreads<128, 0>);
  return mode == 1   ? run(conv_sp_kernel<64, 1>, sp::kThreads<64, 1>)
         : mode == 2 ? run(conv_sp_kernel<64, 2>, sp::kThreads<64, 2>)
                     : run(conv_sp_kernel<64, 0>, sp::kThreads<64, 0>);
}

cudaError_t launch_wgrad_update(const WgradUpdateArgs& a, cudaStream_t stream) {
  static_assert(sizeof(WgradUpdateArgs) <= 4096, "kernel parameter size");
  if (a.nl < 1 || a.nl > kWgradMaxLayers) return cudaErrorInvalidValue;
  if (a.G <= 0) return cudaSuccess;
  if (a.Kd <= 0 || !a.sgd.w || (a.sgd.mom != 0.f && !a.sgd.u)) return cudaErrorInvalidValue;
  int64_t tiles = 0;
  for (int l = 0; l < a.nl; ++l) {
    const WgradUpdateLayer& ly = a.L[l];
    if (ly.M <= 0 || ly.N <= 0) return cudaErrorInvalidValue;
    // operand boxes as the kernel expects them (64-wide MN-major boxes, or full K-major tiles),
    // with the same layouts in every layer
    if (ly.A.mn_major ? ly.A.box_rows != 64 : ly.A.box_rows != BM) return cudaErrorInvalidValue;
    if (ly.B.mn_major ? ly.B.box_rows != 64 : ly.B.box_rows != wu::TN) return cudaErrorInvalidValue;
    if (ly.A.mn_major != a.L[0].A.mn_major || ly.B.mn_major != a.L[0].B.mn_major)
      return cudaErrorInvalidValue;
    tiles += (int64_t)((ly.N + wu::TN - 1) / wu::TN) * ((ly.M + BM - 1) / BM) * a.G;
  }
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  // averaging mode, or replica 0's parameters for all: a CTA per tile position (all G replicas
  // of it), at most one per SM
  const int64_t units = (a.avg || a.w_rep0) ? tiles / a.G : tiles;
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  constexpr size_t smem = sizeof(WuSmem) + 1024;
  static_assert(smem <= 232448, "shared memory per CTA");
  static std::atomic<int> attr_dev{-1};  // several threads may launch
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(wgrad_update_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)smem);
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  const int grid = (int)std::min<int64_t>(units, sms);
  launch_pdl(wgrad_update_kernel, dim3(grid), dim3(wu::THREADS), smem, stream, a);
  return cudaGetLastError();
}

bool conv_tile_shape(int hout, int wout, int* rows, int* images) {
  if (wout < 1 || hout < 1 || wout > BM || BM % wout) return false;
  const int per_image = hout * wout;
  if (per_image >= BM) {
    if (per_image % BM) return false;
    *rows = BM / wout;
    *images = 1;
  } else {
    if (BM % per_image) return false;
    *rows = hout;
    *images = BM / per_image;
  }
  return true;
}

bool conv_strip_ok(int hout, int wout, int stride) {
  int rows = 0, images = 0;
  // the kernel-row offsets inside a box must be whole swizzle atoms (8 pixel rows of the
  // channel width): wout a multiple of 8
  return stride == 1 && conv_tile_shape(hout, wout, &rows, &images) && images == 1 &&
         wout % 8 == 0 && rows + 2 <= 256;
}

bool make_tma_map_conv(CUtensorMap* map, const void* base, int ck, int win, int hin, int B, int G,
                       int wout, int hout, int stride, bool strip) {
  std::call_once(g_encode_once, load_encode);
  int rows = 0, images = 0;
  if (!g_encode || (ck != 16 && ck != 32 && ck != 64) || (stride != 1 && stride != 2) ||
      !conv_tile_shape(hout, wout, &rows, &images) || (reinterpret_cast<uintptr_t>(base) & 15))
    return false;
  if (wout * stride > 256 || rows * stride > 256 || images > 256) return false;
  const uint64_t e = 2;
  cuuint64_t dims[5] = {(cuuint64_t)ck, (cuuint64_t)win, (cuuint64_t)hin, (cuuint64_t)B,
                        (cuuint64_t)G};
  cuuint64_t strides[4] = {(cuuint64_t)ck * e, (cuuint64_t)win * ck * e,
                           (cuuint64_t)hin * win * ck * e, (cuuint64_t)B * hin * win * ck * e};
  // the strip form's box has a halo row above and below
  if (strip && !conv_strip_ok(hout, wout, stride)) return false;
  const int box_rows = strip ? rows + 2 : rows * stride;
  cuuint32_t box[5] = {(cuuint32_t)ck, (cuuint32_t)(wout * stride), (cuuint32_t)box_rows,
                       (cuuint32_t)images, 1};
  cuuint32_t estr[5] = {1, (cuuint32_t)stride, (cuuint32_t)stride, 1, 1};
  const CUtensorMapSwizzle sw = ck == 64 ? CU_TENSOR_MAP_SWIZZLE_128B
                                         : (ck == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                     : CU_TENSOR_MAP_SWIZZLE_32B);
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims,
                        strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}

bool conv_wgrad_tc_ok(int cin, int cout, int stride, int hin, int win, int hout, int wout) {
  if ((cin != 16 && cin != 32 && cin != 64) || cout < 16 || cout > 64 || cout % 16) return false;
  if ((stride != 1 && stride != 2) || wout < 1 || wout > 64 || 64 % wout) return false;
  return (hout * wout) % 64 == 0 && win == wout * stride && hin == hout * stride;
}

// Rows at least 8 wide: 16 pixels are then within a row, or two whole rows.  Narrower ones: 16 pixels are
// within a column of the tile's kp / wout (16 to 128) rows.
bool conv_wgrad_geom(int cin, int cout, int stride, int hout, int wout, ConvWgradGeom* gm) {
  const int nb = conv_wgrad_nb(cout);
  gm->cols = wout < 8;
  gm->strips = stride;
  uint32_t cols = 32;
  while (cols < (uint32_t)(3 * (cin == 64 ? 2 : 1) * nb)) cols <<= 1;
  gm->tmem_cols = cols;
  // 128-pixel tiles where an image has them: fewer stage handshakes, less halo
  for (int kp = (hout * wout) % 128 == 0 ? 128 : 64; kp >= 64; kp -= 64) {
    gm->kp = kp;
    gm->inner = gm->cols ? kp / wout : wout;
    gm->rows = (kp / gm->inner - 1) * stride + 3;
    gm->wp = gm->inner + (stride == 1 ? 2 : 1);
    gm->pitch = gm->cols ? (gm->wp + 7) / 8 * 8 : gm->wp;
    // the unread rows of the last strip's operand end at most (fourth row group) one strip row
    // behind the strip; the tile follows it, and this pad where the tile is smaller
    gm->pad = (int)up1k((uint32_t)gm->pitch * cin * 2);
    const size_t stage = gm->strips * (size_t)up1k((uint32_t)(gm->rows * gm->pitch * cin * 2)) +
                         up1k((uint32_t)(kp * nb * 2));
    const size_t fixed = 1024 + gm->pad + (2 * cw::MAX_ST + 1) * 8 + 16;
    const size_t n2 = (cw::kTwoPerSm - fixed) / stage, n1 = (cw::kOnePerSm - fixed) / stage;
    // two CTAs per SM where each still gets three stages: one's handshakes overlap the other's
    gm->per_sm = n2 >= 3 && 2 * cols <= 512 ? 2 : 1;
    gm->stages = (int)std::min<size_t>(cw::MAX_ST, gm->per_sm == 2 ? n2 : n1);
    gm->smem = fixed + gm->stages * stage;
    // (the pixels that a strip row spans and its rows are TMA box extents)
    if (gm->stages >= 2 && gm->rows <= 256 && (gm->wp - 1) * stride + 1 <= 256) return true;
  }
  return false;
}

int conv_wgrad_ctas(int cin, int cout, int stride, int hout, int wout, int B, int G) {
  ConvWgradGeom gm;
  if (!conv_wgrad_geom(cin, cout, stride, hout, wout, &gm)) return 1;  // launch_conv_wgrad_tc rejects it
  const int64_t tiles = (int64_t)B * hout * wout / gm.kp;
  return (int)std::max<int64_t>(1, std::min<int64_t>(tiles, (int64_t)kNumSMs * gm.per_sm / std::max(G, 1)));
}

namespace {
// A box of box_c channels x (span_w, span_h) pixels, every step_w-th / step_h-th of them, of an NHWC bf16
// array [G][B][H][W][C].
bool encode_nhwc(CUtensorMap* map, const void* base, int C, int W, int H, int B, int G, int box_c, int span_w,
                 int span_h, int step_w, int step_h) {
  std::call_once(g_encode_once, load_encode);
  if (!g_encode || (box_c != 16 && box_c != 32 && box_c != 64) || (reinterpret_cast<uintptr_t>(base) & 15) ||
      span_w > 256 || span_h > 256)
    return false;
  const uint64_t e = 2;
  cuuint64_t dims[5] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B, (cuuint64_t)G};
  cuuint64_t strides[4] = {(cuuint64_t)C * e, (cuuint64_t)W * C * e, (cuuint64_t)H * W * C * e,
                           (cuuint64_t)B * H * W * C * e};
  cuuint32_t box[5] = {(cuuint32_t)box_c, (cuuint32_t)span_w, (cuuint32_t)span_h, 1, 1};
  cuuint32_t estr[5] = {1, (cuuint32_t)step_w, (cuuint32_t)step_h, 1, 1};
  const CUtensorMapSwizzle sw = box_c == 64 ? CU_TENSOR_MAP_SWIZZLE_128B
                                            : (box_c == 32 ? CU_TENSOR_MAP_SWIZZLE_64B
                                                           : CU_TENSOR_MAP_SWIZZLE_32B);
  CUresult r = g_encode(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 5, const_cast<void*>(base), dims,
                        strides, box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, sw,
                        CU_TENSOR_MAP_L2_PROMOTION_L2_128B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS;
}
}  // namespace

bool make_conv_wgrad_maps(ConvWgradArgs* a, const ConvWgradGeom& gm, const void* x, const void* dy, int B) {
  const int span = (gm.wp - 1) * a->stride + 1;  // pixels that a strip row spans
  if (gm.cols)
    return encode_nhwc(&a->x_map, x, a->cin, a->win, a->hin, B, a->G, a->cin, 1, span, 1, a->stride) &&
           encode_nhwc(&a->dy_map, dy, a->cout, a->wout, a->hout, B, a->G, a->nb, 1, gm.inner, 1, 1);
  return encode_nhwc(&a->x_map, x, a->cin, a->win, a->hin, B, a->G, a->cin, span, gm.rows, a->stride, 1) &&
         make_tma_map(&a->dy_map, dy, true, a->cout, a->P, a->G, a->cout, (uint64_t)a->P * a->cout, a->nb,
                      gm.kp, 2 * a->nb);
}

cudaError_t launch_conv_wgrad_tc(const ConvWgradArgs& a, cudaStream_t stream) {
  if (a.P <= 0 || a.G <= 0) return cudaSuccess;
  ConvWgradGeom gm;
  if (!conv_wgrad_tc_ok(a.cin, a.cout, a.stride, a.hin, a.win, a.hout, a.wout) || !a.part ||
      !conv_wgrad_geom(a.cin, a.cout, a.stride, a.hout, a.wout, &gm) || a.nb != conv_wgrad_nb(a.cout) ||
      a.P % gm.kp || a.P % (a.hout * a.wout) || a.cpr < 1 || a.cpr > a.P / gm.kp || a.G > 65535)
    return cudaErrorInvalidValue;
  ConvWgradArgs la = a;
  la.geom = gm;
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  static std::atomic<int> attr_dev{-1};  // several threads may launch
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(conv_wgrad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             232448);
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  return launch_pdl(conv_wgrad_tc_kernel, dim3(a.cpr, a.G), dim3(cw::THREADS), gm.smem, stream, la);
}

int tc_tile_n(int Kd) { return (Kd + BK - 1) / BK <= 2 ? 128 : 64; }

int tc_valid_splits(int Kd, int want) {
  const int nk_all = (Kd + BK - 1) / BK;
  if (want < 1) want = 1;
  if (want > nk_all) want = nk_all;
  const int per = (nk_all + want - 1) / want;
  return (nk_all + per - 1) / per;  // every split gets at least one k-block
}

namespace {
bool gemm_pt_off() {
  static const bool off = [] {
    const char* e = std::getenv("LSGD_GEMM_ONE_TILE");
    return e && e[0] == '1';
  }();
  return off;
}

cudaError_t launch_pt(const TcGemmArgs& a, cudaStream_t stream) {
  int dev = 0, sms = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (e != cudaSuccess) return e;
  constexpr size_t smem = sizeof(PtSmem) + 1024;
  static_assert(smem <= 232448, "shared memory per CTA");
  static std::atomic<int> attr_dev{-1};  // several threads may launch
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(gemm_pt_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  const int64_t tiles = (int64_t)((a.N + pt::PBN - 1) / pt::PBN) * ((a.M + BM - 1) / BM) * a.G;
  if (tiles > 0x7fffffffLL) return cudaErrorInvalidValue;
  const int grid = (int)std::min<int64_t>(tiles, sms);
  launch_pdl(gemm_pt_kernel, dim3(grid), dim3(pt::THREADS), smem, stream, a);
  return cudaGetLastError();
}
}  // namespace

cudaError_t launch_gemm_tc(const TcGemmArgs& a, cudaStream_t stream) {
  if (a.M <= 0 || a.N <= 0 || a.G <= 0) return cudaSuccess;
  if (a.Kd <= 0 || a.G > 65535) return cudaErrorInvalidValue;
  // The TMA boxes must deliver exactly the tiles the kernel expects (expect-tx byte counts and
  // shared-memory extents depend on it).
  const int bn = tc_tile_n(a.Kd);
  // (a K-major A of at most box_rows rows may come in a shorter box of whole 8-row swizzle atoms)
  if (a.A.mn_major ? a.A.box_rows != 64
                   : a.A.box_rows != BM && (a.A.box_rows < 8 || a.A.box_rows > BM || a.A.box_rows % 8 ||
                                            a.M > a.A.box_rows || a.conv))
    return cudaErrorInvalidValue;
  if (a.B.mn_major ? a.B.box_rows != 64 : a.B.box_rows != bn) return cudaErrorInvalidValue;  // 64 or, short, 128
  if ((a.epi == EPI_BIAS || a.epi == EPI_BIAS_RELU) && !a.bias) return cudaErrorInvalidValue;
  if (a.epi == EPI_MASK && !a.mask) return cudaErrorInvalidValue;
  if (!a.C) return cudaErrorInvalidValue;
  if (a.conv) {
    // K-major tap slices of cv_ck channels on both sides; 64-wide N tiles, four stages, no split
    int rows = 0, images = 0;
    if ((a.cv_ck != 16 && a.cv_ck != 32 && a.cv_ck != 64) || (a.cv_stride != 1 && a.cv_stride != 2) ||
        !conv_tile_shape(a.cv_hout, a.cv_wout, &rows, &images) || a.splits > 1 ||
        a.A.mn_major || a.B.mn_major || a.bias_colsum)
      return cudaErrorInvalidValue;
    if (a.M % (a.cv_hout * a.cv_wout)) return cudaErrorInvalidValue;  // whole images
    dim3 gridc((a.N + 63) / 64, (a.M + BM - 1) / BM, a.G);
    if (gridc.y > 65535) return cudaErrorInvalidValue;
    return launch_one_tile<64>(a, gridc, 9, stream);
  }
  // the bias column sums need the whole mini-batch in one tile, and the masked data gradient
  if (a.bias_colsum && (a.M > BM || a.epi != EPI_MASK || (!a.bsgd.w && !a.bias_grad)))
    return cudaErrorInvalidValue;
  const int splits = a.splits > 1 ? a.splits : 1;
  if (splits > 1) {
    const int nk_all = (a.Kd + BK - 1) / BK, per = (nk_all + splits - 1) / splits;
    if (a.epi != EPI_STORE || (int64_t)(splits - 1) * per >= nk_all) return cudaErrorInvalidValue;
    if ((int64_t)a.G * splits > 65535) return cudaErrorInvalidValue;
  }
  constexpr int BN = 128;
  dim3 grid((a.N + BN - 1) / BN, (a.M + BM - 1) / BM, a.G * splits);
  if (grid.y > 65535) return cudaErrorInvalidValue;
  static_assert(BM == kTcTileM, "tile height");
  // Short reductions (the weight gradient's k = B_loc) need only two stages; the smaller shared
  // footprint lets three CTAs share an SM so one CTA's epilogue overlaps the others' loads.
  if ((a.Kd + BK - 1) / BK <= 2) return launch_one_tile<BN>(a, grid, (a.Kd + BK - 1) / BK, stream);
  // Wide products (at least 2048 output columns, no split): the persistent kernel -- the forward
  // (K-major weights) and, since its epilogue prefetches the tile's ReLU mask, the data gradient
  // (MN-major weights).  Narrower layers give it too few 128 x 256 tiles to fill the SMs
  // (measured: MLP 3072-4096x3-100 forward 0.36 -> 0.27 ms per step, backward 0.333 -> 0.322 ms;
  // MLP 3072-1024-1024-10 0.29 -> 0.35 ms per step, so it stays on the one-tile kernel).
  if (splits == 1 && a.N >= 2048 && a.B.box_rows == 64 && (a.A.mn_major || a.A.box_rows == BM) && !gemm_pt_off())
    return launch_pt(a, stream);
  // Other long reductions: 64-wide N tiles, one or two CTAs per SM.  (128-wide ones read the
  // activations half as often and were no faster where they leave three SMs in four a CTA: 31.6, 16.5
  // and 13.2 us against 31.6, 14.5 and 12.4 for the products of MLP 3072-1024-1024-10, K = 16.)
  constexpr int BN2 = 64;
  const int nk_all = (a.Kd + BK - 1) / BK;
  dim3 grid2((a.N + BN2 - 1) / BN2, (a.M + BM - 1) / BM, a.G * splits);
  return launch_one_tile<BN2>(a, grid2, (nk_all + splits - 1) / splits, stream);
}

}  // namespace lsgd
