// Grouped SIMT GEMM with the dense layers' fused epilogues (sm_103a).
//
// The fp32 path (pure fp32 mode: tensor cores cannot give fp32-exact products) and the reference
// for the tcgen05 kernel's tests.  A(m, k) and B(k, n) take arbitrary element strides, so one kernel
// serves the forward (act x W^T), data-gradient (dZ x W) and weight-gradient (dZ^T x act) products
// of Eq. 2's local gradient.
//
// A thread owns 4 or 8 rows -- 4 ty + i and, of 8, BT / 2 + 4 ty + i -- by 2, 4 or 8 columns, and
// multiplies with the packed two-lane fma.rn.f32x2.  The next 16- or 32-deep k slice is in registers
// while this one is multiplied (16 covered the loads' latency only at BT = 128: 638 against 567 us
// for the whole case below), and slices alternate between two shared-memory buffers (one barrier
// per slice).  Element (k, r) of a slice lies in row k at the group of four (r / 4) ^ f(k / 4): the
// transposing stores of a k-contiguous operand (four or eight lanes to a row) and the reads along r
// then both spread over all banks.  Three forms, all of them with one chain of multiply-adds
// in k order per output and split, and the splits' sums in order:
//   BT = 128  256 threads, 8 x 8: wherever such tiles fill the chip (weight gradients);
//   BT = 64   128 threads, 8 x 4: wherever these give every SM a CTA (a mini-batch's forward over a
//             long k, split over CTAs).  64 threads of 8 x 8 need fewer shared-memory reads but
//             leave one warp to a scheduler, which covers no latency: 89 us against 45 for
//             64 x 1024 x 3072, K = 4;
//   BT = 32   128 threads, 4 x 2: the rest (an unsplit data gradient, at most 32 rows or columns):
//             33 us for 64 x 1024 x 1024, K = 4, where 64 x 64 tiles occupied 64 of 152 SMs and
//             took 58.
// Measured, MLP 3072-1024-1024-10, K = 4, B = 64, per step: forward 173 -> 82 us, backward
// 221 -> 112 us against 4 x 4 outputs per thread of a 64 x 64 tile with scalar loads and two
// barriers per slice.
#include <algorithm>

#include "common.cuh"
#include "lsgd_internal.h"

namespace lsgd {
namespace {

template <int BT>
struct Form {
  static constexpr int BK = BT <= 64 ? 32 : 16;            // k slice
  static constexpr int THREADS = BT == 128 ? 256 : 128;
  static constexpr int RG = BT == 32 ? 1 : 2;              // groups of four rows per thread
  static constexpr int CN = BT == 128 ? 8 : BT == 64 ? 4 : 2;  // columns per thread
  static constexpr int TX = BT / CN;                       // threads across the tile
  static constexpr int NL = BT * BK / 4 / THREADS;         // groups of four an operand's slice gives a thread
  static constexpr int SLICE = 2 * BK * BT;                // floats of one buffer: A then B
  static_assert(TX * (BT / (4 * RG)) == THREADS, "the threads tile the outputs");
};

// The groups' place in their row: see above.
template <int BT>
__device__ __forceinline__ int swz(int group, int k) {
  return Form<BT>::BK == 32 ? group ^ ((k >> 2) & 7) : group ^ (((k >> 2) & 3) << 1);
}

// One thread's groups of four of a BT x BK operand slice, element (r, k) at base + r rs + k ks
// (r < nr, k < k_hi: the rest are zero), along k where k is contiguous and along r otherwise.  The
// groups' addresses advance by a slice per load.
template <typename T, int BT>
struct SliceLoader {
  using F = Form<BT>;
  const T* p[F::NL];  // the groups' first elements in the next slice
  int64_t step, along;  // between slices; between a group's elements
  bool kc, vec;
  int left[F::NL];    // rows from the group's first to the edge (<= 0: none)

  __device__ __forceinline__ void place(int i, int& r, int& k) const {
    const int e = threadIdx.x + F::THREADS * i;
    r = kc ? e / (F::BK / 4) : (e % (BT / 4)) * 4;
    k = kc ? (e % (F::BK / 4)) * 4 : e / (BT / 4);
  }
  __device__ __forceinline__ void init(const T* base, int64_t rs, int64_t ks, int nr, int k_lo) {
    kc = ks == 1;
    step = (int64_t)F::BK * ks;
    along = kc ? 1 : rs;
    // groups of four are whole, aligned vectors
    vec = (kc || rs == 1) && (kc ? rs : ks) % 4 == 0 && k_lo % 4 == 0 &&
          (reinterpret_cast<uintptr_t>(base) & (4 * sizeof(T) - 1)) == 0;
#pragma unroll
    for (int i = 0; i < F::NL; ++i) {
      int r, k;
      place(i, r, k);
      p[i] = base + (int64_t)r * rs + (int64_t)(k_lo + k) * ks;
      left[i] = nr - r;
    }
  }
  __device__ __forceinline__ float4 vec4(const T* q) const {
    if constexpr (sizeof(T) == 4) {
      return __ldg(reinterpret_cast<const float4*>(q));
    } else {
      const uint2 u = __ldg(reinterpret_cast<const uint2*>(q));
      return make_float4(bf2f((uint16_t)(u.x & 0xffffu)), bf2f((uint16_t)(u.x >> 16)),
                         bf2f((uint16_t)(u.y & 0xffffu)), bf2f((uint16_t)(u.y >> 16)));
    }
  }
  // nk: k indices from the slice's first to the end of the range
  __device__ __forceinline__ void load(int nk, float4 (&v)[F::NL]) {
    if (vec && nk >= F::BK) {
#pragma unroll
      for (int i = 0; i < F::NL; ++i) {
        if (left[i] >= (kc ? 1 : 4))
          v[i] = vec4(p[i]);
        else
          v[i] = part(i, kc ? 0 : left[i]);
        p[i] += step;
      }
      return;
    }
#pragma unroll
    for (int i = 0; i < F::NL; ++i) {
      int r, k;
      place(i, r, k);
      v[i] = part(i, kc ? (left[i] > 0 ? nk - k : 0) : (k < nk ? left[i] : 0));
      p[i] += step;
    }
  }
  __device__ __forceinline__ float4 part(int i, int n) const {
    float4 v;
    v.x = n > 0 ? Elem<T>::load(p[i]) : 0.f;
    v.y = n > 1 ? Elem<T>::load(p[i] + along) : 0.f;
    v.z = n > 2 ? Elem<T>::load(p[i] + 2 * along) : 0.f;
    v.w = n > 3 ? Elem<T>::load(p[i] + 3 * along) : 0.f;
    return v;
  }
  __device__ __forceinline__ void store(float* sm, const float4 (&v)[F::NL]) const {
#pragma unroll
    for (int i = 0; i < F::NL; ++i) {
      int r, k;
      place(i, r, k);
      float* d = sm + k * BT + 4 * swz<BT>(r >> 2, k) + (r & 3);
      if (kc) {
        d[0] = v[i].x;
        d[BT] = v[i].y;
        d[2 * BT] = v[i].z;
        d[3 * BT] = v[i].w;
      } else {
        *reinterpret_cast<float4*>(d) = v[i];
      }
    }
  }
};

// NC (2 or 4) consecutive outputs (m, n ..) of group g: the raw sums of a split, or the epilogue.
template <typename TC, typename TM, int EPI, int NC>
__device__ __forceinline__ void store_row(const GemmArgs& a, int splits, int split, int g, int m, int n,
                                          float (&x)[NC]) {
  if (m >= a.M || n >= a.N) return;
  auto put = [&](float* d) {
    if (n + NC <= a.N && (reinterpret_cast<uintptr_t>(d) & (4 * NC - 1)) == 0) {
      if constexpr (NC == 4)
        *reinterpret_cast<float4*>(d) = make_float4(x[0], x[1], x[2], x[3]);
      else
        *reinterpret_cast<float2*>(d) = make_float2(x[0], x[1]);
    } else {
#pragma unroll
      for (int i = 0; i < NC; ++i)
        if (n + i < a.N) d[i] = x[i];
    }
  };
  if (splits > 1) {
    put(a.ws + (((int64_t)g * splits + split) * a.M + m) * a.N + n);
    return;
  }
#pragma unroll
  for (int i = 0; i < NC; ++i) {
    if (n + i >= a.N) break;
    if (EPI == EPI_BIAS || EPI == EPI_BIAS_RELU) x[i] += a.bias[(int64_t)g * a.bias_gs + n + i];
    if (EPI == EPI_BIAS_RELU) x[i] = fmaxf(x[i], 0.f);
    if (EPI == EPI_MASK)
      x[i] = Elem<TM>::load(reinterpret_cast<const TM*>(a.mask) + (int64_t)g * a.mask_gs +
                            (int64_t)m * a.mask_rs + n + i) > 0.f
                 ? x[i]
                 : 0.f;
  }
  TC* C = reinterpret_cast<TC*>(a.C) + (int64_t)g * a.c_gs + (int64_t)m * a.c_rs + n;
  if constexpr (sizeof(TC) == 4) {
    put(C);
  } else {
#pragma unroll
    for (int i = 0; i < NC; ++i)
      if (n + i < a.N) Elem<TC>::store(C + i, x[i]);
  }
}

// The update in the weight gradient's epilogue: it writes no gradient and reads none, 16 bytes a parameter
// instead of 24.  Per step of MLP 3072-1024-1024-10, K = 4, B = 64: 39 + 15 us of gradients and 47 of
// update (their memory's floor 45) are 62 + 24.  The form stays at 128: of 64 it is 67 + 28.
//
// Two rows' outputs (columns n + h span of each, NC at a time) into the local update: everything it reads
// is requested before anything is written.
template <int NH, int NC>
__device__ __forceinline__ void update_rows(const SgdParams& p, const GemmArgs& a, int g, const int (&m)[2],
                                            int n, int span, const float (&x)[2][NH][NC]) {
  const bool mom = p.mom != 0.f;
  float w[2][NH][NC], u[2][NH][NC];
  const int64_t base = (int64_t)g * a.c_gs;
  // whole, aligned groups
  const bool vec = NC == 4 && (a.c_rs & 3) == 0 && ((reinterpret_cast<uintptr_t>(p.w + base) |
                   (mom ? reinterpret_cast<uintptr_t>(p.u + base) : 0)) & 15) == 0;
  auto each = [&](auto&& f) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int h = 0; h < NH; ++h) f(i, h, base + (int64_t)m[i] * a.c_rs + n + h * span, n + h * span);
  };
  each([&](int i, int h, int64_t k, int col) {
    if (m[i] >= a.M) return;
    if (vec && col + NC <= a.N) {
      if constexpr (NC == 4) {
        const float4 q = __ldcs(reinterpret_cast<const float4*>(p.w + k));
        const float4 r = mom ? __ldcs(reinterpret_cast<const float4*>(p.u + k)) : make_float4(0.f, 0.f, 0.f, 0.f);
        w[i][h][0] = q.x, w[i][h][1] = q.y, w[i][h][2] = q.z, w[i][h][3] = q.w;
        u[i][h][0] = r.x, u[i][h][1] = r.y, u[i][h][2] = r.z, u[i][h][3] = r.w;
      }
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c) {
        w[i][h][c] = col + c < a.N ? p.w[k + c] : 0.f;
        u[i][h][c] = col + c < a.N && mom ? p.u[k + c] : 0.f;
      }
    }
  });
  each([&](int i, int h, int64_t k, int col) {
    if (m[i] >= a.M) return;
#pragma unroll
    for (int c = 0; c < NC; ++c)
      sgd_elem_any(w[i][h][c], u[i][h][c], x[i][h][c], p.lr, p.mom, p.wd, p.nesterov != 0, p.sign != 0);
    if (vec && col + NC <= a.N) {
      if constexpr (NC == 4) {
        __stcs(reinterpret_cast<float4*>(p.w + k), make_float4(w[i][h][0], w[i][h][1], w[i][h][2], w[i][h][3]));
        if (mom)
          __stcs(reinterpret_cast<float4*>(p.u + k), make_float4(u[i][h][0], u[i][h][1], u[i][h][2], u[i][h][3]));
      }
    } else {
#pragma unroll
      for (int c = 0; c < NC; ++c)
        if (col + c < a.N) {
          p.w[k + c] = w[i][h][c];
          if (mom) p.u[k + c] = u[i][h][c];
        }
    }
  });
}

// splits > 1: blockIdx.z = g splits + split, k in [split kchunk, (split + 1) kchunk), and the raw
// sums go to ws (splitk_epilogue_kernel applies the epilogue).
template <typename TA, typename TB, typename TC, typename TM, int EPI, int BT>
__global__ void __launch_bounds__(Form<BT>::THREADS, BT == 128 ? 2 : 3) gemm_simt_kernel(
    const __grid_constant__ GemmArgs a, int splits, int kchunk) {
  pdl_begin();
  using F = Form<BT>;
  constexpr int BK = F::BK, RG = F::RG, CN = F::CN, CQ = CN < 4 ? CN : 4;  // columns in one group
  __shared__ __align__(16) float sm[2 * F::SLICE];
  const int g = blockIdx.z / splits, split = blockIdx.z % splits;
  const int k_lo = split * kchunk, k_hi = min(a.Kd, k_lo + kchunk);
  const int m0 = blockIdx.y * BT, n0 = blockIdx.x * BT;
  const int tx = threadIdx.x % F::TX, ty = threadIdx.x / F::TX;
  SliceLoader<TA, BT> la;
  SliceLoader<TB, BT> lb;
  la.init(reinterpret_cast<const TA*>(a.A) + (int64_t)g * a.a_gs + (int64_t)m0 * a.a_rs, a.a_rs, a.a_cs,
          a.M - m0, k_lo);
  lb.init(reinterpret_cast<const TB*>(a.B) + (int64_t)g * a.b_gs + (int64_t)n0 * a.b_cs, a.b_cs, a.b_rs,
          a.N - n0, k_lo);

  u64 acc[4 * RG][CN / 2];
#pragma unroll
  for (int i = 0; i < 4 * RG; ++i)
#pragma unroll
    for (int j = 0; j < CN / 2; ++j) acc[i][j] = 0ull;

  if constexpr (EPI == EPI_SGD) {
    // the tile's parameters and momentum on their way to L2 while the products run
    const int row = threadIdx.x / (F::THREADS / BT), lines = min(BT, a.N - n0) * 4 / 128;
    if (m0 + row < a.M) {
      const int64_t at = (int64_t)g * a.c_gs + (int64_t)(m0 + row) * a.c_rs + n0;
      for (int i = threadIdx.x % (F::THREADS / BT); i < lines; i += F::THREADS / BT) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.sgd.w + at + 32 * i));
        if (a.sgd.mom != 0.f) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.sgd.u + at + 32 * i));
      }
    }
  }
  float4 va[F::NL], vb[F::NL];
  la.load(k_hi - k_lo, va);
  lb.load(k_hi - k_lo, vb);
  int buf = 0;
  for (int k0 = k_lo; k0 < k_hi; k0 += BK, buf ^= 1) {
    float* As = sm + buf * F::SLICE;
    float* Bs = As + BK * BT;
    la.store(As, va);
    lb.store(Bs, vb);
    __syncthreads();  // and every thread is past the products of the slice before last
    if (k0 + BK < k_hi) {
      la.load(k_hi - k0 - BK, va);
      lb.load(k_hi - k0 - BK, vb);
    }
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      const float* ap = As + kk * BT + 4 * swz<BT>(ty, kk);
      float av[4 * RG];
      u64 bv[CN / 2];
#pragma unroll
      for (int h = 0; h < RG; ++h) {
        const float4 f = *reinterpret_cast<const float4*>(ap + h * (BT / 2));
        av[4 * h] = f.x;
        av[4 * h + 1] = f.y;
        av[4 * h + 2] = f.z;
        av[4 * h + 3] = f.w;
      }
      if constexpr (CN >= 4) {
        const float* bp = Bs + kk * BT + 4 * swz<BT>(tx, kk);
#pragma unroll
        for (int h = 0; h < CN / 4; ++h) {
          const ulonglong2 t = *reinterpret_cast<const ulonglong2*>(bp + h * (BT / 2));
          bv[2 * h] = t.x;
          bv[2 * h + 1] = t.y;
        }
      } else {
        bv[0] = *reinterpret_cast<const u64*>(Bs + kk * BT + 4 * swz<BT>(tx >> 1, kk) + 2 * (tx & 1));
      }
#pragma unroll
      for (int i = 0; i < 4 * RG; ++i) {
        const u64 x = pack2(av[i], av[i]);
#pragma unroll
        for (int j = 0; j < CN / 2; ++j) fma2(acc[i][j], x, bv[j]);
      }
    }
  }

  if constexpr (EPI == EPI_SGD) {
#pragma unroll
    for (int i0 = 0; i0 < 4 * RG; i0 += 2) {
      float x[2][CN / CQ][CQ];
      int m[2];
#pragma unroll
      for (int r = 0; r < 2; ++r) {
        m[r] = m0 + 4 * ty + ((i0 + r) & 3) + (i0 >> 2) * (BT / 2);
#pragma unroll
        for (int q = 0; q < CN / 2; ++q) {
          const float2 f = unpack2(acc[i0 + r][q]);
          x[r][q / (CQ / 2)][2 * (q % (CQ / 2))] = f.x;
          x[r][q / (CQ / 2)][2 * (q % (CQ / 2)) + 1] = f.y;
        }
      }
      update_rows<CN / CQ, CQ>(a.sgd, a, g, m, n0 + CQ * tx, BT / 2, x);
    }
    return;
  }
#pragma unroll
  for (int i = 0; i < 4 * RG; ++i) {
    const int m = m0 + 4 * ty + (i & 3) + (i >> 2) * (BT / 2);
#pragma unroll
    for (int h = 0; h < CN / CQ; ++h) {
      float x[CQ];
#pragma unroll
      for (int j = 0; j < CQ / 2; ++j) {
        const float2 f = unpack2(acc[i][h * (CQ / 2) + j]);
        x[2 * j] = f.x;
        x[2 * j + 1] = f.y;
      }
      store_row<TC, TM, EPI, CQ>(a, splits, split, g, m, n0 + CQ * tx + h * (BT / 2), x);
    }
  }
}

// The split partial sums added in split order, then the epilogue: one thread per output.
template <typename TC, typename TM, int EPI>
__global__ void __launch_bounds__(256) splitk_epilogue_kernel(GemmArgs a, int splits) {
  pdl_begin();
  const int64_t mn = (int64_t)a.M * a.N, n_all = (int64_t)a.G * mn;
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n_all; e += stride) {
    const int g = (int)(e / mn), m = (int)((e % mn) / a.N), n = (int)(e % a.N);
    const float* ws = a.ws + (int64_t)g * splits * mn + (int64_t)m * a.N + n;
    float v = 0.f;
    for (int sp = 0; sp < splits; ++sp) v += ws[sp * mn];
    if (EPI == EPI_BIAS || EPI == EPI_BIAS_RELU) v += a.bias[(int64_t)g * a.bias_gs + n];
    if (EPI == EPI_BIAS_RELU) v = fmaxf(v, 0.f);
    if (EPI == EPI_MASK)
      v = (Elem<TM>::load(reinterpret_cast<const TM*>(a.mask) + (int64_t)g * a.mask_gs +
                          (int64_t)m * a.mask_rs + n) > 0.f)
              ? v
              : 0.f;
    Elem<TC>::store(reinterpret_cast<TC*>(a.C) + (int64_t)g * a.c_gs + (int64_t)m * a.c_rs + n, v);
  }
}

template <typename TA, typename TB, typename TC, typename TM, int EPI>
cudaError_t launch_epi(const GemmArgs& a, dim3 grid, int splits, int kchunk, int bt, cudaStream_t s) {
  cudaError_t e;
  if (bt == 128)
    e = launch_pdl(gemm_simt_kernel<TA, TB, TC, TM, EPI, 128>, grid, Form<128>::THREADS, 0, s, a, splits, kchunk);
  else if (bt == 64)
    e = launch_pdl(gemm_simt_kernel<TA, TB, TC, TM, EPI, 64>, grid, Form<64>::THREADS, 0, s, a, splits, kchunk);
  else
    e = launch_pdl(gemm_simt_kernel<TA, TB, TC, TM, EPI, 32>, grid, Form<32>::THREADS, 0, s, a, splits, kchunk);
  if (e != cudaSuccess) return e;
  if (a.splits_left) *a.splits_left = splits;
  if (EPI != EPI_SGD && splits > 1 && !a.splits_left) {
    const int64_t n = (int64_t)a.G * a.M * a.N;
    const int blocks = (int)std::min<int64_t>((n + 255) / 256, (int64_t)kNumSMs * 8);
    launch_pdl(splitk_epilogue_kernel<TC, TM, EPI>, blocks, 256, 0, s, a, splits);
  }
  return cudaGetLastError();
}

template <typename TA, typename TB, typename TC, typename TM>
cudaError_t dispatch_epi(const GemmArgs& a, dim3 grid, int splits, int kchunk, int bt,
                         cudaStream_t s) {
  switch (a.epi) {
    case EPI_STORE:
      return launch_epi<TA, TB, TC, TM, EPI_STORE>(a, grid, splits, kchunk, bt, s);
    case EPI_BIAS:
      return launch_epi<TA, TB, TC, TM, EPI_BIAS>(a, grid, splits, kchunk, bt, s);
    case EPI_BIAS_RELU:
      return launch_epi<TA, TB, TC, TM, EPI_BIAS_RELU>(a, grid, splits, kchunk, bt, s);
    case EPI_MASK:
      return launch_epi<TA, TB, TC, TM, EPI_MASK>(a, grid, splits, kchunk, bt, s);
    case EPI_SGD:
      if constexpr (sizeof(TA) == 4)
        return launch_epi<TA, TB, TC, TM, EPI_SGD>(a, grid, splits, kchunk, bt, s);
    default:
      return cudaErrorInvalidValue;
  }
}

}  // namespace

cudaError_t launch_gemm_simt(const GemmArgs& a, cudaStream_t stream) {
  if (a.M <= 0 || a.N <= 0 || a.G <= 0) return cudaSuccess;
  if (a.Kd < 0 || a.G > 65535) return cudaErrorInvalidValue;
  if ((a.epi == EPI_BIAS || a.epi == EPI_BIAS_RELU) && !a.bias) return cudaErrorInvalidValue;
  if (a.epi == EPI_MASK && !a.mask) return cudaErrorInvalidValue;
  if (a.a_bf16 != a.b_bf16) return cudaErrorInvalidValue;
  if (a.mask && a.mask_bf16 != a.a_bf16) return cudaErrorInvalidValue;
  if (a.epi == EPI_SGD && (a.a_bf16 || !a.sgd.w || (a.sgd.mom != 0.f && !a.sgd.u))) return cudaErrorInvalidValue;
  // Few output tiles over a long reduction (a small layer's forward): cut k into splits of at
  // least 128 so that about two CTAs per SM work, as far as the workspace holds the partials.
  const int64_t tiles = (int64_t)((a.N + 63) / 64) * ((a.M + 63) / 64) * a.G;
  int splits = 1;
  if (a.ws && a.epi != EPI_SGD && a.Kd >= 256 && tiles < kNumSMs) {
    const int64_t want = std::min<int64_t>((2 * kNumSMs + tiles - 1) / tiles, a.Kd / 128);
    const int64_t room = a.ws_floats / ((int64_t)a.G * a.M * a.N);
    splits = (int)std::max<int64_t>(1, std::min<int64_t>({want, room, (int64_t)64}));
  }
  const int kchunk = (int)(((a.Kd + splits - 1) / splits + 15) / 16 * 16);
  splits = kchunk > 0 ? (a.Kd + kchunk - 1) / kchunk : 1;  // every split nonempty
  if (splits < 1) splits = 1;
  // the largest tile that gives every SM a CTA (measured: the comment at the top), 32 where a larger
  // one would be mostly empty
  const int64_t tiles128 = (int64_t)((a.N + 127) / 128) * ((a.M + 127) / 128) * a.G;
  const bool narrow = a.M <= 32 || a.N <= 32;
  const int bt = narrow ? 32 : tiles128 >= kNumSMs ? 128 : tiles * splits >= kNumSMs ? 64 : 32;
  dim3 grid((a.N + bt - 1) / bt, (a.M + bt - 1) / bt, a.G * splits);
  if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidValue;
  if (a.a_bf16) {
    if (a.c_bf16)
      return dispatch_epi<uint16_t, uint16_t, uint16_t, uint16_t>(a, grid, splits, kchunk, bt, stream);
    return dispatch_epi<uint16_t, uint16_t, float, uint16_t>(a, grid, splits, kchunk, bt, stream);
  }
  if (a.c_bf16) return cudaErrorInvalidValue;
  return dispatch_epi<float, float, float, float>(a, grid, splits, kchunk, bt, stream);
}

}  // namespace lsgd
