// 3x3 convolutions (zero padding 1) on the fp32 cores, G replicas per launch.
//
// The fp32 mode's convolutions (tensor cores cannot give fp32-exact products) and the SIMT form of
// the bf16 ones.  All three products of a layer run as register-tiled shared-memory kernels on the
// packed two-lane fp32 multiply-add (fma.rn.f32x2: two roundings, each that of fmaf, in one issue
// slot).  They keep that pipe about half busy: the moves that put one input into both lanes, the staging
// between barriers and the uneven last CTAs take the rest.
#include <algorithm>

#include "common.cuh"
#include "lsgd_internal.h"

namespace lsgd {
namespace {

// Four consecutive elements of an activation tensor as fp32.
__device__ __forceinline__ float4 load4(const float* p) { return __ldg(reinterpret_cast<const float4*>(p)); }
__device__ __forceinline__ float4 load4(const uint16_t* p) {
  const uint2 u = __ldg(reinterpret_cast<const uint2*>(p));
  return make_float4(bf2f((uint16_t)(u.x & 0xffffu)), bf2f((uint16_t)(u.x >> 16)),
                     bf2f((uint16_t)(u.y & 0xffffu)), bf2f((uint16_t)(u.y >> 16)));
}

// A tile of pixels: ti images x th rows x tw columns (powers of two) of the output grid, chosen so
// that images narrower than the tile still fill it.
struct Tile {
  int tw, th, ti;      // log2
  int nx, ny;          // tiles across and down an image
  int tiles;           // tiles of one replica
};

int log2_ceil(int v) {
  int l = 0;
  while ((1 << l) < v) ++l;
  return l;
}

Tile tile_of(int B, int H, int W, int px_log2) {
  Tile t;
  t.tw = std::max(3, std::min(5, log2_ceil(W)));
  t.th = std::min(px_log2 - t.tw, log2_ceil(H));
  t.ti = px_log2 - t.tw - t.th;
  t.nx = (W + (1 << t.tw) - 1) >> t.tw;
  t.ny = (H + (1 << t.th) - 1) >> t.th;
  t.tiles = ((B + (1 << t.ti) - 1) >> t.ti) * t.nx * t.ny;
  return t;
}

// ---------------------------------------------------------------------------------------------
// Forward and data gradient: out[g][b][y][x][co] = sum over taps t and ci of
// in[g][b][y S + t / 3 - 1][x S + t % 3 - 1][ci] w_t[co][ci].  The data gradient is this with the
// output gradient as input and w_t[ci][co] = w[co][8 - t][ci] (flip); a stride-2 layer's reads the
// output gradient with zeros between its pixels (up).
//
// A CTA computes 256 pixels x 16 channels, a thread 8 consecutive pixels x 4 channels (2 packed pairs).
// Eight input channels at a time, the tile's input with its halo is staged as one plane per channel
// and their weights as [channel][tap][16].  Per channel and kernel row a thread loads 10 inputs (17 at
// stride 2) and 12 weights for 48 packed multiply-adds: 22 words through the shared-memory pipe's 32
// lanes a cycle against 24 cycles of multiply-adds (4 pixels x 8 channels: 30 words, that pipe bound).
// Four lanes share a pixel group and eight a weight group, so a load's lanes do not conflict.  A
// slice's loads are all requested before the barrier that frees the staging buffers.  The eight
// channels' products are summed by themselves and then added to the running sum, which halves the
// length of the longest chain of roundings at 16 channels and keeps it at 72 + Cin / 8 for any Cin.
// The 16-channel tile over 256 pixels reads each input once per 16 outputs; wider tiles of 32
// channels leave too few CTAs on the later, smaller stages.
// KS = 2, where at most two CTAs per SM would leave the schedulers two warps each (a late stage: 256
// CTAs): a second 128 threads take the odd groups of eight channels, and their sums are added at the
// end.  64 channels of 8 x 8 pixels: 43 -> 38 us, a whole pass of two steps 6.50 -> 6.15 ms; at up to four
// CTAs per SM it gains nothing more (6.16).  Plain fmaf, without the packing moves, is slower (52 us), and
// so are copies of the next slice in flight during this one's products (6.96 ms at KS = 1).
// Measured, ResNet-20 in fp32, K = 4, B = 64, per step: 1.45 ms forward and data gradients (1.65 ms with
// 4 pixels x 8 channels, weight stores in 16-way conflicts and the shortcut added element by element;
// 7.3 ms with one thread per pixel that loaded a weight per multiply-add).
constexpr int kFwThreads = 128, kFwPxLog2 = 8, kFwCo = 16, kFwCi = 8, kFwPx = 8;
constexpr int kFwWPitch = kFwCo + 4;  // a tap's weights; 20 floats: eight channels by four taps, as a warp
                                      // stores them, spread over eight groups of four banks (16: over two banks)

constexpr int kFwMaxSmem = 100 * 1024;

struct ConvFwArgs {
  const void* in;
  const void* w;
  int64_t w_gs;
  float* out;
  int B, Hi, Wi, Ci, Ho, Wo, Co;
  int up, flip;
  Tile t;
  int pr, pc, pitch;  // patch rows and columns per image, row pitch (floats)
  // the block's shortcut: out += sc_dout * (sc_act > 0) at (y / sc_s, x / sc_s) where both are whole
  const float* sc_dout;
  const void* sc_act;
  int sc_s, sc_H, sc_W, sc_C;
};

template <typename TA, int S, int KS>
__global__ void __launch_bounds__(kFwThreads * KS, 4 / KS)
    conv3x3_simt_kernel(const __grid_constant__ ConvFwArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) float fw_sm[];
  constexpr int NT = kFwThreads * KS, CI = kFwCi * KS, NW = CI * 9 * kFwCo / NT;
  const int plane = (a.pr * a.pitch) << a.t.ti;
  float* patch = fw_sm;                                   // [CI][ti][pr][pitch]
  float* ws = patch + CI * plane;                         // [CI][9][kFwWPitch]
  int2* table = reinterpret_cast<int2*>(ws + CI * 9 * kFwWPitch);  // per patch pixel: source, place
  const int tid = threadIdx.x, ht = tid % kFwThreads, half = tid / kFwThreads;
  const int g = blockIdx.z, co0 = blockIdx.y * kFwCo;
  int tile = blockIdx.x;
  const int x0 = (tile % a.t.nx) << a.t.tw;
  tile /= a.t.nx;
  const int y0 = (tile % a.t.ny) << a.t.th;
  const int b0 = (tile / a.t.ny) << a.t.ti;
  const int npx = (a.pr * a.pc) << a.t.ti;
  for (int e = tid; e < npx; e += NT) {
    const int px = e % a.pc, r = e / a.pc, py = r % a.pr, im = r / a.pr;
    int iy = y0 * S + py - 1, ix = x0 * S + px - 1;
    bool in = b0 + im < a.B && iy >= 0 && ix >= 0;
    if (a.up) {
      in = in && !((iy | ix) & 1);
      iy >>= 1;
      ix >>= 1;
    }
    in = in && iy < a.Hi && ix < a.Wi;
    table[e] = make_int2(in ? ((b0 + im) * a.Hi + iy) * a.Wi + ix : -1, (im * a.pr + py) * a.pitch + px);
  }
  const TA* in = reinterpret_cast<const TA*>(a.in) + (int64_t)g * a.B * a.Hi * a.Wi * a.Ci;
  const TA* w = reinterpret_cast<const TA*>(a.w) + (int64_t)g * a.w_gs;

  const int cog = tid & 3, px = (ht >> 2) * kFwPx;  // four channels; first pixel
  const int gx = px & ((1 << a.t.tw) - 1), gr = px >> a.t.tw;
  const int gy = gr & ((1 << a.t.th) - 1), gi = gr >> a.t.th;
  const float* prow = patch + (gi * a.pr + gy * S) * a.pitch + gx * S;
  const float* wrow = ws + 4 * cog;

  u64 sum[kFwPx][2];
#pragma unroll
  for (int p = 0; p < kFwPx; ++p) sum[p][0] = sum[p][1] = 0ull;

  __syncthreads();  // the table
  const bool quads = (a.Ci & 3) == 0;
  // weight i of this thread in a slice: consecutive threads on consecutive elements of the tensor
  auto weight_at = [&](int i, int& co, int& t, int& c) {
    const int e = tid + i * NT;
    if (!a.flip)
      c = e % CI, t = (e / CI) % 9, co = e / (9 * CI);
    else
      co = e % kFwCo, t = (e / kFwCo) % 9, c = e / (9 * kFwCo);
  };
  auto weight_src = [&](int c0, int co, int t, int c) {
    return a.flip ? w + ((int64_t)(c0 + c) * 9 + 8 - t) * a.Co + co0 + co
                  : w + ((int64_t)(co0 + co) * 9 + t) * a.Ci + c0 + c;
  };
  const int h0 = half * kFwCi;  // the half's channels of a slice
  auto put = [&](int place, int c, const float4& v) {
    float* d = patch + c * plane + place;
    d[0] = v.x;
    d[plane] = v.y;
    d[2 * plane] = v.z;
    d[3 * plane] = v.w;
  };
  for (int c0 = 0; c0 < a.Ci; c0 += CI) {
    const int nc = min(CI, a.Ci - c0);
    // all of a slice's loads, the weights' first, before the barrier
    float wv[NW];
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      int co, t, c;
      weight_at(i, co, t, c);
      wv[i] = 0.f;
      if (c < nc && co0 + co < a.Co) wv[i] = Elem<TA>::load(weight_src(c0, co, t, c));
    }
    if (quads) {
      constexpr int NB = 3;
      for (int e0 = ht; e0 - ht < npx; e0 += NB * kFwThreads) {
        int2 s[NB];
        float4 v[NB][2];
#pragma unroll
        for (int i = 0; i < NB; ++i) {
          const int e = e0 + i * kFwThreads;
          s[i] = e < npx ? table[e] : make_int2(-1, -1);
#pragma unroll
          for (int h = 0; h < 2; ++h)
            v[i][h] = s[i].x >= 0 && h0 + 4 * h < nc ? load4(in + (int64_t)s[i].x * a.Ci + c0 + h0 + 4 * h)
                                                     : make_float4(0.f, 0.f, 0.f, 0.f);
        }
        if (e0 == ht) __syncthreads();
#pragma unroll
        for (int i = 0; i < NB; ++i) {
          if (s[i].y < 0) break;
          put(s[i].y, h0, v[i][0]);
          put(s[i].y, h0 + 4, v[i][1]);
        }
      }
    } else {
      __syncthreads();
      for (int e = tid; e < npx; e += NT) {
        const int2 s = table[e];
        for (int c = 0; c < nc; ++c)
          patch[c * plane + s.y] = s.x >= 0 ? Elem<TA>::load(in + (int64_t)s.x * a.Ci + c0 + c) : 0.f;
      }
    }
#pragma unroll
    for (int i = 0; i < NW; ++i) {
      int co, t, c;
      weight_at(i, co, t, c);
      ws[(c * 9 + t) * kFwWPitch + co] = wv[i];
    }
    __syncthreads();
    u64 acc[kFwPx][2];
#pragma unroll
    for (int p = 0; p < kFwPx; ++p) acc[p][0] = acc[p][1] = 0ull;
    for (int c = h0; c < min(nc, h0 + kFwCi); ++c) {
#pragma unroll
      for (int kh = 0; kh < 3; ++kh) {
        const float* r = prow + c * plane + kh * a.pitch;
        constexpr int NV = (kFwPx - 1) * S + 3;
        float v[NV];
#pragma unroll
        for (int i = 0; i + 4 <= NV; i += 4) {
          const float4 f = *reinterpret_cast<const float4*>(r + i);
          v[i] = f.x;
          v[i + 1] = f.y;
          v[i + 2] = f.z;
          v[i + 3] = f.w;
        }
        if (S == 1) {
          const float2 f = *reinterpret_cast<const float2*>(r + NV - 2);
          v[NV - 2] = f.x;
          v[NV - 1] = f.y;
        } else {
          v[NV - 1] = r[NV - 1];
        }
#pragma unroll
        for (int kw = 0; kw < 3; ++kw) {
          const ulonglong2 wq = *reinterpret_cast<const ulonglong2*>(wrow + (c * 9 + kh * 3 + kw) * kFwWPitch);
#pragma unroll
          for (int p = 0; p < kFwPx; ++p) {
            const u64 x = pack2(v[p * S + kw], v[p * S + kw]);
            fma2(acc[p][0], x, wq.x);
            fma2(acc[p][1], x, wq.y);
          }
        }
      }
    }
#pragma unroll
    for (int p = 0; p < kFwPx; ++p) {
      add2(sum[p][0], acc[p][0]);
      add2(sum[p][1], acc[p][1]);
    }
  }

  if constexpr (KS == 2) {
    // the second half's sums to the first, where the staging buffers were
    u64* other = reinterpret_cast<u64*>(fw_sm) + ht;
    __syncthreads();
    if (half) {
#pragma unroll
      for (int p = 0; p < kFwPx; ++p)
#pragma unroll
        for (int q = 0; q < 2; ++q) other[(2 * p + q) * kFwThreads] = sum[p][q];
    }
    __syncthreads();
    if (half) return;
#pragma unroll
    for (int p = 0; p < kFwPx; ++p)
#pragma unroll
      for (int q = 0; q < 2; ++q) add2(sum[p][q], other[(2 * p + q) * kFwThreads]);
  }

  const int b = b0 + gi, y = y0 + gy;
  if (b >= a.B || y >= a.Ho) return;
  const int co = co0 + 4 * cog;
  const int64_t img = (int64_t)g * a.B + b;
  const bool sc_row = a.sc_dout && y % a.sc_s == 0, whole = ((a.Co | a.sc_C) & 3) == 0;
  auto sc_at = [&](int x) { return ((img * a.sc_H + y / a.sc_s) * a.sc_W + x / a.sc_s) * a.sc_C + co; };
  float4 act[kFwPx], d[kFwPx];  // the shortcut's, requested together
#pragma unroll
  for (int p = 0; p < kFwPx; ++p) {
    const int x = x0 + gx + p;
    const bool on = sc_row && whole && co < a.Co && x < a.Wo && x % a.sc_s == 0;
    act[p] = d[p] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (on) {
      act[p] = load4(reinterpret_cast<const TA*>(a.sc_act) + sc_at(x));
      d[p] = load4(a.sc_dout + sc_at(x));
    }
  }
#pragma unroll
  for (int p = 0; p < kFwPx; ++p) {
    const int x = x0 + gx + p;
    if (x >= a.Wo) break;
    const float2 lo = unpack2(sum[p][0]), hi = unpack2(sum[p][1]);
    float o[4] = {lo.x, lo.y, hi.x, hi.y};
    o[0] = act[p].x > 0.f ? o[0] + d[p].x : o[0];
    o[1] = act[p].y > 0.f ? o[1] + d[p].y : o[1];
    o[2] = act[p].z > 0.f ? o[2] + d[p].z : o[2];
    o[3] = act[p].w > 0.f ? o[3] + d[p].w : o[3];
    if (sc_row && !whole && x % a.sc_s == 0) {
      const int64_t e = sc_at(x);
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (co + i < a.Co && Elem<TA>::load(reinterpret_cast<const TA*>(a.sc_act) + e + i) > 0.f)
          o[i] += a.sc_dout[e + i];
    }
    float* dst = a.out + ((img * a.Ho + y) * a.Wo + x) * a.Co + co;
    if ((a.Co & 3) == 0) {
      if (co < a.Co) *reinterpret_cast<float4*>(dst) = make_float4(o[0], o[1], o[2], o[3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (co + i < a.Co) dst[i] = o[i];
    }
  }
}

template <typename TA, int S, int KS>
cudaError_t launch_fw_ks(const ConvFwArgs& a, dim3 grid, size_t smem, cudaStream_t s) {
  static std::atomic<int> attr_dev{-1};  // several threads may launch
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(conv3x3_simt_kernel<TA, S, KS>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             kFwMaxSmem);
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  return launch_pdl(conv3x3_simt_kernel<TA, S, KS>, grid, dim3(kFwThreads * KS), smem, s, a);
}

template <typename TA, int S>
cudaError_t launch_fw(ConvFwArgs a, int G, cudaStream_t s) {
  a.t = tile_of(a.B, a.Ho, a.Wo, kFwPxLog2);
  a.pr = ((1 << a.t.th) - 1) * S + 3;
  a.pc = ((1 << a.t.tw) - 1) * S + 3;
  a.pitch = (a.pc + 3) / 4 * 4;  // rows start on 16 bytes
  const dim3 grid(a.t.tiles, (a.Co + kFwCo - 1) / kFwCo, G);
  if (grid.y > 65535 || grid.z > 65535) return cudaErrorInvalidValue;
  auto smem = [&](int ks) {
    return (size_t)ks * kFwCi * (((a.pr * a.pitch) << a.t.ti) + 9 * kFwWPitch) * 4 +
           (size_t)((a.pr * a.pc) << a.t.ti) * sizeof(int2);
  };
  if constexpr (S == 1) {
    if (a.Ci > kFwCi && (int64_t)grid.x * grid.y * grid.z <= 2 * kNumSMs && smem(2) <= kFwMaxSmem)
      return launch_fw_ks<TA, S, 2>(a, grid, smem(2), s);
  }
  return launch_fw_ks<TA, S, 1>(a, grid, smem(1), s);
}

// ---------------------------------------------------------------------------------------------
// Weight gradient: part[g][q][co][t][ci] = sum over the pixels of range q of
// dy[p][co] x[p S + tap t][ci]; the ranges' partials are added in order by a second kernel.
//
// A CTA takes 16 output x 16 input channels and a range of 128-pixel tiles, staged as they lie in
// memory (64 bytes a pixel) by asynchronous copies, the next tile's while this one is summed.  Warp
// w works on kernel row w % 3; its 16 lanes of a half cover 4 x 4 blocks of 4 output x 4 input
// channels, and the four half-warps of a kernel row take rows r, r + 4, ... of the tile.  A thread
// walks its row four pixels at a time: one load per pixel of dy and of x (two at stride 2; the
// columns that the three kernel columns share stay in registers), 24 packed multiply-adds.  At the end
// the four rows' sums are added in a fixed order.
// An accumulator's chain is a tile range's pixels / 4: at most 32 kWgRangeTiles = 2,048 roundings, however
// many replicas share the launch.
// Measured, ResNet-20 in fp32, K = 4, B = 64, per step: 0.78 ms (46.7 ms with 16 pixels staged
// between two barriers and a shared-memory load per multiply-add).
constexpr int kWgThreads = 192, kWgPxLog2 = 7, kWgRangeTiles = 64;
constexpr int64_t kSmemPerSm = 228 * 1024;  // of which each CTA takes 1 KB besides its own

struct ConvWgArgs {
  const void* x;
  const void* dy;
  float* part;
  int B, Hi, Wi, Ci, Ho, Wo, Co;
  int nq, ci_blocks;
  Tile t;
  int pr, pc, xpitch, dpitch;  // x patch rows and columns per image; row pitches in pixels of 16 floats
};

__device__ __forceinline__ void cp_async(float* dst, const void* src, int bytes, bool in) {
  const uint32_t d = (uint32_t)__cvta_generic_to_shared(dst);
  const int n = in ? bytes : 0;
  if (bytes == 16)
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
  else
    asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(n) : "memory");
}

// One pixel's 16 channels c0 .. c0 + 15 (zeros from C on, and all zeros if !in) to dst; four lanes
// (q = 0 .. 3) per pixel.
template <typename TA>
__device__ __forceinline__ void stage_px(float* dst, const TA* base, int64_t px, int C, int c0, int q,
                                         bool in) {
  const int c = c0 + 4 * q;
  const TA* src = base + (in ? px * C + c : 0);
  if constexpr (sizeof(TA) == 4) {
    if ((C & 3) == 0) {
      const bool ok = in && c < C;
      cp_async(dst + 4 * q, ok ? src : base, 16, ok);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const bool ok = in && c + i < C;
        cp_async(dst + 4 * q + i, ok ? src + i : base, 4, ok);
      }
    }
  } else {
    float v[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) v[i] = in && c + i < C ? Elem<TA>::load(src + i) : 0.f;
    *reinterpret_cast<float4*>(dst + 4 * q) = make_float4(v[0], v[1], v[2], v[3]);
  }
}

template <typename TA, int S>
__global__ void __launch_bounds__(kWgThreads, 3) conv_wgrad_simt_kernel(const __grid_constant__ ConvWgArgs a) {
  pdl_begin();
  extern __shared__ __align__(16) float wg_sm[];
  const int rows = 1 << (a.t.th + a.t.ti);   // rows of the tile
  const int dfl = rows * a.dpitch * 16, xfl = (a.pr << a.t.ti) * a.xpitch * 16;  // floats
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int g = blockIdx.z, q = blockIdx.x;
  const int co0 = (blockIdx.y / a.ci_blocks) * 16, ci0 = (blockIdx.y % a.ci_blocks) * 16;
  const int t_lo = (int)((int64_t)q * a.t.tiles / a.nq), t_hi = (int)((int64_t)(q + 1) * a.t.tiles / a.nq);
  const TA* dy = reinterpret_cast<const TA*>(a.dy) + (int64_t)g * a.B * a.Ho * a.Wo * a.Co;
  const TA* x = reinterpret_cast<const TA*>(a.x) + (int64_t)g * a.B * a.Hi * a.Wi * a.Ci;

  auto stage = [&](int tile, float* buf) {
    const int x0 = (tile % a.t.nx) << a.t.tw;
    tile /= a.t.nx;
    const int y0 = (tile % a.t.ny) << a.t.th, b0 = (tile / a.t.ny) << a.t.ti;
    for (int e = tid; e < rows << (a.t.tw + 2); e += kWgThreads) {
      const int p = e >> 2, c = p & ((1 << a.t.tw) - 1), r = p >> a.t.tw;
      const int y = y0 + (r & ((1 << a.t.th) - 1)), b = b0 + (r >> a.t.th), xx = x0 + c;
      const bool in = b < a.B && y < a.Ho && xx < a.Wo;
      stage_px(buf + (r * a.dpitch + c) * 16, dy, ((int64_t)b * a.Ho + y) * a.Wo + xx, a.Co, co0, e & 3, in);
    }
    float* xb = buf + dfl;
    for (int r = warp; r < a.pr << a.t.ti; r += kWgThreads / 32) {
      const int im = r / a.pr, iy = y0 * S + (r - im * a.pr) - 1, b = b0 + im;
      const bool row_in = b < a.B && iy >= 0 && iy < a.Hi;
      for (int e = lane; e < a.pc * 4; e += 32) {
        const int c = e >> 2, ix = x0 * S + c - 1;
        const bool in = row_in && ix >= 0 && ix < a.Wi;
        stage_px(xb + (r * a.xpitch + c) * 16, x, ((int64_t)b * a.Hi + iy) * a.Wi + ix, a.Ci, ci0, e & 3, in);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };

  const int kh = warp % 3, slice = 2 * (warp / 3) + (lane >> 4);
  const int cob = (lane >> 2) & 3, cib = lane & 3;
  u64 acc[3][4][2];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int o = 0; o < 4; ++o) acc[k][o][0] = acc[k][o][1] = 0ull;

  if (t_lo < t_hi) stage(t_lo, wg_sm);
  for (int t = t_lo; t < t_hi; ++t) {
    float* buf = wg_sm + ((t - t_lo) & 1) * (dfl + xfl);
    if (t + 1 < t_hi) {
      stage(t + 1, wg_sm + ((t + 1 - t_lo) & 1) * (dfl + xfl));
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    for (int r = slice; r < rows; r += 4) {
      const int im = r >> a.t.th, y = r & ((1 << a.t.th) - 1);
      const float* dr = buf + r * a.dpitch * 16 + 4 * cob;
      const float* xr = buf + dfl + (im * a.pr + y * S + kh) * a.xpitch * 16 + 4 * cib;
      constexpr int NX = 3 * S + 3;  // columns under four pixels
      ulonglong2 xv[NX];
#pragma unroll
      for (int i = 0; i < 3 - S; ++i) xv[i] = *reinterpret_cast<const ulonglong2*>(xr + i * 16);
      for (int c = 0; c < 1 << a.t.tw; c += 4) {
        float4 d[4];
#pragma unroll
        for (int p = 0; p < 4; ++p) d[p] = *reinterpret_cast<const float4*>(dr + (c + p) * 16);
#pragma unroll
        for (int i = 3 - S; i < NX; ++i)
          xv[i] = *reinterpret_cast<const ulonglong2*>(xr + (c * S + i) * 16);
#pragma unroll
        for (int p = 0; p < 4; ++p) {
          const u64 dd[4] = {pack2(d[p].x, d[p].x), pack2(d[p].y, d[p].y), pack2(d[p].z, d[p].z),
                             pack2(d[p].w, d[p].w)};
#pragma unroll
          for (int k = 0; k < 3; ++k)
#pragma unroll
            for (int o = 0; o < 4; ++o) {
              fma2(acc[k][o][0], dd[o], xv[p * S + k].x);
              fma2(acc[k][o][1], dd[o], xv[p * S + k].y);
            }
        }
#pragma unroll
        for (int i = 0; i < 3 - S; ++i) xv[i] = xv[i + 4 * S];
      }
    }
    __syncthreads();  // the buffer is free for the tile after next
  }

  // the four rows' sums: (0 + 1) + (2 + 3), across the half-warps, then through shared memory
  float* red = wg_sm;  // [3][16 lanes][48]
  float v[48];
#pragma unroll
  for (int k = 0; k < 3; ++k)
#pragma unroll
    for (int o = 0; o < 4; ++o)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const float2 f = unpack2(acc[k][o][h]);
        v[(k * 4 + o) * 4 + 2 * h] = f.x;
        v[(k * 4 + o) * 4 + 2 * h + 1] = f.y;
      }
#pragma unroll
  for (int i = 0; i < 48; ++i) v[i] += __shfl_xor_sync(0xffffffffu, v[i], 16);
  if (warp >= 3 && lane < 16)
#pragma unroll
    for (int i = 0; i < 48; ++i) red[(kh * 48 + i) * 16 + lane] = v[i];
  __syncthreads();
  if (warp < 3 && lane < 16) {
    float* out = a.part + ((int64_t)g * a.nq + q) * a.Co * 9 * a.Ci;
#pragma unroll
    for (int k = 0; k < 3; ++k)
#pragma unroll
      for (int o = 0; o < 4; ++o) {
        const int co = co0 + 4 * cob + o, ci = ci0 + 4 * cib;
        if (co >= a.Co) continue;
        float* dst = out + ((int64_t)co * 9 + kh * 3 + k) * a.Ci + ci;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int e = (k * 4 + o) * 4 + i;
          if (ci + i < a.Ci) dst[i] = v[e] + red[(kh * 48 + e) * 16 + lane];
        }
      }
  }
}

// The staging's geometry at stride S, and its shared memory.
size_t wg_staging(ConvWgArgs& a, int S) {
  a.pr = ((1 << a.t.th) - 1) * S + 3;
  a.pc = ((1 << a.t.tw) - 1) * S + 3;
  // odd row pitches: the two half-warps of a warp, a row apart, then read different banks
  a.xpitch = a.pc | 1;
  a.dpitch = (1 << a.t.tw) | 1;
  const size_t floats = (size_t)((a.dpitch << (a.t.th + a.t.ti)) + (a.pr << a.t.ti) * a.xpitch) * 16;
  return std::max<size_t>(2 * floats, 3 * 48 * 16) * 4;
}

template <typename TA, int S>
cudaError_t launch_wg(ConvWgArgs a, int G, cudaStream_t s) {
  const size_t smem = wg_staging(a, S);
  const dim3 grid(a.nq, ((a.Co + 15) / 16) * a.ci_blocks, G);
  if (grid.y > 65535 || grid.z > 65535 || smem > 160 * 1024) return cudaErrorInvalidValue;
  static std::atomic<int> attr_dev{-1};  // several threads may launch
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (attr_dev != dev) {
    e = cudaFuncSetAttribute(conv_wgrad_simt_kernel<TA, S>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             160 * 1024);
    if (e != cudaSuccess) return e;
    attr_dev = dev;
  }
  return launch_pdl(conv_wgrad_simt_kernel<TA, S>, grid, dim3(kWgThreads), smem, s, a);
}

}  // namespace

cudaError_t launch_conv3x3_simt(const ConvSimtArgs& c, cudaStream_t s) {
  if (c.G < 1 || c.B < 1 || (c.stride != 1 && c.stride != 2) || c.cin < 1 || c.cout < 1)
    return cudaErrorInvalidValue;
  ConvFwArgs a{};
  a.in = c.in;
  a.w = c.w;
  a.w_gs = c.w_gs;
  a.out = c.out;
  a.B = c.B;
  if (!c.dgrad) {
    a.Hi = c.hin, a.Wi = c.win, a.Ci = c.cin, a.Ho = c.hout, a.Wo = c.wout, a.Co = c.cout;
  } else {
    a.Hi = c.hout, a.Wi = c.wout, a.Ci = c.cout, a.Ho = c.hin, a.Wo = c.win, a.Co = c.cin;
    a.flip = 1;
    a.up = c.stride == 2;
    a.sc_dout = c.sc_dout;
    a.sc_act = c.sc_act;
    a.sc_s = c.stride;
    a.sc_H = c.hout, a.sc_W = c.wout, a.sc_C = c.cout;
  }
  if ((int64_t)a.B * a.Hi * a.Wi > 0x7fffffffLL) return cudaErrorInvalidValue;
  const bool two = !c.dgrad && c.stride == 2;
  if (c.bf16) return two ? launch_fw<uint16_t, 2>(a, c.G, s) : launch_fw<uint16_t, 1>(a, c.G, s);
  return two ? launch_fw<float, 2>(a, c.G, s) : launch_fw<float, 1>(a, c.G, s);
}

// Ranges of one replica: as many CTAs over the replicas and channel blocks as are resident, in one wave -- per
// SM three, or the two or one whose staging its shared memory holds (stride 2, and outputs one or two rows
// high) -- and at least one tile each.  (Four per SM ran as a wave and a third: 55 against 46 us at 64
// channels, 41 against 38 at 16.  Three at stride 2, where two fit: 36.6 against 30.1 us for 16 x 16 pixels,
// 42.5 against 34.2 for 8 x 8, K = 4, B = 64.)
// At most kWgRangeTiles tiles each, in as many waves as that takes, so that many replicas or a large batch
// do not lengthen the fp32 chains: K = 64, B = 128, 16 x 16 pixels of 32 channels would otherwise be one range
// of 256 tiles, 8,192 roundings.  (The ranges, and so the last bits of a replica's gradient, depend on how
// many replicas share the launch, as the tensor-core kernel's do.)
int conv_wgrad_simt_ranges(int G, int B, int hout, int wout, int cin, int cout, int stride) {
  ConvWgArgs a{};
  a.t = tile_of(B, hout, wout, kWgPxLog2);
  const int blocks = ((cout + 15) / 16) * ((cin + 15) / 16), tiles = a.t.tiles;
  const int64_t per_sm = std::max<int64_t>(1, std::min<int64_t>(3, kSmemPerSm / (wg_staging(a, stride) + 1024)));
  const int64_t wave = std::min<int64_t>(tiles, per_sm * kNumSMs / ((int64_t)G * blocks));
  return (int)std::max<int64_t>(wave, (tiles + kWgRangeTiles - 1) / kWgRangeTiles);
}

cudaError_t launch_conv_wgrad_simt(const ConvSimtArgs& c, const void* dy, float* part, cudaStream_t s) {
  if (c.G < 1 || c.B < 1 || (c.stride != 1 && c.stride != 2) || c.cin < 1 || c.cout < 1)
    return cudaErrorInvalidValue;
  ConvWgArgs a{};
  a.x = c.in;
  a.dy = dy;
  a.part = part;
  a.B = c.B;
  a.Hi = c.hin, a.Wi = c.win, a.Ci = c.cin, a.Ho = c.hout, a.Wo = c.wout, a.Co = c.cout;
  a.ci_blocks = (c.cin + 15) / 16;
  a.t = tile_of(c.B, c.hout, c.wout, kWgPxLog2);
  a.nq = conv_wgrad_simt_ranges(c.G, c.B, c.hout, c.wout, c.cin, c.cout, c.stride);
  if (c.bf16)
    return c.stride == 2 ? launch_wg<uint16_t, 2>(a, c.G, s) : launch_wg<uint16_t, 1>(a, c.G, s);
  return c.stride == 2 ? launch_wg<float, 2>(a, c.G, s) : launch_wg<float, 1>(a, c.G, s);
}

}  // namespace lsgd
