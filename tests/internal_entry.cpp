// Plain-C doors to launchers that have no entry point of their own, for the tests that look at them one
// at a time: everything is passed as integers and device pointers.  Host code only, built by _internal.py.
#include "lsgd_internal.h"

using namespace lsgd;

namespace {
ConvSimtArgs simt(int bf16, int G, int B, int hout, int wout, int cin, int cout, int stride) {
  ConvSimtArgs a{};
  a.bf16 = bf16 != 0;
  a.G = G, a.B = B, a.hin = hout * stride, a.win = wout * stride, a.cin = cin;
  a.hout = hout, a.wout = wout, a.cout = cout, a.stride = stride;
  return a;
}
}  // namespace

extern "C" {

int t_wgrad_simt_ranges(int G, int B, int hout, int wout, int cin, int cout, int stride) {
  return conv_wgrad_simt_ranges(G, B, hout, wout, cin, cout, stride);
}

int t_wgrad_simt(int G, int B, int hout, int wout, int cin, int cout, int stride, const float* x,
                 const float* dy, float* part, void* stream) {
  ConvSimtArgs a = simt(0, G, B, hout, wout, cin, cout, stride);
  a.in = x;
  return (int)launch_conv_wgrad_simt(a, dy, part, (cudaStream_t)stream);
}

// A data gradient with the BatchNorm-backward epilogue on the super-pixel kernel: in = dy [G][B][hi][wi][ck],
// w as ConvSpArgs has it.  With part NULL nothing is launched; the partials per replica, or minus the error.
int t_conv_sp_bwd(int G, int B, int hi, int wi, int ck, int N, int phases, const uint16_t* dy,
                  const uint16_t* w, float* out, const uint16_t* mask, const float* y, const float* mean,
                  const float* rstd, const float* sc_dout, const uint16_t* sc_out, int sc_C, int sc_stride,
                  float* part, void* stream) {
  const int64_t per = (int64_t)N * 9 * ck, px = (int64_t)B * hi * wi;
  ConvSpArgs a{};
  a.w = w, a.w_gs = per, a.w_ps = phases ? G * per : 0;
  a.ck = ck, a.N = N, a.stride = 1, a.phases = phases, a.hi = hi, a.wi = wi, a.B = B, a.G = G;
  a.out = out, a.out_gs = px * (phases ? 4 : 1) * N;
  a.bwd.mask = mask, a.bwd.y = y, a.bwd.mean = mean, a.bwd.rstd = rstd;
  a.bwd.sc_dout = sc_dout, a.bwd.sc_out = sc_out, a.bwd.sc_gs = px * sc_C, a.bwd.sc_C = sc_C;
  a.bwd.sc_stride = sc_stride;
  const int n = conv_sp_parts(a);
  if (!part || n == 0) return n;
  a.bwd.part = reinterpret_cast<float2*>(part), a.bwd.part_gs = n;
  const cudaError_t e = launch_conv_sp(a, dy, (cudaStream_t)stream);
  return e == cudaSuccess ? n : -(int)e;
}

}  // extern "C"
