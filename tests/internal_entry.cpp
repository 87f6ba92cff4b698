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

}  // extern "C"
