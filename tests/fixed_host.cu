// The fixed-point functions of csrc/dgpe_fixed.cuh compiled for the host, for test_fixed_host.py.
#include "dgpe_fixed.cuh"

using namespace dgpe;

namespace {
fxw words(long long re, long long im) { return {fx_hi(re), fx_lo(re), fx_hi(im), fx_lo(im)}; }
}  // namespace

extern "C" {
// a w / 2^64 (dir < 0) or a conj(w) / 2^64
void host_twiddle(int dir, const long long *a, const long long *w, long long *out) {
  const fxc r = dir < 0 ? fx_twiddle<-1>({a[0], a[1]}, words(w[0], w[1])) : fx_twiddle<+1>({a[0], a[1]}, words(w[0], w[1]));
  out[0] = r.re;
  out[1] = r.im;
}
}
