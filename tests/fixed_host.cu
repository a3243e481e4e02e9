// The fixed-point functions of csrc/dgpe_fixed.cuh compiled for the host, for test_fixed_host.py.
#include <cmath>
#include <vector>

#include "dgpe_fixed.cuh"

using namespace dgpe;

namespace {
// One line of the real-time sweep k_cn_fx, interior points only: al, be = alpha and 2 beta (FP64 pairs) of m
// points, ginv = 1 / gamma, r = dt / (4 h^2).
struct Z {
  double re, im;
};
Z mul(Z a, Z b) { return {a.re * b.re - a.im * b.im, a.re * b.im + a.im * b.re}; }
Z operator+(Z a, Z b) { return {a.re + b.re, a.im + b.im}; }
void sweep(int m, double r, const Z *al, const Z *be, Z ginv, Z *psi) {
  const int h = m / 2, n = h + 2;
  auto exponent = [&](const Z *t) {
    double mx = 0.0;
    for (int i = 0; i < n && i < m; ++i) mx = std::fmax(mx, std::sqrt(t[i].re * t[i].re + t[i].im * t[i].im));
    int e = 0;
    std::frexp(mx * (1.0 + 1e-15), &e);
    return mx > 0.0 ? std::min(-e, 60) : 60;
  };
  const int ka = exponent(al), kb = exponent(be);
  auto coef = [&](const Z *t, int i, int k) {
    return i < m ? fx_words(std::llrint(std::ldexp(t[i].re, kFxCoefBits + k)), std::llrint(std::ldexp(t[i].im, kFxCoefBits + k))) : fxw{0, 0, 0, 0};
  };
  std::vector<fxc> y(m);
  std::vector<Z> out(m);
  auto forward = [&](bool bottom, int nf) {
    fxv v = {{0, 0}, kFxMinExp};
    for (int s = 0; s < nf; ++s) {
      const int i = bottom ? m - 1 - s : s;
      const fxc t = fx_coef(v.v, coef(al, s, ka));
      v = fx_forward(psi[i].re, psi[i].im, fx_key(cplx<double>{psi[i].re, psi[i].im}), t, v.e + 3 - ka);
      y[i] = fx_pack(v);
    }
    return Z{fx_to(v.v.re, v.e + 1086), fx_to(v.v.im, v.e + 1086)};
  };
  const Z yt = forward(false, h), yb = forward(true, m - 1 - h);
  const Z xh = mul(ginv, psi[h] + mul(al[h], yt) + mul(al[m - 1 - h], yb));
  out[h] = {2.0 * xh.re - psi[h].re, 2.0 * xh.im - psi[h].im};
  const Z cx = {-r * xh.im, r * xh.re};
  const int ex = std::max(fx_key(cplx<double>{cx.re, cx.im}) >> 20, kFxMinBiased);
  for (int bottom = 0; bottom < 2; ++bottom) {
    const int nf = bottom ? m - 1 - h : h;
    fxc t = {fx_from<6>(cx.re, ex), fx_from<6>(cx.im, ex)};
    int et = ex - 1081;
    for (int j = 0; j < nf; ++j) {
      const int q = nf - 1 - j, i = bottom ? h + 1 + j : h - 1 - j;
      const fxv x = fx_backward(fx_unpack(y[i]), t, et);
      const fxc b = fx_coef(x.v, coef(be, q, kb));
      t = fx_coef(x.v, coef(al, q + 1, ka));
      et = x.e + 3 - ka;
      out[i] = {fx_to_int(b.re, x.e + 3 - kb + 1086) - psi[i].re, fx_to_int(b.im, x.e + 3 - kb + 1086) - psi[i].im};
    }
  }
  for (int i = 0; i < m; ++i) psi[i] = out[i];
}
}  // namespace

extern "C" {
// a w / 2^64 (dir < 0) or a conj(w) / 2^64
void host_twiddle(int dir, const long long *a, const long long *w, long long *out) {
  const fxc r = dir < 0 ? fx_twiddle<-1>({a[0], a[1]}, fx_words(w[0], w[1])) : fx_twiddle<+1>({a[0], a[1]}, fx_words(w[0], w[1]));
  out[0] = r.re;
  out[1] = r.im;
}
void host_sweep(int m, double r, const double *al, const double *be, const double *ginv, double *psi) {
  auto z = [](const double *p) { return reinterpret_cast<const Z *>(p); };
  sweep(m, r, z(al), z(be), *z(ginv), reinterpret_cast<Z *>(psi));
}
// the potential step of one point, theta = (v + g |z|^2) with v 2^58; 0 where it is out of range
int host_phase(int imag, double *z, long long v, double g) {
  const fxs zero = fx_scalar(0.0);
  return imag ? fx_phase<true>(z[0], z[1], v, fx_scalar(g), zero, 1000, 0) : fx_phase<false>(z[0], z[1], v, fx_scalar(g), zero, 1000, 0);
}
// (cos theta, -sin theta) 2^60 of theta 2^58; e^-theta = p 2^(n - 60)
void host_cis(long long th, long long *out) {
  const fxc c = fx_cis(th);
  out[0] = c.re;
  out[1] = c.im;
}
long long host_exp(long long th, int *n) { return fx_exp(th, *n); }
// the butterfly of radix p in place on p complex values
void host_butterfly(int dir, int p, long long *v) {
  fxc *z = reinterpret_cast<fxc *>(v);
  auto go = [&](auto radix) {
    constexpr int P = decltype(radix)::value;
    if (p != P) return;
    if (dir < 0) fx_bf<-1, P>(z);
    else fx_bf<+1, P>(z);
  };
  go(std::integral_constant<int, 2>{});
  go(std::integral_constant<int, 3>{});
  go(std::integral_constant<int, 4>{});
  go(std::integral_constant<int, 5>{});
  go(std::integral_constant<int, 6>{});
  go(std::integral_constant<int, 7>{});
  go(std::integral_constant<int, 8>{});
  go(std::integral_constant<int, 9>{});
  go(std::integral_constant<int, 10>{});
}
}
