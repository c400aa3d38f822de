// The FP64 transforms' fixed-point arithmetic (csrc/fixed64.cuh) on the host: one pencil through
// the stages that fft_device.cuh's fx_pencil_fft runs, its threads one after the other.
#include "fixed64.cuh"

#include <vector>

namespace mhd {

template <int R, int DIR>
void stage(std::vector<cfx> &b, int n, int ns, const TwFx *tw, int s) {
  std::vector<cfx> o(n);
  for (int j = 0; j < n / R; ++j) {
    cfx v[8];
    const int k = j % ns;
    v[0] = fx_shift(b[j], s);
    for (int r = 1; r < R; ++r) v[r] = fx_mul<DIR>(b[j + r * (n / R)], tw[s * n + r * k * (n / (ns * R))]);
    fx_dft<R, DIR>(v);
    for (int r = 0; r < R; ++r) o[(j / ns) * ns * R + k + r * ns] = v[r];
  }
  b = o;
}

template <int DIR>
void fft(int n, int zp, double *data) {
  const std::vector<TwFx> table = fp64_twiddles(n);
  const TwFx *tw = table.data();
  const int g = n / 8;
  int lg = 0;
  while ((2 << lg) <= g) ++lg;
  // parts of up to 32 threads (a warp's), merged in order
  FxPart p{0, 0, 0};
  for (int w0 = 0; w0 < g; w0 += 32) {
    const int w1 = w0 + 32 < g ? w0 + 32 : g;
    FxPart q{0, 0, 0};
    for (int t = w0; t < w1; ++t)
      for (int r = 0; r < 8; ++r) {
        if (zp && (r == 3 || r == 4)) continue;
        for (int c = 0; c < 2; ++c) {
          const uint32_t e = fx_exp(fx_hi(data[2 * (t + r * g) + c]));
          q.m = e > q.m ? e : q.m;
        }
      }
    for (int t = w0; t < w1; ++t) {
      uint32_t a = 0;
      for (int r = 0; r < 8; ++r) {
        if (zp && (r == 3 || r == 4)) continue;
        for (int c = 0; c < 2; ++c) a += fx_size(fx_hi(data[2 * (t + r * g) + c]), q.m);
      }
      q.a = a > q.a ? a : q.a;
      q.t += (a >> 3) + 1u;
    }
    p = w0 ? fx_merge(p, q) : q;
  }
  const FxScale sc = fx_scale(p, lg);
  std::vector<cfx> b(n);
  for (int j = 0; j < g; ++j) {
    cfx v[8];
    for (int r = 0; r < 8; ++r) {
      const double *x = data + 2 * (j + r * g);
      v[r] = cfx{fx_from_double(fx_hi(x[0]), fx_lo(x[0]), sc.ek), fx_from_double(fx_hi(x[1]), fx_lo(x[1]), sc.ek)};
    }
    if (zp) fx_dft8<DIR, true>(v);
    else fx_dft8<DIR, false>(v);
    for (int r = 0; r < 8; ++r) b[8 * j + r] = v[r];
  }
  int left = sc.shift;
  for (int ns = 8; ns < n;) {
    const int r = n / ns >= 8 ? 8 : n / ns, l2 = r == 8 ? 3 : r == 4 ? 2 : 1;
    const int s = left < l2 ? left : l2;
    if (r == 8) stage<8, DIR>(b, n, ns, tw, s);
    else if (r == 4) stage<4, DIR>(b, n, ns, tw, s);
    else stage<2, DIR>(b, n, ns, tw, s);
    left -= s;
    ns *= r;
  }
  const uint32_t be = sc.ek + (uint32_t)sc.shift + 1u;
  for (int i = 0; i < n; ++i) {
    data[2 * i] = sc.bad ? fx_double(0x7ff80000u, 0u) : fx_to_double(b[i].re, be);
    data[2 * i + 1] = sc.bad ? fx_double(0x7ff80000u, 0u) : fx_to_double(b[i].im, be);
  }
}
}  // namespace mhd

// One transform of n complex values in place; dir +1 inverse, -1 forward; zp: inputs 3 and 4 of
// the first stage are known zeros.
extern "C" void fixed64_fft(int n, int dir, int zp, double *data) {
  if (dir > 0) mhd::fft<+1>(n, zp, data);
  else mhd::fft<-1>(n, zp, data);
}
