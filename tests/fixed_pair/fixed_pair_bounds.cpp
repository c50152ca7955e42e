// Host build of csrc/fixed_pair.cuh: errors of its dot products, of 1/r from a difference
// and of the conversion to FP64, against quadruple precision.
#include <cmath>
#include <cstdint>
#include <random>

static float g_est = 0.f;  // error added to the FP32 estimate of 1/sqrt
#define FX_HOST_ERR g_est
#include "../../paper_1909_11085_gb300/csrc/fixed_pair.cuh"

using namespace stk;
#if defined(__x86_64__)
typedef __float128 Q;
#else
typedef long double Q;
#endif

static Q pow2(int e) {
  Q r = 1;
  for (; e > 0; --e) r *= 2;
  for (; e < 0; ++e) r /= 2;
  return r;
}

// Differences of points in a cube of half-width 1 (separation up to sep) with vectors whose
// components span `span` binary orders.  out: least and largest error of the dot product in its
// units (2^-60 of the product of the vectors' scales), largest relative error of 1/r and, less a
// unit where it is negative, of the dot product's conversion.
extern "C" void bounds(int count, double sep, int span, double *out) {
  std::mt19937_64 g(17);
  std::uniform_real_distribution<double> U(-1, 1);
  out[0] = out[1] = out[2] = out[3] = 0;
  for (int i = 0; i < count; ++i) {
    double x[3], y[3], v[3];
    for (int k = 0; k < 3; ++k) {
      x[k] = std::ldexp(std::floor(std::ldexp(U(g), 50)), -50);  // exact on the grid
      y[k] = std::ldexp(std::floor(std::ldexp(sep < 2 ? x[k] + sep * U(g) : U(g), 50)), -50);
      v[k] = std::ldexp(U(g), -(int)(g() % (span + 1)));
    }
    int64_t X[3], Y[3], J[3];
    uint32_t xf = kFxExact, yf = kFxExact;
    for (int k = 0; k < 3; ++k) {
      X[k] = fx_coord(x[k], 2, xf);
      Y[k] = fx_coord(y[k], 2, yf);
    }
    int32_t dh[3], dl[3], vh[3], vl[3];
    int a, b;
    if (!fx_diff(X, Y, xf, yf, 2, J, dh, dl, a)) continue;
    const int e = fx_block(v, vh, vl);
    Q dot = 0, r2 = 0;
    for (int k = 0; k < 3; ++k) {
      const Q d = (Q)x[k] - (Q)y[k];
      dot += d * v[k];
      r2 += d * d;
    }
    const int64_t V = fx_dot(dh, dl, vh, vl);
    const double err = (double)((Q)V - dot * pow2(60 - a - e));
    out[0] = std::fmin(out[0], err);
    out[1] = std::fmax(out[1], err);
    const double conv = fx_to_double(V, 1026 + e + a);
    const Q lost = (Q)conv * pow2(60 - a - e) - V;  // of a negative V, one unit more is cut
    const double unit = V < 0 ? 1.0 : 0.0;
    if (V) out[3] = std::fmax(out[3], (std::fabs((double)lost) - unit) / std::fabs((double)V));
    g_est = (float)(2.4e-7 * U(g));
    const Q ri = (Q)fx_rsqrt(fx_norm2(dh, dl), b) * pow2(b - 62 - a);
    out[2] = std::fmax(out[2], std::fabs((double)((ri * ri * r2 - 1) / 2)));
  }
}
