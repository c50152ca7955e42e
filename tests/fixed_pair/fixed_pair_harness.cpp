// Host build of csrc/fixed_pair.cuh: errors of the fixed point pair and of the
// same pair in FP64 against extended precision, in units of the pair's natural
// size (|q|/r for the single layer, |psi||n|/r^2 for the double layer).
#include <cmath>
#include <cstdint>
#include <random>

static float g_est = 0.f;  // error added to the FP32 estimate of 1/sqrt
#define FX_HOST_ERR g_est
#include "../../paper_1909_11085_gb300/csrc/fixed_pair.cuh"

using namespace stk;
typedef long double Q;

template <int KIND>
static void exact(const double *x, const double *y, const double *q, const double *n,
                  const double *p, Q *u) {
  Q d[3], r2 = 0, dq = 0, dn = 0, dp = 0;
  for (int k = 0; k < 3; ++k) {
    d[k] = (Q)x[k] - y[k];
    r2 += d[k] * d[k];
    dq += d[k] * q[k];
    dn += d[k] * n[k];
    dp += d[k] * p[k];
  }
  const Q r = sqrtl(r2);
  for (int k = 0; k < 3; ++k) {
    u[k] = 0;
    if (KIND & K_SL) u[k] += q[k] / r + d[k] * dq / (r2 * r);
    if (KIND & K_DL) u[k] += d[k] * dp * dn / (r2 * r2 * r);
  }
}

template <int KIND>
static void fp64(const double *x, const double *y, const double *q, const double *n,
                 const double *p, double *u) {
  double d[3];
  for (int k = 0; k < 3; ++k) d[k] = x[k] - y[k];
  auto dot = [&](const double *v) { return std::fma(d[0], v[0], std::fma(d[1], v[1], d[2] * v[2])); };
  const double ri = 1.0 / std::sqrt(dot(d)), ri2 = ri * ri;
  const double dq = dot(q), dn = dot(n), dp = dot(p);
  const double c = KIND == K_SL ? dq * ri2
                   : KIND == K_DL ? dp * dn * (ri2 * ri2 * ri)
                                  : std::fma(dp * dn, ri2, dq) * ri2;
  for (int k = 0; k < 3; ++k) u[k] = KIND == K_DL ? d[k] * c : std::fma(d[k], c, q[k]) * ri;
}

// count random pairs in a cube of half-width size about shift, sources within
// sep of their targets (0: anywhere); planar: one coordinate equal, normals
// along it, a zero density component.  out: pairs that took the FP64 form, rms
// and largest error of the fixed form, rms and largest of FP64.
template <int KIND>
static void run(int count, double size, double shift, double sep, int planar, double *out) {
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> U(-1, 1);
  int E;
  std::frexp(size + std::fabs(shift), &E);
  double s1 = 0, s2 = 0, m1 = 0, m2 = 0;
  int slow = 0;
  for (int i = 0; i < count; ++i) {
    double x[3], y[3], q[3], n[3], p[3];
    for (int k = 0; k < 3; ++k) {
      x[k] = shift + size * U(g);
      y[k] = sep > 0 ? x[k] + sep * U(g) : shift + size * U(g);
      if (std::fabs(y[k]) >= std::ldexp(1, E)) y[k] = x[k];
      q[k] = std::ldexp(U(g), (int)(8 * U(g)));
      n[k] = U(g);
      p[k] = 3e-3 * U(g);
    }
    if (planar) {
      y[2] = x[2];
      n[0] = n[1] = q[1] = 0;
    }
    g_est = (float)(2.4e-7 * U(g));
    SrcFx S;
    S.thr = kFxExact;
    uint32_t xf = kFxExact;
    int64_t X[3];
    for (int k = 0; k < 3; ++k) {
      X[k] = fx_coord(x[k], E, xf);
      S.y[k] = fx_coord(y[k], E, S.thr);
      S.q[k] = q[k];
    }
    S.eq = (int16_t)fx_block(q, S.qh, S.ql);
    const int en = fx_block(n, S.nh, S.nl);
    S.epn = (int16_t)(en + fx_block(p, S.ph, S.pl));
    double a[3] = {0, 0, 0}, b[3];
    if (!fx_pair<KIND>(X, xf, E, S, a)) {
      ++slow;
      continue;
    }
    Q u[3];
    exact<KIND>(x, y, q, n, p, u);
    fp64<KIND>(x, y, q, n, p, b);
    double r = 0, qm = 0, pm = 0, nm = 0;
    Q e1 = 0, e2 = 0;
    for (int k = 0; k < 3; ++k) {
      r += (x[k] - y[k]) * (x[k] - y[k]);
      qm = std::fmax(qm, std::fabs(q[k]));
      pm = std::fmax(pm, std::fabs(p[k]));
      nm = std::fmax(nm, std::fabs(n[k]));
      e1 += (a[k] - u[k]) * (a[k] - u[k]);
      e2 += (b[k] - u[k]) * (b[k] - u[k]);
    }
    const double sc = ((KIND & K_SL) ? qm / std::sqrt(r) : 0) + ((KIND & K_DL) ? pm * nm / r : 0);
    const double f1 = (double)sqrtl(e1) / sc, f2 = (double)sqrtl(e2) / sc;
    s1 += f1 * f1;
    s2 += f2 * f2;
    m1 = std::fmax(m1, f1);
    m2 = std::fmax(m2, f2);
  }
  const int n = count - slow > 0 ? count - slow : 1;
  out[0] = slow;
  out[1] = std::sqrt(s1 / n);
  out[2] = m1;
  out[3] = std::sqrt(s2 / n);
  out[4] = m2;
}

extern "C" void fixed_pair_errors(int kind, int count, double size, double shift, double sep,
                                  int planar, double *out) {
  if (kind == K_SL) run<K_SL>(count, size, shift, sep, planar, out);
  else if (kind == K_DL) run<K_DL>(count, size, shift, sep, planar, out);
  else run<K_SLDL>(count, size, shift, sep, planar, out);
}

// Largest relative error of fx_rsqrt over random arguments and the ends of its range.
extern "C" double fixed_rsqrt_error(int count) {
  std::mt19937_64 g(3);
  double worst = 0;
  const int64_t ends[] = {1ll << 58, (1ll << 58) + 1, 1ll << 59, (1ll << 60) - 1, 1ll << 60,
                          (1ll << 60) + 1, (3ll << 60) - 1};
  for (int i = 0; i < count + 7; ++i) {
    int64_t W = i < 7 ? ends[i] : (int64_t)(g() >> 2);
    if (W < (1ll << 58)) W += 1ll << 58;
    if (W >= 3ll << 60) W >>= 1;
    g_est = (float)(2.4e-7 * ((double)(int64_t)g() / 9.3e18));
    int b;
    const Q y = (Q)fx_rsqrt(W, b) / (Q)(1ull << 62) * (1 << b);
    const Q w = (Q)W / (Q)(1ll << 60);
    worst = std::fmax(worst, (double)fabsl((y * y * w - 1) / 2));
  }
  return worst;
}

// Coordinates on the grid and back; returns the largest error in quanta and
// whether the inexact flag was ever clear for a coordinate that lost bits.
extern "C" int fixed_coord_check(int count, int E, double *worst) {
  std::mt19937_64 g(4);
  std::uniform_real_distribution<double> U(-1, 1);
  *worst = 0;
  int lies = 0;
  for (int i = 0; i < count; ++i) {
    const double v = i == 0 ? 0.0 : i == 1 ? 5e-324 : i == 2 ? -std::ldexp(1 - 1e-16, E)
                                                   : std::ldexp(U(g), E - (int)(g() % 80));
    uint32_t f = kFxExact;
    const int64_t X = fx_coord(v, E, f);
    const Q e = fabsl((Q)X - (Q)v * ldexpl(1, 62 - E));
    *worst = std::fmax(*worst, (double)e);
    if (e != 0 && f == kFxExact) ++lies;
  }
  return lies;
}
