// Host build of csrc/fixed_pair.cuh: pairs whose difference is nearly
// perpendicular to the normal and density, component by component (a plane
// seen from just beside it).
#include <cmath>
#include <cstdint>
#include <random>

#include "../../paper_1909_11085_gb300/csrc/fixed_pair.cuh"

using namespace stk;
typedef long double Q;

// Sources on the plane z = z0 with normals along z, densities along z up to `tilt` of their
// length, half-width size; targets at a height up to h above it.  out: pairs that took the
// FP64 form, largest error of the double layer against
// |d| sum |d_k n_k| sum |d_k psi_k| / r^5.
extern "C" void planar_errors(int count, double size, double z0, double h, double tilt,
                              double *out) {
  std::mt19937_64 g(5);
  std::uniform_real_distribution<double> U(-1, 1);
  int E;
  std::frexp(std::fmax(size, std::fabs(z0) + h), &E);
  out[0] = out[1] = 0;
  for (int i = 0; i < count; ++i) {
    const double x[3] = {size * U(g), size * U(g), z0 + h * std::fabs(U(g))},
                 y[3] = {size * U(g), size * U(g), z0};
    const double q[3] = {U(g), U(g), U(g)}, n[3] = {0, 0, 1 + U(g) / 4},
                 p[3] = {tilt * U(g), tilt * U(g), 1 + U(g) / 4};
    SrcFx S;
    S.thr = kFxExact;
    uint32_t xf = kFxExact;
    int64_t X[3];
    for (int k = 0; k < 3; ++k) {
      X[k] = fx_coord(x[k], E, xf);
      S.y[k] = fx_coord(y[k], E, S.thr);
      S.q[k] = q[k];
    }
    S.eq = (int16_t)fx_block(q, S.qh, S.ql, S.thr, kFxRoundQ);
    const int en = fx_block(n, S.nh, S.nl, S.thr, kFxRoundN);
    S.epn = (int16_t)(en + fx_block(p, S.ph, S.pl, S.thr, kFxRoundP));
    double a[3] = {0, 0, 0};
    if (!fx_pair<K_DL>(X, xf, E, S, a)) {
      ++out[0];
      continue;
    }
    Q d[3], r2 = 0, dn = 0, dp = 0, an = 0, ap = 0, err = 0;
    for (int k = 0; k < 3; ++k) {
      d[k] = (Q)x[k] - y[k];
      r2 += d[k] * d[k];
      dn += d[k] * n[k];
      dp += d[k] * p[k];
      an += fabsl(d[k] * n[k]);
      ap += fabsl(d[k] * p[k]);
    }
    const Q r = sqrtl(r2), c = 1 / (r2 * r2 * r);
    for (int k = 0; k < 3; ++k) {
      const Q e = a[k] - d[k] * dp * dn * c;
      err += e * e;
    }
    if (an * ap > 0) out[1] = std::fmax(out[1], (double)(sqrtl(err) / (r * an * ap * c)));
  }
}
