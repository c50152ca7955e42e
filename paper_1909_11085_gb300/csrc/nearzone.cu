// nearzone.cu -- near-zone search on a patch surface (Sec. 3.2, the closest-
// point search, steps a-e): for each target x, the patch of the surface
// closest to x when x lies within d_eps of it, with the closest point
// y = P(u*, v*), the unit normal there and the distance.
//
// A patch is the image of [-1, 1]^2 under the degree-q tensor-product
// interpolant through its (q+1) x (q+1) Clenshaw-Curtis nodes
// (u_i, v_j) = (cos(i pi/q), cos(j pi/q)), node index i (q+1) + j.
//  a. k_nz_boxes: each patch's node box, grown by d_eps and by 5% of its
//     diagonal (the interpolant may leave the nodes' box);
//  b. k_nz_grid / k_nz_cells: a spatial hash -- a uniform grid whose spacing
//     H is at least every box side, so that each box covers at most 2 x 2 x 2
//     cells -- and the (cell, patch) keys of every box;
//  c. the keys sorted (the library's radix sort); a target's cell key then
//     finds the patches whose boxes cover its cell (binary search), and the
//     exact box test keeps those whose box contains it;
//  d. for each of those, the closest point by Newton's method on
//     |x - P(u, v)|^2 with the Gauss-Newton Hessian, a backtracking (Armijo)
//     line search and projection onto [-1, 1]^2, started at the nearest node;
//  e. the nearest patch (ties to the lower index) is kept if its distance is
//     at most d_eps.
// Few targets lie near the surface, and FP64 runs at 1/64 of the FP32 rate on
// GB300, where a warp instruction is charged in full however few of its lanes
// are active.  So the work is arranged in three steps:
//  * k_nz_mark finds the targets inside at least one grown box (an FP32 test
//    that no such target fails, then the FP64 one), writes "none" for the rest
//    and counts the targets of each grid cell; k_nz_scatter lists them cell by
//    cell, so that a warp's 32 targets share their candidate patches and read
//    the same coefficients;
//  * k_nz_search, a warp per 32 listed targets, queues (target, patch) pairs
//    and takes 32 of them at a time, one per lane: nearest node and
//    Gauss-Newton in FP32 on coordinates relative to the patch's centre;
//  * the pairs that can still be their target's nearest within d_eps are
//    finished in FP64: Newton steps from the FP32 point, the gradient in FP64
//    and the Hessian (with the curvature term) in FP32, until a step is below
//    1e-11, which the next would shorten by 1e-5 or more.
// The interpolant is evaluated from its Chebyshev coefficients (relative to
// the patch's centre), which take two multiply-adds per degree for a basis
// value and its derivative where the barycentric form takes two divisions.  A
// pair that FP32 cannot settle (a target on a node, a step that does not
// decrease the distance, no convergence, a Hessian near singular) and one whose
// closest point lies beside a node's parameter (kNzNodeGap) takes the
// plain FP64 iteration (nz_closest), the search's definition.
// 2^20 targets against 320 patches (63.9 k hits): see k_nz_search.
// Results are FP64; the normal is (dP/du x dP/dv) / |dP/du x dP/dv|.
#include <cfloat>
#include <cmath>

#include "../../include/stokesgpu.h"
#include "common.cuh"
#include "prep.cuh"

namespace stk {
stk_status report_error(stk_status s, const char *msg);
}

namespace {

using namespace stk;

constexpr int kNzMaxN1 = 13;  // q <= 12
constexpr int kNzCells = 8;   // cells per patch box
constexpr int kNzThreads = 128;

struct NzGrid {
  double org[3];
  double H;
  int64_t dims[3];
};

// Per patch: centre of its node box, the bound rp (below) and the largest
// coordinate sum of a node relative to the centre.
struct NzMeta {
  double c[3];
  float rp, scale;
};
// Coefficients and nodes of a patch relative to its centre, n1 x n1 each.
struct NzPatches {
  const double *nodes;   // caller nodes [npatch][n1 n1][3]
  const double *boxes;   // [npatch][6] grown boxes
  const float *boxes32;  // the same rounded to FP32
  const double *rp;
  const NzMeta *meta;
  const double2 *c64;    // [npatch][n1 n1][2]: (x, y), (z, 0)
  const float4 *c32;     // [npatch][n1 n1]
  const float4 *x32;     // [npatch][n1 n1] nodes
};

// Grown box, bound and Chebyshev coefficients of each patch: on the CC nodes
// the coefficients are the type-I cosine transform of the values, in u and v.
__global__ void __launch_bounds__(kNzThreads) k_nz_boxes(const double *__restrict__ nodes,
                                                         int n1sq, double d_eps,
                                                         double *__restrict__ boxes,
                                                         float *__restrict__ boxes32,
                                                         double *__restrict__ rp,
                                                         NzMeta *__restrict__ meta,
                                                         double2 *__restrict__ c64,
                                                         float4 *__restrict__ c32,
                                                         float4 *__restrict__ x32) {
  __shared__ double s[6][kNzThreads];
  __shared__ double sr[kNzThreads];
  __shared__ double ct[2 * kNzMaxN1];
  __shared__ double F[3][kNzMaxN1 * kNzMaxN1], G[3][kNzMaxN1 * kNzMaxN1];
  const int p = blockIdx.x;
  // the largest distance between two corners of a node cell: every point of
  // the patch lies within it of a node, up to the interpolant's small
  // deviation from the bilinear cell
  const int n1 = (int)lrint(sqrt((double)n1sq));
  double cm = 0.0;
  for (int e = threadIdx.x; e < (n1 - 1) * (n1 - 1); e += blockDim.x) {
    const int i = e / (n1 - 1), j = e % (n1 - 1);
    const double *c00 = nodes + ((size_t)p * n1sq + i * n1 + j) * 3;
    const double *c01 = c00 + 3, *c10 = c00 + 3 * n1, *c11 = c10 + 3;
    const double *cs[4] = {c00, c01, c10, c11};
    for (int a = 0; a < 4; ++a)
      for (int b = a + 1; b < 4; ++b) {
        const double dx = cs[a][0] - cs[b][0], dy = cs[a][1] - cs[b][1], dz = cs[a][2] - cs[b][2];
        cm = fmax(cm, dx * dx + dy * dy + dz * dz);
      }
  }
  sr[threadIdx.x] = cm;
  double lo[3] = {DBL_MAX, DBL_MAX, DBL_MAX}, hi[3] = {-DBL_MAX, -DBL_MAX, -DBL_MAX};
  for (int e = threadIdx.x; e < n1sq; e += blockDim.x)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const double v = nodes[((size_t)p * n1sq + e) * 3 + k];
      lo[k] = fmin(lo[k], v);
      hi[k] = fmax(hi[k], v);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    s[k][threadIdx.x] = lo[k];
    s[3 + k][threadIdx.x] = hi[k];
  }
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        s[k][threadIdx.x] = fmin(s[k][threadIdx.x], s[k][threadIdx.x + o]);
        s[3 + k][threadIdx.x] = fmax(s[3 + k][threadIdx.x], s[3 + k][threadIdx.x + o]);
      }
      sr[threadIdx.x] = fmax(sr[threadIdx.x], sr[threadIdx.x + o]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    rp[p] = 1.1 * sqrt(sr[0]);
    const double dx = s[3][0] - s[0][0], dy = s[4][0] - s[1][0], dz = s[5][0] - s[2][0];
    const double grow = d_eps + 0.05 * sqrt(dx * dx + dy * dy + dz * dz);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      boxes[6 * p + k] = s[k][0] - grow;
      boxes[6 * p + 3 + k] = s[3 + k][0] + grow;
      boxes32[6 * p + k] = (float)(s[k][0] - grow);
      boxes32[6 * p + 3 + k] = (float)(s[3 + k][0] + grow);
    }
  }
  const double cen[3] = {0.5 * (s[0][0] + s[3][0]), 0.5 * (s[1][0] + s[4][0]),
                         0.5 * (s[2][0] + s[5][0])};
  if (threadIdx.x == 0) {
    NzMeta m;
    for (int k = 0; k < 3; ++k) m.c[k] = cen[k];
    m.rp = (float)(1.1 * sqrt(sr[0]));
    m.scale = (float)((s[3][0] - cen[0]) + (s[4][0] - cen[1]) + (s[5][0] - cen[2]));
    meta[p] = m;
  }
  const int q = n1 - 1;
  for (int m = threadIdx.x; m < 2 * q; m += blockDim.x) ct[m] = cospi((double)m / q);
  for (int e = threadIdx.x; e < n1sq; e += blockDim.x) {
#pragma unroll
    for (int k = 0; k < 3; ++k) F[k][e] = nodes[((size_t)p * n1sq + e) * 3 + k] - cen[k];
    x32[(size_t)p * n1sq + e] = make_float4((float)F[0][e], (float)F[1][e], (float)F[2][e], 0.f);
  }
  __syncthreads();
  // along v, then along u
  for (int pass = 0; pass < 2; ++pass) {
    for (int t = threadIdx.x; t < 3 * n1sq; t += blockDim.x) {
      const int k = t / n1sq, e = t % n1sq, i = e / n1, j = e % n1;
      const int deg = pass ? i : j;
      double a = 0.0;
      for (int m = 0; m < n1; ++m) {
        const double f = pass ? G[k][m * n1 + j] : F[k][i * n1 + m];
        const double wm = (m == 0 || m == q) ? 0.5 : 1.0;
        a = fma(wm * ct[(deg * m) % (2 * q)], f, a);
      }
      a *= ((deg == 0 || deg == q) ? 1.0 : 2.0) / q;
      if (pass) F[k][e] = a;
      else G[k][e] = a;
    }
    __syncthreads();
  }
  for (int e = threadIdx.x; e < n1sq; e += blockDim.x) {
    const size_t o = (size_t)p * n1sq + e;
    c64[2 * o] = make_double2(F[0][e], F[1][e]);
    c64[2 * o + 1] = make_double2(F[2][e], 0.0);
    c32[o] = make_float4((float)F[0][e], (float)F[1][e], (float)F[2][e], 0.f);
  }
}

__global__ void __launch_bounds__(kNzThreads) k_nz_grid(const double *__restrict__ boxes,
                                                        int npatch, NzGrid *__restrict__ g) {
  __shared__ double s[7][kNzThreads];
  double lo[3] = {DBL_MAX, DBL_MAX, DBL_MAX}, hi[3] = {-DBL_MAX, -DBL_MAX, -DBL_MAX}, side = 0.0;
  for (int p = threadIdx.x; p < npatch; p += blockDim.x)
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      lo[k] = fmin(lo[k], boxes[6 * p + k]);
      hi[k] = fmax(hi[k], boxes[6 * p + 3 + k]);
      side = fmax(side, boxes[6 * p + 3 + k] - boxes[6 * p + k]);
    }
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    s[k][threadIdx.x] = lo[k];
    s[3 + k][threadIdx.x] = hi[k];
  }
  s[6][threadIdx.x] = side;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        s[k][threadIdx.x] = fmin(s[k][threadIdx.x], s[k][threadIdx.x + o]);
        s[3 + k][threadIdx.x] = fmax(s[3 + k][threadIdx.x], s[3 + k][threadIdx.x + o]);
      }
      s[6][threadIdx.x] = fmax(s[6][threadIdx.x], s[6][threadIdx.x + o]);
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    double H = s[6][0] > 0.0 ? s[6][0] * (1.0 + 1e-9) : 1.0;
    // cell keys c0 + d0 (c1 + d1 c2) must fit 64 bits: a coarser grid only
    // puts more boxes in a cell
    double d[3];
    while (true) {
#pragma unroll
      for (int k = 0; k < 3; ++k) d[k] = floor((s[3 + k][0] - s[k][0]) / H) + 1.0;
      if (d[0] * d[1] * d[2] <= 4.0e18) break;
      H *= 2.0;
    }
    g->H = H;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      g->org[k] = s[k][0];
      g->dims[k] = (int64_t)d[k];
    }
  }
}

__device__ __forceinline__ bool nz_cell(const NzGrid &g, const double x[3], int64_t c[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    const double f = floor((x[k] - g.org[k]) / g.H);
    if (!(f >= 0.0) || f >= (double)g.dims[k]) return false;
    c[k] = (int64_t)f;
  }
  return true;
}

__global__ void k_nz_cells(const double *__restrict__ boxes, int npatch,
                           const NzGrid *__restrict__ gp, uint64_t *__restrict__ keys,
                           int32_t *__restrict__ vals) {
  const NzGrid g = *gp;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < npatch * kNzCells;
       e += gridDim.x * blockDim.x) {
    const int p = e / kNzCells, c = e % kNzCells;
    int64_t cl[3], ch[3], cc[3];
    bool ok = true;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      cl[k] = (int64_t)floor((boxes[6 * p + k] - g.org[k]) / g.H);
      ch[k] = (int64_t)floor((boxes[6 * p + 3 + k] - g.org[k]) / g.H);
      cl[k] = cl[k] < 0 ? 0 : cl[k];
      ch[k] = ch[k] >= g.dims[k] ? g.dims[k] - 1 : ch[k];
      cc[k] = cl[k] + ((c >> k) & 1);
      ok = ok && cc[k] <= ch[k];
    }
    keys[e] = ok ? (uint64_t)(cc[0] + g.dims[0] * (cc[1] + g.dims[1] * cc[2])) : ~0ull;
    vals[e] = p;
  }
}

// Lagrange basis on the CC nodes and its derivative at t (barycentric form;
// at a node, the differentiation matrix row).
__device__ void nz_basis(int n1, const double *xk, const double *wk, double t, double *L,
                         double *D) {
  int hit = -1;
  for (int k = 0; k < n1; ++k)
    if (fabs(t - xk[k]) < 1e-14) hit = k;
  if (hit >= 0) {
    double dd = 0.0;
    for (int k = 0; k < n1; ++k) {
      L[k] = k == hit ? 1.0 : 0.0;
      D[k] = 0.0;
      if (k != hit) {
        D[k] = (wk[k] / wk[hit]) / (xk[hit] - xk[k]);
        dd -= D[k];
      }
    }
    D[hit] = dd;
    return;
  }
  // l_k = (w_k / (t - x_k)) / S and l_k' = l_k (sum_m w_m / (t - x_m)^2 / S - 1 / (t - x_k)),
  // with D[] holding 1 / (t - x_k) until the end
  double S = 0.0, S2 = 0.0;
  for (int k = 0; k < n1; ++k) {
    const double r = 1.0 / (t - xk[k]);
    const double a = wk[k] * r;
    L[k] = a;
    D[k] = r;
    S += a;
    S2 += a * r;
  }
  const double iS = 1.0 / S, sig = S2 * iS;
  for (int k = 0; k < n1; ++k) {
    L[k] *= iS;
    D[k] = L[k] * (sig - D[k]);
  }
}

// P(u, v), dP/du, dP/dv of one patch.
__device__ void nz_eval(int n1, const double *__restrict__ X, const double *xk, const double *wk,
                        double u, double v, double P[3], double Pu[3], double Pv[3]) {
  double Lu[kNzMaxN1], Du[kNzMaxN1], Lv[kNzMaxN1], Dv[kNzMaxN1];
  nz_basis(n1, xk, wk, u, Lu, Du);
  nz_basis(n1, xk, wk, v, Lv, Dv);
#pragma unroll
  for (int c = 0; c < 3; ++c) P[c] = Pu[c] = Pv[c] = 0.0;
  for (int i = 0; i < n1; ++i) {
    double T[3] = {0.0, 0.0, 0.0}, Tv[3] = {0.0, 0.0, 0.0};
    for (int j = 0; j < n1; ++j) {
      const double *xp = X + 3 * (i * n1 + j);
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        T[c] = fma(Lv[j], xp[c], T[c]);
        Tv[c] = fma(Dv[j], xp[c], Tv[c]);
      }
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      P[c] = fma(Lu[i], T[c], P[c]);
      Pu[c] = fma(Du[i], T[c], Pu[c]);
      Pv[c] = fma(Lu[i], Tv[c], Pv[c]);
    }
  }
}

// The same by a warp.  Every sum is one lane's, over the terms of the forms above in their
// order (and sig is rounded before the difference, as there), so the results are theirs bit
// for bit.  Lanes 0 .. n1 - 1 hold the u basis, 16 .. 16 + n1 - 1 the v basis; then a lane
// takes up to three of the 6 n1 row sums, and lanes 0 .. 8 the sums over the rows.
__device__ __forceinline__ void nz_basis_warp(int n1, const double *xk, const double *wk, double u,
                                              double v, int lane, double &L, double &D) {
  const int half = lane & 16, k = (lane & 15) < n1 ? lane & 15 : 0;
  const double t = half ? v : u;
  const unsigned on = __ballot_sync(kFull, (lane & 15) < n1 && fabs(t - xk[k]) < 1e-14);
  const unsigned mine = (on >> half) & 0xffffu;
  const int hit = mine ? 31 - __clz(mine) : -1;
  const double r = hit >= 0 ? (k == hit ? 0.0 : (wk[k] / wk[hit]) / (xk[hit] - xk[k]))
                            : 1.0 / (t - xk[k]);
  const double a = wk[k] * r;
  double S = 0.0, S2 = 0.0;  // with a node hit: the sum of the row's other entries
  for (int m = 0; m < n1; ++m) {
    const double am = __shfl_sync(kFull, a, half + m), rm = __shfl_sync(kFull, r, half + m);
    if (hit < 0) {
      S += am;
      S2 += am * rm;
    } else if (m != hit) {
      S -= rm;
    }
  }
  if (hit >= 0) {
    L = k == hit ? 1.0 : 0.0;
    D = k == hit ? S : r;
  } else {
    const double iS = 1.0 / S, sig = __dmul_rn(S2, iS);
    L = a * iS;
    D = L * (sig - r);
  }
}
__device__ __noinline__ void nz_eval_warp(int n1, const double *__restrict__ X, const double *xk,
                                          const double *wk, double u, double v, int lane,
                                          double *P, double *Pu, double *Pv) {
  static_assert(kNzMaxN1 <= 16 && 6 * kNzMaxN1 <= 3 * kWarp, "a basis per half warp, three sums per lane");
  double L, D;
  nz_basis_warp(n1, xk, wk, u, v, lane, L, D);
  double T[3] = {0.0, 0.0, 0.0};  // sum s = 6 i + c (values, c < 3) or 6 i + 3 + c (v derivatives)
  for (int j = 0; j < n1; ++j) {
    const double lj = __shfl_sync(kFull, L, 16 + j), dj = __shfl_sync(kFull, D, 16 + j);
#pragma unroll
    for (int m = 0; m < 3; ++m) {
      const int s = lane + kWarp * m, i = s / 6, c = s % 3;
      if (i < n1) T[m] = fma(s % 6 < 3 ? lj : dj, X[3 * (i * n1 + j) + c], T[m]);
    }
  }
  const int out = lane < 9 ? lane / 3 : 0, c = lane % 3;  // P, P_u, P_v
  double acc = 0.0;
  for (int i = 0; i < n1; ++i) {
    const double li = __shfl_sync(kFull, L, i), di = __shfl_sync(kFull, D, i);
    const int s = 6 * i + c + (out == 2 ? 3 : 0);
    const double t0 = __shfl_sync(kFull, T[0], s & 31), t1 = __shfl_sync(kFull, T[1], s & 31),
                 t2 = __shfl_sync(kFull, T[2], s & 31);
    acc = fma(out == 1 ? di : li, s < 32 ? t0 : s < 64 ? t1 : t2, acc);
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    P[q] = __shfl_sync(kFull, acc, q);
    Pu[q] = __shfl_sync(kFull, acc, 3 + q);
    Pv[q] = __shfl_sync(kFull, acc, 6 + q);
  }
}

// The node of a patch nearest to x: squared distance and its (u, v).
__device__ double nz_nearest_node(int n1, const double *__restrict__ X, const double *xk,
                                  const double x[3], double &u, double &v) {
  double best = DBL_MAX;
  for (int e = 0; e < n1 * n1; ++e) {
    const double *xp = X + 3 * e;
    const double d = (xp[0] - x[0]) * (xp[0] - x[0]) + (xp[1] - x[1]) * (xp[1] - x[1]) +
                     (xp[2] - x[2]) * (xp[2] - x[2]);
    if (d < best) {
      best = d;
      u = xk[e / n1];
      v = xk[e % n1];
    }
  }
  return best;
}

__device__ double nz_nearest_node_warp(int n1, const double *__restrict__ X, const double *xk,
                                       const double x[3], int lane, double &u, double &v) {
  double best = DBL_MAX;
  int at = n1 * n1;  // the first of the nearest ones
  for (int e = lane; e < n1 * n1; e += kWarp) {
    const double *xp = X + 3 * e;
    const double d = (xp[0] - x[0]) * (xp[0] - x[0]) + (xp[1] - x[1]) * (xp[1] - x[1]) +
                     (xp[2] - x[2]) * (xp[2] - x[2]);
    if (d < best) {
      best = d;
      at = e;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double d = __shfl_xor_sync(kFull, best, o);
    const int e = __shfl_xor_sync(kFull, at, o);
    if (d < best || (d == best && e < at)) {
      best = d;
      at = e;
    }
  }
  if (at < n1 * n1) {
    u = xk[at / n1];
    v = xk[at % n1];
  }
  return best;
}

// Closest point of a patch to x, from the start (u, v): by each thread, or (WARP) by a
// warp for one x, with the same results.
template <bool WARP>
__device__ __forceinline__ void nz_eval_by(int n1, const double *__restrict__ X, const double *xk,
                                           const double *wk, double u, double v, int lane,
                                           double P[3], double Pu[3], double Pv[3]) {
  if (WARP) nz_eval_warp(n1, X, xk, wk, u, v, lane, P, Pu, Pv);
  else nz_eval(n1, X, xk, wk, u, v, P, Pu, Pv);
}
template <bool WARP>
__device__ double nz_closest(int n1, const double *__restrict__ X, const double *xk,
                             const double *wk, const double x[3], int lane, double &u, double &v,
                             double y[3], double nn[3]) {
  double P[3], Pu[3], Pv[3];
  nz_eval_by<WARP>(n1, X, xk, wk, u, v, lane, P, Pu, Pv);
  double f = 0.0;
#pragma unroll
  for (int c = 0; c < 3; ++c) f += (P[c] - x[c]) * (P[c] - x[c]);
  for (int it = 0; it < 40; ++it) {
    double gu = 0.0, gv = 0.0, huu = 0.0, huv = 0.0, hvv = 0.0;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      const double r = P[c] - x[c];
      gu += r * Pu[c];
      gv += r * Pv[c];
      huu += Pu[c] * Pu[c];
      huv += Pu[c] * Pv[c];
      hvv += Pv[c] * Pv[c];
    }
    // active set: a parameter on its bound whose gradient points out of the
    // square stays there, and the step solves for the other one alone
    const bool fu = (u <= -1.0 && gu > 0.0) || (u >= 1.0 && gu < 0.0);
    const bool fv = (v <= -1.0 && gv > 0.0) || (v >= 1.0 && gv < 0.0);
    if (fu && fv) break;  // a corner that is a constrained minimum
    const double det = huu * hvv - huv * huv;
    double su, sv;
    if (fu) {
      su = 0.0;
      sv = hvv > 1e-300 ? -gv / hvv : -gv;
    } else if (fv) {
      su = huu > 1e-300 ? -gu / huu : -gu;
      sv = 0.0;
    } else if (det > 1e-300) {
      su = -(hvv * gu - huv * gv) / det;
      sv = -(huu * gv - huv * gu) / det;
    } else {
      su = -gu;
      sv = -gv;
    }
    const double slope = gu * su + gv * sv;  // half the directional derivative of f
    double a = 1.0, un = u, vn = v, Pn[3], Pun[3], Pvn[3], fn = f;
    bool moved = false;
    for (int ls = 0; ls < 40; ++ls) {
      un = fmin(1.0, fmax(-1.0, u + a * su));
      vn = fmin(1.0, fmax(-1.0, v + a * sv));
      nz_eval_by<WARP>(n1, X, xk, wk, un, vn, lane, Pn, Pun, Pvn);
      fn = 0.0;
#pragma unroll
      for (int c = 0; c < 3; ++c) fn += (Pn[c] - x[c]) * (Pn[c] - x[c]);
      // Armijo decrease.  Near the minimum the decrease a step buys is below
      // the rounding of |x - P|^2 (about 1e-16 |x|^2; the distance is flat
      // along the surface), so a full Newton step shorter than 1e-6 in the
      // parameters is taken without the test
      if (fn <= f + 2e-4 * a * slope || (ls == 0 && fabs(su) + fabs(sv) < 1e-6)) {
        moved = true;
        break;
      }
      a *= 0.5;
    }
    if (!moved) break;
    const double step = fabs(un - u) + fabs(vn - v);
    u = un;
    v = vn;
    f = fn;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      P[c] = Pn[c];
      Pu[c] = Pun[c];
      Pv[c] = Pvn[c];
    }
    // converged: the parameters are in [-1, 1] and a step below 1e-12 is at
    // the level of the rounding in the gradient (coordinates of order 1e2)
    if (step < 1e-12) break;
  }
  const double cx = Pu[1] * Pv[2] - Pu[2] * Pv[1], cy = Pu[2] * Pv[0] - Pu[0] * Pv[2],
               cz = Pu[0] * Pv[1] - Pu[1] * Pv[0];
  const double cl = sqrt(cx * cx + cy * cy + cz * cz);
  nn[0] = cx / cl;
  nn[1] = cy / cl;
  nn[2] = cz / cl;
#pragma unroll
  for (int c = 0; c < 3; ++c) y[c] = P[c];
  return sqrt(f);
}

// A target's grid cell as the position of its first (cell, patch) key, and
// whether it lies in one of the cell's grown boxes.
__device__ __forceinline__ int64_t nz_first_key(const NzGrid &g, const uint64_t *__restrict__ keys,
                                                int64_t nkeys, const double x[3], uint64_t &key) {
  int64_t c[3];
  if (!nz_cell(g, x, c)) return nkeys;
  key = (uint64_t)(c[0] + g.dims[0] * (c[1] + g.dims[1] * c[2]));
  int64_t lo = 0, hi = nkeys;  // first entry with keys[i] >= key
  while (lo < hi) {
    const int64_t mid = (lo + hi) / 2;
    if (keys[mid] < key) lo = mid + 1;
    else hi = mid;
  }
  return lo;
}

// x inside grown box p.  Rounding to FP32 keeps the order of numbers, so a
// target outside the rounded box is outside the box.
__device__ __forceinline__ bool nz_in_box(const NzPatches &Q, int p, const double x[3],
                                          const float xf[3]) {
  const float *bf = Q.boxes32 + 6 * (size_t)p;
  if (xf[0] < bf[0] || xf[1] < bf[1] || xf[2] < bf[2] || xf[0] > bf[3] || xf[1] > bf[4] ||
      xf[2] > bf[5])
    return false;
  const double *b = Q.boxes + 6 * (size_t)p;
  return x[0] >= b[0] && x[1] >= b[1] && x[2] >= b[2] && x[0] <= b[3] && x[1] <= b[4] &&
         x[2] <= b[5];
}

// Targets inside at least one grown box: their cell (the position of its first
// key) and their rank among the cell's targets; the others get "none" (patch
// -1, distance -1, zero parameters, point and normal) and cell -1.
__global__ void __launch_bounds__(kNzThreads) k_nz_mark(
    NzPatches Q, const NzGrid *__restrict__ gp, const uint64_t *__restrict__ keys,
    const int32_t *__restrict__ vals, int64_t nkeys, const double *__restrict__ trg, int64_t nt,
    int32_t *__restrict__ cell, int32_t *__restrict__ rank, int32_t *__restrict__ count,
    int32_t *__restrict__ patch_out, double *__restrict__ uv_out, double *__restrict__ y_out,
    double *__restrict__ n_out, double *__restrict__ dist_out) {
  const NzGrid g = *gp;
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nt;
       t += (int64_t)gridDim.x * blockDim.x) {
    const double x[3] = {trg[3 * t], trg[3 * t + 1], trg[3 * t + 2]};
    const float xf[3] = {(float)x[0], (float)x[1], (float)x[2]};
    bool any = false;
    uint64_t key = 0;
    const int64_t lo = nz_first_key(g, keys, nkeys, x, key);
    for (int64_t i = lo; i < nkeys && keys[i] == key && !any; ++i) any = nz_in_box(Q, vals[i], x, xf);
    if (any) {
      cell[t] = (int32_t)lo;
      rank[t] = atomicAdd(count + lo, 1);
    } else {
      cell[t] = -1;
      patch_out[t] = -1;
      uv_out[2 * t] = uv_out[2 * t + 1] = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) y_out[3 * t + k] = n_out[3 * t + k] = 0.0;
      dist_out[t] = -1.0;
    }
  }
}

// The marked targets, cell by cell (their order within a cell differs between
// runs; no result depends on it).
__global__ void k_nz_scatter(int64_t nt, const int32_t *__restrict__ cell,
                             const int32_t *__restrict__ rank, const int32_t *__restrict__ offs,
                             int32_t *__restrict__ list) {
  for (int64_t t = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; t < nt;
       t += (int64_t)gridDim.x * blockDim.x)
    if (cell[t] >= 0) list[offs[cell[t]] + rank[t]] = (int32_t)t;
}

// ---- FP32 stage
// The sum over the coefficients needs each basis value once: the v basis is
// kept in registers (unrolled over n1, N1 at compile time for the library's
// default order, otherwise up to the largest), the u basis runs along.
#define NZ_FOR_V(j) \
  _Pragma("unroll") for (int j = 0; j < (N1 ? N1 : kNzMaxN1); ++j) if (N1 || j < n1)

template <typename R>
__device__ __forceinline__ void nz_next(R t2, R &T0, R &T1, R &D0, R &D1) {
  // T_{k+1} = 2 t T_k - T_{k-1}, D_{k+1} = 2 T_k + 2 t D_k - D_{k-1}; t2 = 2 t
  const R T2 = t2 * T1 - T0, D2 = R(2) * T1 + (t2 * D1 - D0);
  T0 = T1;
  T1 = T2;
  D0 = D1;
  D1 = D2;
}

// r = P - x, P_u and P_v at (u, v).
template <int N1>
__device__ __forceinline__ void nz_eval32(int n1, const float4 *__restrict__ C, float u, float v,
                                          const float (&x)[3], float (&r)[3], float (&Pu)[3],
                                          float (&Pv)[3]) {
  constexpr int M = N1 ? N1 : kNzMaxN1;
  float Tv[M], Dv[M];
  {
    float T0 = 1.f, T1 = v, D0 = 0.f, D1 = 1.f;
#pragma unroll
    for (int j = 0; j < M; ++j) {
      Tv[j] = T0;
      Dv[j] = D0;
      nz_next(2.f * v, T0, T1, D0, D1);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) {
    r[c] = -x[c];
    Pu[c] = Pv[c] = 0.f;
  }
  float T0 = 1.f, T1 = u, D0 = 0.f, D1 = 1.f;
#pragma unroll 1
  for (int i = 0; i < n1; ++i) {
    float a[3] = {0.f, 0.f, 0.f}, b[3] = {0.f, 0.f, 0.f};
    NZ_FOR_V(j) {
      const float4 c4 = __ldg(C + i * n1 + j);
      a[0] = fmaf(Tv[j], c4.x, a[0]);
      a[1] = fmaf(Tv[j], c4.y, a[1]);
      a[2] = fmaf(Tv[j], c4.z, a[2]);
      b[0] = fmaf(Dv[j], c4.x, b[0]);
      b[1] = fmaf(Dv[j], c4.y, b[1]);
      b[2] = fmaf(Dv[j], c4.z, b[2]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      r[c] = fmaf(T0, a[c], r[c]);
      Pu[c] = fmaf(D0, a[c], Pu[c]);
      Pv[c] = fmaf(T0, b[c], Pv[c]);
    }
    nz_next(2.f * u, T0, T1, D0, D1);
  }
}

// r . P_uu, r . P_uv, r . P_vv at (u, v): the curvature term of the Hessian.
template <int N1>
__device__ __forceinline__ void nz_curv32(int n1, const float4 *__restrict__ C, float u, float v,
                                          const float (&r)[3], float (&h)[3]) {
  constexpr int M = N1 ? N1 : kNzMaxN1;
  float Tv[M], Dv[M], Ev[M];
  {
    float T0 = 1.f, T1 = v, D0 = 0.f, D1 = 1.f, E0 = 0.f, E1 = 0.f;
#pragma unroll
    for (int j = 0; j < M; ++j) {
      Tv[j] = T0;
      Dv[j] = D0;
      Ev[j] = E0;
      const float E2 = 4.f * D1 + (2.f * v * E1 - E0);
      nz_next(2.f * v, T0, T1, D0, D1);
      E0 = E1;
      E1 = E2;
    }
  }
  h[0] = h[1] = h[2] = 0.f;
  float T0 = 1.f, T1 = u, D0 = 0.f, D1 = 1.f, E0 = 0.f, E1 = 0.f;
#pragma unroll 1
  for (int i = 0; i < n1; ++i) {
    float a = 0.f, b = 0.f, e = 0.f;
    NZ_FOR_V(j) {
      const float4 c4 = __ldg(C + i * n1 + j);
      const float c = fmaf(r[0], c4.x, fmaf(r[1], c4.y, r[2] * c4.z));
      a = fmaf(Tv[j], c, a);
      b = fmaf(Dv[j], c, b);
      e = fmaf(Ev[j], c, e);
    }
    h[0] = fmaf(E0, a, h[0]);
    h[1] = fmaf(D0, b, h[1]);
    h[2] = fmaf(T0, e, h[2]);
    const float E2 = 4.f * D1 + (2.f * u * E1 - E0);
    nz_next(2.f * u, T0, T1, D0, D1);
    E0 = E1;
    E1 = E2;
  }
}

// r = P - x (x relative to the patch's centre), P_u and P_v at (u, v) in FP64.
template <int N1>
__device__ __forceinline__ void nz_eval64(int n1, const double2 *__restrict__ C, double u, double v,
                                          const double (&x)[3], double (&r)[3], double (&Pu)[3],
                                          double (&Pv)[3]) {
  constexpr int M = N1 ? N1 : kNzMaxN1;
  double Tv[M], Dv[M];
  {
    double T0 = 1.0, T1 = v, D0 = 0.0, D1 = 1.0;
#pragma unroll
    for (int j = 0; j < M; ++j) {
      Tv[j] = T0;
      Dv[j] = D0;
      if (j + 1 < M) nz_next(2.0 * v, T0, T1, D0, D1);
    }
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) r[c] = Pu[c] = Pv[c] = 0.0;
  double T0 = 1.0, T1 = u, D0 = 0.0, D1 = 1.0;
#pragma unroll 1
  for (int i = 0; i < n1; ++i) {
    double a[3] = {0.0, 0.0, 0.0}, b[3] = {0.0, 0.0, 0.0};
    NZ_FOR_V(j) {
      const double2 cxy = __ldg(C + 2 * (i * n1 + j));
      const double cz = __ldg(reinterpret_cast<const double *>(C + 2 * (i * n1 + j) + 1));
      a[0] = fma(Tv[j], cxy.x, a[0]);
      a[1] = fma(Tv[j], cxy.y, a[1]);
      a[2] = fma(Tv[j], cz, a[2]);
      b[0] = fma(Dv[j], cxy.x, b[0]);
      b[1] = fma(Dv[j], cxy.y, b[1]);
      b[2] = fma(Dv[j], cz, b[2]);
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) {
      r[c] = fma(T0, a[c], r[c]);
      Pu[c] = fma(D0, a[c], Pu[c]);
      Pv[c] = fma(T0, b[c], Pv[c]);
    }
    nz_next(2.0 * u, T0, T1, D0, D1);
  }
#pragma unroll
  for (int c = 0; c < 3; ++c) r[c] -= x[c];
}
#undef NZ_FOR_V

// The step of a Newton iteration with gradient g and Hessian h (uu, uv, vv) at
// (u, v), and which parameters its active set holds (bit 0: u, bit 1: v): a
// parameter on its bound whose gradient points out of the square stays there.
__device__ __forceinline__ int nz_step32(float gu, float gv, const float (&h)[3], bool fu, bool fv,
                                         float &su, float &sv) {
  su = sv = 0.f;
  if (fu && fv) return 3;
  if (fu) {
    sv = -gv / h[2];
    return 1;
  }
  if (fv) {
    su = -gu / h[0];
    return 2;
  }
  const float det = h[0] * h[2] - h[1] * h[1];
  su = -(h[2] * gu - h[1] * gv) / det;
  sv = -(h[0] * gv - h[1] * gu) / det;
  return 0;
}

constexpr int kNzIter32 = 16;        // FP32 Gauss-Newton iterations
constexpr float kNzStop32 = 2e-5f;   // FP32 step at which FP64 takes over
constexpr int kNzIter64 = 5;

// Nearest node and Gauss-Newton of one (target, patch) pair in FP32.
// Returns false when the pair needs the plain FP64 iteration.
template <int N1>
__device__ __forceinline__ bool nz_pair32(int n1, const float4 *__restrict__ C, float u, float v,
                                          const float (&x)[3], float &uo, float &vo, float &d) {
  float r[3], Pu[3], Pv[3];
  nz_eval32<N1>(n1, C, u, v, x, r, Pu, Pv);
  float f = fmaf(r[0], r[0], fmaf(r[1], r[1], r[2] * r[2]));
  bool ok = false;
  for (int it = 0; it < kNzIter32; ++it) {
    const float gu = fmaf(r[0], Pu[0], fmaf(r[1], Pu[1], r[2] * Pu[2]));
    const float gv = fmaf(r[0], Pv[0], fmaf(r[1], Pv[1], r[2] * Pv[2]));
    const float h[3] = {fmaf(Pu[0], Pu[0], fmaf(Pu[1], Pu[1], Pu[2] * Pu[2])),
                        fmaf(Pu[0], Pv[0], fmaf(Pu[1], Pv[1], Pu[2] * Pv[2])),
                        fmaf(Pv[0], Pv[0], fmaf(Pv[1], Pv[1], Pv[2] * Pv[2]))};
    const bool fu = (u <= -1.f && gu > 0.f) || (u >= 1.f && gu < 0.f);
    const bool fv = (v <= -1.f && gv > 0.f) || (v >= 1.f && gv < 0.f);
    float su, sv;
    if (nz_step32(gu, gv, h, fu, fv, su, sv) == 3) {
      ok = true;
      break;
    }
    const float un = fminf(1.f, fmaxf(-1.f, u + su)), vn = fminf(1.f, fmaxf(-1.f, v + sv));
    const float step = fabsf(un - u) + fabsf(vn - v), full = fabsf(su) + fabsf(sv);
    u = un;
    v = vn;
    nz_eval32<N1>(n1, C, u, v, x, r, Pu, Pv);
    const float fn = fmaf(r[0], r[0], fmaf(r[1], r[1], r[2] * r[2]));
    // the full step is taken as nz_closest takes it (Armijo decrease, or a
    // step below the rounding of f); one that would need backtracking is not
    const bool down = fn <= fmaf(2e-4f, gu * su + gv * sv, f * (1.f + 1e-6f));
    if (!(down || full < 1e-3f)) break;
    f = fn;
    if (step < kNzStop32) {
      ok = true;
      break;
    }
  }
  uo = u;
  vo = v;
  d = sqrtf(f);
  return ok && d < 3e18f;  // false for NaN too
}

// The plain FP64 iteration from the nearest node (out of line: rare).  res: u, v, y, n.
template <bool WARP>
__device__ __noinline__ double nz_pair_plain(int n1, const double *__restrict__ X, const double *xk,
                                             const double *wk, const double *x, double d_eps,
                                             double rp, int lane, double *res) {
  const double xx[3] = {x[0], x[1], x[2]};
  double u, v, y[3], nn[3];
  // every point of the patch lies within rp of a node
  const double d2 = WARP ? nz_nearest_node_warp(n1, X, xk, xx, lane, u, v)
                         : nz_nearest_node(n1, X, xk, xx, u, v);
  if (sqrt(d2) - rp > d_eps) return DBL_MAX;
  const double d = nz_closest<WARP>(n1, X, xk, wk, xx, lane, u, v, y, nn);
  res[0] = u;
  res[1] = v;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    res[2 + k] = y[k];
    res[5 + k] = nn[k];
  }
  return d;
}

// Finishes a pair in FP64 from the FP32 point.  res: u, v, y, n.  Returns the
// distance, or a negative number when the plain iteration has to take it.
template <int N1>
__device__ __forceinline__ double nz_pair64(int n1, const float4 *__restrict__ C32,
                                            const double2 *__restrict__ C64, const NzMeta &m,
                                            const double (&xg)[3], float uf, float vf,
                                            double (&res)[8]) {
  const double x[3] = {xg[0] - m.c[0], xg[1] - m.c[1], xg[2] - m.c[2]};
  double u = uf, v = vf, r[3], Pu[3], Pv[3];
  float cur[3] = {0.f, 0.f, 0.f};
  for (int it = 0; it < kNzIter64; ++it) {
    nz_eval64<N1>(n1, C64, u, v, x, r, Pu, Pv);
    const double gu = fma(r[0], Pu[0], fma(r[1], Pu[1], r[2] * Pu[2]));
    const double gv = fma(r[0], Pv[0], fma(r[1], Pv[1], r[2] * Pv[2]));
    const float a[3] = {(float)Pu[0], (float)Pu[1], (float)Pu[2]};
    const float b[3] = {(float)Pv[0], (float)Pv[1], (float)Pv[2]};
    if (it == 0) {
      const float rf[3] = {(float)r[0], (float)r[1], (float)r[2]};
      nz_curv32<N1>(n1, C32, uf, vf, rf, cur);
    }
    const float gn[3] = {fmaf(a[0], a[0], fmaf(a[1], a[1], a[2] * a[2])),
                         fmaf(a[0], b[0], fmaf(a[1], b[1], a[2] * b[2])),
                         fmaf(b[0], b[0], fmaf(b[1], b[1], b[2] * b[2]))};
    const float h[3] = {gn[0] + cur[0], gn[1] + cur[1], gn[2] + cur[2]};
    // well inside the region where Newton and Gauss-Newton have one limit
    if (!(h[0] > 0.1f * gn[0] && h[2] > 0.1f * gn[2] &&
          h[0] * h[2] - h[1] * h[1] > 0.1f * (gn[0] * gn[2] - gn[1] * gn[1])))
      return -1.0;
    const bool fu = (u <= -1.0 && gu > 0.0) || (u >= 1.0 && gu < 0.0);
    const bool fv = (v <= -1.0 && gv > 0.0) || (v >= 1.0 && gv < 0.0);
    float su, sv;
    nz_step32((float)gu, (float)gv, h, fu, fv, su, sv);
    const double un = fmin(1.0, fmax(-1.0, u + (double)su)), vn = fmin(1.0, fmax(-1.0, v + (double)sv));
    const double du = un - u, dv = vn - v, step = fabs(du) + fabs(dv);
    if (!(step < 1e-3)) return -1.0;
    u = un;
    v = vn;
    if (step < 1e-11) {  // the point moves by P_u du + P_v dv, exact to step^2
      double d2 = 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        r[k] += fma(Pu[k], du, Pv[k] * dv);
        d2 = fma(r[k], r[k], d2);
        res[2 + k] = xg[k] + r[k];
      }
      const double cx = Pu[1] * Pv[2] - Pu[2] * Pv[1], cy = Pu[2] * Pv[0] - Pu[0] * Pv[2],
                   cz = Pu[0] * Pv[1] - Pu[1] * Pv[0];
      const double il = 1.0 / sqrt(cx * cx + cy * cy + cz * cz);
      res[0] = u;
      res[1] = v;
      res[5] = cx * il;
      res[6] = cy * il;
      res[7] = cz * il;
      return sqrt(d2);
    }
  }
  return -1.0;
}

constexpr int kNzWarps = 4;
constexpr int kNzQueue = 64;   // queued pairs of a warp (32 are taken at a time)
constexpr int kNzRefine = 96;  // pairs waiting for FP64

struct NzWarpSmem {
  double x[kWarp][3];       // the warp's targets
  double res[kWarp][8];     // best so far: u, v, y, n
  double bd[kWarp];         //   distance
  int32_t bp[kWarp];        //   patch
  int32_t bplain[kWarp];    //   bit 0: the distance is the plain iteration's, bit 1: only it may be
  float best[kWarp];        // no nearer patch can be further than this (FP32 bound)
  int32_t qp[kNzQueue];     // queued pairs: patch
  int32_t qs[kNzQueue];     //   target slot
  int32_t rp[kNzRefine];    // pairs for FP64: patch
  int32_t rs[kNzRefine];    //   target slot, | 32: plain iteration
  float ru[kNzRefine], rv[kNzRefine];
  float rd[kNzRefine];      //   lower bound of the distance
};

// FP32 stage of the first n (<= 32) queued pairs.
template <int N1>
__device__ __forceinline__ void nz_stage32(NzWarpSmem &sm, const NzPatches &Q, int n1,
                                           const float *xk, float d_eps, int n, int &nref,
                                           int lane) {
  bool keep = false, plain = false;
  int p = 0, slot = 0;
  float u = 0.f, v = 0.f, d = 0.f;
  if (lane < n) {
    p = sm.qp[lane];
    slot = sm.qs[lane];
    const NzMeta m = Q.meta[p];
    const float x[3] = {(float)(sm.x[slot][0] - m.c[0]), (float)(sm.x[slot][1] - m.c[1]),
                        (float)(sm.x[slot][2] - m.c[2])};
    // FP32 rounding of a distance here, with a margin of some ten
    const float tol = 4e-5f * (m.scale + fabsf(x[0]) + fabsf(x[1]) + fabsf(x[2]));
    const float4 *X = Q.x32 + (size_t)p * n1 * n1;
    float best = INFINITY;
    int at = 0;
    for (int e = 0; e < n1 * n1; ++e) {
      const float4 y = __ldg(X + e);
      const float a = y.x - x[0], b = y.y - x[1], c = y.z - x[2];
      const float dd = fmaf(a, a, fmaf(b, b, c * c));
      if (dd < best) {
        best = dd;
        at = e;
      }
    }
    const float lb = sqrtf(best) - m.rp - tol;
    plain = !(best < INFINITY);                            // squares beyond FP32's range
    keep = plain || !(lb > d_eps || lb > sm.best[slot]);  // NaN: kept
    if (keep) {
      // a target on a node is at distance exactly 0, which only the plain
      // iteration's interpolant gives
      if (!(best > 0.f)) {
        const double *Y = Q.nodes + (size_t)p * n1 * n1 * 3, *xg = sm.x[slot];
        for (int e = 0; e < n1 * n1; ++e)
          plain = plain || (Y[3 * e] == xg[0] && Y[3 * e + 1] == xg[1] && Y[3 * e + 2] == xg[2]);
      }
      plain = plain || !nz_pair32<N1>(n1, Q.c32 + (size_t)p * n1 * n1, xk[at / n1], xk[at % n1], x,
                                      u, v, d);
      if (!plain) {
        atomicMin(reinterpret_cast<int *>(&sm.best[slot]), __float_as_int(d + tol));
        d -= tol;
        keep = !(d > d_eps);
      }
    }
  }
  __syncwarp();
  if (keep && !plain && d > sm.best[slot]) keep = false;
  const unsigned b = __ballot_sync(kFull, keep);
  if (keep) {
    const int o = nref + __popc(b & ((1u << lane) - 1u));
    sm.rp[o] = p;
    sm.rs[o] = plain ? (slot | 32) : slot;
    sm.ru[o] = u;
    sm.rv[o] = v;
    sm.rd[o] = d;
  }
  nref += __popc(b);
  __syncwarp();
}

// The barycentric basis of the plain iteration loses eps / |t - x_k| of its derivatives
// when a parameter t comes near a node x_k: the normals are good to about 2e-15 / |t - x_k|
// (11 nodes; arcs and spheres, coordinates up to 100), those of the Chebyshev form to
// 1e-14 everywhere.  The plain iteration is the search's definition, so where the two
// could differ by more than 1e-9 of a normal's size it takes the pair; closer to a node
// than kNzNodeNone, where its derivatives hold fewer than six digits, the Chebyshev form's
// stand.  Random targets: 22 kNzNodeGap of the pairs, some 14 of the 63.9 k hits of k_nz_search's
// figures, which take the call from 1.02 to 1.27 ms (the Armijo test fails in the noise, so
// such a pair takes all 40 iterations).
constexpr double kNzNodeGap = 1e-5, kNzNodeNone = 1e-9;
// kNzBeside: t lies that far from a node; kNzAtNode: closer (the ends of the square, which
// the plain iteration meets exactly, aside).
constexpr int kNzBeside = 1, kNzAtNode = 2;
__device__ __forceinline__ int nz_by_node(int n1, const double *xkd, const float *xk, double t) {
  int by = 0;
  const float tf = (float)t;
  for (int k = 0; k < n1; ++k)
    if (fabsf(tf - xk[k]) < 2.f * (float)kNzNodeGap) {  // few: FP64 only for these
      const double gap = fabs(t - xkd[k]);
      if (gap < kNzNodeNone) by |= fabs(t) < 1.0 ? kNzAtNode : 0;
      else if (gap < kNzNodeGap) by |= kNzBeside;
    }
  return by;
}
// Distances closer than this share of the coordinates' size could be equal, to each other
// or to d_eps: some thirty times the rounding of the interpolants' sums.
constexpr double kNzTie = 1e-13;
__device__ __forceinline__ double nz_size(const NzMeta &m, const double *x) {
  return fabs(x[0]) + fabs(x[1]) + fabs(x[2]) + (double)m.scale;
}
__device__ __forceinline__ bool nz_beside_node(int n1, const double *xkd, const float *xk,
                                               double t) {
  bool beside = false;
  const float tf = (float)t;
  for (int k = 0; k < n1; ++k)
    if (fabsf(tf - xk[k]) < 2.f * (float)kNzNodeGap) {  // few: FP64 only for these
      const double gap = fabs(t - xkd[k]);
      beside = beside || (gap < kNzNodeGap && gap >= kNzNodeNone);
    }
  return beside;
}

// The plain iteration of the lanes' (p, slot) pairs where `plain`: a warp per pair, or a
// thread per pair where there are many (a thread alone takes 1.8 ms for its 40 iterations,
// a warp 0.25).
constexpr int kNzPlainLanes = 8;
// keep: the distance alone.
__device__ __noinline__ double nz_plain(const NzWarpSmem &sm, const NzPatches &Q, int n1,
                                        const double *xkd, const double *wkd, double d_eps,
                                        bool plain, bool keep, int p, int slot, int lane, double d,
                                        double *res) {
  unsigned todo = __ballot_sync(kFull, plain);
  const size_t pn = (size_t)n1 * n1 * 3;
  double r[8];
  if (__popc(todo) > kNzPlainLanes) {
    if (plain)
      d = nz_pair_plain<false>(n1, Q.nodes + p * pn, xkd, wkd, sm.x[slot], d_eps, Q.rp[p], lane, r);
    if (plain && !keep)
      for (int q = 0; q < 8; ++q) res[q] = r[q];
    return d;
  }
  for (; todo; todo &= todo - 1) {
    const int l = __ffs(todo) - 1;
    const int lp = __shfl_sync(kFull, p, l), ls = __shfl_sync(kFull, slot, l);
    const double ld = nz_pair_plain<true>(n1, Q.nodes + lp * pn, xkd, wkd, sm.x[ls], d_eps,
                                          Q.rp[lp], lane, r);
    if (lane == l) d = ld;
    if (lane == l && !keep)
      for (int q = 0; q < 8; ++q) res[q] = r[q];
  }
  return d;
}

// The distances of the lanes' pairs (p, slot) where `tie`, and of their targets' best patches so
// far, by the plain iteration.
__device__ __noinline__ double nz_tie(NzWarpSmem &sm, const NzPatches &Q, int n1, const double *xkd,
                                      const double *wkd, double d_eps, bool tie, bool plain,
                                      bool keep, int p, int slot, int lane, double d, double *res) {
  d = nz_plain(sm, Q, n1, xkd, wkd, d_eps, tie && !plain, keep, p, slot, lane, d, res);
  const int how = tie ? sm.bplain[slot] : 1;
  const bool other = !(how & 1);
  double bres[8];
  const double bd = nz_plain(sm, Q, n1, xkd, wkd, d_eps, other, how & 2, other ? sm.bp[slot] : 0,
                             slot, lane, 0.0, bres);
  if (other) {
    sm.bd[slot] = bd;
    sm.bplain[slot] = how | 1;
    if (!(how & 2))
      for (int q = 0; q < 8; ++q) sm.res[slot][q] = bres[q];
  }
  return d;
}

// FP64 stage of the waiting pairs.
template <int N1>
__device__ __forceinline__ void nz_stage64(NzWarpSmem &sm, const NzPatches &Q, int n1,
                                           const float *xk, const double *xkd, const double *wkd,
                                           double d_eps, int &nref, int lane) {
  int n = 0;  // drop the pairs that another patch has beaten since
  for (int e0 = 0; e0 < nref; e0 += kWarp) {
    const int e = e0 + lane;
    int p = 0, s = 0;
    float u = 0.f, v = 0.f, d = 0.f;
    bool keep = false;
    if (e < nref) {
      p = sm.rp[e];
      s = sm.rs[e];
      u = sm.ru[e];
      v = sm.rv[e];
      d = sm.rd[e];
      keep = (s & 32) || !(d > sm.best[s & 31]);
    }
    const unsigned b = __ballot_sync(kFull, keep);
    __syncwarp();
    if (keep) {
      const int o = n + __popc(b & ((1u << lane) - 1u));
      sm.rp[o] = p;
      sm.rs[o] = s;
      sm.ru[o] = u;
      sm.rv[o] = v;
    }
    n += __popc(b);
    __syncwarp();
  }
  for (int e0 = 0; e0 < n; e0 += kWarp) {
    const int e = e0 + lane;
    const bool act = e < n;
    double d = DBL_MAX, res[8];
    int p = 0, slot = -1 - lane;
    bool plain = false, keep = false;
    if (act) {
      p = sm.rp[e];
      slot = sm.rs[e] & 31;
      const double x[3] = {sm.x[slot][0], sm.x[slot][1], sm.x[slot][2]};
      plain = sm.rs[e] & 32;
      if (!plain) {
        d = nz_pair64<N1>(n1, Q.c32 + (size_t)p * n1 * n1, Q.c64 + 2 * (size_t)p * n1 * n1,
                          Q.meta[p], x, sm.ru[e], sm.rv[e], res);
        const int by = nz_by_node(n1, xkd, xk, res[0]) | nz_by_node(n1, xkd, xk, res[1]);
        keep = d >= 0.0 && (by & kNzAtNode);
        plain = !(d >= 0.0) || by == kNzBeside ||
                fabs(d - d_eps) <= kNzTie * nz_size(Q.meta[p], x);
      }
    }
    if (__any_sync(kFull, plain))
      d = nz_plain(sm, Q, n1, xkd, wkd, d_eps, plain, keep, p, slot, lane, d, res);
    // the nearest patch of a target, ties to the lower index; pairs of one
    // target take turns.  Two patches that meet in an edge hold its nodes as the same
    // numbers, and the plain iteration finds the same distance to it from both; the
    // Chebyshev sums, relative to each patch's own centre, only to rounding.  So distances
    // that could be equal are those of the plain iteration.
    const unsigned grp = __match_any_sync(kFull, slot);
    const int turn = __popc(grp & ((1u << lane) - 1u));
    for (int k = 0; __any_sync(kFull, act && k <= turn); ++k) {
      const bool now = act && k == turn;
      bool tie = false;
      if (now && sm.bp[slot] >= 0) {
        tie = fabs(d - sm.bd[slot]) <= kNzTie * nz_size(Q.meta[p], sm.x[slot]) &&
              !(plain && (sm.bplain[slot] & 1));
      }
      if (__any_sync(kFull, tie)) {
        d = nz_tie(sm, Q, n1, xkd, wkd, d_eps, tie, plain, keep, p, slot, lane, d, res);
        plain = plain || tie;
      }
      if (now && (d < sm.bd[slot] || (d == sm.bd[slot] && p < sm.bp[slot]))) {
        sm.bd[slot] = d;
        sm.bp[slot] = p;
        sm.bplain[slot] = (plain ? 1 : 0) | (keep ? 2 : 0);
#pragma unroll
        for (int q = 0; q < 8; ++q) sm.res[slot][q] = res[q];
      }
      __syncwarp();
    }
  }
  nref = 0;
}

// 2^20 targets in a vessel against its 320 wall patches (q = 10), 63.9 k within
// d_eps: 46.4 ms as one thread per target in FP64 alone (3.4 of 32 lanes
// active, FP64 pipe 92% busy), 1.05 ms in this form (0.75 without the plain iterations
// beside nodes); the call 46.8 -> 1.3 ms.  Bound: the FP64 pipe (75% of the active cycles;
// FMA 9%), with 16.6 lanes active, since each warp finishes its own 32 targets' pairs, and
// at the end the plain iterations.  Three CTAs per SM: the FP64 basis values live in
// registers.  Other orders than q = 10 take N1 = 0, whose loops are unrolled to the largest:
// 200,000 targets at q = 4, 6, 8, 12 6.2, 8.8, 11.7, 19.1 -> 0.48, 0.57, 0.69, 0.81 ms.
template <int N1>
__global__ void __launch_bounds__(kNzWarps *kWarp, 3) k_nz_search(
    NzPatches Q, int q, const NzGrid *__restrict__ gp, const uint64_t *__restrict__ keys,
    const int32_t *__restrict__ vals, int64_t nkeys, const double *__restrict__ trg,
    const int32_t *__restrict__ list, const int32_t *__restrict__ nlist,
    int32_t *__restrict__ next, double d_eps, int32_t *__restrict__ patch_out,
    double *__restrict__ uv_out, double *__restrict__ y_out, double *__restrict__ n_out,
    double *__restrict__ dist_out) {
  __shared__ double xkd[kNzMaxN1], wkd[kNzMaxN1];
  __shared__ float xk[kNzMaxN1];
  __shared__ NzWarpSmem smem[kNzWarps];
  const int n1 = N1 ? N1 : q + 1;
  if (threadIdx.x < n1) {
    xkd[threadIdx.x] = cos(3.14159265358979323846 * threadIdx.x / q);
    xk[threadIdx.x] = (float)xkd[threadIdx.x];
    wkd[threadIdx.x] = ((threadIdx.x & 1) ? -1.0 : 1.0) * ((threadIdx.x == 0 || threadIdx.x == q) ? 0.5 : 1.0);
  }
  __syncthreads();
  NzWarpSmem &sm = smem[threadIdx.x / kWarp];
  const int lane = threadIdx.x & (kWarp - 1);
  const NzGrid g = *gp;
  const int64_t nl = *nlist;
  const float d_eps32 = __double2float_ru(d_eps);
  while (true) {
    int64_t base = 0;
    if (lane == 0) base = atomicAdd(next, 1);
    base = __shfl_sync(kFull, base, 0) * kWarp;
    if (base >= nl) break;
    const bool has = base + lane < nl;
    const int64_t t = has ? list[base + lane] : 0;
    double x[3] = {0.0, 0.0, 0.0};
    uint64_t key = 0;
    int64_t i = nkeys;
    if (has) {
#pragma unroll
      for (int k = 0; k < 3; ++k) x[k] = trg[3 * t + k];
      i = nz_first_key(g, keys, nkeys, x, key);
    }
    const float xf[3] = {(float)x[0], (float)x[1], (float)x[2]};
#pragma unroll
    for (int k = 0; k < 3; ++k) sm.x[lane][k] = x[k];
    sm.bd[lane] = DBL_MAX;
    sm.bp[lane] = -1;
    sm.best[lane] = INFINITY;
    __syncwarp();
    int nq = 0, nref = 0;
    while (true) {
      const bool more = i < nkeys && keys[i] == key;
      const bool any = __any_sync(kFull, more);
      if (any) {
        int p = 0;
        bool in = false;
        if (more) {
          p = vals[i++];
          in = nz_in_box(Q, p, x, xf);
        }
        const unsigned b = __ballot_sync(kFull, in);
        if (in) {
          const int o = nq + __popc(b & ((1u << lane) - 1u));
          sm.qp[o] = p;
          sm.qs[o] = lane;
        }
        nq += __popc(b);
        __syncwarp();
      }
      if (nq >= kWarp || (!any && nq > 0)) {
        const int n = min(nq, kWarp);
        nz_stage32<N1>(sm, Q, n1, xk, d_eps32, n, nref, lane);
        const int rest = nq - n;  // < 32: to the front
        int qp = 0, qs = 0;
        if (lane < rest) {
          qp = sm.qp[n + lane];
          qs = sm.qs[n + lane];
        }
        __syncwarp();
        if (lane < rest) {
          sm.qp[lane] = qp;
          sm.qs[lane] = qs;
        }
        nq = rest;
        __syncwarp();
        if (nref > kNzRefine - kWarp) nz_stage64<N1>(sm, Q, n1, xk, xkd, wkd, d_eps, nref, lane);
      }
      if (!any && nq == 0) break;
    }
    if (nref) nz_stage64<N1>(sm, Q, n1, xk, xkd, wkd, d_eps, nref, lane);
    __syncwarp();
    if (has) {
      const bool near = sm.bp[lane] >= 0 && sm.bd[lane] <= d_eps;
      patch_out[t] = near ? sm.bp[lane] : -1;
      uv_out[2 * t] = near ? sm.res[lane][0] : 0.0;
      uv_out[2 * t + 1] = near ? sm.res[lane][1] : 0.0;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        y_out[3 * t + k] = near ? sm.res[lane][2 + k] : 0.0;
        n_out[3 * t + k] = near ? sm.res[lane][5 + k] : 0.0;
      }
      dist_out[t] = near ? sm.bd[lane] : -1.0;
    }
    __syncwarp();
  }
}

struct NzLayout {
  size_t boxes, boxes32, rp, meta, c64, c32, x32, grid, ka, va, kb, vb, hist, hist_scan, list, cell,
      rank, count, offs, total;
};

NzLayout nz_layout(int32_t npatch, int32_t q, int64_t nt) {
  NzLayout L;
  size_t off = 0;
  auto take = [&](size_t bytes) {
    const size_t o = off;
    off += (bytes + 255) & ~(size_t)255;
    return o;
  };
  const size_t nk = (size_t)npatch * kNzCells;
  L.boxes = take(sizeof(double) * 6 * (size_t)npatch);
  L.boxes32 = take(sizeof(float) * 6 * (size_t)npatch);
  L.rp = take(sizeof(double) * (size_t)npatch);
  L.meta = take(sizeof(NzMeta) * (size_t)npatch);
  const size_t nodes = (size_t)npatch * (size_t)(q + 1) * (size_t)(q + 1);
  L.c64 = take(2 * sizeof(double2) * nodes);
  L.c32 = take(sizeof(float4) * nodes);
  L.x32 = take(sizeof(float4) * nodes);
  L.grid = take(sizeof(NzGrid));
  L.ka = take(sizeof(uint64_t) * nk);
  L.va = take(sizeof(int32_t) * nk);
  L.kb = take(sizeof(uint64_t) * nk);
  L.vb = take(sizeof(int32_t) * nk);
  const size_t he = radix_hist_entries((int64_t)nk);
  L.hist = take(sizeof(int32_t) * he);
  L.hist_scan = take(sizeof(int32_t) * (he + 1));
  const size_t nt1 = (size_t)(nt > 0 ? nt : 1);
  L.list = take(sizeof(int32_t) * nt1);
  L.cell = take(sizeof(int32_t) * nt1);
  L.rank = take(sizeof(int32_t) * nt1);
  L.count = take(sizeof(int32_t) * (nk + 1));  // per cell, then the search's queue head
  L.offs = take(sizeof(int32_t) * (nk + 1));
  L.total = off + 256;
  return L;
}

}  // namespace

extern "C" {

stk_status stokes_near_search_workspace_size(int32_t npatch, int32_t q, int64_t nt,
                                             size_t *bytes) {
  if (!bytes) return report_error(STK_EINVAL, "bytes is NULL");
  if (npatch < 0) return report_error(STK_EINVAL, "npatch must be >= 0");
  if (nt < 0 || nt > 0x7fffffff) return report_error(STK_EINVAL, "nt must be in [0, 2^31 - 1]");
  if (q < 2 || q > kNzMaxN1 - 1) return report_error(STK_EUNSUPPORTED, "q must be in [2, 12]");
  *bytes = nz_layout(npatch, q, nt).total;
  return STK_OK;
}

stk_status stokes_near_patch_search(const double *nodes, int32_t npatch, int32_t q,
                                    const double *trg, int64_t nt, double d_eps, int32_t *patch,
                                    double *uv, double *y, double *n, double *dist,
                                    void *workspace, size_t workspace_bytes, void *stream) {
  size_t need = 0;
  stk_status s = stokes_near_search_workspace_size(npatch, q, nt, &need);
  if (s != STK_OK) return s;
  if (!(d_eps >= 0.0) || !std::isfinite(d_eps))
    return report_error(STK_EINVAL, "d_eps must be finite and >= 0");
  if (nt == 0) return STK_OK;
  if (!trg || !patch || !uv || !y || !n || !dist)
    return report_error(STK_EINVAL, "trg or an output is NULL");
  cudaStream_t st = reinterpret_cast<cudaStream_t>(stream);
  if (npatch == 0) {
    // no surface: nothing is near
    if (cudaMemsetAsync(patch, 0xff, sizeof(int32_t) * (size_t)nt, st) != cudaSuccess)
      return report_error(STK_ECUDA, "cudaMemsetAsync failed");
    return STK_OK;
  }
  if (!nodes) return report_error(STK_EINVAL, "nodes is NULL");
  if (!workspace || workspace_bytes < need) return report_error(STK_ENOMEM, "workspace too small");
  const NzLayout L = nz_layout(npatch, q, nt);
  const uintptr_t u = reinterpret_cast<uintptr_t>(workspace);
  char *ws = reinterpret_cast<char *>((u + 255) & ~(uintptr_t)255);
  double *boxes = reinterpret_cast<double *>(ws + L.boxes);
  NzGrid *grid = reinterpret_cast<NzGrid *>(ws + L.grid);
  uint64_t *ka = reinterpret_cast<uint64_t *>(ws + L.ka), *kb = reinterpret_cast<uint64_t *>(ws + L.kb);
  int32_t *va = reinterpret_cast<int32_t *>(ws + L.va), *vb = reinterpret_cast<int32_t *>(ws + L.vb);
  const int n1 = q + 1;
  double *rp = reinterpret_cast<double *>(ws + L.rp);
  float *boxes32 = reinterpret_cast<float *>(ws + L.boxes32);
  NzMeta *meta = reinterpret_cast<NzMeta *>(ws + L.meta);
  double2 *c64 = reinterpret_cast<double2 *>(ws + L.c64);
  float4 *c32 = reinterpret_cast<float4 *>(ws + L.c32), *x32 = reinterpret_cast<float4 *>(ws + L.x32);
  const int64_t nk = (int64_t)npatch * kNzCells;
  int32_t *count = reinterpret_cast<int32_t *>(ws + L.count);
  int32_t *offs = reinterpret_cast<int32_t *>(ws + L.offs);
  if (cudaMemsetAsync(count, 0, sizeof(int32_t) * (size_t)(nk + 1), st) != cudaSuccess)
    return report_error(STK_ECUDA, "cudaMemsetAsync failed");
  k_nz_boxes<<<npatch, kNzThreads, 0, st>>>(nodes, n1 * n1, d_eps, boxes, boxes32, rp, meta, c64,
                                            c32, x32);
  k_nz_grid<<<1, kNzThreads, 0, st>>>(boxes, npatch, grid);
  k_nz_cells<<<(int)((nk + 255) / 256), 256, 0, st>>>(boxes, npatch, grid, ka, va);
  count_launches(3);
  const int which = radix_sort(ka, va, kb, vb, nk, 64, reinterpret_cast<int32_t *>(ws + L.hist),
                               reinterpret_cast<int32_t *>(ws + L.hist_scan), st);
  const uint64_t *keys = which ? kb : ka;
  const int32_t *vals = which ? vb : va;
  int32_t *list = reinterpret_cast<int32_t *>(ws + L.list);
  int32_t *cell = reinterpret_cast<int32_t *>(ws + L.cell);
  int32_t *rank = reinterpret_cast<int32_t *>(ws + L.rank);
  const NzPatches Q{nodes, boxes, boxes32, rp, meta, c64, c32, x32};
  int64_t blocks = (nt + kNzThreads - 1) / kNzThreads;
  if (blocks > 65535) blocks = 65535;
  k_nz_mark<<<(int)blocks, kNzThreads, 0, st>>>(Q, grid, keys, vals, nk, trg, nt, cell, rank, count,
                                                patch, uv, y, n, dist);
  launch_scan(count, nk, offs, nullptr, st);
  k_nz_scatter<<<(int)blocks, kNzThreads, 0, st>>>(nt, cell, rank, offs, list);
  int dev = 0, sms = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess)
    return report_error(STK_ECUDA, "cannot query the device");
  const int64_t warps = (nt + kWarp - 1) / kWarp;
  const int grid_s = (int)min((int64_t)sms * 3, (warps + kNzWarps - 1) / kNzWarps);
  if (n1 == 11)  // the library's default order (q = 10): its loops unrolled exactly
    k_nz_search<11><<<grid_s, kNzWarps * kWarp, 0, st>>>(Q, q, grid, keys, vals, nk, trg, list,
                                                        offs + nk, count + nk, d_eps, patch, uv, y,
                                                        n, dist);
  else
    k_nz_search<0><<<grid_s, kNzWarps * kWarp, 0, st>>>(Q, q, grid, keys, vals, nk, trg, list,
                                                       offs + nk, count + nk, d_eps, patch, uv, y,
                                                       n, dist);
  count_launches(3);
  if (cudaGetLastError() != cudaSuccess) return report_error(STK_ECUDA, "near-zone search launch failed");
  return STK_OK;
}

}  // extern "C"
