// fmm_fp64.cu -- the FP64 form of the FMM's far field on the GPU (Sec. 3.1,
// "Far evaluation"): the evaluations of fmm_passes.cuh (S2M, M2M, X-list
// sources, L2L, L2T and W-list densities) blocked by CTA and run as fixed
// point pairs (fixed_pair.cuh), and the dense M2L as products with a table of
// kernel values in fixed point.
//
// Evaluations (k_f64_eval): a CTA takes up to 32 target points of one box and
// all their sources, 128 at a time in shared memory, in coordinates relative
// to the box's centre; its 256 threads are (target, source slice) columns,
// summed in slice order.  FP64 pairs written out cost some 50 FP64
// instructions (square root and division) at 64 cycles per warp; a fixed point
// pair costs 10 of them.
//
// Dense M2L: the surfaces of two boxes of one depth are boundary points of two
// p^3 lattices, so the (p^3 boundary)^2 kernel evaluations of a box pair
// take only (2p - 1)^3 displacements.  k_f64_setup tabulates the kernel there
// at half-width 1 for each of the 316 box offsets (9 values: the symmetric
// Stokeslet and the source), k_f64_uc2e rounds each box's densities, and
// add_vlist sums 12 products per surface point pair.  Both are block fixed
// point of 54 bits in two parts of 27, so that a product is 3 integer
// multiply-adds (16 cycles against the 68 of an FP64 one) and a sum over 64
// points is exact.  What is lost is relative to the largest kernel value of an
// offset times the largest density of a box: 2^-55 of each operand's rounding and,
// of either sign, up to 2^-54 for the product of the low parts, where a partial sum in
// FP64 is rounded by 2^-53 of itself.  So that forces and sources, on one exponent, are
// of one size, the viscosity goes with the forces: the table holds the Stokeslet of
// viscosity 1 (errors below 1e-15 at viscosities of 1e-9 to 1e6, random operators; with
// the viscosity in the table 1.6e-9 at 1e-9).
//
// 65,524 points, p = 4 (131,570 V-list pairs, 4,532 W-list): see k_f64_eval.
#include "fixed_pair.cuh"
#include "fmm_fast.cuh"
#include "fmm_fp64.cuh"
#include "prep.cuh"

namespace stk {
namespace fmm {

namespace {

constexpr int kEvalThreads = 256;
constexpr int kEvalTile = 128;    // sources staged at a time
// Most targets per CTA: 32 check points, and 16 points in L2T, where a leaf can
// hold both many points and many W-list boxes (staging a source for 16 targets
// costs 5% of their pairs; the longest CTAs halve).
constexpr int kEvalTargets = 32, kL2tTargets = 16;

enum EvalMode { E_S2M, E_M2M, E_DCHK, E_L2T };

struct EvalSmem {
  SrcFx src[kEvalTile];
  double y[kEvalTile][3];            // positions relative to the box's centre
  double s0[kEvalTile];              // source strengths (equivalent densities)
  int64_t id[kEvalTile];             // point, or box * ns + surface point
  double sum[3][kEvalThreads];
};

// The FP64 form of a pair from the caller's (or the passes') own values.
__device__ __noinline__ void f64_point(const Pass &P, const double *x, const double *y, int64_t i,
                                       double *acc) {
  const double d[3] = {x[0] - y[0], x[1] - y[1], x[2] - y[2]};
  const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
  if (!(r2 > 0.0)) return;
  const double r = sqrt(r2), ir = 1.0 / r, w = P.w[i];
  if (P.f) {
    const double q[3] = {P.csl * (w * P.f[3 * i]), P.csl * (w * P.f[3 * i + 1]),
                         P.csl * (w * P.f[3 * i + 2])};
    const double c = (d[0] * q[0] + d[1] * q[1] + d[2] * q[2]) * (ir / r2);
    for (int a = 0; a < 3; ++a) acc[a] += q[a] * ir + d[a] * c;
  }
  if (P.phi) {
    const double *nn = P.nrm + 3 * i, *ph = P.phi + 3 * i;
    const double c = P.cdl * w * (d[0] * ph[0] + d[1] * ph[1] + d[2] * ph[2]) *
                     (d[0] * nn[0] + d[1] * nn[1] + d[2] * nn[2]) / (r2 * r2 * r);
    for (int a = 0; a < 3; ++a) acc[a] += d[a] * c;
  }
}
__device__ __noinline__ void f64_equivalent(const Pass &P, const double *x, const double *y,
                                            const double *e, int nc, double *acc) {
  const double d[3] = {x[0] - y[0], x[1] - y[1], x[2] - y[2]};
  const double r2 = d[0] * d[0] + d[1] * d[1] + d[2] * d[2];
  if (!(r2 > 0.0)) return;
  const double ri = 1.0 / sqrt(r2), ri3 = ri * ri * ri;
  const double c = P.csl * (d[0] * e[0] + d[1] * e[1] + d[2] * e[2]) * ri3;
  const double s = nc == 4 ? P.csrc * e[3] * ri3 : 0.0;
  for (int a = 0; a < 3; ++a) acc[a] += P.csl * e[a] * ri + d[a] * (c + s);
}

// Box geometry in whole units of the root's size / 2^22 (a box of depth d <= 21
// has half-width 2^(21 - d)): differences of centres and the bounds below are
// integer work, where FP64 would cost as much as the pairs of a small tile.
__device__ __forceinline__ int half_units(int32_t d) { return 1 << (kMaxTreeDepth - d); }
__device__ __forceinline__ void centre_units(const Tree &t, int32_t b, int32_t d, int32_t (&c)[3]) {
#pragma unroll
  for (int k = 0; k < 3; ++k) c[k] = (2 * t.anchor[3 * b + k] + 1) << (kMaxTreeDepth - d);
}
__device__ __forceinline__ double unit_size(const Tree &t) { return t.root_size * 0x1p-22; }
// Exponent E of a grid holding coordinates up to m units: m units < 2^E.
__device__ __forceinline__ int grid_exponent(const Tree &t, int m) {
  return (32 - fx_clz((uint32_t)m)) + fx_field(t.root_size) - 1022 - 22;
}
__device__ __forceinline__ bool in_range(int e) { return e <= kFxMaxExp && e >= -kFxMaxExp; }

// table_offset(), or -1 where the densities or the kernel do not fit the table.
__device__ __forceinline__ int in_table(const Pass &P, int32_t b, int32_t a) {
  const int o = table_offset(P.t, b, a);
  return o >= 0 && P.eexp[a] != kBadExp && in_range(P.kexp[o]) ? o : -1;
}

// One thread's column: sources sl, sl + nsl, ... of the staged tile.  equiv:
// densities dens (nc components) of surface points, else points.
template <int KIND>
__device__ __forceinline__ void eval_tile(const Pass &P, const EvalSmem &sm, int m, int sl, int nsl,
                                          int E, const double (&xl)[3], const double *dens, int nc,
                                          double (&acc)[3]) {
  int64_t X[3];
  uint32_t thr = in_range(E) ? kFxExact : kFxNever;
#pragma unroll
  for (int k = 0; k < 3; ++k) X[k] = fx_coord(xl[k], E, thr);
  for (int j = sl; j < m; j += nsl) {
    if (!fx_pair<KIND>(X, thr, E, sm.src[j], acc, KIND == K_EQ ? sm.s0[j] : 0.0)) {
      double a[3] = {acc[0], acc[1], acc[2]}, x[3] = {xl[0], xl[1], xl[2]};
      if (KIND == K_EQ) f64_equivalent(P, x, sm.y[j], dens + (size_t)nc * sm.id[j], nc, a);
      else f64_point(P, x, sm.y[j], sm.id[j], a);
      acc[0] = a[0];
      acc[1] = a[1];
      acc[2] = a[2];
    }
  }
}

// Adds the points of leaf box a (leaf l) at the CTA's targets.
__device__ __forceinline__ void add_points(const Pass &P, EvalSmem &sm, const double (&cb)[3],
                                           const int32_t (&cu)[3], int ext, int32_t a, int32_t l,
                                           int sl, int nsl, const double (&xl)[3],
                                           double (&acc)[3]) {
  int32_t au[3], m = ext;
  const int32_t da = P.t.depth[a], ra = half_units(da);
  centre_units(P.t, a, da, au);
  for (int k = 0; k < 3; ++k) m = max(m, abs(au[k] - cu[k]) + ra + ra / 32 + 1);
  const int E = grid_exponent(P.t, m);
  const int64_t i0 = P.t.leaf_ptr[l], i1 = P.t.leaf_ptr[l + 1];
  for (int64_t t0 = i0; t0 < i1; t0 += kEvalTile) {
    const int n = (int)min((int64_t)kEvalTile, i1 - t0);
    __syncthreads();
    if ((int)threadIdx.x < n) {
      const int64_t i = t0 + threadIdx.x;
      SrcFx &S = sm.src[threadIdx.x];
      uint32_t thr = in_range(E) ? kFxExact : kFxNever;
      double nn[3], pp[3];
      const double ws = P.csl * P.w[i], wd = P.cdl * P.w[i];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double y = P.pts[3 * i + k] - cb[k];
        sm.y[threadIdx.x][k] = y;
        S.y[k] = fx_coord(y, E, thr);
        S.q[k] = P.f ? ws * P.f[3 * i + k] : 0.0;
        nn[k] = P.phi ? P.nrm[3 * i + k] : 0.0;
        pp[k] = P.phi ? wd * P.phi[3 * i + k] : 0.0;
      }
      const int eq = fx_block(S.q, S.qh, S.ql), en = fx_block(nn, S.nh, S.nl, thr, kFxRoundN),
                ep = fx_block(pp, S.ph, S.pl, thr, kFxRoundP);
      if (!(in_range(eq) && in_range(en) && in_range(ep))) thr = kFxNever;
      S.eq = (int16_t)eq;
      S.epn = (int16_t)(en + ep);
      S.thr = thr;
      sm.id[threadIdx.x] = i;
    }
    __syncthreads();
    if (sl < nsl) {
      if (!P.phi) eval_tile<K_SL>(P, sm, n, sl, nsl, E, xl, nullptr, 0, acc);
      else if (!P.f) eval_tile<K_DL>(P, sm, n, sl, nsl, E, xl, nullptr, 0, acc);
      else eval_tile<K_SLDL>(P, sm, n, sl, nsl, E, xl, nullptr, 0, acc);
    }
  }
}

// Adds the equivalent densities dens (nc components, radius rel x half-width)
// of the boxes list(0 .. count) at the CTA's targets.
// The grid holds coordinates up to `reach` units, which the lists of a tree keep;
// a box beyond (a caller's own lists) takes the FP64 form.
template <class List>
__device__ __forceinline__ void add_equivalents(const Pass &P, EvalSmem &sm,
                                                const int32_t (&cu)[3], int reach, int64_t count,
                                                List list, double rel, const double *dens, int nc,
                                                int sl, int nsl, const double (&xl)[3],
                                                double (&acc)[3]) {
  const int64_t total = count * P.ns;
  const int E = grid_exponent(P.t, reach);
  const double unit = unit_size(P.t);
  for (int64_t g0 = 0; g0 < total; g0 += kEvalTile) {
    const int n = (int)min((int64_t)kEvalTile, total - g0);
    __syncthreads();
    if ((int)threadIdx.x < n) {
      const int64_t g = g0 + threadIdx.x;
      const int32_t a = list(g / P.ns), da = P.t.depth[a];
      const int j = (int)(g % P.ns);
      int32_t au[3];
      centre_units(P.t, a, da, au);
      const double rad = rel * (half_units(da) * unit);
      SrcFx &S = sm.src[threadIdx.x];
      uint32_t thr = in_range(E) ? kFxExact : kFxNever;
      const int64_t id = (int64_t)a * P.ns + j;
      const double *e = dens + (size_t)nc * id;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        const double y = fma(rad, P.surf[3 * j + k], (au[k] - cu[k]) * unit);
        sm.y[threadIdx.x][k] = y;
        S.y[k] = fx_coord(y, E, thr);
        S.q[k] = P.csl * e[k];
      }
      const double s0 = nc == 4 ? P.csrc * e[3] : 0.0;
      const int eq = fx_block(S.q, S.qh, S.ql);
      if (!in_range(eq) || !(fabs(s0) < 1e90)) thr = kFxNever;
      S.eq = (int16_t)eq;
      S.epn = 0;
      S.thr = thr;
      sm.s0[threadIdx.x] = s0;
      sm.id[threadIdx.x] = id;
    }
    __syncthreads();
    if (sl < nsl) eval_tile<K_EQ>(P, sm, n, sl, nsl, E, xl, dens, nc, acc);
  }
}

// ----------------------------------------------------------------- dense M2L
constexpr int kLimb = 27;  // value = (h 2^28 + l) 2^(e - 54), |h| <= 2^26, |l| <= 2^27

__device__ __forceinline__ int2_t to_limbs(double v, int e) {
  const int64_t V = llrint(ldexp(v, 54 - e));
  int2_t r;
  r.h = (int32_t)((V + ((int64_t)1 << kLimb)) >> (kLimb + 1));
  r.l = (int32_t)(V - ((int64_t)r.h << (kLimb + 1)));
  return r;
}

// Kernel values of one box offset (blockIdx.x) at half-width 1.
constexpr int kTableThreads = 128;
__device__ __forceinline__ void table_values(const Pass &P, int o, int m, double (&v)[9]) {
  const int D = 2 * P.p - 1;
  const int mi[3] = {m / (D * D), (m / D) % D, m % D}, oi[3] = {o / 49, (o / 7) % 7, o % 7};
  const double delta = 2.0 * kInner / (P.p - 1);
  double d[3], r2 = 0.0;
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    d[k] = delta * (mi[k] - (P.p - 1)) - 2.0 * (oi[k] - 3);
    r2 = fma(d[k], d[k], r2);
  }
  const double ri = r2 > 0.0 ? 1.0 / sqrt(r2) : 0.0, ri3 = ri * ri * ri;
  const double csl = 0.5 * P.csrc;  // of viscosity 1
  int c = 0;
#pragma unroll
  for (int a = 0; a < 3; ++a)
#pragma unroll
    for (int b = a; b < 3; ++b) v[c++] = csl * ((a == b ? ri : 0.0) + d[a] * d[b] * ri3);
#pragma unroll
  for (int a = 0; a < 3; ++a) v[c++] = P.csrc * d[a] * ri3;
}

// Set-up of a call: surfaces, lattice and twiddles (block 343) and the kernel
// table, a block per box offset.
__global__ void __launch_bounds__(kTableThreads) k_f64_setup(Pass P) {
  __shared__ int top;
  if (blockIdx.x == gridDim.x - 1) {
    fill_setup(P, threadIdx.x, blockDim.x);
    return;
  }
  const int o = blockIdx.x, M = table_entries(P.p), mp = table_pad(P.p);
  const int oi[3] = {o / 49 - 3, (o / 7) % 7 - 3, o % 7 - 3};
  if (oi[0] >= -1 && oi[0] <= 1 && oi[1] >= -1 && oi[1] <= 1 && oi[2] >= -1 && oi[2] <= 1) return;
  if (threadIdx.x == 0) top = 0;
  __syncthreads();
  double v[9];
  int f = 0;
  for (int m = threadIdx.x; m < M; m += kTableThreads) {
    table_values(P, o, m, v);
    for (int c = 0; c < 9; ++c) f = max(f, fx_field(v[c]));
  }
  atomicMax(&top, f);
  __syncthreads();
  const int e = top - 1022;
  if (threadIdx.x == 0) P.kexp[o] = e;
  int2_t *T = P.ktab + (size_t)o * 9 * mp;
  for (int m = threadIdx.x; m < mp; m += kTableThreads) {
    if (m < M) table_values(P, o, m, v);
    for (int c = 0; c < 9; ++c) T[(size_t)c * mp + m] = m < M ? to_limbs(v[c], e) : int2_t{0, 0};
  }
}

// UC2E, a CTA per box: the upward density, and for the kernel table its fixed
// point form scaled to half-width 1 and viscosity 1 (forces by 1 / (r mu), sources by
// 1 / r^2).
__global__ void __launch_bounds__(256) k_f64_uc2e(Pass P) {
  __shared__ int top;
  const int rows = P.nc * P.ns;
  const int32_t b = P.box0 + blockIdx.x;
  if (threadIdx.x == 0) top = -1;
  for (int i = threadIdx.x; i < rows; i += blockDim.x) UC2E()(P, (int64_t)blockIdx.x * rows + i);
  if (!P.ktab) return;
  __syncthreads();
  double c[3], r;
  box_geom(P.t, b, P.depth, c, r);
  const double sf = P.csl / (0.5 * P.csrc) / r, sq = 1.0 / (r * r);
  const double *u = P.up + (size_t)b * rows;
  int f = -1;  // -1: all zero; 0: subnormal
  for (int i = threadIdx.x; i < rows; i += blockDim.x) {
    const double v = u[i] * ((i % P.nc) < 3 ? sf : sq);
    if (v != 0.0 || u[i] != 0.0) f = max(f, fx_field(v));
  }
  f = __reduce_max_sync(kFull, f);
  if ((threadIdx.x & 31) == 0) atomicMax(&top, f);
  __syncthreads();
  const int e = top >= 0 ? top - 1022 : 0;
  const bool ok = in_range(e);  // so that the sums' FP64 exponents are
  if (threadIdx.x == 0) P.eexp[b] = ok ? e : kBadExp;
  for (int i = threadIdx.x; i < 4 * P.ns; i += blockDim.x) {
    const int j = i / 4, k = i % 4;
    const double v = k < P.nc ? u[P.nc * j + k] * (k < 3 ? sf : sq) : 0.0;
    P.edens[((size_t)b * P.ns + j) * 4 + k] = ok ? to_limbs(v, e) : int2_t{0, 0};
  }
}

__device__ __forceinline__ void copy16(void *dst, const void *src) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                   (uint32_t)__cvta_generic_to_shared(dst)),
               "l"(src)
               : "memory");
}

constexpr int kM2lBlock = 64;  // surface points per exact sum: 256 products of 2^52 fit 63 bits

// Two buffers of a table and a box's densities, and the points' lattice positions.
size_t m2l_smem(int p, int ns) {
  return 2 * sizeof(int2_t) * (9 * (size_t)table_pad(p) + 4 * (size_t)ns) + sizeof(int32_t) * ns;
}

// Adds the V-list densities of box b at its check point t (source points of
// slice sl of nsl), one entry after another: the offset's table and the
// entry's densities in shared memory (dyn), the next entry's copied meanwhile.
// Entries outside the table are skipped; returns whether there are any.
__device__ bool add_vlist(const Pass &P, unsigned char *dyn, int32_t b, int t, int sl, int nsl,
                          double (&u)[3]) {
  const int mp = table_pad(P.p), D = 2 * P.p - 1, ns = P.ns, tid = threadIdx.x;
  const size_t buf_bytes = sizeof(int2_t) * (9 * (size_t)mp + 4 * (size_t)ns);
  const bool act = sl < nsl;
  const int j0 = act ? ns * sl / nsl : 0, j1 = act ? ns * (sl + 1) / nsl : 0;
  auto lin = [&](int i) {
    return (P.sidx[3 * i] * D + P.sidx[3 * i + 1]) * D + P.sidx[3 * i + 2];
  };
  const int base = lin(t) + ((P.p - 1) * D + (P.p - 1)) * D + (P.p - 1);
  int32_t *ljs = reinterpret_cast<int32_t *>(dyn + 2 * buf_bytes);  // lattice positions
  for (int i = tid; i < ns; i += blockDim.x) ljs[i] = lin(i);
  const int32_t v1 = P.t.v_ptr[b + 1];
  auto fetch = [&](int32_t a, int off, int buf) {
    unsigned char *dst = dyn + (size_t)buf * buf_bytes;
    const unsigned char *st = reinterpret_cast<const unsigned char *>(P.ktab + (size_t)off * 9 * mp);
    const unsigned char *se = reinterpret_cast<const unsigned char *>(P.edens + (size_t)a * ns * 4);
    const int nt = 9 * mp / 2, ne = 2 * ns;  // 16-byte units
    for (int i = tid; i < nt; i += blockDim.x) copy16(dst + 16 * i, st + 16 * i);
    for (int i = tid; i < ne; i += blockDim.x) copy16(dst + 16 * (nt + i), se + 16 * i);
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  bool odd = false;
  auto next = [&](int32_t v, int32_t &a, int &off) {  // the next entry in the table, or v1
    for (; v < v1; ++v) {
      a = P.t.v_idx[v];
      off = in_table(P, b, a);
      if (off >= 0) break;
      odd = true;
    }
    return v;
  };
  // hh of nj points is below nj 2^54
  const int up = 8 - (32 - fx_clz((uint32_t)min(j1 - j0, kM2lBlock)));
  int32_t a = 0, an = 0;
  int off = 0, offn = 0, buf = 0;
  int32_t v = next(P.t.v_ptr[b], a, off);
  if (v < v1) fetch(a, off, 0);
  while (v < v1) {
    const int32_t vn = next(v + 1, an, offn);
    if (vn < v1) {
      fetch(an, offn, buf ^ 1);
      asm volatile("cp.async.wait_group 1;" ::: "memory");
    } else {
      asm volatile("cp.async.wait_group 0;" ::: "memory");
    }
    __syncthreads();
    const int2_t *T = reinterpret_cast<const int2_t *>(dyn + (size_t)buf * buf_bytes);
    const int4 *Ed = reinterpret_cast<const int4 *>(T + 9 * (size_t)mp);
    // sums in units of 2^(ek + ee - 52 - up), as many bits below as the block leaves
    const int eb = 1086 + P.kexp[off] + P.eexp[a] - 52 - up;
    for (int jb = j0; jb < j1; jb += kM2lBlock) {
      const int je = min(j1, jb + kM2lBlock);
      int64_t hh[3] = {0, 0, 0}, cr[3] = {0, 0, 0};
      for (int j = jb; j < je; ++j) {
        const int2_t *K = T + (base - ljs[j]);
        const int4 e01 = Ed[2 * j], e23 = Ed[2 * j + 1];
        const int32_t eh[4] = {e01.x, e01.z, e23.x, e23.z}, el[4] = {e01.y, e01.w, e23.y, e23.w};
        // kernel value of (velocity, density): xx xy xz yy yz zz, then sx sy sz
        constexpr int sym[3][4] = {{0, 1, 2, 6}, {1, 3, 4, 7}, {2, 4, 5, 8}};
        int2_t kv[9];
#pragma unroll
        for (int c = 0; c < 9; ++c) kv[c] = K[(size_t)c * mp];
#pragma unroll
        for (int q = 0; q < 3; ++q)
#pragma unroll
          for (int c = 0; c < 4; ++c) {
            const int2_t w = kv[sym[q][c]];
            hh[q] = fx_mad(w.h, eh[c], hh[q]);
            cr[q] = fx_mad(w.h, el[c], cr[q]);
            cr[q] = fx_mad(w.l, eh[c], cr[q]);
          }
      }
#pragma unroll
      for (int q = 0; q < 3; ++q) {
        const int64_t rest = (cr[q] + ((int64_t)1 << (kLimb - up))) >> (kLimb + 1 - up);
        u[q] += fx_to_double((hh[q] << up) + rest, eb);
      }
    }
    __syncthreads();
    v = vn;
    a = an;
    off = offn;
    buf ^= 1;
  }
  return odd;
}

// 65,524 points, p = 4, one thread per output in FP64 -> this: DCHK 93 -> 4.4 ms
// (the M2L 3.9 of them: 36 multiply-adds of 5 cycles per surface point pair
// and warp, and 11 shared-memory reads beside them), L2T 16.1 -> 0.86 (1.64 with
// the box geometry in FP64 per staged source), M2M 2.4 -> 0.13, S2M 0.94 -> 0.14;
// the far field 139 -> 5.9 ms.
template <int MODE>
__global__ void __launch_bounds__(kEvalThreads, 2) k_f64_eval(Pass P) {
  extern __shared__ __align__(16) unsigned char dyn[];  // E_DCHK with the kernel table
  __shared__ EvalSmem sm;
  int32_t b, leaf = -1;
  if (MODE == E_S2M || MODE == E_L2T) {
    leaf = blockIdx.x;
    b = P.t.leaf_box[leaf];
  } else {
    b = P.box0 + blockIdx.x;
  }
  const int32_t depth = P.t.depth[b];
  if (MODE == E_S2M && depth < kFirstDepth) return;
  if (MODE == E_M2M && P.t.child_ptr[b] >= P.t.child_ptr[b + 1]) return;
  double cb[3], r;
  box_geom(P.t, b, depth, cb, r);
  int32_t cu[3];
  centre_units(P.t, b, depth, cu);
  // furthest coordinates, in units: targets, and the lists' surfaces (children
  // and W boxes within 3 r + 1.05 r / 2, V boxes within 6 r + 1.05 r; the
  // parent's surface is at 2.95 * 2 r about a centre r off)
  const int ru = half_units(depth), ext = 3 * ru, near_reach = 4 * ru, far_reach = 8 * ru;
  const int64_t p0 = MODE == E_L2T ? P.t.leaf_ptr[leaf] : 0;
  const int nt = MODE == E_L2T ? (int)(P.t.leaf_ptr[leaf + 1] - p0) : P.ns;
  const double rad = MODE == E_DCHK ? kInner * r : kOuter * r;
  constexpr int most = MODE == E_L2T ? kL2tTargets : kEvalTargets;
  const int nch = (nt + most - 1) / most;
  for (int ch = blockIdx.y; ch < nch; ch += gridDim.y) {
    const int a0 = (int)((int64_t)nt * ch / nch), tn = (int)((int64_t)nt * (ch + 1) / nch) - a0;
    const int nsl = kEvalThreads / tn, t = a0 + threadIdx.x % tn, sl = threadIdx.x / tn;
    double xl[3], acc[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int k = 0; k < 3; ++k)
      xl[k] = MODE == E_L2T ? P.pts[3 * (p0 + t) + k] - cb[k] : rad * P.surf[3 * t + k];
    if (MODE == E_S2M) add_points(P, sm, cb, cu, ext, b, leaf, sl, nsl, xl, acc);
    if (MODE == E_M2M) {
      const int32_t c0 = P.t.child_ptr[b];
      add_equivalents(P, sm, cu, near_reach, P.t.child_ptr[b + 1] - c0,
                      [c0](int64_t s) { return c0 + (int32_t)s; }, kInner, P.up, P.nc, sl, nsl, xl,
                      acc);
    }
    if (MODE == E_DCHK) {
      const int32_t v0 = P.t.v_ptr[b], v1 = P.t.v_ptr[b + 1];
      if (!P.spec && !P.ktab) {
        const int32_t *vi = P.t.v_idx + v0;
        add_equivalents(P, sm, cu, far_reach, v1 - v0, [vi](int64_t s) { return vi[s]; }, kInner, P.up,
                        P.nc, sl, nsl, xl, acc);
      } else if (!P.spec && add_vlist(P, dyn, b, t, sl, nsl, acc)) {
        for (int32_t v = v0; v < v1; ++v) {  // entries the kernel table does not hold
          const int32_t a = P.t.v_idx[v];
          if (in_table(P, b, a) < 0)
            add_equivalents(P, sm, cu, far_reach, 1, [a](int64_t) { return a; }, kInner, P.up, P.nc, sl,
                            nsl, xl, acc);
        }
      }
      for (int32_t v = P.t.x_ptr[b]; v < P.t.x_ptr[b + 1]; ++v) {
        const int32_t a = P.t.x_idx[v], l = P.t.box_leaf[a];
        if (l >= 0) add_points(P, sm, cb, cu, ext, a, l, sl, nsl, xl, acc);
      }
      if (depth > kFirstDepth) {
        const int32_t pb = P.t.parent[b];
        add_equivalents(P, sm, cu, far_reach, 1, [pb](int64_t) { return pb; }, kOuter, P.dn, 3, sl, nsl,
                        xl, acc);
      }
    }
    if (MODE == E_L2T) {
      if (depth >= kFirstDepth)
        add_equivalents(P, sm, cu, near_reach, 1, [b](int64_t) { return b; }, kOuter, P.dn, 3, sl, nsl, xl,
                        acc);
      const int32_t *wi = P.t.w_idx + P.t.w_ptr[b];
      add_equivalents(P, sm, cu, near_reach, P.t.w_ptr[b + 1] - P.t.w_ptr[b],
                      [wi](int64_t s) { return wi[s]; }, kInner, P.up, P.nc, sl, nsl, xl, acc);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < 3; ++k) sm.sum[k][threadIdx.x] = sl < nsl ? acc[k] : 0.0;
    __syncthreads();
    for (int v = threadIdx.x; v < 3 * tn; v += kEvalThreads) {
      const int tt = v / 3, k = v % 3;
      double u = 0.0;
      for (int s = 0; s < nsl; ++s) u += sm.sum[k][s * tn + tt];
      if (MODE == E_L2T) {
        double *o = P.out + 3 * (p0 + a0 + tt) + k;
        *o = (P.accumulate ? *o : 0.0) + u;
      } else {
        const size_t at = (size_t)b * 3 * P.ns + 3 * (a0 + tt) + k;
        P.chk[at] = MODE == E_DCHK && P.spec ? P.m2l[at] + u : u;
      }
    }
    __syncthreads();
  }
}

template <class F>
__global__ void __launch_bounds__(256) k_f64_pass(Pass P, int64_t n) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t e = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; e < n; e += stride) F()(P, e);
}

}  // namespace

cudaError_t far_field_fp64(const Pass &P0, const int32_t *depth_ptr, int32_t max_depth, int sms,
                           cudaStream_t st) {
  Pass P = P0;
  const int ns = P.ns, nch = (ns + kEvalTargets - 1) / kEvalTargets;
  int launches = 0;
  auto pass = [&](auto f, int64_t n) {
    if (n <= 0) return;
    const int64_t g = (n + 255) / 256, most = (int64_t)sms * 8;
    k_f64_pass<decltype(f)><<<(unsigned)(g < most ? g : most), 256, 0, st>>>(P, n);
    ++launches;
  };
  auto at_depth = [&](int32_t d) {
    P.depth = d;
    P.box0 = depth_ptr[d];
    P.box1 = depth_ptr[d + 1];
    return (int64_t)(P.box1 - P.box0);
  };
  k_f64_setup<<<P.ktab ? 344 : 1, kTableThreads, 0, st>>>(P);
  ++launches;
  const size_t table_smem = P.ktab ? m2l_smem(P.p, ns) : 0;
  if (table_smem) {
    // the limit belongs to the kernel, not to the call: one value for every order, so that
    // host threads with plans of different orders do not lower each other's
    const cudaError_t e = cudaFuncSetAttribute(
        k_f64_eval<E_DCHK>, cudaFuncAttributeMaxDynamicSharedMemorySize,
        (int)m2l_smem(kTableMaxP, surface_count(kTableMaxP)));
    if (e != cudaSuccess) return e;
  }
  k_f64_eval<E_S2M><<<dim3(P.t.nleaf, nch), kEvalThreads, 0, st>>>(P);
  ++launches;
  for (int32_t d = max_depth; d >= kFirstDepth; --d) {
    const int64_t nb = at_depth(d);
    if (nb <= 0) continue;
    if (d < max_depth) {
      k_f64_eval<E_M2M><<<dim3((unsigned)nb, nch), kEvalThreads, 0, st>>>(P);
      ++launches;
    }
    k_f64_uc2e<<<(unsigned)nb, 256, 0, st>>>(P);
    ++launches;
  }
  for (int32_t d = kFirstDepth; d <= max_depth; ++d) {
    const int64_t nb = at_depth(d), nf = freq_count(P.p);
    if (nb <= 0) continue;
    if (P.spec) {
      pass(UFFT(), nb * nf * P.nc);
      // per box and frequency over its V-list: with the spectral products blocked
      // by parent a missing child or neighbour idles its lanes (65,524 points, far
      // field 33.3 ms against 13.3)
      pass(KMUL(), nb * nf);
      pass(IFFT(), nb * ns);
    }
    k_f64_eval<E_DCHK><<<dim3((unsigned)nb, nch), kEvalThreads, table_smem, st>>>(P);
    ++launches;
    pass(DC2E(), nb * 3 * ns);
  }
  // leaves of up to 256 points take one target chunk per CTA
  k_f64_eval<E_L2T><<<dim3(P.t.nleaf, 256 / kL2tTargets), kEvalThreads, 0, st>>>(P);
  ++launches;
  count_launches(launches);
  return cudaGetLastError();
}

}  // namespace fmm
}  // namespace stk
