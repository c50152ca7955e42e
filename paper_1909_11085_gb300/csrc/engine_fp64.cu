// engine_fp64.cu -- FP64 evaluation of the Stokes single- and double-layer
// sums (Eq. "sl_stokes", the double-layer kernel of Sec. 2.1, summed as in
// Sec. 3.1).  Same work items as the mixed engine: a warp takes up to 128
// targets against the item's source segments, read with warp-uniform
// (broadcast) loads.  On GB300 the FP64 pipe runs at about 1/64 of the FP32
// rate, so a pair written in FP64 alone is bound by it: k_engine_fp64, which
// remains for inputs that fixed point does not fit.  k_engine_fx evaluates the
// differences, dot products and reciprocals in fixed point (fixed_pair.cuh).
// Both are launched; the packing decides on the device which of them works.
#include "common.cuh"
#include "fixed_pair.cuh"
#include "prep.cuh"

namespace stk {

template <int T, int KIND>
__device__ __forceinline__ void seg64(const SrcRec64 *__restrict__ rec, int64_t s, int64_t e,
                                      int sg, int b, const double (&x)[T][3],
                                      double (&acc)[T][3]) {
  for (int64_t k = s + sg; k < e; k += b) {
    const SrcRec64 &R = rec[k];
    const double yx = R.y[0], yy = R.y[1], yz = R.y[2];
    double qx = 0, qy = 0, qz = 0, nx = 0, ny = 0, nz = 0, px = 0, py = 0, pz = 0;
    if (KIND & K_SL) { qx = R.q[0]; qy = R.q[1]; qz = R.q[2]; }
    if (KIND & K_DL) {
      nx = R.n[0]; ny = R.n[1]; nz = R.n[2];
      px = R.p[0]; py = R.p[1]; pz = R.p[2];
    }
#pragma unroll
    for (int t = 0; t < T; ++t) {
      const double dx = x[t][0] - yx, dy = x[t][1] - yy, dz = x[t][2] - yz;
      const double r2 = dx * dx + dy * dy + dz * dz;
      const double ri = r2 > 0.0 ? rsqrt(r2) : 0.0;  // zero-distance pair contributes nothing
      const double ri2 = ri * ri;
      if (KIND == K_SL) {
        const double c = (dx * qx + dy * qy + dz * qz) * ri2;
        acc[t][0] += (qx + dx * c) * ri;
        acc[t][1] += (qy + dy * c) * ri;
        acc[t][2] += (qz + dz * c) * ri;
      } else if (KIND == K_DL) {
        const double c = (dx * px + dy * py + dz * pz) * (dx * nx + dy * ny + dz * nz) *
                         (ri2 * ri2 * ri);
        acc[t][0] += dx * c;
        acc[t][1] += dy * c;
        acc[t][2] += dz * c;
      } else {
        const double dq = dx * qx + dy * qy + dz * qz;
        const double dp = dx * px + dy * py + dz * pz;
        const double dn = dx * nx + dy * ny + dz * nz;
        const double c = (dq + dp * dn * ri2) * ri2;
        acc[t][0] += (qx + dx * c) * ri;
        acc[t][1] += (qy + dy * c) * ri;
        acc[t][2] += (qz + dz * c) * ri;
      }
    }
  }
}

template <int T>
__device__ void run_item64(const EngineParams &P, const Item &it, int b, int lane) {
  const int G = kWarp / b, tgl = lane % G, sg = lane / G;
  const int tn = it.tn_part & 0xFF, part = it.tn_part >> 8;
  double x[T][3], acc[T][3];
  bool valid[T];
#pragma unroll
  for (int t = 0; t < T; ++t) {
    const int li = tgl + G * t;
    valid[t] = li < tn;
    const int gi = it.t0 + (valid[t] ? li : 0);
    const int ci = P.tperm ? P.tperm[gi] : gi;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      x[t][k] = valid[t] ? P.trg64[3 * (size_t)ci + k] : 1e300;
      acc[t][k] = 0.0;
    }
  }
  for (int e = it.seg0; e < it.seg1; ++e) {
    const int sid = P.seg_list ? P.seg_list[e] : e;
    const int64_t s = P.range_ptr[sid], en = P.range_ptr[sid + 1];
    const int kind = seg_kind(P, sid);
    if (kind == K_SL)
      seg64<T, K_SL>(P.rec64, s, en, sg, b, x, acc);
    else if (kind == K_DL)
      seg64<T, K_DL>(P.rec64, s, en, sg, b, x, acc);
    else
      seg64<T, K_SLDL>(P.rec64, s, en, sg, b, x, acc);
  }
  for (int o = G; o < kWarp; o <<= 1)
#pragma unroll
    for (int t = 0; t < T; ++t)
#pragma unroll
      for (int k = 0; k < 3; ++k) acc[t][k] += __shfl_xor_sync(kFull, acc[t][k], o);
  if (sg == 0) {
    double *out = P.part_out + ((size_t)part * (size_t)P.nt + (size_t)it.t0) * 3;
#pragma unroll
    for (int t = 0; t < T; ++t)
      if (valid[t]) {
        const int li = tgl + G * t;
#pragma unroll
        for (int k = 0; k < 3; ++k) out[3 * li + k] = acc[t][k];
      }
  }
}

__global__ void __launch_bounds__(kWarpsPerCta *kWarp, 4) k_engine_fp64(EngineParams P, FxParams F) {
  if (F.state && fx_use(*F.state, F.ns, F.nt)) return;  // k_engine_fx does the call
  const int lane = threadIdx.x & (kWarp - 1);
  const int n_items = *P.n_items;
  while (true) {
    int idx = 0;
    if (lane == 0) idx = atomicAdd(P.item_counter, 1);
    idx = __shfl_sync(kFull, idx, 0);
    if (idx >= n_items) break;
    const int id = P.item_order ? P.item_order[idx] : idx;
    const Item it = P.items[id];
    const int tn = it.tn_part & 0xFF;
    if (P.policy == 1) {
      if (tn <= 32)
        run_item64<1>(P, it, 1, lane);
      else if (tn <= 64)
        run_item64<2>(P, it, 1, lane);
      else if (tn <= 96)
        run_item64<3>(P, it, 1, lane);
      else
        run_item64<4>(P, it, 1, lane);
    } else if (tn <= 8)
      run_item64<1>(P, it, 4, lane);
    else if (tn <= 16)
      run_item64<2>(P, it, 4, lane);
    else if (tn <= 24)
      run_item64<3>(P, it, 4, lane);
    else if (tn <= 32)
      run_item64<4>(P, it, 4, lane);
    else if (tn <= 48)
      run_item64<3>(P, it, 2, lane);
    else if (tn <= 64)
      run_item64<4>(P, it, 2, lane);
    else if (tn <= 96)
      run_item64<3>(P, it, 1, lane);
    else
      run_item64<4>(P, it, 1, lane);
  }
}

// ------------------------------------------------------------ fixed point
// The FP64 form of a pair that fixed point cannot hold, from the caller's values (j: the
// source).
template <int KIND>
__device__ __noinline__ void fx_slow(const FxParams &F, const double *xp, const double *yp,
                                     int64_t j, const double *q, double *acc) {
  const double dx = xp[0] - yp[0], dy = xp[1] - yp[1], dz = xp[2] - yp[2];
  const double r2 = dx * dx + dy * dy + dz * dz;
  if (!(r2 > 0.0)) return;  // zero-distance pair contributes nothing
  const double ri = rsqrt(r2), ri2 = ri * ri;
  double c = 0.0;
  if (KIND & K_DL) {
    const double wc = (F.w ? F.w[j] : 1.0) * F.cdl;
    const double *n = F.nrm + 3 * j, *p = F.phi + 3 * j;
    c = (dx * (wc * p[0]) + dy * (wc * p[1]) + dz * (wc * p[2])) *
        (dx * n[0] + dy * n[1] + dz * n[2]);
  }
  const double d[3] = {dx, dy, dz};
  if (KIND & K_SL) {
    c = (dx * q[0] + dy * q[1] + dz * q[2] + c * ri2) * ri2;
    for (int k = 0; k < 3; ++k) acc[k] += (q[k] + d[k] * c) * ri;
  } else {
    c *= ri2 * ri2 * ri;
    for (int k = 0; k < 3; ++k) acc[k] += d[k] * c;
  }
}

template <int KIND>
__device__ __forceinline__ void seg_fx(const EngineParams &P, const FxParams &F,
                                       const SrcFx *__restrict__ rec, int64_t s, int64_t e, int b,
                                       int E, const int64_t (&X)[3], uint32_t xthr,
                                       const double *xp, double (&acc)[3]) {
  for (int64_t k = s; k < e; k += b) {
    const SrcFx &S = rec[k];
    if (!fx_pair<KIND>(X, xthr, E, S, acc)) {
      double a[3] = {acc[0], acc[1], acc[2]};
      fx_slow<KIND>(F, xp, P.src64 + 3 * (size_t)k, k, S.q, a);
      acc[0] = a[0];
      acc[1] = a[1];
      acc[2] = a[2];
    }
  }
}

// An item's tn targets and b source slices make tn b columns, one per lane,
// 32 to a pass over the item's sources; b is chosen so that the last pass is
// nearly full (a pair costs some 700 cycles of a warp, its loads nothing).  The
// slices' sums meet in shared memory and are added in slice order.
constexpr int kFxCols = 256, kFxSlices = 16;

//
// Bound: the FP64 pipe, 9 instructions of about 68 cycles per warp and SL + DL
// pair, with some 190 integer and FP32 instructions beside them (six CTAs per
// SM so that one warp's integer part overlaps another's FP64 part).  SL + DL of
// 34,816 points on themselves: 71.5 -> 19.9 ms (k_engine_fp64 -> this), near
// field of 262,096 points: 44.3 -> 7.5 ms (24.2 ms with items of 128 targets,
// whose last round left the GPU idle).
// Double layer of a flat wall of 4,096 points at z = 10 at targets 0.1 and less above it
// (faint dots, summed exactly): 0.41 ms, 0.32 in general position, 1.0 in k_engine_fp64.
template <int KMODE>
__global__ void __launch_bounds__(kWarpsPerCta *kWarp, 6) k_engine_fx(EngineParams P, FxParams F) {
  __shared__ double sums[kWarpsPerCta][3][kFxCols];
  const FxState fs = *F.state;
  if (!fx_use(fs, F.ns, F.nt)) return;  // k_engine_fp64 does the call
  const int E = fx_exp(fs);
  double(*R)[kFxCols] = sums[threadIdx.x / kWarp];
  const int lane = threadIdx.x & (kWarp - 1);
  const int n_items = *P.n_items;
  while (true) {
    int idx = 0;
    if (lane == 0) idx = atomicAdd(P.item_counter, 1);
    idx = __shfl_sync(kFull, idx, 0);
    if (idx >= n_items) break;
    const Item it = P.items[P.item_order ? P.item_order[idx] : idx];
    const int tn = it.tn_part & 0xFF, part = it.tn_part >> 8;
    // slices: fewest lanes idle, at most kFxCols columns
    int b = 1;
    for (int c = 2, idle = ((tn + 31) & ~31) - tn, cols = tn;
         c <= kFxSlices && idle * 16 > cols && c * tn <= kFxCols; ++c) {
      const int n = c * tn, w = ((n + 31) & ~31) - n;
      if (w * cols < idle * n) {
        idle = w;
        cols = n;
        b = c;
      }
    }
    const int ncol = b * tn;
    for (int c0 = 0; c0 < ncol; c0 += kWarp) {
      const int col = min(c0 + lane, ncol - 1);
      const int sl = col / tn, t = it.t0 + col % tn;
      const double *xp = P.trg64 + 3 * (size_t)(P.tperm ? P.tperm[t] : t);
      int64_t X[3];
      uint32_t xthr = kFxExact;
      double acc[3];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        X[k] = fx_coord(xp[k], E, xthr);
        acc[k] = 0.0;
      }
      for (int e = it.seg0; e < it.seg1; ++e) {
        int sid = P.seg_list ? P.seg_list[e] : e;
        const int64_t s = P.range_ptr[sid] + sl;
        int64_t en = P.range_ptr[sid + 1];
        if (KMODE && P.seg_list)  // contiguous segments as one, so that slices come out even
          while (e + 1 < it.seg1 && P.range_ptr[sid = P.seg_list[e + 1]] == en) {
            en = P.range_ptr[sid + 1];
            ++e;
          }
        if (KMODE ? KMODE == K_SL : !(sid & 1))
          seg_fx<K_SL>(P, F, F.rec, s, en, b, E, X, xthr, xp, acc);
        else if (KMODE ? KMODE == K_DL : true)
          seg_fx<K_DL>(P, F, F.rec, s, en, b, E, X, xthr, xp, acc);
        else
          seg_fx<K_SLDL>(P, F, F.rec, s, en, b, E, X, xthr, xp, acc);
      }
      if (c0 + lane < ncol)
#pragma unroll
        for (int k = 0; k < 3; ++k) R[k][col] = acc[k];
    }
    __syncwarp();
    double *out = P.part_out + ((size_t)part * (size_t)P.nt + (size_t)it.t0) * 3;
    for (int v = lane; v < 3 * tn; v += kWarp) {
      const int t = v / 3, k = v % 3;
      double a = R[k][t];
      for (int sl = 1; sl < b; ++sl) a += R[k][sl * tn + t];
      out[v] = a;
    }
    __syncwarp();
  }
}

// The largest exponent field of this thread's coordinates of the sources and (when they
// differ) targets.
__device__ __forceinline__ int fx_range_of(int64_t ns, const double *__restrict__ src, int64_t nt,
                                           const double *__restrict__ trg, int64_t i0,
                                           int64_t step) {
  const int64_t n = 3 * ns, m = n + 3 * nt;
  int f = 0;
  for (int64_t i = i0; i < m; i += step) f = max(f, fx_field(i < n ? src[i] : trg[i - n]));
  return f;
}

// This thread's records of the sources on the grid of exponent E; trg: the targets whose
// inexact coordinates are counted too (for the double layer's faint dots).
__device__ __forceinline__ void fx_records_of(int64_t ns, const double *__restrict__ src, int64_t nt,
                                              const double *__restrict__ trg,
                                              const double *__restrict__ f,
                                              const double *__restrict__ nrm,
                                              const double *__restrict__ phi,
                                              const double *__restrict__ w, double csl, double cdl,
                                              int E, int64_t i0, int64_t step,
                                              SrcFx *__restrict__ rec, int &bad, int &inexact,
                                              int &trg_inexact) {
  bad = inexact = trg_inexact = 0;
  for (int64_t j = i0; j < ns; j += step) {
    SrcFx R;
    const double wj = w ? w[j] : 1.0;
    double n[3], p[3];
    R.thr = kFxExact;
    for (int k = 0; k < 3; ++k) {
      R.y[k] = fx_coord(src[3 * j + k], E, R.thr);
      R.q[k] = f ? wj * csl * f[3 * j + k] : 0.0;
      n[k] = phi ? nrm[3 * j + k] : 0.0;
      p[k] = phi ? wj * cdl * phi[3 * j + k] : 0.0;
    }
    const int eq = fx_block(R.q, R.qh, R.ql, R.thr, kFxRoundQ),
              en = fx_block(n, R.nh, R.nl, R.thr, kFxRoundN),
              ep = fx_block(p, R.ph, R.pl, R.thr, kFxRoundP);
    const bool ok = eq <= kFxMaxExp && eq >= -kFxMaxExp && en <= kFxMaxExp && en >= -kFxMaxExp &&
                    ep <= kFxMaxExp && ep >= -kFxMaxExp;
    R.eq = (int16_t)eq;
    R.epn = (int16_t)(en + ep);
    bad |= !ok;
    inexact += R.thr >= kFxInexact;
    rec[j] = R;
  }
  for (int64_t i = i0; phi && i < nt; i += step) {
    uint32_t thr = kFxExact;
    for (int k = 0; k < 3; ++k) fx_coord(trg[3 * i + k], E, thr);
    trg_inexact += thr != kFxExact;
  }
}

// This thread's records of the plain FP64 form.
__device__ __forceinline__ void fp64_records_of(int64_t ns, const double *__restrict__ src,
                                                const double *__restrict__ f,
                                                const double *__restrict__ nrm,
                                                const double *__restrict__ phi,
                                                const double *__restrict__ w, double csl,
                                                double cdl, int64_t i0, int64_t step,
                                                SrcRec64 *__restrict__ rec) {
  for (int64_t j = i0; j < ns; j += step) {
    SrcRec64 R;
    const double wj = w ? w[j] : 1.0;
    for (int k = 0; k < 3; ++k) {
      R.y[k] = src[3 * j + k];
      R.q[k] = f ? wj * csl * f[3 * j + k] : 0.0;
      R.n[k] = phi ? nrm[3 * j + k] : 0.0;
      R.p[k] = phi ? wj * cdl * phi[3 * j + k] : 0.0;
    }
    rec[j] = R;
  }
}

__device__ __forceinline__ bool fx_exp_fits(int E) { return E <= kFxMaxExp && E >= -kFxMaxExp; }

__global__ void k_fx_range(int64_t ns, const double *__restrict__ src, int64_t nt,
                           const double *__restrict__ trg, FxState *__restrict__ st) {
  int f = fx_range_of(ns, src, nt, trg, blockIdx.x * (int64_t)blockDim.x + threadIdx.x,
                      (int64_t)gridDim.x * blockDim.x);
  f = __reduce_max_sync(kFull, f);
  if ((threadIdx.x & 31) == 0) atomicMax(&st->field, f);
}

__global__ void k_pack_fx(int64_t ns, const double *__restrict__ src, int64_t nt,
                          const double *__restrict__ trg, const double *__restrict__ f,
                          const double *__restrict__ nrm, const double *__restrict__ phi,
                          const double *__restrict__ w, double csl, double cdl,
                          FxState *__restrict__ st, SrcFx *__restrict__ rec) {
  const int E = st->field - 1022;
  if (!fx_exp_fits(E)) return;
  int bad, inexact, trg_inexact;
  fx_records_of(ns, src, nt, trg, f, nrm, phi, w, csl, cdl, E,
                blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x, rec,
                bad, inexact, trg_inexact);
  inexact = __reduce_add_sync(kFull, inexact);
  trg_inexact = __reduce_add_sync(kFull, trg_inexact);
  bad = __any_sync(kFull, bad);
  if ((threadIdx.x & 31) != 0) return;
  if (bad) st->bad = 1;
  if (inexact) atomicAdd(&st->inexact, inexact);
  if (trg_inexact) atomicAdd(&st->trg_inexact, trg_inexact);
}

__global__ void k_pack_fp64(int64_t ns, const double *__restrict__ src,
                            const double *__restrict__ f, const double *__restrict__ nrm,
                            const double *__restrict__ phi, const double *__restrict__ w,
                            double csl, double cdl, const FxState *__restrict__ fx, int64_t nt,
                            SrcRec64 *__restrict__ rec) {
  if (fx && fx_use(*fx, ns, nt)) return;
  fp64_records_of(ns, src, f, nrm, phi, w, csl, cdl,
                  blockIdx.x * (int64_t)blockDim.x + threadIdx.x, (int64_t)gridDim.x * blockDim.x,
                  rec);
}

// The three of them in one block, for few points, where a launch costs more than its work
// (single layer of 64 points on themselves 75 -> 68 us, 500 83 -> 81, 2,000 142 -> 152).
constexpr int kPackThreads = 256;
constexpr int64_t kPackFew = 512;
__global__ void __launch_bounds__(kPackThreads)
    k_pack_few(int64_t ns, const double *__restrict__ src, int64_t nt,
               const double *__restrict__ trg, const double *__restrict__ f,
               const double *__restrict__ nrm, const double *__restrict__ phi,
               const double *__restrict__ w, double csl, double cdl, FxState *__restrict__ st,
               SrcFx *__restrict__ recfx, SrcRec64 *__restrict__ rec) {
  __shared__ FxState s;
  const bool first = (threadIdx.x & 31) == 0;
  if (threadIdx.x == 0) s = FxState{0, 0, 0, 0};
  __syncthreads();
  const int m = __reduce_max_sync(kFull, fx_range_of(ns, src, nt, trg, threadIdx.x, kPackThreads));
  if (first) atomicMax(&s.field, m);
  __syncthreads();
  const int E = s.field - 1022;
  if (fx_exp_fits(E)) {
    int bad, inexact, trg_inexact;
    fx_records_of(ns, src, nt, trg, f, nrm, phi, w, csl, cdl, E, threadIdx.x, kPackThreads, recfx,
                  bad, inexact, trg_inexact);
    bad = __any_sync(kFull, bad);
    inexact = __reduce_add_sync(kFull, inexact);
    trg_inexact = __reduce_add_sync(kFull, trg_inexact);
    if (first) {
      atomicOr(&s.bad, bad);
      atomicAdd(&s.inexact, inexact);
      atomicAdd(&s.trg_inexact, trg_inexact);
    }
  }
  __syncthreads();
  if (threadIdx.x == 0) *st = s;
  if (!fx_use(s, ns, nt))
    fp64_records_of(ns, src, f, nrm, phi, w, csl, cdl, threadIdx.x, kPackThreads, rec);
}

static int pack_grid(int64_t n) {
  int64_t g = (n + 255) / 256;
  return (int)(g < 1 ? 1 : g > 4096 ? 4096 : g);
}

void launch_pack_fp64(int64_t ns, const double *src, const double *f, const double *nrm,
                      const double *phi, const double *w, double csl, double cdl, SrcRec64 *rec,
                      cudaStream_t st) {
  k_pack_fp64<<<pack_grid(ns), 256, 0, st>>>(ns, src, f, nrm, phi, w, csl, cdl, nullptr, 0, rec);
  count_launches(1);
}

void launch_fx_range(int64_t ns, const double *src, int64_t nt, const double *trg, FxState *fx,
                     cudaStream_t st) {
  k_fx_range<<<pack_grid(3 * ns + 3 * nt), 256, 0, st>>>(ns, src, nt, trg, fx);
  count_launches(1);
}

void launch_fx_records(int64_t n, const double *pts, const double *f, const double *nrm,
                       const double *phi, const double *w, double csl, double cdl, FxState *fx,
                       SrcFx *rec, cudaStream_t st) {
  k_pack_fx<<<pack_grid(n), 256, 0, st>>>(n, pts, 0, nullptr, f, nrm, phi, w, csl, cdl, fx, rec);
  count_launches(1);
}

void launch_pack_fx(int64_t ns, const double *src, int64_t nt, const double *trg, const double *f,
                    const double *nrm, const double *phi, const double *w, double csl, double cdl,
                    FxState *fx, SrcFx *recfx, SrcRec64 *rec, cudaStream_t st) {
  if (ns + nt <= kPackFew) {
    k_pack_few<<<1, kPackThreads, 0, st>>>(ns, src, nt, trg, f, nrm, phi, w, csl, cdl, fx, recfx, rec);
    count_launches(1);
    return;
  }
  launch_fx_range(ns, src, nt, trg, fx, st);
  k_pack_fx<<<pack_grid(ns > nt ? ns : nt), 256, 0, st>>>(ns, src, nt, trg, f, nrm, phi, w, csl, cdl,
                                                          fx, recfx);
  k_pack_fp64<<<pack_grid(ns), 256, 0, st>>>(ns, src, f, nrm, phi, w, csl, cdl, fx, nt, rec);
  count_launches(2);
}

cudaError_t launch_engine_fp64(const EngineParams &P, const FxParams &F, int grid, int grid_fx,
                               cudaStream_t stream) {
  if (!F.state) {
    // the plain engine alone
  } else if (P.kind_alternating) {
    k_engine_fx<0><<<grid_fx, kWarpsPerCta * kWarp, 0, stream>>>(P, F);
  } else if (P.kind == K_SL) {
    k_engine_fx<K_SL><<<grid_fx, kWarpsPerCta * kWarp, 0, stream>>>(P, F);
  } else if (P.kind == K_DL) {
    k_engine_fx<K_DL><<<grid_fx, kWarpsPerCta * kWarp, 0, stream>>>(P, F);
  } else {
    k_engine_fx<K_SLDL><<<grid_fx, kWarpsPerCta * kWarp, 0, stream>>>(P, F);
  }
  k_engine_fp64<<<grid, kWarpsPerCta * kWarp, 0, stream>>>(P, F);
  count_launches(F.state ? 2 : 1);
  return cudaGetLastError();
}

cudaError_t engine_fp64_occupancy(int *blocks_per_sm, int *blocks_per_sm_fx) {
  cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm, k_engine_fp64,
                                                                kWarpsPerCta * kWarp, 0);
  if (e != cudaSuccess) return e;
  return cudaOccupancyMaxActiveBlocksPerMultiprocessor(blocks_per_sm_fx, k_engine_fx<K_SLDL>,
                                                       kWarpsPerCta * kWarp, 0);
}

}  // namespace stk
