// adjoint.cu -- gradients of L = sum_i g_i . u(x_i), u = SL[f] + DL[phi], with
// respect to the densities, the source positions and normals and the target
// positions.  The pair terms are the derivatives of the two kernels (the
// single layer of Eq. "sl_stokes", the double layer of Sec. 2.1), with d = x - y,
// q = w f / (8 pi mu), psi = 6 w phi / (8 pi):
//   s = g.q/r + (d.g)(d.q)/r^3
//     ds/dq   = g/r + d (d.g)/r^3
//     ds/dd   = [g (d.q) + q (d.g) - (g.q) d]/r^3 - 3 (d.g)(d.q) d/r^5
//   t = (d.g)(d.psi)(d.n)/r^5
//     dt/dpsi = (d.g)(d.n) d/r^5,   dt/dn = (d.g)(d.psi) d/r^5
//     dt/dd   = [g (d.psi)(d.n) + psi (d.g)(d.n) + n (d.g)(d.psi)]/r^5 - 5 t d/r^2
// dL/dx_i = sum_j d(s + t)/dd,  dL/dy_j = -sum_i d(s + t)/dd.  Nothing O(N^2) is
// stored: two passes recompute the pair terms.  The source-major pass gives,
// per source, dL/df, dL/dphi, dL/dn and dL/dy (a sum over targets); the
// target-major pass gives dL/dx (a sum over sources).
//
// Both passes tile their inputs through shared memory in CTAs of 128 output
// points (Morton-sorted, so a CTA is spatially compact) and split the inputs
// over blockIdx.y for occupancy.  The mixed form works in FP32 in the CTA's
// local frame (positions split hi/lo as in the forward records) with a
// two-sum per tile; a pair with |r| < alpha h_j is left out of the FP32 sum
// and listed for its output point (up to kAdjNearCap); k_adj_near then
// evaluates the listed pairs in FP64 (difference, 1/|r| and the pair terms) in
// input order and adds them to the point's partial.  Keeping FP64 out of the
// FP32 pass keeps its registers, and so its occupancy, those of FP32 code.
// An output point with more near pairs than the list holds is rescanned by
// k_adj_near with the FP32 pass's own frame and test.  The FP64 form evaluates
// the differences, dot products and reciprocals of a pair in fixed point
// (fixed_pair.cuh) where its inputs fit, and in double otherwise.
#include <cfloat>

#include "common.cuh"
#include "prep.cuh"

namespace stk {

constexpr int kAdjThreads = 128;

// Pair terms.  For the source-major pass the own point is the source (q, psi,
// n fixed) and g comes from the input; for the target-major pass the own
// point is the target (g fixed).  acc layout (source-major): 0..2 ds/dq,
// 3..5 dt/dpsi / psi-scale, 6..8 dt/dn, 9..11 -d(s+t)/dd; (target-major):
// 0..2 d(s+t)/dd.
template <typename R, bool SRC>
__device__ __forceinline__ void adj_pair(R dx, R dy, R dz, R ri, const R (&g)[3], const R (&q)[3],
                                         const R (&p)[3], const R (&n)[3], int has_sl, int has_dl,
                                         R *acc) {
  const R ri2 = ri * ri, ri3 = ri * ri2, ri5 = ri3 * ri2;
  const R dg = dx * g[0] + dy * g[1] + dz * g[2];
  R gx = 0, gy = 0, gz = 0;
  if (has_sl) {
    const R dq = dx * q[0] + dy * q[1] + dz * q[2];
    const R gq = g[0] * q[0] + g[1] * q[1] + g[2] * q[2];
    if (SRC) {
      const R c = dg * ri3;
      acc[0] += g[0] * ri + dx * c;
      acc[1] += g[1] * ri + dy * c;
      acc[2] += g[2] * ri + dz * c;
    }
    const R a = dq * ri3, b = dg * ri3, cd = -gq * ri3 - R(3) * dg * dq * ri5;
    gx += g[0] * a + q[0] * b + dx * cd;
    gy += g[1] * a + q[1] * b + dy * cd;
    gz += g[2] * a + q[2] * b + dz * cd;
  }
  if (has_dl) {
    const R dp = dx * p[0] + dy * p[1] + dz * p[2];
    const R dn = dx * n[0] + dy * n[1] + dz * n[2];
    const R a = dg * dn * ri5, b = dg * dp * ri5;
    if (SRC) {
      acc[3] += dx * a;
      acc[4] += dy * a;
      acc[5] += dz * a;
      acc[6] += dx * b;
      acc[7] += dy * b;
      acc[8] += dz * b;
    }
    const R e = dp * dn * ri5, t5 = R(5) * b * dn * ri2;  // 5 t / r^2, t = (d.g)(d.psi)(d.n)/r^5
    gx += g[0] * e + p[0] * a + n[0] * b - dx * t5;
    gy += g[1] * e + p[1] * a + n[1] * b - dy * t5;
    gz += g[2] * e + p[2] * a + n[2] * b - dz * t5;
  }
  if (SRC) {
    acc[9] -= gx;
    acc[10] -= gy;
    acc[11] -= gz;
  } else {
    acc[0] += gx;
    acc[1] += gy;
    acc[2] += gz;
  }
}

template <bool SRC>
struct NAcc {
  static constexpr int value = SRC ? 12 : 3;
};

// ---------------------------------------------------------------- FP32 pass
// Two output points per thread, one in each half of the packed FP32
// instructions (an input's values are duplicated into both halves), 128 output
// points per CTA of 64 threads.  One output per thread issued 81% of its slots
// at 63% of the FMA pipe; packed, the pipe is the bound (81 of its operations
// per source-major pair, 65 per target-major one).  Per half the operations,
// their order and their rounding are those the scalar form compiled to (which
// product of a sum is fused differs between the passes: FIRST), so the sums are
// what one output per thread gave, bit for bit.
// 34,816 points on themselves: source-major 4.01 -> 3.03 ms, target-major
// 3.46 -> 2.55 ms (FMA pipe 83% and 81% of its cycles).
constexpr int kAdjPack = kAdjThreads / 2;  // threads of a packed CTA

__device__ __forceinline__ float2 a2(float2 a, float2 b) { return __fadd2_rn(a, b); }
__device__ __forceinline__ float2 m2(float2 a, float2 b) { return __fmul2_rn(a, b); }
__device__ __forceinline__ float2 f2(float2 a, float2 b, float2 c) { return __ffma2_rn(a, b, c); }
__device__ __forceinline__ float2 both(float v) { return make_float2(v, v); }
__device__ __forceinline__ float2 neg2(float2 a) { return make_float2(-a.x, -a.y); }
// a b + c d, the first or the second product fused into the sum
template <bool FIRST>
__device__ __forceinline__ float2 sum2(float2 a, float2 b, float2 c, float2 d) {
  return FIRST ? f2(a, b, m2(c, d)) : f2(c, d, m2(a, b));
}
template <bool FIRST>
__device__ __forceinline__ float2 dot2(const float2 (&a)[3], const float2 (&b)[3]) {
  return f2(a[2], b[2], sum2<FIRST>(a[0], b[0], a[1], b[1]));
}

template <bool SRC, int KIND>
__device__ __forceinline__ void adj_pair2(const float2 (&d)[3], float2 ri, const float2 (&g)[3],
                                          const float2 (&q)[3], const float2 (&p)[3],
                                          const float2 (&n)[3], float2 *acc) {
  const float2 ri2 = m2(ri, ri), ri3 = m2(ri, ri2), ri5 = m2(ri3, ri2);
  const float2 dg = dot2<true>(d, g);
  float2 gx[3] = {both(0.f), both(0.f), both(0.f)};
  if (KIND & K_SL) {
    const float2 dq = dot2<SRC>(d, q), gq = dot2<SRC>(g, q);
    const float2 a = m2(dq, ri3), b = m2(dg, ri3);
    if (SRC)
#pragma unroll
      for (int k = 0; k < 3; ++k) acc[k] = a2(acc[k], f2(g[k], ri, m2(d[k], b)));
    const float2 t = m2(m2(both(3.f), dg), dq);
    const float2 cd = f2(neg2(t), ri5, m2(neg2(gq), ri3));
#pragma unroll
    for (int k = 0; k < 3; ++k) gx[k] = f2(d[k], cd, sum2<SRC>(g[k], a, q[k], b));
  }
  if (KIND & K_DL) {
    const float2 dp = dot2<true>(d, p), dn = dot2<true>(d, n);
    const float2 a = m2(m2(dg, dn), ri5), b = m2(m2(dg, dp), ri5);
    if (SRC)
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        acc[3 + k] = f2(d[k], a, acc[3 + k]);
        acc[6 + k] = f2(d[k], b, acc[6 + k]);
      }
    const float2 e = m2(m2(dp, dn), ri5), t5 = m2(m2(m2(both(5.f), b), dn), ri2), mt5 = neg2(t5);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float2 w = f2(d[k], mt5, f2(n[k], b, sum2<SRC>(g[k], e, p[k], a)));
      gx[k] = a2(gx[k], w);
    }
  }
#pragma unroll
  for (int k = 0; k < 3; ++k)
    if (SRC) acc[9 + k] = a2(acc[9 + k], neg2(gx[k]));
    else acc[k] = a2(acc[k], gx[k]);
}

template <bool SRC, int KIND>
__global__ void __launch_bounds__(kAdjPack, SRC ? 8 : 12) k_adj_mixed(AdjParams A) {
  constexpr int NA = NAcc<SRC>::value;
  __shared__ float4 sP[kAdjThreads];   // local position, hh
  __shared__ float4 sG[kAdjThreads];   // g (src-major) or q (trg-major)
  __shared__ float4 sN[SRC ? 1 : kAdjThreads];   // n (trg-major)
  __shared__ float4 sPs[SRC ? 1 : kAdjThreads];  // psi (trg-major)
  __shared__ int32_t sI[kAdjThreads];  // caller index
  __shared__ float sums[2 * NA][kAdjThreads];  // compensated sums (hi, lo)
  __shared__ float red[6][kAdjPack / kWarp];
  const SrcRec *orec = reinterpret_cast<const SrcRec *>(A.out_rec);
  const SrcRec *irec = reinterpret_cast<const SrcRec *>(A.in_rec);
  const int tid = threadIdx.x;
  const int64_t o0 = (int64_t)blockIdx.x * kAdjThreads;
  bool valid[2];
  int64_t oc[2];
  SrcRec Ro[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    valid[h] = o0 + tid + h * kAdjPack < A.nout;
    oc[h] = A.operm[valid[h] ? o0 + tid + h * kAdjPack : o0];
    Ro[h] = orec[oc[h]];
  }

  // CTA origin: centre of the output points' bounding box, as hi/lo splits
  const SrcRec R0 = orec[A.operm[o0]];
  float oh[3], ol[3];
  {
    float mn[3], mx[3];  // (an invalid half repeats the first point)
#pragma unroll
    for (int k = 0; k < 3; ++k) mn[k] = INFINITY, mx[k] = -INFINITY;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const float r[3] = {(Ro[h].yh.x - R0.yh.x) + (Ro[h].q.w - R0.q.w),
                          (Ro[h].yh.y - R0.yh.y) + (Ro[h].n.w - R0.n.w),
                          (Ro[h].yh.z - R0.yh.z) + (Ro[h].p.w - R0.p.w)};
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        mn[k] = fminf(mn[k], r[k]);
        mx[k] = fmaxf(mx[k], r[k]);
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) {
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        mn[k] = fminf(mn[k], __shfl_xor_sync(kFull, mn[k], o));
        mx[k] = fmaxf(mx[k], __shfl_xor_sync(kFull, mx[k], o));
      }
      if (tid % kWarp == 0) {
        red[k][tid / kWarp] = mn[k];
        red[3 + k][tid / kWarp] = mx[k];
      }
    }
    __syncthreads();
    const float first[3] = {R0.yh.x, R0.yh.y, R0.yh.z}, low[3] = {R0.q.w, R0.n.w, R0.p.w};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const float lo = fminf(red[k][0], red[k][1]), hi = fmaxf(red[3 + k][0], red[3 + k][1]);
      split_hl((double)first[k] + (double)low[k] + 0.5 * ((double)lo + hi), oh[k], ol[k]);
    }
  }
  float2 own[3], v1[3], on[3], op[3];  // position; g (trg-major) or q; n; psi
  float2 own_hh;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const float o[3] = {to_local(Ro[h].yh.x, Ro[h].q.w, oh[0], ol[0]),
                        to_local(Ro[h].yh.y, Ro[h].n.w, oh[1], ol[1]),
                        to_local(Ro[h].yh.z, Ro[h].p.w, oh[2], ol[2])};
    if (valid[h] && blockIdx.y == 0) {  // the frame, for a rescan of an overflowing list
      float *fr = A.oframe + 9 * (size_t)oc[h];
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        fr[k] = o[k];
        fr[3 + k] = oh[k];
        fr[6 + k] = ol[k];
      }
    }
    const float q[3] = {Ro[h].q.x, Ro[h].q.y, Ro[h].q.z}, n[3] = {Ro[h].n.x, Ro[h].n.y, Ro[h].n.z},
                p[3] = {Ro[h].p.x, Ro[h].p.y, Ro[h].p.z};
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      (h ? own[k].y : own[k].x) = o[k];
      (h ? v1[k].y : v1[k].x) = q[k];
      (h ? on[k].y : on[k].x) = n[k];
      (h ? op[k].y : op[k].x) = p[k];
    }
    (h ? own_hh.y : own_hh.x) = Ro[h].yh.w;
  }

  float2 ps[NA];
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    ps[a] = both(0.f);
#pragma unroll
    for (int h = 0; h < 2; ++h)
      sums[a][tid + h * kAdjPack] = sums[NA + a][tid + h * kAdjPack] = 0.f;
  }

  // the tiles of split y / nsub, its part y % nsub
  const int64_t split = blockIdx.y / A.nsub, sub = blockIdx.y % A.nsub;
  const int64_t s0 = A.nin * split / A.nsplit, s1 = A.nin * (split + 1) / A.nsplit;
  const int64_t tiles = (s1 - s0 + kAdjThreads - 1) / kAdjThreads;
  const int64_t i0 = s0 + kAdjThreads * (tiles * sub / A.nsub);
  const int64_t i1 = min(s1, s0 + kAdjThreads * (tiles * (sub + 1) / A.nsub));
  for (int64_t tb = i0; tb < i1; tb += kAdjThreads) {
    __syncthreads();
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int s = tid + h * kAdjPack;
      if (tb + s < i1) {
        const int32_t ic = A.iperm[tb + s];
        const SrcRec R = irec[ic];
        sP[s] = make_float4(to_local(R.yh.x, R.q.w, oh[0], ol[0]),
                            to_local(R.yh.y, R.n.w, oh[1], ol[1]),
                            to_local(R.yh.z, R.p.w, oh[2], ol[2]), R.yh.w);
        sG[s] = make_float4(R.q.x, R.q.y, R.q.z, 0.f);
        if (!SRC) {
          sN[s] = make_float4(R.n.x, R.n.y, R.n.z, 0.f);
          sPs[s] = make_float4(R.p.x, R.p.y, R.p.z, 0.f);
        }
        sI[s] = ic;
      }
    }
    __syncthreads();
    const int m = (int)min((int64_t)kAdjThreads, i1 - tb);
    for (int kk = 0; kk < m; ++kk) {
      const float4 P = sP[kk], G = sG[kk];
      const float2 in[3] = {both(P.x), both(P.y), both(P.z)};
      const float2 gi[3] = {both(G.x), both(G.y), both(G.z)};
      float2 d[3];  // x - y: the target is the input (src-major) or the own point
#pragma unroll
      for (int k = 0; k < 3; ++k) d[k] = SRC ? a2(in[k], neg2(own[k])) : a2(own[k], neg2(in[k]));
      const float2 r2 = f2(d[0], d[0], f2(d[1], d[1], m2(d[2], d[2])));
      const bool near0 = r2.x < (SRC ? own_hh.x : P.w), near1 = r2.y < (SRC ? own_hh.y : P.w);
      const float2 ri = make_float2(near0 ? 0.f : rsqrt_ftz(r2.x), near1 ? 0.f : rsqrt_ftz(r2.y));
      if (SRC) {
        adj_pair2<SRC, KIND>(d, ri, gi, v1, op, on, ps);
      } else {
        float2 n2[3], p2[3];
        if (KIND & K_DL) {
          const float4 N = sN[kk], Q = sPs[kk];
          n2[0] = both(N.x), n2[1] = both(N.y), n2[2] = both(N.z);
          p2[0] = both(Q.x), p2[1] = both(Q.y), p2[2] = both(Q.z);
        }
        adj_pair2<SRC, KIND>(d, ri, v1, gi, p2, n2, ps);
      }
      if (near0 || near1) {  // listed for the FP64 pass
#pragma unroll
        for (int h = 0; h < 2; ++h)
          if ((h ? near1 : near0) && valid[h]) {
            const int slot = atomicAdd(A.near_cnt + oc[h], 1);
            if (slot < A.near_cap) A.near_idx[(size_t)oc[h] * A.near_cap + slot] = sI[kk];
          }
      }
    }
#pragma unroll
    for (int a = 0; a < NA; ++a) {
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int s = tid + h * kAdjPack;
        float hi = sums[a][s], lo = sums[NA + a][s];
        two_sum_acc(hi, lo, h ? ps[a].y : ps[a].x);
        sums[a][s] = hi;
        sums[NA + a][s] = lo;
      }
      ps[a] = both(0.f);
    }
  }
#pragma unroll
  for (int h = 0; h < 2; ++h)
    if (valid[h]) {
      const int s = tid + h * kAdjPack;
      double *out = A.partial + ((size_t)blockIdx.y * (size_t)A.nout + (size_t)oc[h]) * NA;
#pragma unroll
      for (int a = 0; a < NA; ++a) out[a] = (double)sums[a][s] + (double)sums[NA + a][s];
    }
}

// ---------------------------------------------------------------- near pairs
// FP64 pair terms of output point oc with input ic (zero distance: nothing).
template <bool SRC>
__device__ __forceinline__ void adj_near_pair(const AdjParams &A, int64_t oc, int32_t ic,
                                              double (&ad)[NAcc<SRC>::value]) {
  const SrcRec *orec = reinterpret_cast<const SrcRec *>(A.out_rec);
  const SrcRec *irec = reinterpret_cast<const SrcRec *>(A.in_rec);
  const double *xa = SRC ? A.in64 + 3 * (size_t)ic : A.out64 + 3 * (size_t)oc;
  const double *ya = SRC ? A.out64 + 3 * (size_t)oc : A.in64 + 3 * (size_t)ic;
  const double ddx = xa[0] - ya[0], ddy = xa[1] - ya[1], ddz = xa[2] - ya[2];
  const double rr = ddx * ddx + ddy * ddy + ddz * ddz;
  if (!(rr > 0.0)) return;
  const SrcRec Ro = orec[oc], Ri = irec[ic];
  const double rid = 1.0 / sqrt(rr);
  // own values: g (target-major) or q, psi, n (source-major); the input's the others
  const SrcRec &S = SRC ? Ro : Ri, &Tg = SRC ? Ri : Ro;
  const double g[3] = {Tg.q.x, Tg.q.y, Tg.q.z}, q[3] = {S.q.x, S.q.y, S.q.z},
               p[3] = {S.p.x, S.p.y, S.p.z}, n[3] = {S.n.x, S.n.y, S.n.z};
  adj_pair<double, SRC>(ddx, ddy, ddz, rid, g, q, p, n, A.has_sl, A.has_dl, ad);
}

// One thread per output point: its listed near pairs, sorted by input index,
// in FP64, added to the point's first partial.  A point whose list overflowed
// is rescanned over all inputs (in index order) with the FP32 pass's frame
// and test, so the same pairs are found.
template <bool SRC>
__global__ void __launch_bounds__(kAdjThreads) k_adj_near(AdjParams A) {
  constexpr int NA = NAcc<SRC>::value;
  for (int64_t oc = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; oc < A.nout;
       oc += (int64_t)gridDim.x * blockDim.x) {
    const int32_t c = A.near_cnt[oc];
    if (c == 0) continue;
    double ad[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) ad[a] = 0.0;
    if (c <= A.near_cap) {
      int32_t idx[kAdjNearCap];
      for (int k = 0; k < c; ++k) {  // insertion sort
        const int32_t v = A.near_idx[(size_t)oc * A.near_cap + k];
        int m = k;
        while (m > 0 && idx[m - 1] > v) {
          idx[m] = idx[m - 1];
          --m;
        }
        idx[m] = v;
      }
      for (int k = 0; k < c; ++k) adj_near_pair<SRC>(A, oc, idx[k], ad);
    } else {
      const SrcRec *orec = reinterpret_cast<const SrcRec *>(A.out_rec);
      const SrcRec *irec = reinterpret_cast<const SrcRec *>(A.in_rec);
      const float *fr = A.oframe + 9 * (size_t)oc;
      const float ox = fr[0], oy = fr[1], oz = fr[2];
      const float oh[3] = {fr[3], fr[4], fr[5]}, ol[3] = {fr[6], fr[7], fr[8]};
      const float own_hh = orec[oc].yh.w;
      for (int64_t ic = 0; ic < A.nin; ++ic) {
        const SrcRec R = irec[ic];
        const float px = to_local(R.yh.x, R.q.w, oh[0], ol[0]);
        const float py = to_local(R.yh.y, R.n.w, oh[1], ol[1]);
        const float pz = to_local(R.yh.z, R.p.w, oh[2], ol[2]);
        const float dx = SRC ? px - ox : ox - px, dy = SRC ? py - oy : oy - py,
                    dz = SRC ? pz - oz : oz - pz;
        const float r2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
        const float hh = SRC ? own_hh : R.yh.w;
        if (r2 < hh) adj_near_pair<SRC>(A, oc, (int32_t)ic, ad);
      }
    }
    double *out = A.partial + (size_t)oc * NA;  // the first input split
#pragma unroll
    for (int a = 0; a < NA; ++a) out[a] += ad[a];
  }
}

// ---------------------------------------------------------------- FP64 pass
template <bool SRC>
__global__ void __launch_bounds__(kAdjThreads) k_adj_fp64(AdjParams A) {
  if (A.fx && fx_adj_use(*A.fx, A.nout + A.nin)) return;  // k_adj_fx does the call
  constexpr int NA = NAcc<SRC>::value;
  __shared__ double sP[kAdjThreads][3];
  __shared__ double sA[kAdjThreads][3];
  __shared__ double sN[kAdjThreads][3];
  __shared__ double sPs[kAdjThreads][3];
  const SrcRec64 *orec = reinterpret_cast<const SrcRec64 *>(A.out_rec);
  const SrcRec64 *irec = reinterpret_cast<const SrcRec64 *>(A.in_rec);
  const int tid = threadIdx.x;
  const int64_t o_sorted = (int64_t)blockIdx.x * kAdjThreads + tid;
  const bool valid = o_sorted < A.nout;
  const int64_t oc = valid ? A.operm[o_sorted] : 0;
  SrcRec64 Ro;
  if (valid) Ro = orec[oc];
  double acc[NA];
#pragma unroll
  for (int a = 0; a < NA; ++a) acc[a] = 0.0;
  const int64_t parts = (int64_t)A.nsplit * A.nsub;
  const int64_t i0 = A.nin * blockIdx.y / parts, i1 = A.nin * (blockIdx.y + 1) / parts;
  for (int64_t tb = i0; tb < i1; tb += kAdjThreads) {
    const int64_t k = tb + tid;
    if (k < i1) {
      const SrcRec64 R = irec[A.iperm[k]];
      for (int c = 0; c < 3; ++c) {
        sP[tid][c] = R.y[c];
        sA[tid][c] = R.q[c];
        sN[tid][c] = R.n[c];
        sPs[tid][c] = R.p[c];
      }
    }
    __syncthreads();
    const int m = (int)min((int64_t)kAdjThreads, i1 - tb);
    if (valid) {
      for (int kk = 0; kk < m; ++kk) {
        const double dx = SRC ? sP[kk][0] - Ro.y[0] : Ro.y[0] - sP[kk][0];
        const double dy = SRC ? sP[kk][1] - Ro.y[1] : Ro.y[1] - sP[kk][1];
        const double dz = SRC ? sP[kk][2] - Ro.y[2] : Ro.y[2] - sP[kk][2];
        const double r2 = dx * dx + dy * dy + dz * dz;
        const double ri = r2 > 0.0 ? rsqrt(r2) : 0.0;
        double g[3], q[3], pp[3], nn[3];
        for (int c = 0; c < 3; ++c) {
          if (SRC) {
            g[c] = sA[kk][c];
            q[c] = Ro.q[c];
            pp[c] = Ro.p[c];
            nn[c] = Ro.n[c];
          } else {
            g[c] = Ro.q[c];
            q[c] = sA[kk][c];
            pp[c] = sPs[kk][c];
            nn[c] = sN[kk][c];
          }
        }
        adj_pair<double, SRC>(dx, dy, dz, ri, g, q, pp, nn, A.has_sl, A.has_dl, acc);
      }
    }
    __syncthreads();
  }
  if (valid) {
    double *out = A.partial + ((size_t)blockIdx.y * (size_t)A.nout + (size_t)oc) * NA;
#pragma unroll
    for (int a = 0; a < NA; ++a) out[a] = acc[a];
  }
}

// ------------------------------------------------ FP64 pass in fixed point
// The FP64 form of a pair that fixed point cannot hold.
template <bool SRC>
__device__ __noinline__ void adj_fx_slow(const SrcRec64 *T, const SrcRec64 *S, int has_sl,
                                         int has_dl, double *acc) {
  const double dx = T->y[0] - S->y[0], dy = T->y[1] - S->y[1], dz = T->y[2] - S->y[2];
  const double r2 = dx * dx + dy * dy + dz * dz;
  if (!(r2 > 0.0)) return;  // zero-distance pair contributes nothing
  const double g[3] = {T->q[0], T->q[1], T->q[2]}, q[3] = {S->q[0], S->q[1], S->q[2]},
               p[3] = {S->p[0], S->p[1], S->p[2]}, n[3] = {S->n[0], S->n[1], S->n[2]};
  adj_pair<double, SRC>(dx, dy, dz, rsqrt(r2), g, q, p, n, has_sl, has_dl, acc);
}

// Exponents of the sources' normals (fx_block's), which their records only hold
// added to those of psi.
__global__ void k_adj_nexp(int64_t ns, const double *__restrict__ nrm,
                           int32_t *__restrict__ nexp) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < ns;
       j += (int64_t)gridDim.x * blockDim.x) {
    const int f = max(fx_field(nrm[3 * j]), max(fx_field(nrm[3 * j + 1]), fx_field(nrm[3 * j + 2])));
    nexp[j] = f ? f - 1022 : 0;
  }
}

// One output point per thread; the inputs' records are read with warp-uniform
// loads.  With c = (d.g)/r^3, t = (d.g)/r^5, w = d.q + (d.psi)(d.n)/r^2:
//   ds/dq = g/r + c d,  dt/dpsi = a d,  dt/dn = b d,  a = t (d.n),  b = t (d.psi)
//   d(s+t)/dd = g w/r^3 + q c + psi a + n b - d [(g.q)/r^3 + t (3 d.q + 5 (d.psi)(d.n)/r^2)]
// The terms along the own point's vectors only need the sums of their scalars
// (own: q c + psi a + n b source-major, g w/r^3 target-major); the vectors are
// multiplied in once at the end.
//
// Bound: the FP64 pipe, 31 (source-major) and 23 (target-major) instructions of
// about 68 cycles per warp and pair of both layers, where k_adj_fp64, with the
// differences, dot products and the reciprocal square root in FP64 as well,
// takes about 100 and 80.  34,816 points on themselves, both passes: 365 -> 118 ms
// (double layer 235 -> 89, single layer 218 -> 67); 1,088 points 1.86 -> 0.42 ms, with
// splits of at least 32 inputs.  Error against 64 bits (extended precision sums,
// 544 points): at most 6.5e-16 where k_adj_fp64's is 9.6e-16.
template <bool SRC, int KIND>
__global__ void __launch_bounds__(kAdjThreads, 4) k_adj_fx(AdjParams A) {
  constexpr int NA = NAcc<SRC>::value;
  const FxState fs = *A.fx;
  if (!fx_adj_use(fs, A.nout + A.nin)) return;  // k_adj_fp64 does the call
  const int E = fx_exp(fs);
  const int64_t o_sorted = (int64_t)blockIdx.x * kAdjThreads + threadIdx.x;
  if (o_sorted >= A.nout) return;
  const int64_t oc = A.operm[o_sorted];
  const SrcRec64 *orec = reinterpret_cast<const SrcRec64 *>(A.out_rec);
  const SrcRec64 *irec = reinterpret_cast<const SrcRec64 *>(A.in_rec);
  const SrcFx own = A.out_fx[oc];
  const int own_en = SRC && (KIND & K_DL) ? A.nexp[oc] : 0;
  double acc[NA], sum[3] = {0.0, 0.0, 0.0};
#pragma unroll
  for (int i = 0; i < NA; ++i) acc[i] = 0.0;
  const int64_t parts = (int64_t)A.nsplit * A.nsub;
  const int64_t i0 = A.nin * blockIdx.y / parts, i1 = A.nin * (blockIdx.y + 1) / parts;
  for (int64_t k = i0; k < i1; ++k) {
    const int32_t ic = A.iperm[k];
    const SrcFx &in = A.in_fx[ic];
    const SrcFx &T = SRC ? in : own, &S = SRC ? own : in;
    int64_t J[3];
    int32_t dh[3], dl[3];
    int ea, eb, z, z3;
    // dots in units of 2^(e - 60): field 1086 + e - 60
    double dg = 0.0, dp = 0.0, dn = 0.0;
    bool fits = fx_diff(T.y, S.y, T.thr, S.thr, E, J, dh, dl, ea);
    if (fits) {
      const int64_t vg = fx_dot(dh, dl, T.qh, T.ql);
      const int bg = 1026 + T.eq + ea;
      if (!(KIND & K_DL) || !fx_faint(vg)) dg = fx_to_double(vg, bg);
      else fits = fx_faint_dot(vg, J, dh, T.qh, T.ql, fx_is_exact(T.thr, S.thr & ~kFxRoundQ, kFxRoundQ),
                               bg, dg);
      if (KIND & K_DL) {
        const int en = SRC ? own_en : A.nexp[ic];
        const int64_t vp = fx_dot(dh, dl, S.ph, S.pl), vn = fx_dot(dh, dl, S.nh, S.nl);
        const int bp = 1026 + S.epn - en + ea, bn = 1026 + en + ea;
        if (!fx_faint(vp)) dp = fx_to_double(vp, bp);
        else fits = fits && fx_faint_dot(vp, J, dh, S.ph, S.pl, fx_is_exact(T.thr, S.thr, kFxRoundP),
                                         bp, dp);
        if (!fx_faint(vn)) dn = fx_to_double(vn, bn);
        else fits = fits && fx_faint_dot(vn, J, dh, S.nh, S.nl, fx_is_exact(T.thr, S.thr, kFxRoundN),
                                         bn, dn);
      }
    }
    if (!fits) {
      double s[NA];
      for (int i = 0; i < NA; ++i) s[i] = acc[i];
      adj_fx_slow<SRC>(SRC ? irec + ic : orec + oc, SRC ? orec + oc : irec + ic, KIND & K_SL,
                       KIND & K_DL, s);
      for (int i = 0; i < NA; ++i) acc[i] = s[i];
      continue;
    }
    double d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) d[i] = fx_to_double(J[i], 1023 + ea);
    const uint64_t Y = fx_rsqrt(fx_norm2(dh, dl), eb);  // 2^ea / r = Y 2^(eb - 62)
    const uint64_t Z = fx_mul62(Y, Y, z), W = fx_mul62(Z, Y, z3);
    const double i1r = fx_round(Y, 1022 + eb - ea), i2r = fx_round(Z, 1022 + 2 * (eb - ea) - z);
    const double i3r = fx_round(W, 1022 + 3 * (eb - ea) - z - z3);
    const double c = dg * i3r, t = c * i2r;
    double e, cd, a = 0.0, b = 0.0, pd = 0.0;  // cd: the bracket above
    if (KIND & K_DL) {
      a = t * dn;
      b = t * dp;
      pd = dp * dn;
    }
    if (KIND & K_SL) {
      const double dq = fx_to_double(fx_dot(dh, dl, S.qh, S.ql), 1026 + S.eq + ea);
      const double gq = fx_to_double(fx_dot(T.qh, T.ql, S.qh, S.ql), 1026 + T.eq + S.eq);
      const double w = KIND & K_DL ? fx_fma(pd, i2r, dq) : dq;
      e = i3r * w;
      // 3 d.q + 5 (w - d.q)
      const double v = KIND & K_DL ? fx_fma(5.0, w, -2.0 * dq) : 3.0 * dq;
      cd = fx_fma(t, v, i3r * gq);
    } else {
      const double p5 = pd * i2r;
      e = p5 * i3r;
      cd = 5.0 * (t * p5);
    }
    if (SRC) {
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        if (KIND & K_SL) acc[i] = fx_fma(d[i], c, fx_fma(in.q[i], i1r, acc[i]));
        if (KIND & K_DL) {
          acc[3 + i] = fx_fma(d[i], a, acc[3 + i]);
          acc[6 + i] = fx_fma(d[i], b, acc[6 + i]);
        }
        acc[9 + i] = fx_fma(d[i], cd, fx_fma(-in.q[i], e, acc[9 + i]));
      }
      if (KIND & K_SL) sum[0] += c;
      if (KIND & K_DL) {
        sum[1] += a;
        sum[2] += b;
      }
    } else {
      const SrcRec64 &R = irec[ic];
#pragma unroll
      for (int i = 0; i < 3; ++i) {
        acc[i] = fx_fma(-d[i], cd, acc[i]);
        if (KIND & K_SL) acc[i] = fx_fma(in.q[i], c, acc[i]);
        if (KIND & K_DL) acc[i] = fx_fma(R.n[i], b, fx_fma(R.p[i], a, acc[i]));
      }
      sum[0] += e;
    }
  }
  const SrcRec64 &Ro = orec[oc];
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    if (SRC) {
      if (KIND & K_SL) acc[9 + i] = fx_fma(-Ro.q[i], sum[0], acc[9 + i]);
      if (KIND & K_DL)
        acc[9 + i] = fx_fma(-Ro.n[i], sum[2], fx_fma(-Ro.p[i], sum[1], acc[9 + i]));
    } else {
      acc[i] = fx_fma(Ro.q[i], sum[0], acc[i]);
    }
  }
  double *out = A.partial + ((size_t)blockIdx.y * (size_t)A.nout + (size_t)oc) * NA;
#pragma unroll
  for (int i = 0; i < NA; ++i) out[i] = acc[i];
}

// Sums the input splits in order and writes the caller's gradients.
__global__ void k_adj_finish_src(int64_t ns, int32_t nsplit, const double *__restrict__ part,
                                 const double *__restrict__ w, double csl, double cdl,
                                 double *grad_f, double *grad_phi, double *grad_n, double *grad_y) {
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < ns;
       j += (int64_t)gridDim.x * blockDim.x) {
    double a[12] = {0};
    for (int s = 0; s < nsplit; ++s)
      for (int k = 0; k < 12; ++k) a[k] += part[((size_t)s * ns + j) * 12 + k];
    const double wj = w[j];
    for (int k = 0; k < 3; ++k) {
      if (grad_f) grad_f[3 * j + k] = wj * csl * a[k];
      if (grad_phi) grad_phi[3 * j + k] = wj * cdl * a[3 + k];
      if (grad_n) grad_n[3 * j + k] = a[6 + k];
      if (grad_y) grad_y[3 * j + k] = a[9 + k];
    }
  }
}

__global__ void k_adj_finish_trg(int64_t nt, int32_t nsplit, const double *__restrict__ part,
                                 double *grad_x) {
  for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nt;
       i += (int64_t)gridDim.x * blockDim.x) {
    double a[3] = {0, 0, 0};
    for (int s = 0; s < nsplit; ++s)
      for (int k = 0; k < 3; ++k) a[k] += part[((size_t)s * nt + i) * 3 + k];
    for (int k = 0; k < 3; ++k) grad_x[3 * i + k] = a[k];
  }
}

void launch_adj_nexp(int64_t ns, const double *nrm, int32_t *nexp, cudaStream_t st) {
  int64_t g = (ns + 255) / 256;
  if (g > 4096) g = 4096;
  k_adj_nexp<<<(int)(g < 1 ? 1 : g), 256, 0, st>>>(ns, nrm, nexp);
  count_launches(1);
}

template <bool SRC>
static void launch_adj_fx(const AdjParams &A, dim3 grid, cudaStream_t st) {
  if (A.fx) {
    if (!A.has_dl) k_adj_fx<SRC, K_SL><<<grid, kAdjThreads, 0, st>>>(A);
    else if (!A.has_sl) k_adj_fx<SRC, K_DL><<<grid, kAdjThreads, 0, st>>>(A);
    else k_adj_fx<SRC, K_SLDL><<<grid, kAdjThreads, 0, st>>>(A);
    count_launches(1);
  }
  k_adj_fp64<SRC><<<grid, kAdjThreads, 0, st>>>(A);  // with A.fx the device picks one of them
}

template <bool SRC>
static void launch_adj_mixed(const AdjParams &A, dim3 grid, cudaStream_t st) {
  if (!A.has_dl) k_adj_mixed<SRC, K_SL><<<grid, kAdjPack, 0, st>>>(A);
  else if (!A.has_sl) k_adj_mixed<SRC, K_DL><<<grid, kAdjPack, 0, st>>>(A);
  else k_adj_mixed<SRC, K_SLDL><<<grid, kAdjPack, 0, st>>>(A);
}

cudaError_t launch_adjoint(bool mixed, bool src_major, const AdjParams &A, cudaStream_t st) {
  const dim3 grid((unsigned)((A.nout + kAdjThreads - 1) / kAdjThreads),
                  (unsigned)(A.nsplit * A.nsub));
  if (mixed) {
    cudaMemsetAsync(A.near_cnt, 0, sizeof(int32_t) * (size_t)A.nout, st);
    int64_t gn = (A.nout + kAdjThreads - 1) / kAdjThreads;
    if (gn > 65535) gn = 65535;
    if (src_major) {
      launch_adj_mixed<true>(A, grid, st);
      k_adj_near<true><<<(int)gn, kAdjThreads, 0, st>>>(A);
    } else {
      launch_adj_mixed<false>(A, grid, st);
      k_adj_near<false><<<(int)gn, kAdjThreads, 0, st>>>(A);
    }
    count_launches(1);
  } else {
    if (src_major) launch_adj_fx<true>(A, grid, st);
    else launch_adj_fx<false>(A, grid, st);
  }
  count_launches(1);
  return cudaGetLastError();
}

void launch_adj_finish(bool src_major, int64_t n, int32_t nsplit, const double *part,
                       const double *w, double csl, double cdl, double *grad_f, double *grad_phi,
                       double *grad_n, double *grad_y, double *grad_x, cudaStream_t st) {
  const int threads = 256;
  int64_t g = (n + threads - 1) / threads;
  if (g > 4096) g = 4096;
  if (g < 1) g = 1;
  if (src_major)
    k_adj_finish_src<<<(int)g, threads, 0, st>>>(n, nsplit, part, w, csl, cdl, grad_f, grad_phi,
                                                 grad_n, grad_y);
  else
    k_adj_finish_trg<<<(int)g, threads, 0, st>>>(n, nsplit, part, grad_x);
  count_launches(1);
}

}  // namespace stk
