// near.cu -- the near pairs of the mixed-precision sums (Eq. "sl_stokes" and
// the double-layer kernel of Sec. 2.1, summed as in Sec. 3.1).
//
// The mixed engine leaves out of its FP32 sums every candidate pair with
// |r| < alpha h_j, where FP32 cancellation in x - y would dominate the error.
// This kernel adds exactly those pairs back, with the difference x - y and
// 1/|r| in FP64 (near_contrib).  It walks the same work items as the engine
// and takes the same decisions with the same arithmetic (frame_origin,
// local_coord, box_dist2, pair_r2 in common.cuh), so every pair is summed by
// exactly one of the two kernels.
//
// One warp per item, persistent, items in the engine's cost order:
//  1. the item's frame and its targets' local coordinates, as the engine
//     stored them (so the decisions below match the engine's bit for bit);
//  2. the candidate sources the engine listed for the item: each lane takes
//     one, computes its local coordinates and tests it against every target
//     (two per packed FP32 instruction) into a bit mask;
//  3. near pairs go to a queue in shared memory in a fixed order; a full
//     queue is evaluated one pair per lane (the FP64 pipe of GB300 runs at
//     1/64 of the FP32 rate, so it is only ever fed full warps), and the
//     values are added per target in queue order (compensated FP32), which
//     makes the result independent of scheduling;
//  4. the item's sums are added to its targets' partial results.
// The self pair (target and source are the same caller point) contributes
// nothing and is not queued.
//
// An item whose list overflowed (its targets straddle a jump of the Morton
// order, so its box is large) is left to k_near_over: a CTA scans the item's
// sources with the engine's test and each of its warps takes the candidates
// through eight targets of its own.  A pair is added for its target in the
// same order as by one warp for all of them, so the sums are the same; one warp
// took up to 4.7 ms for such an item while the rest of the GPU had finished
// (139,264 x 204,800 points, k_near: 4.73 -> 0.62 ms; 1.50 with the targets split
// over warps that each scan the sources).  The U-list near field's items hold some 60
// targets, four per warp of such a CTA, each of which tests all candidates: where so many of
// its lists overflow that warps with an item each fill the GPU (alpha well above 1),
// k_near_all takes all its items in one launch instead (1,048,928 points, alpha 8: 21.2 ms
// a step with a CTA per item, 14.3 so; alpha 4: 4.93 and 4.14).
#include <climits>

#include "common.cuh"
#include "prep.cuh"

namespace stk {

namespace {

constexpr int kNearWarps = 4;
constexpr int kNearMinBlocks = 8;
constexpr int kNearQueue = 192;  // pairs queued per warp
constexpr int kNearSegWin = 32;  // segments per window

template <int TARGETS>
struct __align__(16) NearSmem {
  float xs[3][TARGETS];     // targets: local coordinates (slots to a multiple of 8; padding
                            //   far away),
  int32_t sid[TARGETS];     //   caller index (self pairs; -1: none)
  float sv[kWarp][3];       // values of one round of evaluations
  float acc[2][3][TARGETS]; // per-target compensated sums (hi, lo)
  int32_t qj[kNearQueue];   // queued pair: source index | kind << 30
  uint8_t qt[kNearQueue];   //   target within the unit
};

// Evaluates the queued pairs, one per lane per round, and adds each value to
// its target's sum; pairs of one target are added in queue order.
template <class Smem>
__device__ void eval_queue(Smem &sm, const EngineParams &P, int32_t t0, int qn, int lane) {
  for (int e0 = 0; e0 < qn; e0 += kWarp) {
    const int e = e0 + lane;
    const bool act = e < qn;
    float v[3] = {0.f, 0.f, 0.f};
    int li = -1 - lane;  // idle lanes get keys of their own
    if (act) {
      li = sm.qt[e];
      const uint32_t jj = (uint32_t)sm.qj[e];
      const int64_t j = jj & 0x3fffffffu;
      const int32_t gi = t0 + li;
      const int64_t ci = P.tperm ? P.tperm[gi] : gi;
      const SrcRec r = P.rec[j];
      if (!near_contrib(P.trg64 + 3 * ci, P.src64 + 3 * j, r.q, r.n, r.p, (int)(jj >> 30), v))
        v[0] = v[1] = v[2] = 0.f;
    }
    sm.sv[lane][0] = v[0];
    sm.sv[lane][1] = v[1];
    sm.sv[lane][2] = v[2];
    const unsigned grp = __match_any_sync(kFull, li);
    __syncwarp();
    if (act && lane == __ffs(grp) - 1) {  // the group's first lane adds its members in order
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        float h = sm.acc[0][k][li], l = sm.acc[1][k][li];
        for (unsigned m = grp; m; m &= m - 1) two_sum_acc(h, l, sm.sv[__ffs(m) - 1][k]);
        sm.acc[0][k][li] = h;
        sm.acc[1][k][li] = l;
      }
    }
    __syncwarp();
  }
}

// Tests up to 32 candidates, one per lane (local coordinates y; hh < 0: none),
// against the unit's tn targets, two per packed FP32 instruction; near pairs are
// queued by candidate (lane), then by target.
template <int TARGETS>
__device__ __forceinline__ void test_candidates(NearSmem<TARGETS> &sm, const EngineParams &P,
                                                int32_t t0, int tn, const float (&y)[3], float hh,
                                                int32_t j, uint32_t kb, int &qn, int lane) {
  constexpr int W = (TARGETS + kWarp - 1) / kWarp;
  const int tn8 = (tn + 7) & ~7;
  // x + (-y) is the IEEE x - y
  const float2 ny0 = make_float2(-y[0], -y[0]), ny1 = make_float2(-y[1], -y[1]),
               ny2 = make_float2(-y[2], -y[2]);
  unsigned mask[W];
#pragma unroll
  for (int w = 0; w < W; ++w) {
    mask[w] = 0u;
    if (w * kWarp < tn) {
#pragma unroll
      for (int i = 0; i < (TARGETS < kWarp ? TARGETS : kWarp); i += 2) {
        const int ti = w * kWarp + i;
        if (ti >= tn8) break;
        const float2 X0 = *reinterpret_cast<const float2 *>(&sm.xs[0][ti]);
        const float2 X1 = *reinterpret_cast<const float2 *>(&sm.xs[1][ti]);
        const float2 X2 = *reinterpret_cast<const float2 *>(&sm.xs[2][ti]);
        const int2 S2 = *reinterpret_cast<const int2 *>(&sm.sid[ti]);
        const float2 d0 = __fadd2_rn(X0, ny0), d1 = __fadd2_rn(X1, ny1), d2 = __fadd2_rn(X2, ny2);
        const float2 r2 = __ffma2_rn(d0, d0, __ffma2_rn(d1, d1, __fmul2_rn(d2, d2)));
        if (is_near(r2.x, hh) && S2.x != j) mask[w] |= 1u << i;
        if (is_near(r2.y, hh) && S2.y != j) mask[w] |= 2u << i;
      }
    }
  }
  int cnt = 0;
#pragma unroll
  for (int w = 0; w < W; ++w) cnt += __popc(mask[w]);
  int incl = cnt;
#pragma unroll
  for (int o = 1; o < kWarp; o <<= 1) {
    const int v = __shfl_up_sync(kFull, incl, o);
    if (lane >= o) incl += v;
  }
  const int total = __shfl_sync(kFull, incl, kWarp - 1);
  if (total == 0) return;
  const int base = incl - cnt;  // this lane's first entry within the round
  const int32_t jq = (int32_t)((uint32_t)j | kb);
  // the round's entries [done, done + room) go to the queue; a full queue is
  // evaluated before the rest
  for (int done = 0;;) {
    const int room = kNearQueue - qn;
    int idx = base;
#pragma unroll
    for (int w = 0; w < W; ++w)
      for (unsigned m = mask[w]; m; m &= m - 1, ++idx)
        if (idx >= done && idx < done + room) {
          const int pos = qn + idx - done;
          sm.qt[pos] = (uint8_t)(w * kWarp + __ffs(m) - 1);
          sm.qj[pos] = jq;
        }
    const int n_emit = min(room, total - done);
    qn += n_emit;
    done += n_emit;
    if (done == total) break;
    __syncwarp();
    eval_queue(sm, P, t0, qn, lane);
    qn = 0;
  }
}

// Targets [t0, t0 + tn) in the local coordinates the engine stored.
template <int TARGETS>
__device__ __forceinline__ void load_targets(NearSmem<TARGETS> &sm, const EngineParams &P,
                                             int32_t t0, int tn, int lane) {
  const int tn8 = (tn + 7) & ~7;
  for (int li = lane; li < tn8; li += kWarp) {
    // slots beyond the targets: padding, never near (|r|^2 = inf)
    float x[3] = {1e30f, 1e30f, 1e30f};
    int32_t self = -1;  // caller index when targets are the sources
    if (li < tn) {
      const int32_t gi = t0 + li;
      if (P.self_index) self = P.tperm ? P.tperm[gi] : gi;
      const float *xl = P.xloc + 3 * (size_t)gi;
#pragma unroll
      for (int k = 0; k < 3; ++k) {
        x[k] = xl[k];
        sm.acc[0][k][li] = sm.acc[1][k][li] = 0.f;
      }
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) sm.xs[k][li] = x[k];
    sm.sid[li] = self;
  }
  __syncwarp();
}

// Evaluates what is queued and adds the near sums to the targets' partial results.
template <int TARGETS>
__device__ __forceinline__ void finish_unit(NearSmem<TARGETS> &sm, const EngineParams &P,
                                            int32_t t0, int tn, int part, int qn, int lane) {
  __syncwarp();
  if (qn) eval_queue(sm, P, t0, qn, lane);
  for (int li = lane; li < tn; li += kWarp) {
    double v[3];
    bool any = false;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      v[k] = (double)sm.acc[0][k][li] + (double)sm.acc[1][k][li];
      any |= sm.acc[0][k][li] != 0.f || sm.acc[1][k][li] != 0.f;
    }
    if (any) {
      double *o = P.part_out + ((size_t)part * (size_t)P.nt + (size_t)(t0 + li)) * 3;
      o[0] += v[0];
      o[1] += v[1];
      o[2] += v[2];
    }
  }
  __syncwarp();
}

// Takes an item's listed candidates through its targets.
__device__ __forceinline__ void test_listed(NearSmem<kItemMax> &sm, const EngineParams &P, int32_t id,
                                            int32_t ncl, int32_t t0, int tn, const float (&oh)[3],
                                            const float (&ol)[3], int &qn, int lane) {
  const int32_t *cl = P.cand_list + (size_t)id * (size_t)P.cand_cap;
  const int n_list = min(ncl, P.cand_cap);
  for (int p0 = 0; p0 < n_list; p0 += kWarp) {
    const int pp = p0 + lane;
    float y[3] = {0.f, 0.f, 0.f}, hh = -1.f;  // hh < 0: idle lane, never near
    int32_t j = -1;
    uint32_t kb = 0;
    if (pp < n_list) {
      const uint32_t e = (uint32_t)cl[pp];
      j = (int32_t)(e & 0x3fffffffu);
      kb = e & 0xc0000000u;
      const float4 yh = __ldg(&P.rec[j].yh);
      y[0] = to_local(yh.x, __ldg(&P.rec[j].q.w), oh[0], ol[0]);
      y[1] = to_local(yh.y, __ldg(&P.rec[j].n.w), oh[1], ol[1]);
      y[2] = to_local(yh.z, __ldg(&P.rec[j].p.w), oh[2], ol[2]);
      hh = yh.w;
    }
    test_candidates(sm, P, t0, tn, y, hh, j, kb, qn, lane);
  }
}

// all_from: from this many overflowed items on, k_near_all takes all items.
__global__ void __launch_bounds__(kNearWarps *kWarp, kNearMinBlocks) k_near(EngineParams P,
                                                                          int all_from) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // k_near_over, as room comes free
  __shared__ NearSmem<kItemMax> smem[kNearWarps];
  NearSmem<kItemMax> &sm = smem[threadIdx.x / kWarp];
  const int lane = threadIdx.x & (kWarp - 1);
  const int n_items = *P.n_items;
  // (the engine stopped early: its lists are incomplete)
  if (*P.err_flag || *P.over_cnt >= all_from) return;
  while (true) {
    int idx = 0;
    if (lane == 0) idx = atomicAdd(P.near_counter, 1);
    idx = __shfl_sync(kFull, idx, 0);
    if (idx >= n_items) break;
    const int32_t id = P.item_order ? P.item_order[idx] : idx;
    const int32_t ncl = P.cand_cnt[id];
    if (ncl < 0) continue;  // overflowed: k_near_over
    const Item it = P.items[id];
    const int tn = it.tn_part & 0xFF;
    const float *fr = P.frames + 12 * (size_t)id;
    float oh[3], ol[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      oh[k] = fr[k];
      ol[k] = fr[3 + k];
    }
    load_targets(sm, P, it.t0, tn, lane);
    int qn = 0;
    test_listed(sm, P, id, ncl, it.t0, tn, oh, ol, qn, lane);
    finish_unit(sm, P, it.t0, tn, it.tn_part >> 8, qn, lane);
  }
}

// The items whose lists overflowed, a CTA at a time: all threads test the item's
// sources as the engine did and keep the candidates in source order; each warp
// then takes them through its own kOverTargets targets.
constexpr int kOverWarps = 16;
constexpr int kOverThreads = kOverWarps * kWarp;
constexpr int kOverTargets = kItemMax / kOverWarps;
constexpr int kOverBuf = 2 * kOverThreads;  // candidates kept between two passes over the targets

struct OverSmem {
  NearSmem<kOverTargets> warp[kOverWarps];
  float4 y[kOverBuf];                // candidates: local coordinates, (alpha h)^2
  int32_t j[kOverBuf];               //   source index | kind << 30
  int32_t seg_start[kNearSegWin];    // window of segments: first source (< 2^30),
  int32_t seg_pre[kNearSegWin];      //   sources before it in the window,
  int32_t seg_kind[kNearSegWin];     //   kind bits
  int32_t wsum[kOverWarps];
  int32_t total, item;
};
static_assert(sizeof(OverSmem) <= 48 * 1024, "no opt-in shared memory");

__global__ void __launch_bounds__(kOverThreads, 2) k_near_over(EngineParams P, int all_from) {
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");  // k_near_all
  // (the engine's results only: complete before k_near began); it ends after k_near
  const int n_over = *P.over_cnt;
  if (n_over == 0 || n_over >= all_from || *P.err_flag) {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    return;
  }
  extern __shared__ __align__(16) unsigned char over_smem[];
  OverSmem &sm = *reinterpret_cast<OverSmem *>(over_smem);
  const int tid = threadIdx.x, lane = tid & (kWarp - 1), wid = tid / kWarp;
  NearSmem<kOverTargets> &ws = sm.warp[wid];
  const unsigned lt = (1u << lane) - 1u;
  while (true) {
    __syncthreads();
    if (tid == 0) sm.item = atomicAdd(P.over_head, 1);
    __syncthreads();
    if (sm.item >= n_over) break;
    const int32_t id = P.over_list[sm.item];
    const Item it = P.items[id];
    const int item_tn = it.tn_part & 0xFF;
    const int ta = item_tn * wid / kOverWarps, tn = item_tn * (wid + 1) / kOverWarps - ta;
    const int32_t t0 = it.t0 + ta;
    const float *fr = P.frames + 12 * (size_t)id;
    float oh[3], ol[3], blo[3], bhi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      oh[k] = fr[k];
      ol[k] = fr[3 + k];
      blo[k] = fr[6 + k];
      bhi[k] = fr[9 + k];
    }
    if (tn > 0) load_targets(ws, P, t0, tn, lane);
    int qn = 0, nc = 0;  // pairs queued by this warp; candidates kept (the same in every thread)
    auto take = [&](int n) {  // the first n kept candidates, by every warp
      __syncthreads();
      if (tn > 0)
        for (int p0 = 0; p0 < n; p0 += kWarp) {
          const int pp = p0 + lane;
          float y[3] = {0.f, 0.f, 0.f}, hh = -1.f;
          uint32_t e = 0xffffffffu;
          if (pp < n) {
            const float4 c = sm.y[pp];
            y[0] = c.x;
            y[1] = c.y;
            y[2] = c.z;
            hh = c.w;
            e = (uint32_t)sm.j[pp];
          }
          test_candidates(ws, P, t0, tn, y, hh, (int32_t)(e & 0x3fffffffu), e & 0xc0000000u, qn,
                          lane);
        }
      __syncthreads();
    };
    for (int32_t w0 = it.seg0; w0 < it.seg1; w0 += kNearSegWin) {
      const int nw = min(kNearSegWin, it.seg1 - w0);
      __syncthreads();
      if (wid == 0) {
        int32_t sz = 0;
        if (lane < nw) {
          const int32_t sid = P.seg_list ? P.seg_list[w0 + lane] : w0 + lane;
          const int64_t a = P.range_ptr[sid];
          sz = (int32_t)(P.range_ptr[sid + 1] - a);
          sm.seg_start[lane] = (int32_t)a;
          sm.seg_kind[lane] = seg_kind(P, sid) << 30;
        }
        int incl = sz;
#pragma unroll
        for (int o = 1; o < kWarp; o <<= 1) {
          const int v = __shfl_up_sync(kFull, incl, o);
          if (lane >= o) incl += v;
        }
        if (lane < nw) sm.seg_pre[lane] = incl - sz;
        if (lane == kWarp - 1) sm.total = incl;
      }
      __syncthreads();
      const int total = sm.total;
      for (int p0 = 0; p0 < total; p0 += kOverThreads) {
        const int pp = p0 + tid;
        bool cand = false;
        float4 c = make_float4(0.f, 0.f, 0.f, 0.f);
        uint32_t je = 0;
        if (pp < total) {
          int e = 0;  // last segment starting at or before pp
#pragma unroll
          for (int step = kNearSegWin / 2; step > 0; step >>= 1)
            if (e + step < nw && sm.seg_pre[e + step] <= pp) e += step;
          const int32_t j = sm.seg_start[e] + (pp - sm.seg_pre[e]);
          const SrcRec *r = P.rec + j;
          const float4 yh = __ldg(&r->yh);
          c = make_float4(to_local(yh.x, __ldg(&r->q.w), oh[0], ol[0]),
                          to_local(yh.y, __ldg(&r->n.w), oh[1], ol[1]),
                          to_local(yh.z, __ldg(&r->p.w), oh[2], ol[2]), yh.w);
          cand = is_candidate(box_dist2(c.x, c.y, c.z, blo, bhi), c.w);
          je = (uint32_t)j | (uint32_t)sm.seg_kind[e];
        }
        const unsigned b = __ballot_sync(kFull, cand);
        if (lane == 0) sm.wsum[wid] = __popc(b);
        __syncthreads();
        int before = 0, all = 0;
#pragma unroll
        for (int w = 0; w < kOverWarps; ++w) {
          before += w < wid ? sm.wsum[w] : 0;
          all += sm.wsum[w];
        }
        if (cand) {
          const int o = nc + before + __popc(b & lt);
          sm.y[o] = c;
          sm.j[o] = (int32_t)je;
        }
        nc += all;
        if (nc > kOverBuf - kOverThreads) {
          take(nc);
          nc = 0;
        } else {
          __syncthreads();  // wsum is read before the next round writes it
        }
      }
    }
    if (nc) take(nc);
    if (tn > 0) finish_unit(ws, P, t0, tn, it.tn_part >> 8, qn, lane);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

// All items where many lists overflowed, an item per warp: the warp tests an overflowed item's
// sources 32 at a time, first conservatively on the 16-byte position record; each candidate is
// broadcast and every lane tests its targets.  (Taking these candidates through bit masks costs
// more: most of a candidate's targets are near and would fill the queue several times.)
constexpr int kScanT = kItemMax / kWarp;  // targets per lane
constexpr int kScanMinBlocks = 8;

struct ScanSmem {
  NearSmem<kItemMax> n;
  int32_t seg_start[kNearSegWin];    // window of segments, as in OverSmem
  int32_t seg_pre[kNearSegWin];
  int32_t seg_kind[kNearSegWin];
};

__global__ void __launch_bounds__(kNearWarps *kWarp, kScanMinBlocks) k_near_all(EngineParams P,
                                                                                int all_from) {
  __shared__ ScanSmem smem[kNearWarps];
  const bool mine = *P.over_cnt >= all_from && !*P.err_flag;
  ScanSmem &sm = smem[threadIdx.x / kWarp];
  const int lane = threadIdx.x & (kWarp - 1);
  const unsigned lt = (1u << lane) - 1u;
  const int n_items = *P.n_items;
  while (mine) {
    int idx = 0;
    if (lane == 0) idx = atomicAdd(P.over_head, 1);
    idx = __shfl_sync(kFull, idx, 0);
    if (idx >= n_items) break;
    const int32_t id = P.item_order ? P.item_order[idx] : idx;
    const int32_t ncl = P.cand_cnt[id];
    const Item it = P.items[id];
    const int tn = it.tn_part & 0xFF;
    const float *fr = P.frames + 12 * (size_t)id;
    float oh[3], ol[3], blo[3], bhi[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      oh[k] = fr[k];
      ol[k] = fr[3 + k];
      blo[k] = fr[6 + k];
      bhi[k] = fr[9 + k];
    }
    const float tol0 = 4.8e-7f * (fabsf(oh[0]) + fabsf(oh[1]) + fabsf(oh[2]));
    load_targets(sm.n, P, it.t0, tn, lane);
    int qn = 0;
    if (ncl >= 0) {
      test_listed(sm.n, P, id, ncl, it.t0, tn, oh, ol, qn, lane);
      finish_unit(sm.n, P, it.t0, tn, it.tn_part >> 8, qn, lane);
      continue;
    }
    float x[kScanT][3];
    int32_t self[kScanT];
#pragma unroll
    for (int t = 0; t < kScanT; ++t) {
      const int li = lane + kWarp * t;
      self[t] = li < tn ? sm.n.sid[li] : -1;
#pragma unroll
      for (int k = 0; k < 3; ++k) x[t][k] = li < tn ? sm.n.xs[k][li] : 1e30f;
    }
    for (int32_t w0 = it.seg0; w0 < it.seg1; w0 += kNearSegWin) {
      const int nw = min(kNearSegWin, it.seg1 - w0);
      __syncwarp();
      int32_t sz = 0;
      if (lane < nw) {
        const int32_t sid = P.seg_list ? P.seg_list[w0 + lane] : w0 + lane;
        const int64_t a = P.range_ptr[sid];
        sz = (int32_t)(P.range_ptr[sid + 1] - a);
        sm.seg_start[lane] = (int32_t)a;
        sm.seg_kind[lane] = seg_kind(P, sid) << 30;
      }
      int incl = sz;
#pragma unroll
      for (int o = 1; o < kWarp; o <<= 1) {
        const int v = __shfl_up_sync(kFull, incl, o);
        if (lane >= o) incl += v;
      }
      if (lane < nw) sm.seg_pre[lane] = incl - sz;
      const int total = __shfl_sync(kFull, incl, kWarp - 1);
      __syncwarp();
      for (int p0 = 0; p0 < total; p0 += kWarp) {
        const int pp = p0 + lane;
        bool cand = false;
        int32_t j = 0;
        uint32_t kb = 0;
        float y[3] = {0.f, 0.f, 0.f}, hh = 0.f;
        if (pp < total) {
          int e = 0;  // last segment starting at or before pp
#pragma unroll
          for (int step = kNearSegWin / 2; step > 0; step >>= 1)
            if (e + step < nw && sm.seg_pre[e + step] <= pp) e += step;
          j = sm.seg_start[e] + (pp - sm.seg_pre[e]);
          kb = (uint32_t)sm.seg_kind[e];
          const SrcRec *r = P.rec + j;
          const float4 yh = __ldg(&r->yh);
          hh = yh.w;
          // yh - oh differs from the local coordinate by less than tol (the dropped low parts
          // and one rounding each)
          const float tol = fmaf(4.8e-7f, fabsf(yh.x) + fabsf(yh.y) + fabsf(yh.z), tol0) + 1e-30f;
          const float lo2[3] = {blo[0] - tol, blo[1] - tol, blo[2] - tol};
          const float hi2[3] = {bhi[0] + tol, bhi[1] + tol, bhi[2] + tol};
          if (box_dist2(yh.x - oh[0], yh.y - oh[1], yh.z - oh[2], lo2, hi2) <
              hh * 1.0001f + 1e-30f) {
            y[0] = to_local(yh.x, __ldg(&r->q.w), oh[0], ol[0]);
            y[1] = to_local(yh.y, __ldg(&r->n.w), oh[1], ol[1]);
            y[2] = to_local(yh.z, __ldg(&r->p.w), oh[2], ol[2]);
            cand = is_candidate(box_dist2(y[0], y[1], y[2], blo, bhi), hh);
          }
        }
        for (unsigned cm = __ballot_sync(kFull, cand); cm; cm &= cm - 1) {
          const int l = __ffs(cm) - 1;
          const float y0 = __shfl_sync(kFull, y[0], l), y1 = __shfl_sync(kFull, y[1], l),
                      y2 = __shfl_sync(kFull, y[2], l), h2 = __shfl_sync(kFull, hh, l);
          const int32_t jl = __shfl_sync(kFull, j, l);
          const uint32_t kl = __shfl_sync(kFull, kb, l);
          unsigned nm = 0;  // this lane's near targets
#pragma unroll
          for (int t = 0; t < kScanT; ++t)
            if (t * kWarp < tn) {
              const float r2 =
                  pair_r2(__fsub_rn(x[t][0], y0), __fsub_rn(x[t][1], y1), __fsub_rn(x[t][2], y2));
              if (is_near(r2, h2) && self[t] != jl) nm |= 1u << t;
            }
          if (!__any_sync(kFull, nm != 0)) continue;
          // queue order: by lane, then by target slot
          const int cnt = __popc(nm);
          const unsigned b0 = __ballot_sync(kFull, cnt & 1), b1 = __ballot_sync(kFull, cnt & 2),
                         b2 = __ballot_sync(kFull, cnt & 4);
          int pos = qn + __popc(b0 & lt) + 2 * __popc(b1 & lt) + 4 * __popc(b2 & lt);
          for (unsigned mm = nm; mm; mm &= mm - 1, ++pos) {
            sm.n.qt[pos] = (uint8_t)(lane + kWarp * (__ffs(mm) - 1));
            sm.n.qj[pos] = (int32_t)((uint32_t)jl | kl);
          }
          qn += __popc(b0) + 2 * __popc(b1) + 4 * __popc(b2);
          if (qn > kNearQueue - kScanT * kWarp) {
            __syncwarp();
            eval_queue(sm.n, P, it.t0, qn, lane);
            qn = 0;
          }
        }
      }
    }
    finish_unit(sm.n, P, it.t0, tn, it.tn_part >> 8, qn, lane);
  }
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

}  // namespace

// Overflowed items of the U-list near field from which on a warp each (k_near_all) beats a
// CTA each: as many as its resident warps.  262,096 points, some 4,100 overflowed items at
// alpha 8: 5.5 ms a step with a CTA each, 7.4 with a warp; 524,000 points, 8,300: 8.1 with a
// warp.  Items of direct sums and batches hold 64 to 128 targets, and a CTA each stays the
// better form (64 suspensions, alpha 8: 37.6 ms, 38.4 with a warp each).
constexpr int kAllItems = 4864;

// Runs after the engine on the same stream; P is the engine's parameter block
// (items, segments, records, partial results) and P.near_counter is zeroed.
void launch_near(const EngineParams &P, int sms, int64_t max_items, cudaStream_t st) {
  int64_t grid = (int64_t)sms * kNearMinBlocks;
  const int64_t need = (max_items + kNearWarps - 1) / kNearWarps;
  if (grid > need) grid = need;
  if (grid < 1) grid = 1;
  const bool all = P.seg_list && max_items >= kAllItems;
  const int all_from = all ? kAllItems : INT_MAX;
  k_near<<<(int)grid, kNearWarps * kWarp, 0, st>>>(P, all_from);
  // k_near_over reads and adds to nothing of k_near's: it starts as that one's CTAs end
  // (2 to 6 us of a call when no list has overflowed); k_near_all likewise
  cudaLaunchAttribute early;
  early.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  early.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(2 * sms));
  cfg.blockDim = dim3(kOverThreads);
  cfg.dynamicSmemBytes = sizeof(OverSmem);
  cfg.stream = st;
  cfg.attrs = &early;
  cfg.numAttrs = 1;
  cudaLaunchKernelEx(&cfg, k_near_over, P, all_from);
  count_launches(2);
  if (!all) return;
  cfg.gridDim = dim3((unsigned)grid);
  cfg.blockDim = dim3(kNearWarps * kWarp);
  cfg.dynamicSmemBytes = 0;
  cudaLaunchKernelEx(&cfg, k_near_all, P, all_from);
  count_launches(1);
}

}  // namespace stk
