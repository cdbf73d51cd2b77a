// Tessellation under grid-host aggregation: counts and offsets, then points.
#pragma once
#include "np_engine.h"

namespace nestpar {

// The output offsets number the points of all curves, so under grid-host
// aggregation (serial children spread) they are all that disaggregation needs:
// no records, no block offsets, and no difference in where a point runs between
// curves above and below the threshold (np_stats reports them as the form
// defines them).
//
//   bezier_count   parents: one thread per curve counts its points, a CTA scans
//                  its tile of kPointTile curves and leaves one word per curve
//                  (offset in the tile << 12 | N - 1) and the tile's sums.
//   bezier_points  children: one warp per curve, point j on lane j % 32, each
//                  store of a warp 256 consecutive bytes; neighbouring warps
//                  take neighbouring curves, so the grid writes one moving
//                  window of the output.
//
// What bounds them: the count pass its fixed chain (control points, the exact
// integer count, two scans), the point pass stores and instruction issue. No
// CTA waits for another one's offsets: with both in one kernel each group of
// tiles waited for its look-back before it could store its first point, and a
// CTA held 450-500 curves, too coarse to fill 152 SMs. Measured, one pass of
// random curves (6.2 M and 25 M points, threshold 32 and none): 43.9 -> 15.1 us
// and 64.8 -> 43.2 us; the point grid alone takes 35 us for 25 M points (200 MB
// of stores, 30 us at the copy bandwidth; 68% of the issue slots).
static_assert(kPointBlock % (kPointBlock / 32 * kPointCurves) == 0, "a point CTA's curves lie in one count tile");
constexpr int kPointTile = kPointBlock;   // N <= 4096: an offset in the tile takes 20 bits

// Per tile: a.lb_agg (points, serialised curves, launching curves, their
// points), a.ob_agg (their coarsened blocks, curves). Up to kPointScanTiles tiles
// the point grid's CTAs sum the tiles before theirs themselves, and one CTA
// more takes the statistics; beyond that (a.k set) the count CTA that finishes
// last scans the tiles, a chain of its own (a fence, an atomic and two round
// trips, 3 us) that a small tessellation would wait for. (At 1024 tiles the two
// cost the same: 12.6 + 34.4 us with the scan, 8.2 + 38.9 us without; at 256
// tiles a pass takes 18.4 and 16.5 us.)

// np_stats and the total from what the threads of one CTA counted.
__device__ __forceinline__ void point_stats(const Args& a, unsigned items, unsigned serial, unsigned launched,
                                            unsigned citems, unsigned cblocks, unsigned curves,
                                            unsigned long long total) {
  __shared__ unsigned s_sum[6];
  const int tid = (int)threadIdx.x;
  if (tid < 6) s_sum[tid] = 0u;
  __syncthreads();
  const unsigned v[6] = {items, serial, launched, citems, cblocks, curves};
#pragma unroll
  for (int k = 0; k < 6; k++) {
    const unsigned x = __reduce_add_sync(kFull, v[k]);
    if ((tid & 31) == 0) atomicAdd(&s_sum[k], x);
  }
  __syncthreads();
  if (tid == 0) {
    LevelState* st = a.st;
    for (int k = 0; k < S_N; k++) st->s[k] = 0ull;
    st->s[S_ITEMS] = s_sum[0];
    st->s[S_SERIAL] = s_sum[1];
    st->s[S_LAUNCHP] = s_sum[2];
    st->s[S_CITEMS] = s_sum[3];
    st->s[S_CBLOCKS] = s_sum[4];
    st->s[S_PARENTS] = s_sum[5];
    st->body_iters = 0;
    if ((long long)total > a.cap) st->error |= kErrCapacity;
    a.offsets[a.count_fixed] = (int)min(total, (unsigned long long)INT_MAX);
  }
}

// Statistics and the total from the tiles' sums, by one CTA of kPointTile
// threads; with `scan` the tiles' exclusive prefixes go to a.lb_incl as words
// (at most kPointTop, beyond INT_MAX: nothing fits there, and the offset in the
// tile can be added without wrapping).
constexpr unsigned kPointTop = 0xfff00000u;
__device__ __forceinline__ void point_totals(const Args& a, int ntiles, bool scan) {
  __shared__ uint2 s_scan2[33];
  const int tid = (int)threadIdx.x, count = a.count_fixed;
  const int T = a.threshold < 1 ? 1 : a.threshold;
  const bool never = a.threshold == INT_MAX;
  const int per = ceil_div(ntiles, kPointTile), t0 = min(tid * per, ntiles), t1 = min(t0 + per, ntiles);
  // (the counters fit in 32 bits where all points fit; else they are taken again below)
  unsigned items = 0, serial = 0, launched = 0, citems = 0, cblocks = 0, curves = 0;
  unsigned long long mine = 0;   // points of this thread's tiles: below 2^15 tiles of at most 2^20
#pragma unroll 1
  for (int t = t0; t < t1; t++) {
    const uint4 v = __ldcg(&a.lb_agg[t]), x = __ldcg(&a.ob_agg[t]);
    mine += v.x;
    serial += v.y;
    launched += v.z;
    citems += v.w;
    cblocks += x.x;
    curves += x.y;
  }
  items = (unsigned)mine;
  // a 64-bit scan of sums below 2^36 as two counters: the low 24 bits and the rest
  unsigned e0, e1, lo, hi;
  block_scan2((unsigned)mine & 0xffffffu, (unsigned)(mine >> 24), e0, e1, lo, hi, s_scan2);
  const unsigned long long first = ((unsigned long long)e1 << 24) + e0, total = ((unsigned long long)hi << 24) + lo;
  if (scan) {
    unsigned* prefix = reinterpret_cast<unsigned*>(a.lb_incl);
    unsigned long long at = first;
    for (int t = t0; t < t1; t++) {
      prefix[t] = (unsigned)min(at, (unsigned long long)kPointTop);
      at += __ldcg(&a.lb_agg[t]).x;
    }
  }
  if ((long long)total > a.cap) {
    // curves that do not fit have no children: count those that do (thread by
    // thread over its tiles' curves)
    items = serial = launched = citems = cblocks = 0;
    unsigned long long at = first;
#pragma unroll 1
    for (int t = t0; t < t1; t++) {
#pragma unroll 1
      for (int i = t * kPointTile; i < min(count, (t + 1) * kPointTile); i++) {
        const unsigned w = (unsigned)__ldcg(&a.boff[i]);
        const int N = (w & 4095u) ? (int)(w & 4095u) + 1 : 0;
        if (N == 0 || (long long)(at + (w >> 12)) + N > a.cap) continue;
        items += (unsigned)N;
        if (!never && N >= T) {
          launched++;
          citems += (unsigned)N;
          cblocks += (unsigned)ceil_div(ceil_div(N, a.child_block), a.cfactor);
        } else {
          serial++;
        }
      }
      at += __ldcg(&a.lb_agg[t]).x;
    }
  }
  point_stats(a, items, serial, launched, citems, cblocks, curves, total);
}

__global__ void __launch_bounds__(kPointTile, 4) bezier_count(Args a) {
  NP_PDL_ENTRY();
  __shared__ uint4 s_scan[33];
  __shared__ int s_last;
  const int tid = (int)threadIdx.x, count = a.count_fixed;
  const int ntiles = ceil_div(count, kPointTile);
  const int T = a.threshold < 1 ? 1 : a.threshold;
  const bool never = a.threshold == INT_MAX;   // (launches nothing, whatever N)
#pragma unroll 1
  for (int tile = (int)blockIdx.x; tile < ntiles; tile += (int)gridDim.x) {
    const int i = tile * kPointTile + tid;
    int pid = -1, base = 0, N = 0;
    if (i < count) pid = a.ids ? __ldcg(&a.ids[i]) : i;
    const bool valid = pid >= 0;
    if (valid) BezierBody::count(a, pid, base, N);
    const bool launch = valid && !never && N >= T;
    const unsigned cg = launch ? (unsigned)ceil_div(ceil_div(N, a.child_block), a.cfactor) : 0u;
    // points, launching curves and their points; curves and coarsened blocks
    uint4 ex, tot;
    block_scan4(make_uint4((unsigned)N, launch ? 1u : 0u, launch ? (unsigned)N : 0u, cg), ex, tot, s_scan);
    const int curves = __syncthreads_count(valid);
    if (i < count) a.boff[i] = (int)(ex.x << 12 | (unsigned)(N > 0 ? N - 1 : 0));
    if (tid == 0) {
      a.lb_agg[tile] = make_uint4(tot.x, (unsigned)curves - tot.y, tot.y, tot.z);
      a.ob_agg[tile] = make_uint4(tot.w, (unsigned)curves, 0u, 0u);
    }
  }
  if (!a.k) return;
  __threadfence();
  __syncthreads();
  if (tid == 0) s_last = atomicAdd(a.grp_ctr, 1) == (int)gridDim.x - 1;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  point_totals(a, ntiles, true);
  if (tid == 0) *a.grp_ctr = 0;
}

// A curve's points as integer-weighted sums: with r = 1 / (N - 1)^2, point j is
//   k^2 (r P0) + j k (2 r P1) + j^2 (r P2),  k = N - 1 - j,
// whose weights are exact in FP32 ((N - 1)^2 < 2^24). A warp prepares
// kPointCurves curves at once, one per lane (offset, N, the six products), and
// then runs them one after the other from shuffles: 17 instructions per 32
// points and 14 per curve.
//
// The products keep their 24 bits only while they are normal numbers (r is at
// least 2^-24): a curve with a coordinate below 2^-100 in magnitude, other than
// 0, takes the child body's own form instead, whose weights carry r and whose
// coordinates are not scaled. (Scaled all the same, coordinates of 1e-36 came
// out with a relative error of 1.2e-2 at N = 4096; the test takes 1 us of the
// point grid's 35 for 25 M points, weights that carry r in every curve 2.8.)
//
// Lane l holds curve `i` = its warp's curve l % kPointCurves: id `pid` (-1: none),
// offset and number of points.
__device__ __forceinline__ void point_curves(const Args& a, int i, int pid, unsigned base, int N) {
  const int lane = (int)threadIdx.x & 31;
  float ax = 0.f, ay = 0.f, bx = 0.f, by = 0.f, cx = 0.f, cy = 0.f;
  bool low = false;
  if (pid >= 0) {
    const float* c = a.b.ctrl + 6 * (size_t)pid;
    const float nm1 = (float)(N - 1), r = 1.0f / (nm1 * nm1), r2 = 2.0f * r;
    ax = __ldg(c);
    ay = __ldg(c + 1);
    bx = __ldg(c + 2);
    by = __ldg(c + 3);
    cx = __ldg(c + 4);
    cy = __ldg(c + 5);
    low = fminf(fminf(fminf(fabsf(ax), fabsf(ay)), fminf(fabsf(bx), fabsf(by))), fminf(fabsf(cx), fabsf(cy))) < 0x1p-100f;
    ax *= r;
    ay *= r;
    bx *= r2;
    by *= r2;
    cx *= r;
    cy *= r;
    if (lane < kPointCurves) a.offsets[i] = offset_word(base);
  }
  // (none, or it does not fit: skipped; the capacity is at most INT_MAX)
  if (pid < 0 || offset_word(base) > (int)a.cap - N) N = 0;
  auto scaled = [&](int q) {
    const int n = __shfl_sync(kFull, N, q);
    float2* out = a.b.points + __shfl_sync(kFull, base, q) + lane;
    const float x0 = __shfl_sync(kFull, ax, q), y0 = __shfl_sync(kFull, ay, q), x1 = __shfl_sync(kFull, bx, q),
                y1 = __shfl_sync(kFull, by, q), x2 = __shfl_sync(kFull, cx, q), y2 = __shfl_sync(kFull, cy, q);
    float j = (float)lane, k = (float)(n - 1 - lane);
    for (int left = n - lane; left > 0; left -= 32) {
      const float w0 = k * k, w1 = j * k, w2 = j * j;
      *out = make_float2(w0 * x0 + w1 * x1 + w2 * x2, w0 * y0 + w1 * y1 + w2 * y2);
      out += 32;
      j += 32.0f;
      k -= 32.0f;
    }
  };
  if (!__any_sync(kFull, low)) {
    for (int q = 0; q < kPointCurves; q++) scaled(q);
    return;
  }
  // (a zero stays a zero: no reason by itself)
  bool tiny = false;
  if (low)
    for (int k = 0; k < 6; k++) {
      const float x = fabsf(__ldg(a.b.ctrl + 6 * (size_t)pid + k));
      tiny = tiny || (x > 0.0f && x < 0x1p-100f);
    }
  const unsigned apart = __ballot_sync(kFull, tiny);
#pragma unroll 1
  for (int q = 0; q < kPointCurves; q++) {
    if (!(apart >> q & 1u)) {   // (uniform)
      scaled(q);
      continue;
    }
    const int n = __shfl_sync(kFull, N, q);
    const BezierBody::P p[1] = {
        BezierBody::parent(a.b, __shfl_sync(kFull, pid, q), (int)__shfl_sync(kFull, base, q), n)};
    for (int j = lane; j < n; j += 32) {
      const int idx[1] = {j};
      const BezierBody::F f[1] = {};
      const bool v[1] = {true};
      bool push[1];
      int next[1];
      BezierBody::apply_batch<1>(a.b, p, idx, f, v, push, next);
    }
  }
}

__global__ void __launch_bounds__(256, 6) bezier_points(Args a) {
  NP_PDL_ENTRY();
  const int lane = (int)threadIdx.x & 31;
  const int count = a.count_fixed;
  const int tile = (int)((long long)blockIdx.x * (blockDim.x >> 5) * kPointCurves / kPointTile);   // of all its curves
  const int ntiles = ceil_div(count, kPointTile);
  if (tile >= ntiles) {   // (the one CTA beyond the curves)
    point_totals(a, ntiles, false);
    return;
  }
  // the points before this CTA's tile
  unsigned before = 0;
  if (a.k) {
    before = __ldcg(&reinterpret_cast<const unsigned*>(a.lb_incl)[tile]);
  } else {
    __shared__ unsigned s_part[8];
    for (int t = (int)threadIdx.x; t < tile; t += (int)blockDim.x) before += __ldcg(&a.lb_agg[t].x);
    before = __reduce_add_sync(kFull, before);
    if (lane == 0) s_part[threadIdx.x >> 5] = before;
    __syncthreads();
    before = 0;
#pragma unroll
    for (int k = 0; k < 8; k++) before += s_part[k];
  }
  const int first = ((int)blockIdx.x * ((int)blockDim.x >> 5) + ((int)threadIdx.x >> 5)) * kPointCurves;
  const int i = first + (lane & (kPointCurves - 1));
  unsigned base = 0;
  int N = 0, pid = -1;
  if (i < count) {
    const unsigned w = (unsigned)__ldcg(&a.boff[i]);
    pid = a.ids ? __ldcg(&a.ids[i]) : i;
    base = before + (w >> 12);   // (at most 2^31 or so, or kPointTop and a tile: no wrap)
    N = (int)(w & 4095u) + 1;
  }
  point_curves(a, i, pid, base, N);
}

// Up to kPointFused curves: one grid in place of the two. Each CTA counts the
// curves before its own itself (two a thread at 512), and so does the CTA for
// the totals. What bounds it is the launch and one chain of control points,
// counts and stores. Passes of 1, 64 and 300 curves one after the other: 2.5,
// 3.6 and 4.3 us on the device (4.2, 5.2 and 5.6 with two grids), 4.7 us a call
// on the host (6.1); at 1000 curves the two take the same, at 2048 one takes
// 8.2 us and two 6.0.
__global__ void __launch_bounds__(kPointBlock, 4) bezier_fused(Args a) {
  NP_PDL_ENTRY();
  const int tid = (int)threadIdx.x, lane = tid & 31, wid = tid >> 5;
  const int count = a.count_fixed;
  const int c0 = (int)blockIdx.x * (kPointBlock / 32 * kPointCurves);   // the CTA's first curve
  auto points_of = [&](int i, int& pid) {
    int base = 0, N = 0;
    pid = a.ids ? __ldcg(&a.ids[i]) : i;
    if (pid >= 0) BezierBody::count(a, pid, base, N);
    return N;
  };
  if (c0 >= count) {   // (the one CTA beyond the curves)
    __shared__ uint2 s_scan2[33];
    const int T = a.threshold < 1 ? 1 : a.threshold;
    unsigned items = 0, serial = 0, launched = 0, citems = 0, cblocks = 0, curves = 0;
    auto tally = [&](int i, long long& at, long long cap) {
      int pid;
      const int N = points_of(i, pid);
      if (pid < 0) return;
      curves++;
      at += N;
      if (at > cap) return;   // (does not fit: no children)
      items += (unsigned)N;
      if (a.threshold != INT_MAX && N >= T) {
        launched++;
        citems += (unsigned)N;
        cblocks += (unsigned)ceil_div(ceil_div(N, a.child_block), a.cfactor);
      } else {
        serial++;
      }
    };
    long long at = 0;
#pragma unroll 4
    for (int i = tid; i < count; i += kPointBlock) tally(i, at, LLONG_MAX);
    unsigned e0, e1, total, u1;
    block_scan2(items, 0u, e0, e1, total, u1, s_scan2);
    if ((long long)total > a.cap) {
      // again, in order: a run of curves per thread
      const int per = ceil_div(count, kPointBlock), i0 = min(tid * per, count), i1 = min(i0 + per, count);
      unsigned run = 0;
      int pid;
#pragma unroll 1
      for (int i = i0; i < i1; i++) run += (unsigned)points_of(i, pid);
      unsigned t1;
      __syncthreads();
      block_scan2(run, 0u, e0, e1, t1, u1, s_scan2);
      items = serial = launched = citems = cblocks = curves = 0;
      at = e0;
#pragma unroll 1
      for (int i = i0; i < i1; i++) tally(i, at, a.cap);
    }
    point_stats(a, items, serial, launched, citems, cblocks, curves, total);
    return;
  }
  unsigned before = 0;
  int pid = -1;
#pragma unroll 4
  for (int i = tid; i < c0; i += kPointBlock) before += (unsigned)points_of(i, pid);
  before = __reduce_add_sync(kFull, before);
  const int i = c0 + wid * kPointCurves + (lane & (kPointCurves - 1));
  pid = -1;
  const int N = i < count ? points_of(i, pid) : 0;
  int incl = N;
#pragma unroll
  for (int d = 1; d < kPointCurves; d *= 2) {
    const int o = __shfl_up_sync(kFull, incl, d, kPointCurves);
    if ((lane & (kPointCurves - 1)) >= d) incl += o;
  }
  __shared__ unsigned s_before[kPointBlock / 32], s_own[kPointBlock / 32];
  if (lane == kPointCurves - 1) {
    s_before[wid] = before;
    s_own[wid] = (unsigned)incl;
  }
  __syncthreads();
  unsigned base = (unsigned)(incl - N);
#pragma unroll
  for (int k = 0; k < kPointBlock / 32; k++) base += s_before[k] + (k < wid ? s_own[k] : 0u);
  point_curves(a, i, pid, base, N);
}

}  // namespace nestpar
