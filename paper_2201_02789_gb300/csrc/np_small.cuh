// The loops that run small levels whole: SSSP in a cluster, with a distance
// window; BFS from its start in one CTA, with its visited set in shared memory.
#pragma once
#include "np_loop.cuh"

namespace nestpar {

// ------------------------------------------------------- thread-block clusters

__device__ __forceinline__ unsigned cluster_rank() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_ctarank;" : "=r"(r));
  return r;
}
__device__ __forceinline__ unsigned cluster_size() {
  unsigned r;
  asm volatile("mov.u32 %0, %%cluster_nctarank;" : "=r"(r));
  return r;
}
// All threads of all CTAs of the cluster (a hardware barrier: the CTAs of a
// cluster are resident together); what was written before it, in shared or
// global memory, is visible after it.
__device__ __forceinline__ void cluster_barrier() {
  asm volatile("barrier.cluster.arrive.release.aligned;\n barrier.cluster.wait.acquire.aligned;" ::: "memory");
}
// Address of this CTA's shared variable in CTA `rank` of the cluster.
__device__ __forceinline__ unsigned cluster_addr(const void* p, unsigned rank) {
  unsigned a;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(smem_u32(p)), "r"(rank));
  return a;
}
__device__ __forceinline__ int cluster_ld(unsigned addr) {
  int v;
  asm volatile("ld.shared::cluster.u32 %0, [%1];" : "=r"(v) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ int4 cluster_ld4(unsigned addr) {
  int4 v;
  asm volatile("ld.shared::cluster.v4.u32 {%0, %1, %2, %3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w)
               : "r"(addr)
               : "memory");
  return v;
}
__device__ __forceinline__ void cluster_st4(unsigned addr, int4 v) {
  asm volatile("st.shared::cluster.v4.u32 [%0], {%1, %2, %3, %4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w)
               : "memory");
}

// Positions for the lanes with `take` from one shared counter, one atomic per warp.
__device__ __forceinline__ int warp_slots(bool take, int* counter) {
  const unsigned m = __ballot_sync(kFull, take);
  int base = 0;
  if (m != 0u && (threadIdx.x & 31) == 0) base = atomicAdd(counter, __popc(m));
  return __shfl_sync(kFull, base, 0) + __popc(m & lanemask_lt());
}

// The segments of 32 consecutive items t .. t + 31, one per lane: seg[j].x is
// the first item of segment j, strictly increasing, seg[0].x <= t. A 32-ary
// search finds the segment of item t; no more than 32 segments start among the
// 32 items, so one probe per lane and a ballot-like mask of the starts give
// the others.
__device__ __forceinline__ int warp_segment(const int4* seg, int n, int t) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = n;
  while (hi - lo > 32) {
    const int stride = (hi - lo + 31) >> 5, i = lo + lane * stride;
    const bool p = i < hi && seg[i].x <= t;
    lo += (__popc(__ballot_sync(kFull, p)) - 1) * stride;
    hi = min(hi, lo + stride);
  }
  const int i = lo + lane;
  const bool p = i < hi && seg[i].x <= t;
  const int r = lo + __popc(__ballot_sync(kFull, p)) - 1, j = r + 1 + lane;
  const int at = j < n ? seg[j].x - t : 32;
  return r + __popc(__reduce_or_sync(kFull, at < 32 ? 1u << at : 0u) & (0xffffffffu >> (31 - lane)));
}

// ------------------------------------------------- small-level loop, SSSP form
//
// One cluster of up to 16 CTAs runs whole rounds of the packed SSSP while the
// frontier stays small, and on top of it defers work. Plain frontier
// Bellman-Ford relaxes every vertex lowered in a round at once; on a graph of
// large diameter (a road network) that expands each vertex over a hundred
// times, because far vertices are expanded from distances that nearer ones
// still lower. Here a round expands only the pending vertices with a distance
// of at most `cut`; the others wait in far lists in shared memory. The final
// distances are the same (a vertex is expanded again whenever its distance has
// fallen since, as in the near-far form of delta-stepping, Davidson, Baxter,
// Garland and Owens, IPDPS 2014), the work is not: on a 514 x 514 grid 7 M
// relaxations in 918 rounds instead of 215 M in 899 levels, 4.3 ms instead of 13.3.
//
// What bounds a round is its chain of dependent round trips to L2 (distance
// and row bounds of the parents, then edges, then the reductions) as long as
// no SM has more than a few hundred items: one CTA alone took 10 us for a
// round of 600 parents and 3500 items (its SM's rate of L2 sectors and
// atomics); sixteen take 4.7 us for twice that (4900 cycles of round trips,
// 1200 of the barrier, the rest scans and shared memory). So a round has one
// cluster barrier and nothing else that all wait for:
//   - a vertex that a relaxation lowers goes to its CTA's stage (two stages,
//     alternating); after the barrier each CTA pulls an equal share of all
//     stages through distributed shared memory;
//   - each CTA sends a header (pushes, deferred, wide parents, distances) to
//     every CTA before the barrier, and every CTA takes the same decisions
//     from the same headers;
//   - a parent with kWideItems children or more is published instead of
//     expanded, and all CTAs take a slice of it in the next round (a round more
//     for its children: at 512 an R-MAT graph of 3000 vertices takes 93 us
//     instead of 82, whose hubs all have so many).
// The window steers itself by the size of the rounds, not by the weights: no
// cut until a slowly growing round (by less than twofold: an R-MAT frontier
// grows tenfold and ends in a few levels, where deferring only adds rounds) has
// more than kWinHigh fresh entries; the middle of the distances expanded before
// it is then the cut and an eighth of their span the step; a round that expands
// fewer than kWinHigh / 2 parents raises the cut by the step. (2048: the 514 x
// 514 grid takes 964 rounds at 1024 and 918 at 2048, whose children a pass of
// the cluster's threads still covers.)
//
// An entry of a far list carries the distance its vertex had when it was
// deferred; if the vertex has been lowered since, that lowering pushed an
// entry of its own and the old one is dropped. Nothing separates the CTAs'
// pulls of a round from their relaxations, so a pulled vertex may already have
// been lowered in the same round: its tag is then the round's own, and the
// pulled entry is dropped too, because that lowering pushed one (deferred with
// the new distance as its key, both would be live). So a vertex has at most one
// live entry, and when the grids take over (a frontier too large) the live
// entries are the frontier, no more than there are vertices. Windowed rounds are not Bellman-Ford levels: the
// level cap moves on by the rounds run here, and a run of the loop is bounded
// by its own count of rounds.
constexpr int kSmallParentsMax = 2048;
constexpr int kClThreads = 512;
constexpr int kClMax = 16;                      // CTAs of a cluster at most
constexpr int kClStage = 4096;                  // pushes of one CTA in one round
constexpr int kClPull = 2;                      // entries per thread and round: pulled,
constexpr int kClFar = 2;                       // from the far list,
constexpr int kClWide = 2;                      // slices of wide parents
constexpr int kClEntries = kClPull + kClFar + kClWide;
constexpr int kFarList = kClFar * kClThreads;
constexpr int kWideList = 64;                   // wide parents of one CTA (16 of them: kClWide * kClThreads slices)
constexpr int kWideItems = 2048;
// Children of one CTA in a round beyond which it defers the rest; where half of
// the CTAs have so many, the grids take over (65,536 children or so: about what
// a round and a level of the grids both take 25 us for). Without that the
// cluster went on through such frontiers a budget at a time: R-MAT graphs of
// 20,000 and 40,000 vertices with 16 and 8 edges each took 232 and 243 us
// instead of 153 and 168 (184 and 196 before the cluster loop).
constexpr int kClItems = 4096;
// Children of all published parents together beyond which the grids take over;
// first for a graph with no more vertices than the frontier limit (it cannot
// outgrow the cluster), then for a larger one.
constexpr unsigned kWideSmall = 524288u, kWideLarge = 32768u;
constexpr unsigned kStartItems = 8192;          // of a first frontier of at most 32 vertices of a larger graph
constexpr int kClUnfiltered = 1024;
constexpr int kWinHigh = 2048;
constexpr unsigned kNoCut = 0xffffffffu;
constexpr size_t kClusterSmem =
    sizeof(int) * (2 * (size_t)kClStage + 2 * kFarList + 4 * (size_t)kClEntries * kClThreads + 8 * kWideList);

template <class Body>
__global__ void __launch_bounds__(kClThreads) sssp_cluster(Args a, cudaGraphConditionalHandle h, int K, int in_body) {
  NP_PDL_ENTRY();
  constexpr int KS = 4;                          // items per thread per pass
  extern __shared__ __align__(16) int s_dyn[];
  int4* s_wide = reinterpret_cast<int4*>(s_dyn);                 // published wide parents [2][kWideList]
  int* s_stage = s_dyn + 8 * kWideList;                          // pushes [2][kClStage]
  int* s_far_id = s_stage + 2 * kClStage;                        // the far list
  unsigned* s_far_key = reinterpret_cast<unsigned*>(s_far_id + kFarList);
  // the round's parents and slices: {first item, id, row start, distance}
  int4* s_seg = reinterpret_cast<int4*>(s_far_id + 2 * kFarList);
  // every CTA's header: {pushes (one above the stage's size: more) | wide << 20, parents << 16 | deferred,
  // children of the wide parents, 1 if a CTA had too many children} and {least, largest distance of
  // the round's entries, least deferred distance, -}
  __shared__ __align__(16) int4 s_hdr[2][kClMax][2];
  __shared__ unsigned s_dmin, s_dmax, s_fmin;
  __shared__ unsigned long long s_tot;           // parents and slices << 32 | their items
  __shared__ unsigned s_wide_items;
  __shared__ int s_n, s_nwide, s_ndefer, s_far_n, s_par, s_budget, s_over;
  LevelState* st = a.st;
  const int tid = (int)threadIdx.x, lane = tid & 31;
  const int rank = (int)cluster_rank(), nc = (int)cluster_size();
  const int lg = 31 - __clz(nc);   // (8 or 16 CTAs)
  // the frontier's size limit: np_config.small_parents scaled to the cluster, and what its threads can pull
  const int limit = min(min(a.small_parents, kSmallParentsMax) * (kClMax / 2), kClPull * kClThreads * nc);
  const int high = min(limit, kWinHigh), low = high / 2;
  const int max_levels = __ldcg(&st->max_levels);
  const int L0 = __ldcg(&st->base) + K;
  const int count0 = __ldcg(&st->count[L0 % 3]);
  int L = L0, prev = 0, nfar = 0;
  int rounds_left = max_levels < (1 << 29) ? 2 * max_levels + 4096 : 1 << 30;
  unsigned cut = kNoCut, step = 1;
  unsigned long long n_par = 0, n_items = 0, n_serial = 0, n_levels = 0, n_push = 0;
  int total = count0, wide_all = 0;   // entries and wide parents of all CTAs
  const bool fits = a.n_vertices <= limit;
  const unsigned wide_max = fits ? kWideSmall : kWideLarge;
  bool ran = count0 > 0 && count0 <= limit && L < max_levels;
  if (ran && !fits && count0 <= 32) {
    // a few vertices with many children (a search from a hub): the grids' from
    // the start (every warp of every CTA sees the same; R-MAT 18 from a hub of
    // 26,000 children 265 -> 243 us)
    const int id = lane < count0 ? __ldcg(&((L & 1) ? a.fr1 : a.fr0)[lane]) : -1;
    int row = 0, deg = 0;
    if (id >= 0) Body::count(a, id, row, deg);
    ran = __reduce_add_sync(kFull, min((unsigned)deg, 1u << 24)) <= kStartItems;
  }
  if (ran && tid == 0) {
    if (rank == 0) st->small_n = 0;
    s_n = 0;
    s_nwide = 0;
    s_ndefer = 0;
    s_far_n = 0;
    s_par = 0;
    s_budget = 0;
    s_over = 0;
    s_wide_items = 0u;
    s_tot = 0ull;
    s_dmin = 0xffffffffu;
    s_dmax = 0u;
    s_fmin = 0xffffffffu;
  }
  // Whether the loop runs or not: every CTA has read the level header (base,
  // count, max_levels, the frontier above) before CTA 0 may write it at the
  // end, so all take the same L0 and `ran`; and every CTA is running before its
  // shared memory is written. (A CTA that read the header after that write took
  // a level K later, whose count slot may hold a small old level.)
  cluster_barrier();
  while (ran) {
    const int cur = (L - L0) & 1, nxt = cur ^ 1;
    // ---- the round's size and window, the same in every CTA
    int pre = 0;             // pushes of the CTAs before CTA `lane`
    bool look = false;       // look through the far list
    if (L != L0) {
      const int4 h0 = lane < nc ? s_hdr[cur][lane][0] : make_int4(0, 0, 0, 0);
      int inc = h0.x;
#pragma unroll
      for (int o = 1; o < kClMax; o <<= 1) {
        const int x = __shfl_up_sync(kFull, inc, o);
        if (lane >= o) inc += x;
      }
      const int mine = h0.x & 0xfffff;
      const int sums = __reduce_add_sync(kFull, h0.y);
      pre = (inc & 0xfffff) - mine;
      const int all = __shfl_sync(kFull, inc, nc - 1);
      total = all & 0xfffff;
      wide_all = all >> 20;
      const int far_all = sums & 0xffff, near_all = (int)((unsigned)sums >> 16);
      if (near_all > 0) {
        n_levels++;
        if (L - 1 > 0) n_push += (unsigned)near_all;
      }
      if (total + wide_all + far_all == 0) break;                               // no vertex is pending
      // the grids take over: the frontier, or its children, too many for a cluster
      if (total > limit || __any_sync(kFull, mine > kClStage) || --rounds_left <= 0) break;
      if (wide_all > 0 && __reduce_add_sync(kFull, min((unsigned)h0.z, 1u << 26)) > wide_max) break;
      if (2 * __popc(__ballot_sync(kFull, h0.w != 0)) >= nc) break;
      if (total > high && (cut != kNoCut || (prev > 0 && total >= prev && total < 2 * prev))) {
        // the middle of the last round's distances
        const int4 h1 = lane < nc ? s_hdr[cur][lane][1] : make_int4(-1, 0, 0, 0);
        const unsigned dmin = __reduce_min_sync(kFull, (unsigned)h1.x);
        const unsigned span = __reduce_max_sync(kFull, (unsigned)h1.y) - dmin;
        cut = min(cut, dmin + span / 2);
        step = span / 8 > 0u ? span / 8 : 1u;
      } else if (total + wide_all == 0) {
        // only deferred entries are left: move the cut past the nearest
        const unsigned fmin =
            __reduce_min_sync(kFull, lane < nc ? (unsigned)s_hdr[cur][lane][1].z : 0xffffffffu);
        cut = fmin > 0xfffffffeu - step ? 0xfffffffeu : fmin + step;
        look = true;
      } else if (cut != kNoCut && near_all < low) {
        cut = cut > 0xfffffffeu - step ? 0xfffffffeu : cut + step;
        if (step < (1u << 30)) step += step / 4 + 1;
        look = true;
      }
      if (__any_sync(kFull, h0.w != 0)) look = true;   // some were deferred for their children: within the cut
      prev = total;
    }
    // ---- this CTA's entries: its share of the stages, its far list, its slice of each wide parent
    const int lo = (int)((unsigned)total * (unsigned)rank >> lg), hi = (int)((unsigned)total * (unsigned)(rank + 1) >> lg);
    int pid[kClEntries], base[kClEntries], N[kClEntries];
    unsigned d[kClEntries], key[kClFar];
    bool use[kClEntries];    // expand it in this round, in this CTA
#pragma unroll
    for (int r = 0; r < kClPull; r++) {
      const int i = lo + r * kClThreads + tid;
      pid[r] = -1;
      if (lo + r * kClThreads < hi) {   // (uniform)
        if (L == L0) {
          if (i < hi) pid[r] = __ldcg(&((L & 1) ? a.fr1 : a.fr0)[i]);
        } else {
          int c = 0, off = 0;   // the CTA holding entry i, and its place there
#pragma unroll
          for (int q = 0; q < kClMax; q++) {
            const int x = __shfl_sync(kFull, pre, q);
            if (q < nc && x <= i) {
              c = q;
              off = i - x;
            }
          }
          if (i < hi) pid[r] = cluster_ld(cluster_addr(&s_stage[cur * kClStage + off], (unsigned)c));
        }
      }
    }
#pragma unroll
    for (int r = 0; r < kClFar; r++) {
      const int i = r * kClThreads + tid, e = kClPull + r;
      pid[e] = look && i < nfar ? s_far_id[i] : -1;
      key[r] = look && i < nfar ? s_far_key[i] : kNoCut;
    }
#pragma unroll
    for (int r = 0; r < kClPull + kClFar; r++) {
      use[r] = pid[r] >= 0 && (r < kClPull || key[r < kClPull ? 0 : r - kClPull] <= cut);
      const unsigned long long word = use[r] ? __ldcg(&a.b.dtag[pid[r]]) : 0ull;
      d[r] = (unsigned)(word >> 32);
      base[r] = 0;
      N[r] = 0;
      if (use[r]) Body::count(a, pid[r], base[r], N[r]);
      // (lowered in this round: an entry of the next one)
      if (r < kClPull) use[r] = use[r] && (unsigned)word != (unsigned)(L + 1);
    }
#pragma unroll
    for (int r = 0; r < kClWide; r++) {
      const int e = kClPull + kClFar + r;
      pid[e] = -1;
      base[e] = 0;
      N[e] = 0;
      d[e] = 0u;
      use[e] = false;
      if (wide_all > 0) {   // uniform over the cluster
        const int j = r * kClThreads + tid, c = j / kWideList, k = j % kWideList;
        if (c < nc && k < s_hdr[cur][c][0].x >> 20) {
          const int4 q = cluster_ld4(cluster_addr(&s_wide[cur * kWideList + k], (unsigned)c));
          const int f0 = (int)((long long)q.z * rank >> lg), f1 = (int)((long long)q.z * (rank + 1) >> lg);
          pid[e] = q.x;
          base[e] = q.y + f0;
          N[e] = f1 - f0;
          d[e] = (unsigned)q.w;
          use[e] = f1 > f0;
        }
      }
    }
    if (look) {
      if (tid == 0) {
        s_far_n = 0;
        s_fmin = 0xffffffffu;
      }
      __syncthreads();   // the far list is in registers: it is written again below
    }
    // ---- expand, publish or defer each entry
    auto defer = [&](bool waits, int id, unsigned k) {   // (all lanes of a warp)
      if (!__any_sync(kFull, waits)) return;
      const int q = warp_slots(waits, &s_far_n);
      if (waits) {
        s_far_id[q] = id;
        s_far_key[q] = k;
        atomicMin(&s_fmin, k);
      }
    };
    // room in the far list for this lane's entry (else it is expanded at once)
    auto room = [&](bool waits) {
      if (nfar + (hi - lo) <= kFarList) return waits;   // (uniform)
      const int p = warp_slots(waits, &s_ndefer);
      return waits && p < kFarList - nfar;
    };
    unsigned dlo = 0xffffffffu, dhi = 0u;
#pragma unroll
    for (int r = 0; r < kClPull; r++) {
      if (lo + r * kClThreads >= hi) continue;   // uniform
      if (use[r]) {
        dlo = min(dlo, d[r]);
        dhi = max(dhi, d[r]);
      }
      if (cut != kNoCut) {   // uniform
        bool waits = use[r] && d[r] > cut;
        waits = room(waits);
        use[r] = use[r] && !waits;
        defer(waits, pid[r], d[r]);
      }
    }
    if (look) {   // uniform
#pragma unroll
      for (int r = 0; r < kClFar; r++) {
        if (r * kClThreads >= nfar) continue;   // uniform
        const int e = kClPull + r;
        defer(pid[e] >= 0 && !use[e], pid[e], key[r]);
        use[e] = use[e] && key[r] == d[e];   // lowered since it was deferred: dropped
      }
    }
    // parents with many children go to all CTAs; a warp whose other parents
    // would take the CTA beyond its children defers them, and so does one that
    // finds the list of wide parents full
    unsigned parents = 0, mine = 0, cnt = 0;
    bool big = wide_all > 0;   // slices, or a wide parent expanded here
#pragma unroll
    for (int r = 0; r < kClPull + kClFar; r++)
      if (use[r]) {
        parents++;
        mine += min((unsigned)N[r], 0x1000000u);
      }
    if (__any_sync(kFull, mine > 64u)) {
      unsigned sum = 0;
#pragma unroll
      for (int r = 0; r < kClPull + kClFar; r++) {
        const bool wide = use[r] && N[r] >= kWideItems;
        if (__any_sync(kFull, wide)) {
          const int k = warp_slots(wide, &s_nwide);
          const bool out = room(wide && k >= kWideList);
          defer(out, pid[r], d[r]);
          if (out) {
            s_over = 1;
            parents--;
          }
          if (wide && k < kWideList) {
            s_wide[nxt * kWideList + k] = make_int4(pid[r], base[r], N[r], (int)d[r]);
            atomicAdd(&s_wide_items, min((unsigned)N[r], 1u << 20));
            n_items += (unsigned)N[r];
            n_serial++;
          }
          big = big || (wide && !out && k >= kWideList);
          use[r] = use[r] && (!wide || (!out && k >= kWideList));
        }
        sum += use[r] ? min((unsigned)N[r], 0x10000u) : 0u;
      }
      sum = __reduce_add_sync(kFull, sum);
      int at = 0;
      if (sum > 512u && lane == 0) at = atomicAdd(&s_budget, (int)sum);
      at = __shfl_sync(kFull, at, 0);
      if (at + (int)sum > kClItems) {
        if (lane == 0) s_over = 1;
#pragma unroll
        for (int r = 0; r < kClPull; r++) {
          const bool out = room(use[r]);
          use[r] = use[r] && !out;
          parents -= out ? 1u : 0u;
          defer(out, pid[r], d[r]);
        }
      }
    }
    mine = 0;
#pragma unroll
    for (int r = 0; r < kClEntries; r++) {
      if (!use[r]) continue;
      if (r < kClPull + kClFar) n_items += (unsigned)N[r];
      if (N[r] == 0) {
        use[r] = false;
        continue;
      }
      if (r < kClPull + kClFar) n_serial++;
      mine += (unsigned)N[r];
      cnt++;
    }
    n_par += parents;
    // ---- the round's parents and slices, compacted: one atomic per warp on
    // their number and items together keeps both in the same order
    if (__any_sync(kFull, parents + cnt != 0u)) {
      unsigned it = mine, ct = cnt;
      if (!__any_sync(kFull, big)) {
        // (a warp has below 2^18 items: one scan carries both)
        unsigned w = cnt << 20 | mine;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned x = __shfl_up_sync(kFull, w, o);
          if (lane >= o) w += x;
        }
        it = w & 0xfffffu;
        ct = w >> 20;
      } else {
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const unsigned x = __shfl_up_sync(kFull, it, o), y = __shfl_up_sync(kFull, ct, o);
          if (lane >= o) {
            it += x;
            ct += y;
          }
        }
      }
      unsigned long long at = 0ull;
      if (lane == 31) {
        at = atomicAdd(&s_tot, ((unsigned long long)ct << 32) | it);
      }
      parents = __reduce_add_sync(kFull, parents);
      if (lane == 0) atomicAdd(&s_par, (int)parents);
      if (2 * total > high) {   // (uniform: the next round may need the span)
        dlo = __reduce_min_sync(kFull, dlo);
        dhi = __reduce_max_sync(kFull, dhi);
        if (lane == 0 && dlo <= dhi) {
          atomicMin(&s_dmin, dlo);
          atomicMax(&s_dmax, dhi);
        }
      }
      at = __shfl_sync(kFull, at, 31);
      unsigned first = (unsigned)at + it - mine, j = (unsigned)(at >> 32) + ct - cnt;
#pragma unroll
      for (int r = 0; r < kClEntries; r++)
        if (use[r]) {
          s_seg[j] = make_int4((int)first, pid[r], base[r], (int)d[r]);
          first += (unsigned)N[r];
          j++;
        }
    }
    __syncthreads();
    const int nseg = (int)(s_tot >> 32), items = (int)(unsigned)s_tot;
    // ---- the children
    BodyArgs b = a.b;
    b.L = L;
    // (few children: a filter read before each atomic would only lengthen the
    // chain; many: most fail the filter, and an SM's atomics are the limit)
    b.unfiltered = items <= kClUnfiltered;
    int* next = (L & 1) ? a.fr0 : a.fr1;
    int* stage = s_stage + nxt * kClStage;
    for (int t0 = tid & ~31; t0 < items; t0 += KS * kClThreads) {   // (uniform over the warp)
      typename Body::F f[KS];
      typename Body::P pk[KS];
      bool v[KS];
      int idx[KS];
#pragma unroll
      for (int k = 0; k < KS; k++) {
        const int t = t0 + k * kClThreads + lane;
        v[k] = t < items;
        idx[k] = 0;
        pk[k] = typename Body::P{};
        f[k] = typename Body::F{};
        if (t0 + k * kClThreads < items) {   // (uniform over the warp)
          const int4 q = s_seg[warp_segment(s_seg, nseg, t - lane)];
          idx[k] = t - q.x;
          // (the level-loop bodies do not use N in parent_aux)
          pk[k] = Body::parent_aux(b, q.y, q.z, 0, (unsigned)q.w);
          if (v[k]) f[k] = Body::fetch(b, pk[k], idx[k]);
        }
      }
      bool pf[KS];
      int pv[KS];
      Body::template apply_batch<KS>(b, pk, idx, f, v, pf, pv);
      unsigned m[KS];
      int n = 0;
#pragma unroll
      for (int k = 0; k < KS; k++) {
        m[k] = __ballot_sync(kFull, pf[k]);
        n += __popc(m[k]);
      }
      if (n == 0) continue;
      int pos = 0;
      if (lane == 0) pos = atomicAdd(&s_n, n);
      pos = __shfl_sync(kFull, pos, 0);
#pragma unroll
      for (int k = 0; k < KS; k++) {
        const int at = pos + __popc(m[k] & lanemask_lt());
        pos += __popc(m[k]);
        if (pf[k] && at < kClStage) stage[at] = pv[k];
        if (pos > kClStage) {   // (uniform over the warp) the grids take over after this round
          const bool spill = pf[k] && at >= kClStage;
          const int p = warp_slots(spill, &st->small_n);
          if (spill) next[p] = pv[k];
        }
      }
    }
    __syncthreads();
    nfar = s_far_n;
    if (tid < 32) {
      const int4 h0 = make_int4(min(s_n, kClStage + 1) | min(s_nwide, kWideList) << 20, s_par << 16 | s_far_n,
                                (int)s_wide_items, s_over);
      const int4 h1 = make_int4((int)s_dmin, (int)s_dmax, (int)s_fmin, 0);
      if (lane < nc) {
        cluster_st4(cluster_addr(&s_hdr[nxt][rank][0], (unsigned)lane), h0);
        cluster_st4(cluster_addr(&s_hdr[nxt][rank][1], (unsigned)lane), h1);
      }
      __syncwarp();
      if (lane == 0) {
        s_n = 0;
        s_nwide = 0;
        s_ndefer = 0;
        s_par = 0;
        s_budget = 0;
        s_over = 0;
        s_wide_items = 0u;
        s_tot = 0ull;
        s_dmin = 0xffffffffu;
        s_dmax = 0u;
      }
    }
    cluster_barrier();
    L++;
  }
  if (ran) {
    // ---- the live entries become the frontier of level L
    const int cur = (L - L0) & 1;
    const int own = min(s_hdr[cur][rank][0].x & 0xfffff, kClStage), own_wide = s_hdr[cur][rank][0].x >> 20;
    int* fr = (L & 1) ? a.fr1 : a.fr0;
    const int all = own + own_wide + nfar;
    for (int i0 = 0; i0 < all; i0 += kClThreads) {
      const int i = i0 + tid;
      int id = -1;
      if (i < own) {
        id = s_stage[cur * kClStage + i];
      } else if (i < all) {
        unsigned k;
        if (i < own + own_wide) {
          const int4 q = s_wide[cur * kWideList + i - own];
          id = q.x;
          k = (unsigned)q.w;
        } else {
          id = s_far_id[i - own - own_wide];
          k = s_far_key[i - own - own_wide];
        }
        if ((unsigned)(__ldcg(&a.b.dtag[id]) >> 32) != k) id = -1;
      }
      const int p = warp_slots(id >= 0, &st->small_n);
      if (id >= 0) fr[p] = id;
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n_par += __shfl_xor_sync(kFull, n_par, o);
      n_items += __shfl_xor_sync(kFull, n_items, o);
      n_serial += __shfl_xor_sync(kFull, n_serial, o);
    }
    if (lane == 0) {
      add_stat(st, S_PARENTS, n_par);
      add_stat(st, S_ITEMS, n_items);
      add_stat(st, S_SERIAL, n_serial);
    }
    cluster_barrier();
  }
  if (rank == 0 && tid == 0) {
    int left = count0;
    if (ran) {
      left = __ldcg(&st->small_n);
      for (int k = 0; k < 4; k++) {
        st->ticket[k] = 0;
        st->agg_records[k] = 0;
        st->agg_blocks[k] = 0;
        st->agg_acc[k] = 0ull;
        st->child_ticket[k] = 0;
        st->pack_acc[k] = 0ull;
        st->pack_records[k] = 0;
        st->pack_items[k] = 0;
        st->pack_ticket[k] = 0;
      }
      st->count[L % 3] = left;
      st->count[(L + 1) % 3] = 0;
      st->count[(L + 2) % 3] = 0;
      add_stat(st, S_LEVELS, n_levels);
      add_stat(st, S_PUSHES, n_push);
      st->max_levels = max_levels + (L - L0);
    }
    st->base = L;
    bool more = left > 0 && (ran || L < max_levels);
    if (in_body) {
      // the iteration cap turns a level loop that failed to terminate into an error
      const int it = ++st->body_iters;
      if (more && it > max_levels + 16) {
        st->error |= kErrTimeout;
        more = false;
      }
    }
    cudaGraphSetConditional(h, more ? 1u : 0u);
  }
}

// -------------------------------------------------- first levels of a BFS
//
// One CTA runs the levels from the start of a traversal for as long as they are
// small, with one bit per vertex in shared memory as the visited set: nothing
// has been reached yet, so it starts empty, and a claim is a shared-memory
// operation instead of a compare-and-swap in L2. The thread that claims a vertex
// stores its level, loads its row bounds and queues it with its place among the
// next level's items (one packed atomic per warp: vertices, vertices with
// children, children), so a level needs no scan and one barrier. What is left of
// its chain are two round trips to L2 (edges, row bounds) instead of three, and
// what bounds a larger level is the CTA's instruction issue, not the rate of one
// SM's L2 atomics: 8.3 us a level of 2600 children with the claims in L2, 3.7 here
// (road grid 514 x 514, 602 levels, 5.0 -> 2.2 ms; a 4096-vertex web-like graph of
// 18 levels 90 -> 48 us). A level of 16384 children takes about 6 us, what the
// grids need for one however small; of 32768, 10 (R-MAT 18 then lost 14%).
// When a level has too many parents or children the grids take over from the
// frontier in global memory, and the body-end loop (level_small) is the one that
// runs small levels after that.
constexpr int kBitsQueue = 8192;        // queued parents at most (two queues of {first item, row start})
constexpr int kBitsItems = 16384;       // children of a level (they bound its vertices, counted in 16 bits)
constexpr int kBitsSmem = 216 * 1024;
constexpr int kBitsMaxVertices = 1 << 20;   // 128 KB of bits; at least 5600 queued parents

// Dynamic shared memory for n vertices, and the queue's size in it.
__host__ __device__ inline int bits_words(int n) { return (n + 127) / 128 * 4; }
__host__ __device__ inline int bits_queue(int n) {
  const int q = (kBitsSmem - bits_words(n) * 4) / 16;
  return q < kBitsQueue ? q : kBitsQueue;
}
inline size_t bits_smem(int n) { return (size_t)bits_words(n) * 4 + (size_t)bits_queue(n) * 16; }

__device__ __forceinline__ int warp_segment2(const int2* seg, int n, int t) {
  const int lane = threadIdx.x & 31;
  int lo = 0, hi = n;
  while (hi - lo > 32) {
    const int stride = (hi - lo + 31) >> 5, i = lo + lane * stride;
    const bool p = i < hi && seg[i].x <= t;
    lo += (__popc(__ballot_sync(kFull, p)) - 1) * stride;
    hi = min(hi, lo + stride);
  }
  const int i = lo + lane;
  const bool p = i < hi && seg[i].x <= t;
  const int r = lo + __popc(__ballot_sync(kFull, p)) - 1, j = r + 1 + lane;
  const int at = j < n ? seg[j].x - t : 32;
  return r + __popc(__reduce_or_sync(kFull, at < 32 ? 1u << at : 0u) & (0xffffffffu >> (31 - lane)));
}

template <class Body>
__global__ void __launch_bounds__(1024) bfs_first_levels(Args a, cudaGraphConditionalHandle h, int, int) {
  NP_PDL_ENTRY();
  constexpr int KS = 4;
  extern __shared__ __align__(16) unsigned s_bits[];
  const int words = bits_words(a.n_vertices), cap = bits_queue(a.n_vertices);
  int2* s_queue = reinterpret_cast<int2*>(s_bits + words);   // [2][cap]
  // of level L at L % 3: vertices << 48 | those with children << 32 | their children
  __shared__ unsigned long long s_tot[3];
  LevelState* st = a.st;
  const int tid = (int)threadIdx.x, lane = tid & 31;
  const int limit = min(a.small_parents, kSmallParentsMax) * 4;
  const int max_levels = __ldcg(&st->max_levels);
  const int count0 = __ldcg(&st->count[0]);
  const bool ran = count0 > 0 && count0 <= limit && max_levels > 0;
  for (int i = tid; i < words / 4; i += 1024) reinterpret_cast<uint4*>(s_bits)[i] = make_uint4(0u, 0u, 0u, 0u);
  if (tid < 3) s_tot[tid] = 0ull;
  __syncthreads();
  // queues the vertices id[k] with take[k] for level `to`: their row bounds, all
  // loaded before any is used, and one atomic per warp
  auto push = [&](auto& take, auto& id, int to, int* next) {
    constexpr int M = sizeof(take) / sizeof(take[0]);
    int base[M], N[M];
    unsigned long long mine = 0ull;   // vertices << 48 | with children << 32 | children, of this thread
#pragma unroll
    for (int k = 0; k < M; k++) {
      base[k] = 0;
      N[k] = 0;
      if (take[k]) Body::count(a, id[k], base[k], N[k]);
    }
#pragma unroll
    for (int k = 0; k < M; k++)
      mine += (take[k] ? 1ull << 48 : 0ull) + (N[k] > 0 ? 1ull << 32 : 0ull) + (unsigned)N[k];
    if (!__any_sync(kFull, mine != 0ull)) return;
    unsigned long long inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned long long x = __shfl_up_sync(kFull, inc, o);
      if (lane >= o) inc += x;
    }
    unsigned long long at = 0ull;
    if (lane == 31) at = atomicAdd(&s_tot[to % 3], inc);
    at = __shfl_sync(kFull, at, 31) + inc - mine;
    int pos = (int)(at >> 48), j = (int)(at >> 32 & 0xffffull);
    unsigned first = (unsigned)at;
#pragma unroll
    for (int k = 0; k < M; k++) {
      if (take[k] && next) next[pos++] = id[k];
      if (N[k] > 0) {
        if (j < cap) s_queue[(to & 1) * cap + j] = make_int2((int)first, base[k]);
        j++;
        first += (unsigned)N[k];
      }
    }
  };
  int L = 0, count = count0;
  unsigned long long n_par = 0, n_items = 0, n_serial = 0;
  if (ran) {
    for (int i0 = 0; i0 < count0; i0 += 1024) {   // (the frontier itself is in global memory already)
      const int i = i0 + tid;
      int id[1] = {i < count0 ? __ldcg(&a.fr0[i]) : -1};
      bool take[1] = {id[0] >= 0};
      if (take[0]) atomicOr(&s_bits[id[0] >> 5], 1u << (id[0] & 31));
      push(take, id, 0, nullptr);
    }
    __syncthreads();
    for (;;) {
      const unsigned long long tot = s_tot[L % 3];
      const int segs = (int)(tot >> 32 & 0xffffull);
      const unsigned items = (unsigned)tot;
      count = (int)(tot >> 48);
      // nothing left, or the grids' (a queue that overflowed has more than cap entries)
      if (count == 0 || count > limit || segs > cap || items > (unsigned)kBitsItems || L >= max_levels) break;
      if (tid == 0) s_tot[(L + 2) % 3] = 0ull;   // (read in level L - 1, added to from level L + 1 on)
      n_par += (unsigned)count;
      n_items += items;
      n_serial += (unsigned)segs;
      int* next = (L & 1) ? a.fr0 : a.fr1;
      const int2* queue = s_queue + (L & 1) * cap;
      for (int t0 = tid & ~31; t0 < (int)items; t0 += KS * 1024) {   // (uniform over the warp)
        int v[KS];
#pragma unroll
        for (int k = 0; k < KS; k++) {
          const int t = t0 + k * 1024 + lane;
          v[k] = -1;
          if (t - lane < (int)items) {   // (uniform)
            // (a single traversal: an entry carries no query part)
            const int2 q = queue[warp_segment2(queue, segs, t - lane)];
            if (t < (int)items) v[k] = __ldg(&a.b.col[q.y + t - q.x]);
          }
        }
        bool take[KS];
#pragma unroll
        for (int k = 0; k < KS; k++) {
          const unsigned bit = 1u << (v[k] & 31);
          take[k] = v[k] >= 0 && !(s_bits[v[k] >> 5] & bit) && !(atomicOr(&s_bits[v[k] >> 5], bit) & bit);
          if (take[k]) a.b.level[v[k]] = L + 1;
        }
        push(take, v, L + 1, next);
      }
      __syncthreads();
      L++;
    }
  }
  if (tid == 0) {
    if (ran) {
      st->count[L % 3] = count;
      st->count[(L + 1) % 3] = 0;
      st->count[(L + 2) % 3] = 0;
      add_stat(st, S_LEVELS, (unsigned long long)L);
      add_stat(st, S_PUSHES, n_par - (L > 0 ? (unsigned long long)count0 : 0ull));
      add_stat(st, S_PARENTS, n_par);
      add_stat(st, S_ITEMS, n_items);
      add_stat(st, S_SERIAL, n_serial);
    }
    st->base = L;
    cudaGraphSetConditional(h, count > 0 && L < max_levels ? 1u : 0u);
  }
}

}  // namespace nestpar
