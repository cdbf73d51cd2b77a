// The aggregated child grid of triangle counting: adjacency bitmaps in shared memory.
#pragma once
#include "np_child.cuh"

namespace nestpar {

// Persistent child grid of the grid-host form. A CTA takes the next chunk of
// aggregated blocks (about kTcEdges oriented edges u -> v) from the level's
// ticket and goes through it record by record: the out-list of u is marked in a
// bitmap over the vertices in shared memory, and each warp takes a share of the
// record's edges and reads N+(v) of one after the other, 32 consecutive entries
// at a time, each lane testing its entry's bit. Then the marks are taken back.
//
// What bounds it: the entries read (the sum of |N+(v)| over the edges, 251 M for
// R-MAT 17 with 1.86 M oriented edges, from L1 and L2), about 20 instructions and
// 3 shared-memory wavefronts per 32 of them; 252 us. An intersection per thread
// (a blocked merge of two sorted lists) reads fewer entries, but each lane walks
// lists of its own, uncoalesced and divergent: 709 us. A record costs each warp of
// its CTA about as much as two edges beside its entries, so CTAs are small (128
// threads up to 131,072 vertices, 13 to an SM: 252 us; 256 threads 275; 512
// threads 358); a byte per vertex shared by eight groups of four warps halves the
// instructions of a test but leaves half the warps: 268 us. A vertex's place is
// permuted (bits 5..9 mixed with the next five), because low ids are common in
// R-MAT graphs and the ids' own bits would send a quarter of the tests to one bank.
constexpr int kTcEdges = 256;
constexpr int kTcMaxVertices = 1600 * 1024;   // 200 KB; beyond that the intersection per thread stays

__global__ void __maxnreg__(40) tc_child(BodyArgs b, AggSeg s) {
  NP_PDL_ENTRY();
  extern __shared__ unsigned s_map[];   // [s.words], a multiple of 1024 bits
  __shared__ int s_first;
  const int tid = (int)threadIdx.x, nt = (int)blockDim.x, lane = tid & 31, warp = tid >> 5, nw = nt >> 5;
  auto place = [](int v) { return (unsigned)v ^ ((unsigned)v >> 5 & 0x3e0u); };
  auto has = [&](int v) {
    const unsigned p = place(v);
    return s_map[p >> 5] >> (p & 31) & 1u;
  };
  int nrec = 0, total = 0;
  agg_totals(b.st, b.L, s.mode, nrec, total);
  int* ticket = &b.st->child_ticket[b.L & 3];
  const int span = s.cb * s.cf;                          // edges of an aggregated block
  // (fewer blocks to a chunk where the grid would not have one chunk each)
  const int chunk = max(1, min(kTcEdges / span, total / (int)gridDim.x));
  int first = (int)blockIdx.x * chunk;                   // its first chunk; later ones come from the ticket
  if (first >= total) return;
  for (int i = tid; i < s.words; i += nt) s_map[i] = 0u;
  __syncthreads();
  unsigned long long found = 0;
  int done = 0;
  while (first < total) {   // uniform
    const int last = min(total, first + chunk);
    int j = warp_search(s.boff, 0, nrec, first);
    for (int B = first; B < last; j++) {
      const int4 r = __ldcg(&s.rec[j]);
      const int off = __ldcg(&s.boff[j]);
      const int end = min(last, j + 1 < nrec ? __ldcg(&s.boff[j + 1]) : total);
      const int* nu = b.col + r.y;
      for (int i = tid; i < r.z; i += nt) {
        const unsigned p = place(__ldg(&nu[i]));
        atomicOr(&s_map[p >> 5], 1u << (p & 31));
      }
      const int e0 = (B - off) * span, e1 = min(r.z, (end - off) * span);
      const int share = ceil_div(e1 - e0, nw), a0 = e0 + warp * share, a1 = min(e1, a0 + share);
      __syncthreads();
      for (int x = a0; x < a1; x += 32) {
        int vb = 0, vn = 0;
        if (x + lane < a1) {
          const int v = __ldg(&nu[x + lane]);
          vb = __ldg(&b.row_ptr[v]);
          vn = __ldg(&b.row_ptr[v + 1]) - vb;
        }
        unsigned c = 0;   // (below 2^32: 32 lists of below 2^26 entries a lane)
        const int here = min(32, a1 - x);
        for (int q = 0; q < here; q++) {
          const int* p = b.col + __shfl_sync(kFull, vb, q) + lane;
          int n = __shfl_sync(kFull, vn, q);
          for (; n >= 128; n -= 128, p += 128) {
            const int w0 = __ldg(p), w1 = __ldg(p + 32), w2 = __ldg(p + 64), w3 = __ldg(p + 96);
            c += has(w0) + has(w1) + (has(w2) + has(w3));
          }
          if (n & 64) {
            const int w0 = __ldg(p), w1 = __ldg(p + 32);
            c += has(w0) + has(w1);
            p += 64;
          }
          if (n & 32) {
            c += has(__ldg(p));
            p += 32;
          }
          if (lane < (n & 31)) c += has(__ldg(p));
        }
        found += c;
      }
      __syncthreads();
      for (int i = tid; i < r.z; i += nt) s_map[place(__ldg(&nu[i])) >> 5] = 0u;
      __syncthreads();
      B = end;
    }
    done += last - first;
    // (the next write of s_first is a record's barriers later)
    if (tid == 0) s_first = atomicAdd(ticket, chunk) + (int)gridDim.x * chunk;
    __syncthreads();
    first = s_first;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) found += __shfl_xor_sync(kFull, found, o);
  if (lane == 0 && found) atomicAdd(&b.acc[(blockIdx.x * nw + warp) & (kTcSlots - 1)], found);
  if (tid == 0 && done) add_stat(b.st, S_CBLOCKS, (unsigned long long)done);
}

}  // namespace nestpar
