// Windows inside a CTA: the tokens of one window from the positions, and the selection of its merged sources (Steps 1, 2
// and 4).  Used by the FD kernels, which take one window (or a tile of one) per CTA, and by the map kernel.
#pragma once
#include "common.cuh"

namespace lkv {

// Calls emit(l, i) for every token i of window w, l its rank inside the window in storage (= position) order, from
// whatever thread holds it, and returns the number of tokens.  All threads of the CTA (WARPS warps) take part; the caller
// synchronises before it uses what emit wrote.  A full grid is counted out; otherwise every position is looked at (the
// position arrays are small, and an unsorted one is still taken apart without a gap: it only raises a status bit).
// match: window_search_bytes(cap_in), warp_sum: [WARPS], both in shared memory.
__host__ __device__ inline size_t window_search_bytes(int cap_in) { return size_t((cap_in + 31) / 32) * 8; }

template <int WARPS, typename Emit>
__device__ __forceinline__ int window_tokens(const Geometry& g, const int* __restrict__ pos, int n, int w,
                                             unsigned int* match, int* warp_sum, Emit emit) {
  constexpr int NT = 32 * WARPS;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int w2 = g.w * g.w, tile = w / w2, wr = (w - tile * w2) / g.w, wc = w - tile * w2 - wr * g.w;
  const int rows = g.rows[tile], cols = g.cols[tile], first = g.tile_off[tile], n_grid = g.tile_off[g.n_tiles];
  // rows r with r * w / rows == wr, columns c with c * w / cols == wc
  const int r0 = (wr * rows + g.w - 1) / g.w, r1 = ((wr + 1) * rows + g.w - 1) / g.w;
  const int c0 = (wc * cols + g.w - 1) / g.w, c1 = ((wc + 1) * cols + g.w - 1) / g.w;
  if (!pos && n == n_grid) {
    const int nw = (r1 - r0) * (c1 - c0);
    for (int l = tid; l < nw; l += NT) {
      const int r = l / (c1 - c0);
      emit(l, first + (r0 + r) * cols + c0 + (l - r * (c1 - c0)));
    }
    return nw;
  }
  const int lo = first + r0 * cols, hi = first + r1 * cols;
  const int chunks = (n + 31) >> 5;
  // four consecutive tokens per lane, 128 per warp and step: enough loads in flight that a sample of a few thousand tokens
  // is one or two round trips
#pragma unroll 4
  for (int c = warp * 4; c < chunks; c += WARPS * 4) {
    const int i = c * 32 + lane * 4;
    int p[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) p[k] = i + k < n ? (pos ? pos[i + k] : i + k) : 0;
    unsigned int m = 0;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      bool in = false;
      if (p[k] >= lo && p[k] < hi) {
        const int col = (p[k] - first) % cols;
        in = col >= c0 && col < c1;
      }
      in = in || (w == 0 && (p[k] < 0 || p[k] >= n_grid));   // no such position: counted with window 0
      if (in && i + k < n) m |= 1u << ((lane & 7) * 4 + k);
    }
    m |= __shfl_xor_sync(0xffffffffu, m, 1);
    m |= __shfl_xor_sync(0xffffffffu, m, 2);
    m |= __shfl_xor_sync(0xffffffffu, m, 4);
    if ((lane & 7) == 0 && c + (lane >> 3) < chunks) match[c + (lane >> 3)] = m;
  }
  __syncthreads();
  int nw = 0;
  for (int base = 0; base < chunks; base += NT) {
    const unsigned int m = base + tid < chunks ? match[base + tid] : 0u;
    const int own = __popc(m);
    int x = own;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, x, o);
      if (lane >= o) x += t;
    }
    if (lane == 31) warp_sum[warp] = x;
    __syncthreads();
    int before = nw, total = 0;
#pragma unroll
    for (int k = 0; k < WARPS; ++k) {
      const int s = warp_sum[k];
      if (k < warp) before += s;
      total += s;
    }
    if (base + tid < chunks) match[chunks + base + tid] = before + x - own;   // tokens of the window in front of the word
    nw += total;
    __syncthreads();
  }
  for (int c = warp; c < chunks; c += WARPS) {           // a lane per token: a window may be as dense as the sample
    const unsigned int m = match[c];
    if ((m >> lane) & 1u) emit((int)match[chunks + c] + __popc(m & ((1u << lane) - 1u)), c * 32 + lane);
  }
  return nw;
}

// The lists of one window in shared memory.
struct WindowLists {
  unsigned int* key;     // [max_src + 4] orderable lowest score of every source
  int* into;             // [max_src + 4] destination (rank among the destinations) of selected sources, -1 for the others
  int* best;             // [max_src] destination that attains the lowest score, -1: none
  int* count;            // [max_dst] sources merged into a destination
  int* tok;              // [max_cell] token index by local rank
  unsigned short* part;  // [kParts][max_dst] the same by eighths of the sources (windows of more than 128 sources)
  static constexpr int kParts = 8;
  static __host__ __device__ size_t bytes(int max_cell) {
    const size_t src = (max_cell + 1) / 2;
    return (2 * ((src + 7) & ~size_t(3)) + 2 * src + max_cell + (src > 128 ? kParts / 2 * src : 0)) * 4;
  }
  __device__ static WindowLists at(void* p, int max_cell) {     // p: 16-byte aligned
    const int src = (max_cell + 1) / 2;
    WindowLists w;
    w.key = static_cast<unsigned int*>(p);
    w.into = reinterpret_cast<int*>(w.key + ((src + 7) & ~3));
    w.best = w.into + ((src + 7) & ~3);
    w.count = w.best + src;
    w.tok = w.count + src;
    w.part = reinterpret_cast<unsigned short*>(w.tok + max_cell);
    return w;
  }
};

// The destination (rank among the window's nb) a key of the tiled FD kernel names, -1: none.  A tile whose waits expired
// stores no key, so what stands in its place is whatever the workspace held: it must not become an index.
__host__ __device__ inline int key_partner(unsigned long long key, int nb) {
  const unsigned int to = (unsigned int)key;
  return to < (unsigned int)nb ? (int)to : -1;
}

// Selection: the `removed` sources with the lowest (score, index) are merged into their best destination.  Writes every
// token's partner and place (see Workspace).  key / best / tok are complete in shared memory (synchronised) on entry; all
// threads take part, in whole warps.  Bound by the length of a thread's walk over the other sources, so as many lanes share
// a source as there are threads for (18 of 256: 8).  A source's rank among the sources of its destination is counted the
// same way in windows of up to 128 sources; in larger ones eight warps walk an eighth of the sources each, 32 at a time
// (match_any gives the rank within the 32, a counter per destination and eighth the ones before): 1024 sources 8.0 us with
// one warp for all of them, 2.2 with eight.
__device__ __forceinline__ void select_window(const WindowLists& s, int nw, int removed, int par, int* __restrict__ partner,
                                              int* __restrict__ place) {
  const int tid = threadIdx.x, nthr = blockDim.x, lane = tid & 31, warp = tid >> 5;
  const int na = (nw + 1 - par) >> 1, nb = nw - na;      // sources: local ranks of parity `par`
  const bool ranked = removed > 0 && removed < na;
  int share = 1;                                         // lanes per source
  while (share < 32 && 2 * share * na <= nthr) share *= 2;
  const int mine0 = tid / share, step = nthr / share, sub = tid & (share - 1);
  if (ranked) {
    if (tid < 4) s.key[na + tid] = 0xffffffffu;          // the last group of four keys
    __syncthreads();
    for (int e0 = 0; e0 < na; e0 += step) {
      const int e = min(e0 + mine0, na - 1);             // (whole warps stay together)
      const unsigned int mine = s.key[e];
      int rank = 0;
      for (int k = 4 * sub; k < na; k += 4 * share) {
        const uint4 v = *reinterpret_cast<const uint4*>(s.key + k);
        rank += (v.x < mine) + (v.y < mine) + (v.z < mine) + (v.w < mine);
        if (k < e) rank += (v.x == mine) + (k + 1 < e && v.y == mine) + (k + 2 < e && v.z == mine) + (k + 3 < e && v.w == mine);
      }
      for (int o = share >> 1; o > 0; o >>= 1) rank += __shfl_xor_sync(0xffffffffu, rank, o);
      if (sub == 0) s.into[e] = rank < removed ? s.best[e] : -1;
    }
  } else {
    for (int e = tid; e < na; e += nthr) s.into[e] = removed >= na ? s.best[e] : -1;
  }
  if (na <= 128) {
    for (int e = tid; e < nb; e += nthr) s.count[e] = 0;
    __syncthreads();
    for (int e0 = 0; e0 < na; e0 += step) {
      const int e = min(e0 + mine0, na - 1), to = s.into[e];
      int q = 0;
      if (to >= 0)
        for (int k = 4 * sub; k < e; k += 4 * share) {
          const int4 v = *reinterpret_cast<const int4*>(s.into + k);
          q += (v.x == to) + (k + 1 < e && v.y == to) + (k + 2 < e && v.z == to) + (k + 3 < e && v.w == to);
        }
      for (int o = share >> 1; o > 0; o >>= 1) q += __shfl_xor_sync(0xffffffffu, q, o);
      if (sub == 0 && e0 + mine0 < na) {
        const int i = s.tok[2 * e + par];
        if (to >= 0) atomicAdd(&s.count[to], 1);
        partner[i] = to < 0 ? -2 : s.tok[2 * to + 1 - par];
        place[i] = q;
      }
    }
    __syncthreads();
    for (int e = tid; e < nb; e += nthr) {
      const int i = s.tok[2 * e + 1 - par];
      partner[i] = -1;
      place[i] = s.count[e];
    }
    return;
  }
  const int parts = min(WindowLists::kParts, nthr >> 5), len = ((na + parts - 1) / parts + 31) & ~31;
  for (int k = tid; k < parts * nb; k += nthr) s.part[k] = 0;
  __syncthreads();
  if (warp < parts) {
    unsigned short* count = s.part + warp * nb;
    for (int base = warp * len; base < min(na, (warp + 1) * len); base += 32) {
      const int e = base + lane, to = e < na ? s.into[e] : -1;
      const unsigned int peers = __match_any_sync(0xffffffffu, to);
      const int before = to >= 0 ? count[to] : 0;
      __syncwarp();
      if (to >= 0 && lane == __ffs(peers) - 1) count[to] = (unsigned short)(before + __popc(peers));
      __syncwarp();
      if (e < na) s.best[e] = before + __popc(peers & ((1u << lane) - 1u));    // (its destination is in `into` by now)
    }
  }
  __syncthreads();
  for (int e = tid; e < nb; e += nthr) {
    int run = 0;
    for (int k = 0; k < parts; ++k) {
      const int c = s.part[k * nb + e];
      s.part[k * nb + e] = (unsigned short)run;
      run += c;
    }
    const int i = s.tok[2 * e + 1 - par];
    partner[i] = -1;
    place[i] = run;
  }
  __syncthreads();
  for (int e = tid; e < na; e += nthr) {
    const int i = s.tok[2 * e + par], to = s.into[e];
    partner[i] = to < 0 ? -2 : s.tok[2 * to + 1 - par];
    place[i] = to < 0 ? 0 : s.part[e / len * nb + to] + s.best[e];
  }
}

}  // namespace lkv
