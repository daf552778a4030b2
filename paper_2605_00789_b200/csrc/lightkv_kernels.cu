// liblightkv kernels, part 1: window build, fp32-FMA contractions (FD, xi), selection + merge map,
// weighted merge of hidden states, K/V merge-compaction.  sm_100a.
#include <algorithm>
#include <type_traits>

#include "launch.h"
#include "tc_common.cuh"
#include "windows.cuh"

namespace lkv {

__device__ inline void set_status(uint32_t* status, uint32_t bit) {
  if (status) atomicOr(status, bit);
}

// =====================================================================================================
// Window build ("Window partitioning", Step 1).  One CTA per sample.
// Every token gets its window id from its original grid position; tokens of a window are ranked in
// storage order (positions ascend with storage, so this is position order).  Rank l even -> set A
// (the paper's 1st, 3rd, ... token), odd -> set B.  The SOURCE nodes (the ones that may be merged away: set A,
// or set B in the reverse direction, g.src_par = 1) go to the a_* lists, the destinations to b_tok, window by
// window.
// Stable ranking without sorting: each warp owns a contiguous segment of the tokens and a private row
// of per-window counters; an exclusive prefix over the 32 rows gives every warp its starting rank.
// =====================================================================================================
__global__ void __launch_bounds__(1024)
window_build_kernel(Geometry g, const int* __restrict__ pos_all, const int* __restrict__ n_vis,
                    Workspace ws, uint32_t* status) {
  grid_dependency_wait();
  grid_launch_dependents();                    // in this order: see grid_dependency_sync
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nW = g.n_windows;
  uint16_t* cnt = reinterpret_cast<uint16_t*>(smem_raw);                        // [32][nW]
  int* wsum = reinterpret_cast<int*>(smem_raw + ((size_t(32) * nW * 2 + 15) & ~size_t(15)));  // [nW+1]
  int* asum = wsum + nW + 1;                                                    // [nW+1]

  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  int n = n_vis ? n_vis[b] : ws.cap_in;
  if (n > ws.cap_in) { n = ws.cap_in; if (tid == 0) set_status(status, LIGHTKV_STATUS_COUNT); }
  if (n < 0) n = 0;
  const int* pos = pos_all ? pos_all + size_t(b) * ws.cap_in : nullptr;
  int* tok_win = ws.tok_win + size_t(b) * ws.cap_in;
  int* tok_l = ws.tok_l + size_t(b) * ws.cap_in;
  int* a_tok = ws.a_tok + size_t(b) * ws.cap_a;
  int* a_win = ws.a_win + size_t(b) * ws.cap_a;
  int* b_tok = ws.b_tok + size_t(b) * ws.cap_b;
  unsigned long long* a_key = ws.a_key + size_t(b) * ws.cap_a;

  for (int i = tid; i < 32 * nW; i += blockDim.x) cnt[i] = 0;
  __syncthreads();

  const int seg = (n + 31) / 32;
  const int s0 = min(n, wp * seg), s1 = min(n, s0 + seg);

  // pass A: window id of every token, per-warp per-window counts
  for (int base = s0; base < s1; base += 32) {
    const int i = base + lane;
    const bool act = i < s1;
    const unsigned amask = __ballot_sync(0xffffffffu, act);
    if (act) {
      const int p = pos ? pos[i] : i;
      int w = window_of(g, p);
      const int prev = (i > 0) ? (pos ? pos[i - 1] : i - 1) : -1;
      if (w < 0 || p <= prev) { set_status(status, LIGHTKV_STATUS_POS_ORDER); if (w < 0) w = 0; }
      tok_win[i] = w;
      const unsigned peers = __match_any_sync(amask, w);
      if (lane == __ffs(peers) - 1) cnt[wp * nW + w] += (uint16_t)__popc(peers);
    }
    __syncwarp();
  }
  __syncthreads();

  // exclusive prefix over the 32 warp rows, window totals
  for (int w = tid; w < nW; w += blockDim.x) {
    int run = 0;
    for (int k = 0; k < 32; ++k) {
      const int c = cnt[k * nW + w];
      cnt[k * nW + w] = (uint16_t)run;
      run += c;
    }
    wsum[w] = run;
  }
  __syncthreads();

  // exclusive scans over windows: token offsets (wsum) and A-entry offsets (asum)
  if (wp == 0) {
    const int chunk = (nW + 31) / 32;
    const int lo = min(nW, lane * chunk), hi = min(nW, lo + chunk);
    int s = 0, sa = 0;
    for (int w = lo; w < hi; ++w) { s += wsum[w]; sa += (wsum[w] + 1 - g.src_par) >> 1; }
    int xs = s, xa = sa;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, xs, o), ta = __shfl_up_sync(0xffffffffu, xa, o);
      if (lane >= o) { xs += t; xa += ta; }
    }
    xs -= s; xa -= sa;
    for (int w = lo; w < hi; ++w) {
      const int c = wsum[w];
      wsum[w] = xs; asum[w] = xa;
      xs += c; xa += (c + 1 - g.src_par) >> 1;
    }
    if (lane == 31) { wsum[nW] = xs; asum[nW] = xa; }
  }
  __syncthreads();
  // A sample whose A or B nodes do not fit the plan's capacities (a subset of the grid handed to a plan that was
  // built for full grids) keeps all of its tokens: its windows are published empty, so no later kernel finds an
  // entry, a tile or a window size for it, nothing is indexed past a row, and the status word says so.
  const bool over = asum[nW] > ws.cap_a || wsum[nW] - asum[nW] > ws.cap_b;
  if (over && tid == 0) set_status(status, LIGHTKV_STATUS_COUNT);
  for (int w = tid; w <= nW; w += blockDim.x) {
    ws.win_off[size_t(b) * (nW + 1) + w] = over ? 0 : wsum[w];
    ws.a_off[size_t(b) * (nW + 1) + w] = over ? 0 : asum[w];
  }
  // pass B: local rank, A / B entry lists
  for (int base = s0; base < s1; base += 32) {
    const int i = base + lane;
    const bool act = i < s1;
    const unsigned amask = __ballot_sync(0xffffffffu, act);
    if (act) {
      const int w = tok_win[i];
      const unsigned peers = __match_any_sync(amask, w);
      const int before = cnt[wp * nW + w];
      __syncwarp(amask);
      if (lane == __ffs(peers) - 1) cnt[wp * nW + w] = (uint16_t)(before + __popc(peers));
      __syncwarp(amask);
      const int l = before + __popc(peers & ((1u << lane) - 1u));
      tok_l[i] = l;
      if ((l & 1) != g.src_par) {
        const int e = (wsum[w] - asum[w]) + (l >> 1);
        if (e < ws.cap_b) b_tok[e] = i;
      } else {
        const int e = asum[w] + (l >> 1);
        if (e < ws.cap_a) { a_tok[e] = i; a_win[e] = w; a_key[e] = ~0ull; }
      }
    }
    __syncwarp();
  }
}

cudaError_t launch_window_build(const LayerLaunch& L) {
  const int nW = L.geo.n_windows;
  const size_t smem = ((size_t(32) * nW * 2 + 15) & ~size_t(15)) + size_t(2) * (nW + 1) * sizeof(int);
  const cudaError_t e = ensure_dynamic_smem(window_build_kernel, 200 * 1024);
  if (e != cudaSuccess) return e;
  return launch_kernel(window_build_kernel, L.batch, 1024, smem, L.stream, 1, L.geo, L.a->pos, L.a->n_vis, L.ws, L.a->status);
}

// =====================================================================================================
// FD + best partner, fp32 FMA path (Eq. "similarity", Step 2).
// One CTA per (sample, tile of 32 A entries).  The B entries of the windows the tile touches are
// visited in chunks of 64; G = X_A X_B^T accumulates in registers over k-chunks of 32 staged in smem,
// squared norms accumulate from the same staged tiles.  Every A row then scans the FD of its own
// window's B entries in ascending order (strict <, so ties go to the lowest B index).
// =====================================================================================================
constexpr int FD_TA = 32, FD_TB = 64, FD_KC = 32;

template <typename T>
__device__ inline void load4(const T* p, float (&f)[4]);
template <>
__device__ inline void load4<float>(const float* p, float (&f)[4]) {
  const float4 v = *reinterpret_cast<const float4*>(p);
  f[0] = v.x; f[1] = v.y; f[2] = v.z; f[3] = v.w;
}
template <>
__device__ inline void load4<__nv_bfloat16>(const __nv_bfloat16* p, float (&f)[4]) {
  const uint2 v = *reinterpret_cast<const uint2*>(p);
  f[0] = __uint_as_float(v.x << 16); f[1] = __uint_as_float(v.x & 0xffff0000u);
  f[2] = __uint_as_float(v.y << 16); f[3] = __uint_as_float(v.y & 0xffff0000u);
}

template <typename T>
__global__ void __launch_bounds__(256)
fd_simt_kernel(const T* __restrict__ hidden, int64_t batch_stride, int64_t row_stride, const int* __restrict__ seq_start,
               int vis_begin, int d, int metric, Workspace ws) {
  grid_dependency_sync();
  __shared__ float As[FD_TA][FD_KC + 1];
  __shared__ float Bs[FD_TB][FD_KC + 1];
  __shared__ float Gs[FD_TA][FD_TB + 1];
  __shared__ float a_ss[FD_TA], b_ss[FD_TB];
  __shared__ int a_row[FD_TA], b_row[FD_TB], a_lo[FD_TA], a_hi[FD_TA];

  const int b = blockIdx.y, tid = threadIdx.x;
  const int nW = ws.n_windows;
  const int* win_off = ws.win_off + size_t(b) * (nW + 1);
  const int* a_off = ws.a_off + size_t(b) * (nW + 1);
  const int* a_tok = ws.a_tok + size_t(b) * ws.cap_a;
  const int* a_win = ws.a_win + size_t(b) * ws.cap_a;
  const int* b_tok = ws.b_tok + size_t(b) * ws.cap_b;
  const int n_a = a_off[nW];
  const int e0 = blockIdx.x * FD_TA;
  if (e0 >= n_a) return;
  const int ne = min(FD_TA, n_a - e0);
  const T* x = hidden + size_t(b) * batch_stride + size_t((seq_start ? seq_start[b] : 0) + vis_begin) * row_stride;

  if (tid < FD_TA) {
    if (tid < ne) {
      const int w = a_win[e0 + tid];
      a_row[tid] = a_tok[e0 + tid];
      a_lo[tid] = win_off[w] - a_off[w];
      a_hi[tid] = win_off[w + 1] - a_off[w + 1];
    } else {
      a_row[tid] = -1; a_lo[tid] = 0; a_hi[tid] = 0;
    }
  }
  __syncthreads();
  const int bb0 = a_lo[0], bb1 = a_hi[ne - 1];

  const int tx = tid & 15, ty = tid >> 4;            // 4 B columns x 2 A rows per thread
  float best_f = 3.0e38f;                            // threads < ne: running minimum of their A row
  int best_e = -1;                                   // ... and the B entry that attains it
  float ssa = 0.f;                                   // threads < FD_TA: squared norm of A row tid

  for (int cb = bb0; cb < bb1; cb += FD_TB) {
    const int nb = min(FD_TB, bb1 - cb);
    if (tid < FD_TB) b_row[tid] = tid < nb ? b_tok[cb + tid] : -1;
    float acc[2][4] = {};
    float ssb = 0.f;                                 // threads 32..95: squared norm of B row tid-32
    const bool first = (cb == bb0);
    __syncthreads();
    for (int k0 = 0; k0 < d; k0 += FD_KC) {
      {  // stage A tile: 32 x 32, 4 elements per thread
        const int r = tid >> 3, c = (tid & 7) * 4;
        float f[4] = {0.f, 0.f, 0.f, 0.f};
        if (a_row[r] >= 0 && k0 + c < d) load4<T>(x + size_t(a_row[r]) * row_stride + k0 + c, f);
#pragma unroll
        for (int j = 0; j < 4; ++j) As[r][c + j] = f[j];
      }
#pragma unroll
      for (int half = 0; half < 2; ++half) {  // stage B tile: 64 x 32
        const int r = (tid >> 3) + half * 32, c = (tid & 7) * 4;
        float f[4] = {0.f, 0.f, 0.f, 0.f};
        if (b_row[r] >= 0 && k0 + c < d) load4<T>(x + size_t(b_row[r]) * row_stride + k0 + c, f);
#pragma unroll
        for (int j = 0; j < 4; ++j) Bs[r][c + j] = f[j];
      }
      __syncthreads();
#pragma unroll 8
      for (int kk = 0; kk < FD_KC; ++kk) {
        const float a0 = As[2 * ty][kk], a1 = As[2 * ty + 1][kk];
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float bv = Bs[4 * tx + j][kk];
          acc[0][j] = fmaf(a0, bv, acc[0][j]);
          acc[1][j] = fmaf(a1, bv, acc[1][j]);
        }
      }
      if (first && tid < FD_TA) {
        for (int kk = 0; kk < FD_KC; ++kk) ssa = fmaf(As[tid][kk], As[tid][kk], ssa);
      } else if (tid >= 32 && tid < 32 + FD_TB) {
        for (int kk = 0; kk < FD_KC; ++kk) ssb = fmaf(Bs[tid - 32][kk], Bs[tid - 32][kk], ssb);
      }
      __syncthreads();
    }
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) Gs[2 * ty + i][4 * tx + j] = acc[i][j];
    if (first && tid < FD_TA) a_ss[tid] = ssa;
    if (tid >= 32 && tid < 32 + FD_TB) b_ss[tid - 32] = ssb;
    __syncthreads();
    if (tid < ne) {
      const int lo = max(a_lo[tid], cb), hi = min(a_hi[tid], cb + nb);
      const float na = sqrtf(a_ss[tid]);
      for (int e = lo; e < hi; ++e) {
        float fd;
        if (metric == LIGHTKV_FD_COSINE) {
          const float den = na * sqrtf(b_ss[e - cb]);
          fd = 1.0f - (den > 0.f ? Gs[tid][e - cb] / den : 0.f);
        } else {
          fd = fmaxf(fmaf(-2.0f, Gs[tid][e - cb], a_ss[tid] + b_ss[e - cb]), 0.f);   // |a|^2 + |b|^2 - 2 <a, b>
          if (metric == LIGHTKV_FD_L2) fd = sqrtf(fd);
        }
        if (fd < best_f) { best_f = fd; best_e = e; }
      }
    }
    __syncthreads();
  }
  if (tid < ne && best_e >= 0)
    ws.a_key[size_t(b) * ws.cap_a + e0 + tid] = ((unsigned long long)orderable(best_f) << 32) | (unsigned)best_e;
}

cudaError_t launch_fd_simt(const LayerLaunch& L) {
  const dim3 grid((L.ws.cap_a + FD_TA - 1) / FD_TA, L.batch);
  if (L.dtype == LIGHTKV_BF16)
    return launch_kernel(fd_simt_kernel<__nv_bfloat16>, grid, 256, 0, L.stream, 1,
                         static_cast<const __nv_bfloat16*>(L.a->hidden), L.a->hidden_batch_stride,
                         L.a->hidden_row_stride, L.a->seq_start, L.a->vis_begin, L.hidden, L.divergence, L.ws);
  return launch_kernel(fd_simt_kernel<float>, grid, 256, 0, L.stream, 1, static_cast<const float*>(L.a->hidden),
                       L.a->hidden_batch_stride, L.a->hidden_row_stride, L.a->seq_start, L.a->vis_begin, L.hidden,
                       L.divergence, L.ws);
}

// =====================================================================================================
// xi per head, fp32 FMA path (Eq. "attention-factor" with the causal softmax rows of Eq.
// "attention-matrix").  One CTA per (tile of 32 vision queries, head, sample), longest rows first.  Keys 0..s_i are
// visited in tiles of 32 with an online (running-maximum) softmax that carries two sums per row: all visible
// keys and the prompt keys J.  Output per head: sum_J / sum_all.  With a caller-supplied row
// log-sum-exp only the prompt keys are visited: sum_J exp(logit - lse).
// The eight warps of a CTA take every eighth tile of keys, on their own: a warp loads its keys 32 dimensions at a time
// (cp.async, the next chunk during this one), a lane holds 4 x 8 logits (12 shared-memory loads of 16 bytes per 128 FMAs)
// and keeps its own maximum and sums of its four queries; lanes and warps meet once, at the end.  Two CTAs per SM, for
// any head size.  Bound by latency: four warps per scheduler issue 0.6 instructions a clock (packed FMAs, half as many,
// take the same time).
// 2 x 576 queries x 8 heads of 128 in fp32: 38 us, the next stage with 317 queries 27; with four groups of 128 threads at
// a barrier per key tile of 64 (4 x 4 logits a lane) 60 and 33 (bf16, heads of 256: 152 -> 65); 8 x 8 logits a lane, two warps per scheduler: 43 and 33;
// the head dimension cut over the warps: 46 and 31; two CTAs of a cluster per query tile: 50 and 30.
// =====================================================================================================
constexpr int XI_TQ = 32, XI_TK = 32, XI_WARPS = 8, XI_DIMS = 32;
constexpr int XI_LD = XI_DIMS + 4;                       // pitch of a chunk's rows: eight of them in different banks
__host__ __device__ inline int xi_q_pitch(int dh) { return (dh + 7) / 8 * 8 + 4; }

template <typename T>
struct XiSimtArgs {
  const T* q; int64_t q_bs, q_hs, q_rs;
  const T* k; int64_t k_bs, k_hs, k_rs;
  const float* lse; int64_t lse_bs, lse_hs;        // caller's row log-sum-exp (ATTN_LSE) or nullptr
  float* lse_out; int64_t lse_out_bs, lse_out_hs;  // receives the row log-sum-exp (ATTN_FULL) or nullptr
  const int* n_vis;
  const int* seq_start;                            // first row of each sample in q, k, lse, lse_out (packed batches) or nullptr
  int vis_begin, n_text_after, bidirectional;
  int n_q_heads, n_kv_heads, dh;
  unsigned int sms;                                // SMs of the device
  int wait_first;                                  // as in the tensor-core kernel
  TextSet text;
};

template <typename T>
__global__ void __launch_bounds__(32 * XI_WARPS, 2)
xi_simt_kernel(XiSimtArgs<T> a, Workspace ws) {
  grid_launch_dependents();
  if (a.wait_first) grid_dependency_wait();              // else at the end: it reads nothing FD or the map write
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int dh = a.dh, ldq = xi_q_pitch(dh);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* ring = reinterpret_cast<float*>(smem_raw) + warp * 2 * XI_TK * XI_LD;            // [warps][2][XI_TK][XI_LD]
  float* Qs = reinterpret_cast<float*>(smem_raw) + XI_WARPS * 2 * XI_TK * XI_LD;          // [XI_TQ][ldq]

  // The queries with the most keys first.  Where every CTA is resident at once, two to an SM, the second half starts with
  // the fewest and hands its tiles to the warps in the other direction: the SMs, and the schedulers of an SM, have about
  // the same to do.
  const bool second = gridDim.x <= 2 * a.sms && blockIdx.x >= a.sms;
  const int item = second ? gridDim.x - 1 - (blockIdx.x - a.sms) : blockIdx.x;
  const int tiles = (ws.cap_in + XI_TQ - 1) / XI_TQ, heads = gridDim.x / tiles;           // (heads of all samples)
  const int b = item % heads / a.n_q_heads, h = item % heads % a.n_q_heads, t0 = (tiles - 1 - item / heads) * XI_TQ;
  const int n = a.n_vis ? min(a.n_vis[b], ws.cap_in) : ws.cap_in;
  if (t0 >= n) {
    grid_dependency_wait();
    return;
  }
  const int nq = min(XI_TQ, n - t0);
  const int hk = h / (a.n_q_heads / a.n_kv_heads);
  const int row0 = a.seq_start ? a.seq_start[b] : 0;
  const T* qh = a.q + size_t(b) * a.q_bs + size_t(h) * a.q_hs + size_t(row0) * a.q_rs;
  const T* kh = a.k + size_t(b) * a.k_bs + size_t(hk) * a.k_hs + size_t(row0) * a.k_rs;
  const float scale2 = 1.4426950408889634f / sqrtf((float)dh);      // logits in log2 units
  const int q_pos = a.vis_begin + t0;                                 // of the first query
  const int n_seq = a.vis_begin + n + a.n_text_after;                 // keys of this sample

  auto put = [](float* dst, const T* p, bool in) {      // four values, zeros if not `in`
    if constexpr (sizeof(T) == 4) {
      tc::cp_async16(tc::smem_u32(dst), p, in ? 16u : 0u);
    } else {
      float f[4] = {0.f, 0.f, 0.f, 0.f};
      if (in) load4<T>(p, f);
      *reinterpret_cast<float4*>(dst) = make_float4(f[0], f[1], f[2], f[3]);
    }
  };
  for (int idx = threadIdx.x; idx < XI_TQ * (dh / 4); idx += blockDim.x) {
    const int r = idx / (dh / 4), d = (idx - r * (dh / 4)) * 4;
    put(Qs + r * ldq + d, qh + size_t(q_pos + (r < nq ? r : 0)) * a.q_rs + d, r < nq);
  }
  // last key any row of the tile may see: its own (causal) or the sample's last (bidirectional)
  const int s_last = a.bidirectional ? n_seq - 1 : q_pos + nq - 1;
  const int key_lo = a.lse ? a.text.begin : 0;
  const int key_hi = a.lse ? min(a.text.end, s_last + 1) : s_last + 1;
  const int j_first = key_lo + (second ? XI_WARPS - 1 - warp : warp) * XI_TK;
  // the warp's next chunk: lane (lr, ld4) loads 16 bytes of the rows lr + 4 k
  const int lr = lane >> 3, ld4 = (lane & 7) * 4;
  int load_j = j_first, load_d = 0;
  auto load = [&](int st) {
    if (load_j < key_hi) {
      const int rows = load_d + ld4 < dh ? min(XI_TK, key_hi - load_j) : 0;
      const T* p = kh + size_t(load_j) * a.k_rs + load_d;
      const T* pr = p + size_t(lr) * a.k_rs + ld4;
      float* dst = ring + st * XI_TK * XI_LD + lr * XI_LD + ld4;
#pragma unroll
      for (int k = 0; k < XI_TK / 4; ++k) {
        const bool in = lr + 4 * k < rows;
        put(dst + 4 * k * XI_LD, in ? pr : p, in);
        pr += 4 * a.k_rs;
      }
      load_d += XI_DIMS;
      if (load_d >= dh) { load_d = 0; load_j += XI_WARPS * XI_TK; }
    }
    tc::cp_async_commit();
  };
  tc::cp_async_commit();
  load(0);
  tc::cp_async_wait<1>();
  __syncthreads();                                      // the queries are there

  const int tx = lane & 3, ty = lane >> 2;              // queries ty + 8 i, keys tx + 4 j
  float m_run[4], l_all[4], l_txt[4];                   // maximum in log2 units (given log-sum-exp: that); sums
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    m_run[i] = -INFINITY; l_all[i] = 0.f; l_txt[i] = 0.f;
    if (a.lse) {
      const int r = ty + 8 * i;
      m_run[i] = r < nq ? a.lse[size_t(b) * a.lse_bs + size_t(h) * a.lse_hs + row0 + q_pos + r] * 1.4426950408889634f : 0.f;
    }
  }
  for (int j0 = j_first, st = 0; j0 < key_hi; j0 += XI_WARPS * XI_TK) {
    float acc[4][8] = {};
    for (int d0 = 0; d0 < dh; d0 += XI_DIMS, st ^= 1) {
      load(st ^ 1);
      tc::cp_async_wait<1>();
      __syncwarp();                                     // the chunk is there for all lanes
      const float* Kt = ring + st * XI_TK * XI_LD + tx * XI_LD;
      const float* Qt = Qs + ty * ldq + d0;
      const int dims = min(XI_DIMS, dh - d0);
#pragma unroll 1
      for (int kk = 0; kk < dims; kk += 4) {
        float4 q[4];
#pragma unroll
        for (int i = 0; i < 4; ++i) q[i] = *reinterpret_cast<const float4*>(Qt + 8 * i * ldq + kk);
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const float4 k = *reinterpret_cast<const float4*>(Kt + 4 * j * XI_LD + kk);
#pragma unroll
          for (int i = 0; i < 4; ++i)
            acc[i][j] = fmaf(q[i].w, k.w, fmaf(q[i].z, k.z, fmaf(q[i].y, k.y, fmaf(q[i].x, k.x, acc[i][j]))));
        }
      }
      __syncwarp();                                     // every lane has read it: it is filled next
    }
    const unsigned tile_text = a.text.mask32(j0), text = tile_text >> tx;                  // bits 4 j: this lane's keys
    const bool whole = j0 + XI_TK <= key_hi && (a.bidirectional || j0 + XI_TK - 1 <= q_pos);   // every query sees every key
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int last = min(a.bidirectional ? n_seq - 1 : q_pos + ty + 8 * i, key_hi - 1) - j0 - tx;   // visible: 4 j <= last
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = whole || 4 * j <= last ? acc[i][j] * scale2 : -INFINITY;
      float ref = m_run[i];
      if (!a.lse) {
#pragma unroll
        for (int j = 0; j < 8; ++j) ref = fmaxf(ref, acc[i][j]);
        const float old = m_run[i];
        m_run[i] = ref;
        if (ref == -INFINITY) ref = 0.f;                // none of the lane's keys is visible so far: all terms are 0
        const float resc = exp2f(old - ref);
        l_all[i] *= resc;
        l_txt[i] *= resc;
      }
#pragma unroll
      for (int j = 0; j < 8; ++j) acc[i][j] = exp2f(acc[i][j] - ref);
#pragma unroll
      for (int j = 0; j < 8; ++j) l_all[i] += acc[i][j];
      if (tile_text)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if ((text >> (4 * j)) & 1u) l_txt[i] += acc[i][j];
    }
  }
  // ---- the lanes' and the warps' results of a query meet
  __shared__ float s_m[XI_WARPS][XI_TQ], s_all[XI_WARPS][XI_TQ], s_txt[XI_WARPS][XI_TQ];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    float m = m_run[i];
    if (!a.lse) {
#pragma unroll
      for (int o = 2; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
      const float f = m == -INFINITY ? 0.f : exp2f(m_run[i] - m);
      l_all[i] *= f;
      l_txt[i] *= f;
    }
#pragma unroll
    for (int o = 2; o > 0; o >>= 1) {
      l_all[i] += __shfl_xor_sync(0xffffffffu, l_all[i], o);
      l_txt[i] += __shfl_xor_sync(0xffffffffu, l_txt[i], o);
    }
    if (tx == 0) { s_m[warp][ty + 8 * i] = m; s_all[warp][ty + 8 * i] = l_all[i]; s_txt[warp][ty + 8 * i] = l_txt[i]; }
  }
  tc::cp_async_wait<0>();
  __syncthreads();
  const int r = threadIdx.x;
  if (r < nq) {
    float m = s_m[0][r], all = 0.f, txt = 0.f;          // finite without a given log-sum-exp: key 0 is visible to every query
#pragma unroll
    for (int k = 1; k < XI_WARPS; ++k) m = fmaxf(m, s_m[k][r]);
#pragma unroll
    for (int k = 0; k < XI_WARPS; ++k) {
      const float f = a.lse ? 1.f : exp2f(s_m[k][r] - m);
      all += s_all[k][r] * f;
      txt += s_txt[k][r] * f;
    }
    ws.xi_h[(size_t(b) * ws.cap_in + t0 + r) * a.n_q_heads + h] = a.lse ? txt : txt / all;
    if (a.lse_out)
      a.lse_out[size_t(b) * a.lse_out_bs + size_t(h) * a.lse_out_hs + row0 + q_pos + r] = (m + log2f(all)) * 0.6931471805599453f;
  }
  grid_dependency_wait();
}

template <typename T>
static cudaError_t launch_xi_simt_t(const LayerLaunch& L, bool wait_first) {
  const lightkv_layer_args_t* a = L.a;
  const int dh = L.head_dim;
  const size_t smem = size_t(XI_WARPS * 2 * XI_TK * XI_LD + XI_TQ * xi_q_pitch(dh)) * sizeof(float);   // at most 105 KB: two CTAs per SM
  const unsigned ctas = unsigned((L.ws.cap_in + XI_TQ - 1) / XI_TQ) * unsigned(L.n_q_heads) * unsigned(L.batch);
  XiSimtArgs<T> x;
  x.q = static_cast<const T*>(a->q); x.q_bs = a->q_batch_stride; x.q_hs = a->q_head_stride; x.q_rs = a->q_row_stride;
  x.k = static_cast<const T*>(a->k); x.k_bs = a->k_batch_stride; x.k_hs = a->k_head_stride; x.k_rs = a->k_row_stride;
  x.lse = L.xi_mode == LIGHTKV_XI_ATTN_LSE ? a->lse : nullptr; x.lse_bs = a->lse_batch_stride; x.lse_hs = a->lse_head_stride;
  x.lse_out = L.xi_mode == LIGHTKV_XI_ATTN_FULL ? a->lse_out : nullptr;
  x.lse_out_bs = a->lse_out_batch_stride; x.lse_out_hs = a->lse_out_head_stride;
  x.n_vis = a->n_vis; x.seq_start = a->seq_start;
  x.vis_begin = a->vis_begin; x.n_text_after = a->n_text_after; x.bidirectional = a->bidirectional;
  x.n_q_heads = L.n_q_heads; x.n_kv_heads = L.n_kv_heads; x.dh = dh; x.sms = sm_count();
  x.wait_first = wait_first ? 1 : 0;
  x.text = L.text;
  const cudaError_t e = ensure_dynamic_smem(xi_simt_kernel<T>, 108 * 1024);
  if (e != cudaSuccess) return e;
  return launch_kernel(xi_simt_kernel<T>, dim3(ctas), 32 * XI_WARPS, smem, L.stream, 1, x, L.ws);
}

cudaError_t launch_xi_simt(const LayerLaunch& L, bool wait_first) {
  return L.dtype == LIGHTKV_BF16 ? launch_xi_simt_t<__nv_bfloat16>(L, wait_first) : launch_xi_simt_t<float>(L, wait_first);
}

// ---- xi of a token, the sum over its heads.  They are added in one order everywhere, so that xi and the weights have the same
// bits whichever kernels a call's size, workspace or map event select: head h counts to sum h % 32, in ascending order, and these
// 32 meet as a warp's lanes do in a butterfly over 1, 2, 4, 8 and 16.

// One token, in every lane; the lanes share the heads, two loads in flight.
__device__ __forceinline__ float warp_xi(const float* x, int heads, int lane) {
  float v = 0.f;
#pragma unroll 1
  for (int h = lane; h < heads; h += 64) {
    const float v0 = x[h], v1 = h + 32 < heads ? x[h + 32] : 0.f;
    v = (v + v0) + v1;
  }
#pragma unroll
  for (int o = 1; o <= 16; o <<= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Of eight values a lane, summed over the eight lanes that differ in bits 0 to 2 (first over 1, then 2 and 4): lane l gets value
// xi_value(l & 7).
__host__ __device__ constexpr int xi_value(int l) { return (l & 1) << 2 | (l & 2) | (l & 4) >> 2; }
__device__ __forceinline__ float sum_eight(float (&p)[8], int lane) {
#pragma unroll
  for (int o = 1, left = 4; o <= 4; o <<= 1, left >>= 1)
#pragma unroll
    for (int t = 0; t < left; ++t) {
      const float give = lane & o ? p[t] : p[t + left], keep = lane & o ? p[t + left] : p[t];
      p[t] = keep + __shfl_xor_sync(0xffffffffu, give, o);
    }
  return p[0];
}

// One token by a thread: sixteen heads at a time, groups of four pair by pair.  (Little code and few registers: with all groups
// unrolled, eight loads in flight or a warp's lanes over its tokens' heads a map takes 0.5 to 1.5 us more.)
__device__ __forceinline__ float token_xi(const float* x, int heads) {
  const bool quads = (heads & 3) == 0;                      // (rows of four floats are 16-byte aligned)
  float sum = 0.f;
#pragma unroll 1
  for (int h = 0; h < min(heads, 32); h += 16) {
    float4 s[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) s[m] = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 1
    for (int k = h; k < heads; k += 32) {
      float4 v[4];
      if (quads) {                                          // (clamped, not left out: a load behind a branch waits for the one before)
#pragma unroll
        for (int m = 0; m < 4; ++m) v[m] = *reinterpret_cast<const float4*>(x + min(k + 4 * m, heads - 4));
#pragma unroll
        for (int m = 1; m < 4; ++m)
          if (k + 4 * m >= heads) v[m] = make_float4(0.f, 0.f, 0.f, 0.f);
      } else {
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int c = k + 4 * m, last = heads - 1;
          v[m] = make_float4(x[min(c, last)], x[min(c + 1, last)], x[min(c + 2, last)], x[min(c + 3, last)]);
        }
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          const int c = k + 4 * m;
          v[m] = make_float4(c < heads ? v[m].x : 0.f, c + 1 < heads ? v[m].y : 0.f, c + 2 < heads ? v[m].z : 0.f, c + 3 < heads ? v[m].w : 0.f);
        }
      }
#pragma unroll
      for (int m = 0; m < 4; ++m) { s[m].x += v[m].x; s[m].y += v[m].y; s[m].z += v[m].z; s[m].w += v[m].w; }
    }
    float q[4];
#pragma unroll
    for (int m = 0; m < 4; ++m) q[m] = (s[m].x + s[m].y) + (s[m].z + s[m].w);
    sum += (q[0] + q[1]) + (q[2] + q[3]);
  }
  return sum;
}

// =====================================================================================================
// Selection + merge map (Steps 2-5).  One cluster of 1-8 CTAs per sample (about a token per thread); every
// CTA keeps a contiguous range of the sample's tokens through all phases, phases that read what other
// threads wrote are separated by cluster barriers, prefix sums cross the cluster through distributed shared
// memory.
//   1  xi = sum over heads (token_xi; or given / uniform); every source token (local rank parity src_par): r =
//      removal_count(n_w), selected iff it is among the r entries of its window with the smallest
//      (FD, index) (rank by counting 32-bit keys; skipped when r = |A|); a selected token takes its best B
//   2  survivors (all B, unselected A) get consecutive output slots in storage (= position) order: dst,
//      pos_out, and a group of one member each
//   3  a merged token joins its partner's group (integer atomic on the size); its place in the group is
//      the number of earlier entries of its window with the same partner
//   4  group sizes -> grp_off (scan)
//   5  grp_src: the survivor first, then its merged A tokens in entry order
//   6  weights xi_i / sum over the group, the sum taken in that fixed order
// =====================================================================================================
struct SelectArgs {
  int n_q_heads, xi_mode, cap_out, src_par;
  double keep;
  const int* n_vis;
  const int* pos;
  const float* xi_in;
  int* n_vis_out;
  int* pos_out;
  int* dst;
  float* weight;
  int* grp_off;
  int* grp_src;
  float* xi_out;
  uint32_t* status;
};

// exclusive scan of one value per thread across the CTA; returns the exclusive prefix, total in *total
__device__ inline int block_exclusive_scan(int v, int* warp_sums /* [33] smem */, int* total) {
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
  int x = v;
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += t;
  }
  __syncthreads();                       // warp_sums may still be read from the previous call
  if (lane == 31) warp_sums[wp] = x;
  __syncthreads();
  if (wp == 0) {
    int s = lane < nwarps ? warp_sums[lane] : 0;
    const int own = s;
    for (int o = 1; o < 32; o <<= 1) {
      const int t = __shfl_up_sync(0xffffffffu, s, o);
      if (lane >= o) s += t;
    }
    warp_sums[lane] = s - own;
    if (lane == 31) warp_sums[32] = s;
  }
  __syncthreads();
  *total = warp_sums[32];
  return warp_sums[wp] + x - v;
}

// CLUSTER = false: one CTA per sample, plain launch, block barriers only.
template <bool CLUSTER>
__global__ void __launch_bounds__(1024) select_map_kernel(Workspace ws, SelectArgs a) {
  grid_dependency_sync();
  __shared__ int warp_sums[33];
  __shared__ int cta_total[2];                  // survivors / group members counted by this CTA
  const int cs = CLUSTER ? (int)tc::cluster_nctarank() : 1, rank = CLUSTER ? (int)tc::cluster_ctarank() : 0;
  auto sync_all = [&]() { if (CLUSTER) tc::cluster_sync(); else __syncthreads(); };
  const int b = blockIdx.x / cs, tid = threadIdx.x, nthr = blockDim.x;
  const int gtid = rank * nthr + tid;                        // thread index inside the cluster
  const int nW = ws.n_windows;
  int n = a.n_vis ? min(a.n_vis[b], ws.cap_in) : ws.cap_in;
  if (n < 0) n = 0;
  const int* win_off = ws.win_off + size_t(b) * (nW + 1);
  const int* a_off = ws.a_off + size_t(b) * (nW + 1);
  const int* tok_win = ws.tok_win + size_t(b) * ws.cap_in;
  const int* tok_l = ws.tok_l + size_t(b) * ws.cap_in;
  const unsigned long long* a_key = ws.a_key + size_t(b) * ws.cap_a;
  const int* b_tok = ws.b_tok + size_t(b) * ws.cap_b;
  float* xi = ws.xi + size_t(b) * ws.cap_in;
  int* partner = ws.partner + size_t(b) * ws.cap_in;
  int* slot = ws.slot + size_t(b) * ws.cap_in;
  int* a_partner = ws.a_partner + size_t(b) * ws.cap_a;
  const int* pos = a.pos ? a.pos + size_t(b) * ws.cap_in : nullptr;
  int* dst = a.dst + size_t(b) * ws.cap_in;
  float* weight = a.weight + size_t(b) * ws.cap_in;
  int* grp_off = a.grp_off + size_t(b) * (a.cap_out + 1);
  int* grp_src = a.grp_src + size_t(b) * ws.cap_in;
  int* pos_out = a.pos_out + size_t(b) * a.cap_out;

  // Every CTA of the cluster owns a contiguous range of the sample's tokens; a thread keeps the same tokens
  // in every phase, so what it wrote for a token it may read back without a barrier.
  const int chunk = (n + cs - 1) / cs, lo = min(n, rank * chunk), hi = min(n, lo + chunk);

  // Exclusive scan of `value(i)` over the cluster: CTA `rank` owns [s_lo, s_hi) (at most s_chunk long, the
  // same bound in every CTA), counts it, learns the ranges before it through distributed shared memory,
  // then scans it.  emit(i, prefix) is called for every i; returns the grand total.
  auto cluster_scan = [&](int s_lo, int s_hi, int s_chunk, int which, auto value, auto emit) {
    int before = 0, grand = 0;
    auto exchange = [&](int mine) {
      if (tid == 0) cta_total[which] = mine;
      tc::cluster_sync();
      for (int j = 0; j < cs; ++j) {
        const int t = (int)tc::ld_cluster_u32(tc::map_to_cta(tc::smem_u32(&cta_total[which]), j));
        if (j < rank) before += t;
        grand += t;
      }
    };
    if (s_chunk <= nthr) {                              // one value per thread: a single pass
      const int i = s_lo + tid;
      int total;
      const int ex = block_exclusive_scan(i < s_hi ? value(i) : 0, warp_sums, &total);
      if (CLUSTER) exchange(total); else grand = total;
      if (i < s_hi) emit(i, before + ex);
      return grand;
    }
    if (CLUSTER) {
      int mine = 0;
      for (int base = s_lo; base < s_hi; base += nthr) {
        const int i = base + tid;
        int total;
        block_exclusive_scan(i < s_hi ? value(i) : 0, warp_sums, &total);
        mine += total;
      }
      exchange(mine);
    }
    int carry = before;
    for (int base = s_lo; base < s_hi; base += nthr) {
      const int i = base + tid;
      int total;
      const int ex = block_exclusive_scan(i < s_hi ? value(i) : 0, warp_sums, &total);
      if (i < s_hi) emit(i, carry + ex);
      carry += total;
    }
    return CLUSTER ? grand : carry;
  };

  // phase 1: xi of every token; every A token (even local rank, entry a_off[w] + l / 2) decides whether it is
  // among the r lowest-FD entries of its window and, if so, takes the partner FD found for it
  const uint32_t* key_word = reinterpret_cast<const uint32_t*>(a_key);   // [2e]: best B entry, [2e + 1]: orderable FD
  for (int i = lo + tid; i < hi; i += nthr) {
    float v;
    if (a.xi_mode == LIGHTKV_XI_GIVEN) v = a.xi_in[size_t(b) * ws.cap_in + i];
    else if (a.xi_mode == LIGHTKV_XI_UNIFORM) v = 1.0f;
    else v = token_xi(ws.xi_h + (size_t(b) * ws.cap_in + i) * a.n_q_heads, a.n_q_heads);
    xi[i] = v;
    if (a.xi_out) a.xi_out[size_t(b) * ws.cap_in + i] = v;
    int p = -1;
    const int l = tok_l[i];
    if ((l & 1) == a.src_par) {                        // a source node
      const int w = tok_win[i];
      const int e_lo = a_off[w], e_hi = a_off[w + 1], e = e_lo + (l >> 1);
      if (e < ws.cap_a) {
        const int r = removal_count(win_off[w + 1] - win_off[w], a.keep, a.src_par);
        bool sel;
        if (r <= 0) sel = false;
        else if (r >= e_hi - e_lo) sel = true;
        else {
          // rank in the order (lowest FD, A entry index): entries before e win ties, entries after e lose them
          const uint32_t mine = key_word[2 * e + 1];
          int rk = 0;
          for (int e2 = e_lo; e2 < e; ++e2) rk += (key_word[2 * e2 + 1] <= mine);
          for (int e2 = e + 1; e2 < e_hi; ++e2) rk += (key_word[2 * e2 + 1] < mine);
          sel = rk < r;
        }
        const uint32_t best_e = key_word[2 * e];
        p = (sel && best_e != 0xffffffffu) ? b_tok[best_e] : -1;
        a_partner[e] = p;                              // entry-indexed copy: phase 3 counts over it in order
      }
    }
    partner[i] = p;
  }

  // phase 2: output slot of every surviving token (its own tokens: no barrier needed before); the survivor
  // opens its group with one member
  const int survivors = cluster_scan(lo, hi, chunk, 0, [&](int i) { return partner[i] < 0 ? 1 : 0; },
                                     [&](int i, int prefix) {
                                       if (partner[i] >= 0) return;
                                       slot[i] = prefix;
                                       dst[i] = prefix;
                                       if (prefix >= a.cap_out) return;
                                       pos_out[prefix] = pos ? pos[i] : i;
                                       grp_off[prefix] = 1;
                                     });
  const int n_out = min(survivors, a.cap_out);
  if (gtid == 0) {
    a.n_vis_out[b] = n_out;
    if (survivors > a.cap_out) set_status(a.status, LIGHTKV_STATUS_COUNT);
  }
  sync_all();

  // phase 3: a merged token joins the group of its partner; its place in the group is the number of earlier
  // entries of its window with the same partner (kept in slot[], which a merged token does not use otherwise)
  for (int i = lo + tid; i < hi; i += nthr) {
    const int p = partner[i];
    if (p < 0) continue;
    const int o = slot[p];
    dst[i] = o;
    const int e_lo = a_off[tok_win[i]], e = e_lo + (tok_l[i] >> 1);
    int rk = 0;
    for (int e2 = e_lo; e2 < e; ++e2) rk += (a_partner[e2] == p);
    slot[i] = rk;
    if (o < a.cap_out) atomicAdd(&grp_off[o], 1);
  }
  sync_all();

  // phase 4: group sizes -> group offsets
  const int chunk_o = (n_out + cs - 1) / cs, lo_o = min(n_out, rank * chunk_o), hi_o = min(n_out, lo_o + chunk_o);
  const int members = cluster_scan(lo_o, hi_o, chunk_o, 1, [&](int o) { return grp_off[o]; },
                                   [&](int o, int prefix) { grp_off[o] = prefix; });
  if (gtid == 0) grp_off[n_out] = members;
  sync_all();

  // phase 5: member lists, the surviving token first, then the merged ones in entry order
  for (int i = lo + tid; i < hi; i += nthr) {
    const int o = dst[i];
    if (o >= a.cap_out) continue;
    grp_src[grp_off[o] + (partner[i] < 0 ? 0 : 1 + slot[i])] = i;
  }
  sync_all();

  // phase 6: weights xi_i / (sum of xi over the group), the sum taken in member order
  for (int i = lo + tid; i < hi; i += nthr) {
    if (partner[i] >= 0) continue;
    const int o = slot[i];
    if (o >= a.cap_out) continue;
    const int g0 = grp_off[o], g1 = grp_off[o + 1];
    float den = 0.f;
    for (int c = g0; c < g1; ++c) den += xi[grp_src[c]];
    if (den >= 1e-30f) {
      for (int c = g0; c < g1; ++c) { const int t = grp_src[c]; weight[t] = xi[t] / den; }
    } else {
      set_status(a.status, LIGHTKV_STATUS_ZERO_WEIGHT);
      for (int c = g0; c < g1; ++c) weight[grp_src[c]] = 1.0f / (float)(g1 - g0);
    }
  }
}

cudaError_t launch_select_map(const LayerLaunch& L) {
  const lightkv_layer_args_t* a = L.a;
  SelectArgs s;
  s.n_q_heads = L.n_q_heads; s.xi_mode = L.xi_mode; s.cap_out = L.ws.cap_out; s.keep = L.keep;
  s.src_par = L.geo.src_par;
  s.n_vis = a->n_vis; s.pos = a->pos; s.xi_in = a->xi; s.n_vis_out = a->n_vis_out; s.pos_out = a->pos_out;
  s.dst = a->dst; s.weight = a->weight; s.grp_off = a->grp_off; s.grp_src = a->grp_src;
  s.xi_out = a->xi_out; s.status = a->status;
  // one cluster per sample: 1, 2, 4 or 8 CTAs of 1024 threads, about one token per thread
  const int cs = L.ws.cap_in <= 1024 ? 1 : (L.ws.cap_in <= 2048 ? 2 : (L.ws.cap_in <= 4096 ? 4 : 8));
  if (cs == 1) return launch_kernel(select_map_kernel<false>, L.batch, 1024, 0, L.stream, 1, L.ws, s);
  return launch_kernel(select_map_kernel<true>, L.batch * cs, 1024, 0, L.stream, cs, L.ws, s);
}

// =====================================================================================================
// Merge map behind the streaming FD kernel, which left every token's partner and its place (see Workspace), or, with
// SELECT, behind the tiled one, which left the windows' tokens and keys: the CTAs of a sample then first take its windows
// in turn and select.  Groups, slots and positions need no xi: where xi comes from attention the kernel runs beside the xi
// kernel and leaves the weights to those behind it (weights_kernel, merge_rows_kernel); given or uniform xi is at hand
// (WEIGHTS).  One
// cluster of 1-8 CTAs per sample, TPT consecutive tokens per thread, everything between the first loads and the last
// stores in registers and (distributed) shared memory:
//   1  survivors and group sizes are counted in ONE pair of prefix sums: a survivor's slot, and the offset of its group
//      (its members are 1 + place tokens)
//   2  a merged token reads its partner's slot and offset from the CTA that owns it (WEIGHTS: and puts its index and xi at
//      its place in that CTA's member list; groups of one CTA's survivors are one contiguous range)
//   3  WEIGHTS: xi_i / sum over the group, the sum taken in member order (survivor first)
// Bound by latency: one round trip to L2 for the loads, three cluster barriers, one round of stores: 1.6 us from its wait to
// its end for 576 tokens, 2 for 16 x 432, 4 to 8 for 2880 (5.6, 7 and 10.5 when it also summed xi, behind the xi kernel).  A
// merged token that would need a kernel-wide search for its group costs one remote read here, because the streaming FD
// kernel holds whole windows.
// (select_map_kernel, which starts from keys, takes six dependent rounds through L2.)
// =====================================================================================================
// The weight of a member with `xi` in a group of `size` whose sum is `den`.
__device__ __forceinline__ float member_weight(float xi, float den, int size) {
  return den >= 1e-30f ? xi / den : 1.0f / (float)size;
}

struct MapArgs {
  int xi_mode, cap_in, cap_out, cap_a, cap_b, n_grid;
  const float* xi_in;
  const float* xi_h;                   // WEIGHTS, xi from attention: [B, cap_in, H]
  int n_q_heads;
  const int* n_vis;
  const int* pos;
  int* partner;
  int* place;
  const unsigned long long* key;       // SELECT: [B, blocks, cap_in]
  const int* win_tok;                  // SELECT: [B, n_windows, max_cell + 1]
  int blocks, max_cell, n_windows, src_par;
  double keep;
  int* n_vis_out;
  int* pos_out;
  int* dst;
  int* grp_off;
  int* grp_src;
  float* weight;
  float* xi_out;
  uint32_t* status;
};

template <bool CLUSTER, int TPT, bool SELECT, bool WEIGHTS>
__global__ void __launch_bounds__(1024) map_kernel(const __grid_constant__ MapArgs a) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int nthr = blockDim.x, tid = threadIdx.x, lane = tid & 31, wp = tid >> 5;
  const int span = nthr * TPT;                              // tokens a CTA can own
  int* s_slot = reinterpret_cast<int*>(smem_raw);           // [span] slot of an owned survivor
  int* s_off = s_slot + span;                               // [span] offset of its group
  int* m_tok = s_off + span;                                // WEIGHTS: [cap_in] member list: token index
  float* m_xi = reinterpret_cast<float*>(m_tok + a.cap_in); // WEIGHTS: [cap_in] ... and its xi
  __shared__ int base_off[8];                               // WEIGHTS: first member offset of every CTA
  __shared__ int warp_sums[2][33];
  __shared__ int cta_total[3];                              // survivors, members, sources of this CTA
  const int cs = CLUSTER ? (int)tc::cluster_nctarank() : 1, rank = CLUSTER ? (int)tc::cluster_ctarank() : 0;
  auto sync_all = [&]() { if (CLUSTER) tc::cluster_sync(); else __syncthreads(); };
  const int b = blockIdx.x / cs;
  int n = a.n_vis ? a.n_vis[b] : a.cap_in;
  if (n > a.cap_in) { n = a.cap_in; if (rank == 0 && tid == 0) set_status(a.status, LIGHTKV_STATUS_COUNT); }
  if (n < 0) n = 0;
  const size_t row = size_t(b) * a.cap_in;
  const int chunk = ((n + cs - 1) / cs + TPT - 1) / TPT * TPT;   // tokens per CTA (whole threads)
  const int lo = min(n, rank * chunk), hi = min(n, lo + chunk);
  const int i0 = lo + tid * TPT;

  if (SELECT) {
    const WindowLists lists = WindowLists::at(smem_raw, a.max_cell);          // (before the arrays above are in use)
    for (int w = rank; w < a.n_windows; w += cs) {
      const int* win_tok = a.win_tok + (size_t(b) * a.n_windows + w) * (a.max_cell + 1);
      const int nw = win_tok[0], par = a.src_par, na = (nw + 1 - par) >> 1, nb = nw - na;
      for (int l = tid; l < nw; l += nthr) lists.tok[l] = win_tok[1 + l];
      // (keys by window and source, asked for before the window's tokens and their number are there: no faster, and more keys
      // than tokens where windows differ in size)
      const int removed = nb > 0 ? removal_count(nw, a.keep, par) : 0, blocks = removed > 0 ? min(a.blocks, (nb + kFdTile - 1) / kFdTile) : 0;
      for (int e = tid; e < na; e += nthr) {
        const unsigned long long* k = a.key + size_t(b) * a.blocks * a.cap_in + win_tok[1 + 2 * e + par];
        unsigned long long key = ~0ull;
        for (int ib = 0; ib < blocks; ib += 4) {
          unsigned long long v[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) v[j] = ib + j < blocks ? k[size_t(ib + j) * a.cap_in] : ~0ull;
#pragma unroll
          for (int j = 0; j < 4; ++j) key = min(key, v[j]);
        }
        lists.key[e] = (unsigned int)(key >> 32);
        lists.best[e] = key_partner(key, nb);
      }
      __syncthreads();
      select_window(lists, nw, removed, par, a.partner + row, a.place + row);
      __syncthreads();
    }
    sync_all();
  }

  // ---- loads
  int prt[TPT], plc[TPT], ps[TPT];
  float xi[TPT];
  bool bad = false;
#pragma unroll
  for (int j = 0; j < TPT; ++j) {
    const int i = i0 + j;
    prt[j] = -1; plc[j] = 0; ps[j] = i; xi[j] = 1.0f;
    if (i < hi) {
      if (WEIGHTS && a.xi_mode == LIGHTKV_XI_GIVEN) xi[j] = a.xi_in[row + i];
      if (WEIGHTS && a.xi_h) xi[j] = token_xi(a.xi_h + (row + i) * a.n_q_heads, a.n_q_heads);
      prt[j] = __ldcg(a.partner + row + i);
      plc[j] = __ldcg(a.place + row + i);
      if (a.pos) {
        ps[j] = a.pos[row + i];
        bad = bad || ps[j] <= (i > 0 ? a.pos[row + i - 1] : -1) || ps[j] >= a.n_grid;
      } else {
        bad = bad || i >= a.n_grid;
      }
    }
  }
  if (__any_sync(0xffffffffu, bad) && lane == 0) set_status(a.status, LIGHTKV_STATUS_POS_ORDER);

  // ---- survivors and group members in front of this thread
  int ns = 0, nm = 0, nsrc = 0;
#pragma unroll
  for (int j = 0; j < TPT; ++j)
    if (i0 + j < hi) {
      if (prt[j] < 0) { ++ns; nm += 1 + plc[j]; }
      if (prt[j] != -1) ++nsrc;
    }
  int xs = ns, xm = nm;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int ts = __shfl_up_sync(0xffffffffu, xs, o), tm = __shfl_up_sync(0xffffffffu, xm, o);
    if (lane >= o) { xs += ts; xm += tm; }
  }
  nsrc = __reduce_add_sync(0xffffffffu, nsrc);
  if (tid < 3) cta_total[tid] = 0;
  if (lane == 31) { warp_sums[0][wp] = xs; warp_sums[1][wp] = xm; }
  __syncthreads();
  if (lane == 0 && nsrc) atomicAdd(&cta_total[2], nsrc);
  if (wp == 0) {
    const int nw = nthr >> 5;
    int s = lane < nw ? warp_sums[0][lane] : 0, m = lane < nw ? warp_sums[1][lane] : 0;
    const int own_s = s, own_m = m;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int ts = __shfl_up_sync(0xffffffffu, s, o), tm = __shfl_up_sync(0xffffffffu, m, o);
      if (lane >= o) { s += ts; m += tm; }
    }
    warp_sums[0][lane] = s - own_s;
    warp_sums[1][lane] = m - own_m;
    if (lane == 31) { cta_total[0] = s; cta_total[1] = m; }
  }
  sync_all();
  int before_s = 0, before_m = 0, survivors = 0, members = 0, sources = 0;
  if (CLUSTER) {
    int total[8][3];                                        // all of the cluster's counts in flight
#pragma unroll
    for (int j = 0; j < 8; ++j)
#pragma unroll
      for (int k = 0; k < 3; ++k)
        total[j][k] = j < cs ? (int)tc::ld_cluster_u32(tc::map_to_cta(tc::smem_u32(&cta_total[k]), j)) : 0;
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      if (j < rank) { before_s += total[j][0]; before_m += total[j][1]; }
      if (WEIGHTS && tid == 0) base_off[j] = members;
      survivors += total[j][0];
      members += total[j][1];
      sources += total[j][2];
    }
  } else {
    if (WEIGHTS && tid == 0) base_off[0] = 0;
    survivors = cta_total[0];
    members = cta_total[1];
    sources = cta_total[2];
  }
  // A sample whose A or B nodes do not fit the plan's capacities (a subset of the grid handed to a plan that was built
  // for full grids) keeps all of its tokens, and the status word says so.
  const bool over = sources > a.cap_a || n - sources > a.cap_b;
  if (over) {
    survivors = members = n;
    before_s = before_m = lo;
    xs = xm = ns = nm = 0;
#pragma unroll
    for (int j = 0; j < TPT; ++j) { prt[j] = -1; plc[j] = 0; }
  }
  const int n_out = min(survivors, a.cap_out);
  if (rank == 0 && tid == 0) {
    a.n_vis_out[b] = n_out;
    if (n_out == survivors) a.grp_off[size_t(b) * (a.cap_out + 1) + n_out] = members;   // (cut at cap_out: set below)
    if (over || survivors > a.cap_out) set_status(a.status, LIGHTKV_STATUS_COUNT);
  }
  int slot = over ? i0 : before_s + warp_sums[0][wp] + xs - ns, off = over ? i0 : before_m + warp_sums[1][wp] + xm - nm;
#pragma unroll
  for (int j = 0; j < TPT; ++j) {
    const int i = i0 + j;
    if (i < hi && prt[j] < 0) {
      const int l = i - lo;
      s_slot[l] = slot;
      s_off[l] = off;
      a.dst[row + i] = slot;
      if (slot < a.cap_out) {
        a.pos_out[size_t(b) * a.cap_out + slot] = ps[j];
        a.grp_off[size_t(b) * (a.cap_out + 1) + slot] = off;
        a.grp_src[row + off] = i;
      } else if (slot == a.cap_out) {
        a.grp_off[size_t(b) * (a.cap_out + 1) + slot] = off;   // the groups that are kept end here
      }
      if (WEIGHTS) {
        m_tok[off - before_m] = i;
        m_xi[off - before_m] = xi[j];
      }
      ++slot;
      off += 1 + plc[j];
    }
  }
  sync_all();
  // ---- merged tokens join their partner's group
#pragma unroll
  for (int j = 0; j < TPT; ++j) {
    const int i = i0 + j, p = prt[j];
    if (i < hi && p >= 0) {
      const int r = CLUSTER ? p / chunk : 0, l = p - r * chunk;
      int o, at;
      if (CLUSTER) {
        o = (int)tc::ld_cluster_u32(tc::map_to_cta(tc::smem_u32(&s_slot[l]), r));
        at = (int)tc::ld_cluster_u32(tc::map_to_cta(tc::smem_u32(&s_off[l]), r));
      } else {
        o = s_slot[l]; at = s_off[l];
      }
      at += 1 + plc[j];
      a.dst[row + i] = o;
      if (o < a.cap_out) a.grp_src[row + at] = i;
      if (WEIGHTS) {
        at -= base_off[r];
        if (CLUSTER) {
          tc::st_cluster_u32(tc::map_to_cta(tc::smem_u32(&m_tok[at]), r), (uint32_t)i);
          tc::st_cluster_u32(tc::map_to_cta(tc::smem_u32(&m_xi[at]), r), __float_as_uint(xi[j]));
        } else {
          m_tok[at] = i; m_xi[at] = xi[j];
        }
      }
    }
    if (WEIGHTS && i < hi && a.xi_out) a.xi_out[row + i] = xi[j];
  }
  if (CLUSTER || WEIGHTS) sync_all();                       // nobody reads or writes this CTA's shared memory any more
  if (WEIGHTS) {
#pragma unroll
    for (int j = 0; j < TPT; ++j) {
      const int i = i0 + j;
      if (i < hi && prt[j] < 0 && s_slot[i - lo] < a.cap_out) {
        const int at = s_off[i - lo] - before_m, size = 1 + plc[j];
        float den = 0.f;
        for (int c = 0; c < size; ++c) den += m_xi[at + c];
        for (int c = 0; c < size; ++c) a.weight[row + m_tok[at + c]] = member_weight(m_xi[at + c], den, size);
        if (!(den >= 1e-30f)) set_status(a.status, LIGHTKV_STATUS_ZERO_WEIGHT);
      }
    }
  }
}

cudaError_t launch_map(const LayerLaunch& L, bool select, bool behind_xi) {
  const lightkv_layer_args_t* a = L.a;
  const bool attn = L.xi_mode == LIGHTKV_XI_ATTN_FULL || L.xi_mode == LIGHTKV_XI_ATTN_LSE, weights = !attn || behind_xi;
  MapArgs m;
  m.xi_mode = L.xi_mode; m.xi_in = a->xi; m.xi_h = attn ? L.ws.xi_h : nullptr; m.n_q_heads = L.n_q_heads; m.weight = a->weight; m.xi_out = a->xi_out;
  m.cap_in = L.ws.cap_in; m.cap_out = L.ws.cap_out;
  m.cap_a = L.ws.cap_a; m.cap_b = L.ws.cap_b; m.n_grid = L.n_grid;
  m.n_vis = a->n_vis; m.pos = a->pos; m.partner = L.ws.partner; m.place = L.ws.slot;
  m.key = L.ws.tile_key; m.win_tok = L.ws.win_tok; m.blocks = L.fd_blocks; m.max_cell = L.max_cell; m.n_windows = L.geo.n_windows;
  m.src_par = L.geo.src_par; m.keep = L.keep;
  m.n_vis_out = a->n_vis_out; m.pos_out = a->pos_out; m.dst = a->dst; m.grp_off = a->grp_off;
  m.grp_src = a->grp_src; m.status = a->status;
  // one cluster per sample: as many CTAs of up to 1024 threads as give every thread one token (two beyond 8192), and
  // with windows to select in, as many as there are windows (up to eight) of at least 256 threads
  const int n = L.ws.cap_in;
  int cs = 1;
  while (cs < 8 && (cs * 1024 < n || (select && cs < L.geo.n_windows))) cs *= 2;
  const int tpt = n > 8192 ? 2 : 1;
  const int threads = std::max(select ? 256 : 32, std::min(1024, (((n + cs - 1) / cs + tpt - 1) / tpt + 31) / 32 * 32));
  size_t smem = (size_t(2) * threads * tpt + (weights ? size_t(2) * n : 0)) * 4;
  if (select) smem = std::max(smem, WindowLists::bytes(L.max_cell));
  auto launch = [&](auto kernel) -> cudaError_t {
    const cudaError_t e = ensure_dynamic_smem(kernel, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_kernel(kernel, L.batch * cs, threads, smem, L.stream, cs, m);
  };
  auto form = [&](auto w) {
    constexpr bool W = decltype(w)::value;
    if (tpt == 2) return select ? launch(map_kernel<true, 2, true, W>) : launch(map_kernel<true, 2, false, W>);
    if (cs > 1) return select ? launch(map_kernel<true, 1, true, W>) : launch(map_kernel<true, 1, false, W>);
    return select ? launch(map_kernel<false, 1, true, W>) : launch(map_kernel<false, 1, false, W>);
  };
  return weights ? form(std::true_type()) : form(std::false_type());
}

// Launches of at most four rows an SM do not fill the SMs' memory pipes by number: they get wider CTAs and more members of
// a group in flight per thread: a group of ten tokens is three rounds of loads instead of five (one image of 576 tokens,
// one layer: 39.6 -> 33.3 us a pass).
static bool few_rows(long long rows) { return rows <= 4 * sm_count(); }
static bool few_rows(const LayerLaunch& L) {
  return few_rows((long long)(L.a->vis_begin + L.ws.cap_out + L.a->n_text_after) * L.batch);
}
// The instructions a row's CTA spends on its weights are in nobody's way while a launch is short; a long one is bound by
// memory only as long as little else is issued.  us of compress_layer, a given log-sum-exp, with the merge / by weights_kernel:
// 9.5 MB (2304 tokens x 4096) 28.7 / 31.8, 11 MB (4 x 576) 27.2 / 28.8, 17.5 MB (2 x 2048 x 3584) 39.9 / 42.7, 21 MB (16 x 576 x
// 2048) 46.7 / 46.7, 22 MB (8 x 576 x 4096) 39.9 / 38.8, 27.5 MB (40 x 576 x 1024) 65.5 / 65.5, 30 MB (6 x 1152 x 4096) 53.9 / 51.4,
// 44 MB (16 x 576 x 4096) 73.3 / 68.7, 59.5 MB (2 x 8192 x 3584) 128 / 119, 98 MB (8 x 2880 x 4096) 168 / 151; the same with xi from
// all keys.  (Rows of 1 KB and a hundred samples, 40 MB: 112 / 115.)
bool merge_takes_weights(const LayerLaunch& L) {
  return (long long)(L.a->vis_begin + L.ws.cap_out + L.a->n_text_after) * L.batch * L.hidden * (L.dtype == LIGHTKV_BF16 ? 2 : 4) <= (24ll << 20);
}
// The map behind xi, with the weights.  For a caller that waits for the map alone, where it costs less than weights_kernel does
// beside what the map beside xi saves: in short launches with few heads, whose sums are little work for a sample's CTAs, or few
// tokens, fewer where the map has the longer xi from all keys to run beside.  us of compress_layer, map behind xi / beside it and
// weights_kernel, samples x tokens x heads, given log-sum-exp: 1 x 576 x 32 19.6 / 20.2, 2 x 798 x 32 29.7 / 31.9, 2 x 1024 x 28 28.7
// / 26.5, 4 x 576 x 32 29.8 / 28.8, 2 x 2048 x 28 47.6 / 42.5; 1 x 4096 x 8 22.4 / 26.5, 2 x 2048 x 16 27.1 / 28.4, 16 x 576 x 16 31.0 /
// 31.9, 4 x 2304 x 16 33.3 / 32.8; all keys: 2 x 200 x 32 18.4 / 20.4, 1 x 288 x 32 19.2 / 21.6, 1 x 576 x 32 24.0 / 22.9, 2 x 400 x 32
// 23.6 / 23.1, 2 x 798 x 32 39.0 / 33.7, 4 x 1152 x 32 67.5 / 62.4; 16 x 576 x 16 49.0 / 49.4, 4 x 2304 x 16 75.8 / 76.1.
// And for one whose counts are replaced in place, whatever the launch: the xi kernel reads n_vis item by item, and a map beside it
// would put the smaller counts there.
bool map_behind_xi(const LayerLaunch& L) {
  if (L.a->n_vis == L.a->n_vis_out) return true;
  const long long few_tokens = L.xi_mode == LIGHTKV_XI_ATTN_LSE ? 2000 : 500;
  return L.a->map_event && merge_takes_weights(L) && (L.n_q_heads <= 16 || (long long)L.batch * L.ws.cap_in <= few_tokens);
}

// =====================================================================================================
// xi of the tokens (in the one order, see warp_xi) and the weights of the groups (Eq. "message-passing"), behind
// map_kernel, which knows the groups but runs beside the xi kernel: xi_i / sum over the group, the sum taken in member
// order (survivor first).  A cluster of eight CTAs per sample: a warp sums the heads of eight tokens into
// shared memory; then a thread per group reads its members' sums from the CTAs that hold them.  Bound by
// the length of its chain of loads, shuffles and barriers: 4 to 6 us (32 tokens a warp, or a thread per token: 6 to 12).
// =====================================================================================================
struct WeightArgs {
  int n_q_heads, cap_in, cap_out;
  int chunk;                           // weights_kernel: tokens per CTA
  unsigned magic_chunk;                // div_multiplier(chunk)
  const float* xi_h;                   // [B, cap_in, H]
  const int* n_vis;
  const int* n_vis_out;
  const int* grp_off;
  const int* grp_src;
  const int* dst;
  float* weight;
  float* xi_out;
  uint32_t* status;
};
constexpr int kWeightCtas = 8;

__global__ void __launch_bounds__(1024) weights_kernel(const __grid_constant__ WeightArgs a) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  float* s_xi = reinterpret_cast<float*>(smem_raw);       // [chunk] xi of this CTA's tokens
  const int rank = (int)tc::cluster_ctarank(), b = blockIdx.x / kWeightCtas, tid = threadIdx.x, nthr = blockDim.x;
  const int warp = tid >> 5, lane = tid & 31, H = a.n_q_heads;
  const size_t row = size_t(b) * a.cap_in;
  // a thread's first group is looked up at once, before the counts are there (the lists have the room)
  const int o0 = tid * kWeightCtas + rank;
  const int* go = a.grp_off + size_t(b) * (a.cap_out + 1);
  int g0 = 0, g1 = 0;
  if (o0 < a.cap_out) { g0 = go[o0]; g1 = go[o0 + 1]; }
  const int n = a.n_vis ? max(0, min(a.n_vis[b], a.cap_in)) : a.cap_in, n_out = a.n_vis_out[b];
  const int lo = rank * a.chunk, hi = min(a.cap_in, lo + a.chunk);
  const float* x = a.xi_h + row * H;
  for (int i0 = lo + 8 * warp; i0 < hi; i0 += nthr >> 2) {
    // eight tokens of a warp, the lanes over the heads (addresses are clamped, not loads left out: a load behind a branch
    // waits for the one before); then every lane holds the sum of a token
    float p[8] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    const int last = a.cap_in - 1 - i0;
    for (int h0 = lane; h0 - lane < H; h0 += 64) {
      const float* xh = x + i0 * H + min(h0, H - 1);
      const float* xg = x + i0 * H + min(h0 + 32, H - 1);
      float v[8], w[8];
#pragma unroll
      for (int t = 0; t < 8; ++t) v[t] = xh[min(t, last) * H];
      if (h0 - lane + 32 < H) {
#pragma unroll
        for (int t = 0; t < 8; ++t) w[t] = xg[min(t, last) * H];
#pragma unroll
        for (int t = 0; t < 8; ++t) p[t] = (p[t] + v[t]) + (h0 + 32 < H ? w[t] : 0.f);
      } else {
#pragma unroll
        for (int t = 0; t < 8; ++t) p[t] += h0 < H ? v[t] : 0.f;
      }
    }
    float v = sum_eight(p, lane);
    v += __shfl_xor_sync(0xffffffffu, v, 8);
    v += __shfl_xor_sync(0xffffffffu, v, 16);
    const int i = i0 + xi_value(lane & 7);
    if (lane < 8 && i < hi) {
      s_xi[i - lo] = v;
      if (a.xi_out && i < n) a.xi_out[row + i] = v;
    }
  }
  constexpr int AHEAD = 8;                                // members looked up at once
  const int* gs = a.grp_src + row;
  int tok[AHEAD];
#pragma unroll
  for (int k = 0; k < AHEAD; ++k) tok[k] = gs[min(max(g0 + k, 0), a.cap_in - 1)];
  tc::cluster_sync();
  const uint32_t base = tc::smem_u32(s_xi);
  auto xi_of = [&](int i) {
    const int r = div_magic(i, a.magic_chunk);
    return tc::ld_cluster_f32(tc::map_to_cta(base + uint32_t(i - r * a.chunk) * 4, r));
  };
  for (int o = o0; o < n_out; o += kWeightCtas * nthr) {
    if (o != o0) {
      g0 = go[o];
      g1 = go[o + 1];
#pragma unroll
      for (int k = 0; k < AHEAD; ++k) tok[k] = gs[min(g0 + k, a.cap_in - 1)];
    }
    const int size = g1 - g0;
    float den = 0.f, first[AHEAD];
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) first[k] = k < size ? xi_of(tok[k]) : 0.f;
#pragma unroll
    for (int k = 0; k < AHEAD; ++k) den += first[k];
    for (int g = AHEAD; g < size; ++g) den += xi_of(gs[g0 + g]);
#pragma unroll
    for (int k = 0; k < AHEAD; ++k)
      if (k < size) a.weight[row + tok[k]] = member_weight(first[k], den, size);
    for (int g = AHEAD; g < size; ++g) {
      const int i = gs[g0 + g];
      a.weight[row + i] = member_weight(xi_of(i), den, size);
    }
    if (!(den >= 1e-30f)) set_status(a.status, LIGHTKV_STATUS_ZERO_WEIGHT);
  }
  tc::cluster_sync();                                     // nobody reads this CTA's shared memory any more
}

static WeightArgs weight_args(const LayerLaunch& L) {
  const lightkv_layer_args_t* a = L.a;
  const int chunk = std::max(2, (L.ws.cap_in + kWeightCtas - 1) / kWeightCtas);      // at most kMapMaxTokens / 8; 2: see div_magic
  return {L.n_q_heads, L.ws.cap_in, L.ws.cap_out, chunk, div_multiplier(chunk), L.ws.xi_h, a->n_vis,
          a->n_vis_out, a->grp_off, a->grp_src, a->dst, a->weight, a->xi_out, a->status};
}

cudaError_t launch_weights(const LayerLaunch& L) {
  const WeightArgs w = weight_args(L);
  const int threads = std::min(1024, std::max(4 * w.chunk, 128) / 32 * 32 + 32);       // warps for one round over the tokens
  return launch_kernel(weights_kernel, L.batch * kWeightCtas, threads, size_t(4) * w.chunk, L.stream, kWeightCtas, w);
}

// A sample cut at cap_out has tokens that belong to no group that is kept: their xi is still reported.
__device__ __noinline__ void xi_of_cut_tokens(const WeightArgs& a, int b, int n, int n_out) {
  if (!a.xi_out || a.grp_off[size_t(b) * (a.cap_out + 1) + n_out] >= n) return;
  const int lane = threadIdx.x & 31;
  for (int i = threadIdx.x >> 5; i < n; i += blockDim.x >> 5)
    if (a.dst[size_t(b) * a.cap_in + i] >= a.cap_out) {
      const float v = warp_xi(a.xi_h + (size_t(b) * a.cap_in + i) * a.n_q_heads, a.n_q_heads, lane);
      if (lane == 0) a.xi_out[size_t(b) * a.cap_in + i] = v;
    }
}

// =====================================================================================================
// Weighted merge of the hidden states (Eq. "message-passing", Steps 3-5): one CTA per output row.
// Row o of the vision block is sum over its group of weight_i * x_i in fp32, rounded once to the
// storage type; a group of one has weight exactly 1 and is copied.  Text rows
// before / after the vision block are copied.  Pure 16-byte streaming loads and stores.
// WEIGHTS: the CTA computes its group's weights, too (a warp per member), while its first rows are on their way to L2: one
// kernel less in a row of dependent ones.  See merge_takes_weights.
// =====================================================================================================
template <typename T>
struct MergeArgs {
  const T* src; int64_t src_bs, src_rs;
  T* out; int64_t out_bs, out_rs;
  int d, vis_begin, n_text_after;
  const int* seq_start;
  const int* seq_start_out;
  WeightArgs w;
};

// Registers: with the weights the form for many rows spills at five CTAs per SM (4 x 652 rows of 4096, a pass: 103.9 us; with
// four 100.7).
template <typename T, int MB, bool WEIGHTS>
__global__ void __launch_bounds__(256, MB > 2 ? 3 : WEIGHTS ? 4 : 5) merge_rows_kernel(const __grid_constant__ MergeArgs<T> a) {
  grid_dependency_sync();
  constexpr int V = Vec<T>::n;
  constexpr int AHEAD = 64;                             // members whose weights stay on chip
  __shared__ float s_xi[WEIGHTS ? AHEAD : 1], s_wt[WEIGHTS ? AHEAD : 1];
  const int b = blockIdx.y, row = blockIdx.x, o = row - a.vis_begin;
  const int cap_in = a.w.cap_in, cap_out = a.w.cap_out;
  // (the row's group is looked up before it is known that the row has one: one round trip less)
  const int* go = a.w.grp_off + size_t(b) * (cap_out + 1) + min(max(o, 0), cap_out - 1);
  const int g0 = go[0], g1 = go[1];
  const int n_in = a.w.n_vis ? min(a.w.n_vis[b], cap_in) : cap_in;
  const int n_out = a.w.n_vis_out[b];
  if (WEIGHTS && row == 0) xi_of_cut_tokens(a.w, b, n_in, n_out);
  if (row >= a.vis_begin + n_out + a.n_text_after) return;
  const T* sb = a.src + size_t(b) * a.src_bs + size_t(a.seq_start ? a.seq_start[b] : 0) * a.src_rs;
  T* orow = a.out + size_t(b) * a.out_bs + size_t((a.seq_start_out ? a.seq_start_out[b] : 0) + row) * a.out_rs;
  const int chunks = a.d / V, tid = threadIdx.x, nthr = blockDim.x;
  const bool text = o < 0 || o >= n_out;
  const int* gs = a.w.grp_src + size_t(b) * cap_in + g0;
  float* wt = a.w.weight + size_t(b) * cap_in;
  float* xo = a.w.xi_out ? a.w.xi_out + size_t(b) * cap_in : nullptr;
  const float* xh = a.w.xi_h + size_t(b) * cap_in * a.w.n_q_heads;
  const int count = text ? 1 : g1 - g0;
  if (count == 1) {                                     // copied
    const int i = text ? 0 : gs[0];
    const T* srow = sb + size_t(text ? (o < 0 ? row : row - n_out + n_in) : a.vis_begin + i) * a.src_rs;
    float w = WEIGHTS || text ? 1.0f : wt[i];
    for (int c0 = tid; c0 < chunks; c0 += 2 * nthr) {
      const int c1 = c0 + nthr;
      const uint4 a0 = ld_stream16(srow + c0 * V);
      if (c1 < chunks) {
        const uint4 a1 = ld_stream16(srow + c1 * V);
        st_stream16(orow + c1 * V, a1);
      }
      st_stream16(orow + c0 * V, a0);
    }
    if (text) return;
    if (WEIGHTS && tid < 32) {
      const float v = warp_xi(xh + size_t(i) * a.w.n_q_heads, a.w.n_q_heads, tid);
      w = member_weight(v, v, 1);
      if (tid == 0) {
        wt[i] = w;
        if (xo) xo[i] = v;
        if (!(v >= 1e-30f)) set_status(a.w.status, LIGHTKV_STATUS_ZERO_WEIGHT);
      }
    }
    // an infinite xi leaves no number as its weight, nor as the row
    if (WEIGHTS ? __syncthreads_or(w != w) : w != w) {
      float none[V];
#pragma unroll
      for (int j = 0; j < V; ++j) none[j] = __int_as_float(0x7fffffff);
      for (int c = tid; c < chunks; c += nthr) st_stream16(orow + c * V, pack16(none, T()));
    }
    return;
  }
  const T* vis = sb + size_t(a.vis_begin) * a.src_rs;
  if (WEIGHTS) {
    // the rows are asked for while the weights are computed (prefetches hold no registers)
    for (int g = 0; g < min(count, 8); ++g) {
      const T* r = vis + size_t(gs[g]) * a.src_rs;
      if (tid * V * 2 < a.d) prefetch_l2(r + tid * V * 2);
    }
    const int lane = tid & 31;
    float den = 0.f;
    for (int k0 = 0; k0 < count; k0 += AHEAD) {
      const int m = min(AHEAD, count - k0);
      for (int k = tid >> 5; k < m; k += nthr >> 5) {
        const int i = gs[k0 + k];
        const float v = warp_xi(xh + size_t(i) * a.w.n_q_heads, a.w.n_q_heads, lane);
        if (lane == 0) {
          s_xi[k] = v;
          if (xo) xo[i] = v;
          if (count > AHEAD) wt[i] = v;
        }
      }
      __syncthreads();
      for (int k = 0; k < m; ++k) den += s_xi[k];
      if (count > AHEAD) __syncthreads();           // (s_xi is filled again, or read below)
    }
    if (count <= AHEAD) {
      for (int k = tid; k < count; k += nthr) {
        const float w = member_weight(s_xi[k], den, count);
        s_wt[k] = w;
        wt[gs[k]] = w;
      }
    } else {
      for (int k = tid; k < count; k += nthr) {
        const int i = gs[k];
        const float w = member_weight(wt[i], den, count);
        wt[i] = w;
        if (k < AHEAD) s_wt[k] = w;
      }
    }
    if (tid == 0 && !(den >= 1e-30f)) set_status(a.w.status, LIGHTKV_STATUS_ZERO_WEIGHT);
    __syncthreads();
  }
  // two 16-byte chunks per thread and MB members at a time: 2 MB loads in flight whatever the group's size
  for (int c0 = tid; c0 < chunks; c0 += 2 * nthr) {
    const int c1 = c0 + nthr;
    const bool two = c1 < chunks;
    float acc0[V], acc1[V];
#pragma unroll
    for (int j = 0; j < V; ++j) { acc0[j] = 0.f; acc1[j] = 0.f; }
    for (int g = 0; g < count; g += MB) {
      uint4 va[MB], vb[MB];
      float wv[MB];
#pragma unroll
      for (int u = 0; u < MB; ++u) {
        if (g + u < count) {
          const int i = gs[g + u];
          if (!WEIGHTS) wv[u] = wt[i];
          const T* r = vis + size_t(i) * a.src_rs;
          va[u] = ld_stream16(r + c0 * V);
          if (two) vb[u] = ld_stream16(r + c1 * V);
        }
      }
#pragma unroll
      for (int u = 0; u < MB; ++u) {
        if (g + u < count) {
          if (WEIGHTS) wv[u] = g + u < AHEAD ? s_wt[g + u] : wt[gs[g + u]];
          float f[V];
          unpack16(va[u], f, T());
#pragma unroll
          for (int j = 0; j < V; ++j) acc0[j] = fmaf(wv[u], f[j], acc0[j]);
          if (two) {
            unpack16(vb[u], f, T());
#pragma unroll
            for (int j = 0; j < V; ++j) acc1[j] = fmaf(wv[u], f[j], acc1[j]);
          }
        }
      }
    }
    st_stream16(orow + c0 * V, pack16(acc0, T()));
    if (two) st_stream16(orow + c1 * V, pack16(acc1, T()));
  }
}

cudaError_t launch_merge_rows(const LayerLaunch& L, bool weights) {
  const lightkv_layer_args_t* a = L.a;
  const int rows = a->vis_begin + L.ws.cap_out + a->n_text_after;
  const dim3 grid(rows, L.batch);
  auto run = [&](auto tag) -> cudaError_t {
    using T = decltype(tag);
    const MergeArgs<T> m = {static_cast<const T*>(a->hidden), a->hidden_batch_stride, a->hidden_row_stride,
                            static_cast<T*>(a->hidden_out), a->hidden_out_batch_stride, a->hidden_out_row_stride,
                            L.hidden, a->vis_begin, a->n_text_after, a->seq_start, a->seq_start_out, weight_args(L)};
    if (few_rows(L)) return launch_kernel(weights ? merge_rows_kernel<T, 4, true> : merge_rows_kernel<T, 4, false>, grid, 256, 0, L.stream, 1, m);
    // two chunks per thread: narrow rows get narrow CTAs, and more of them
    const int pairs = (L.hidden / Vec<T>::n + 1) / 2, threads = std::max(64, std::min(256, (pairs + 31) / 32 * 32));
    return launch_kernel(weights ? merge_rows_kernel<T, 2, true> : merge_rows_kernel<T, 2, false>, grid, threads, 0, L.stream, 1, m);
  };
  return L.dtype == LIGHTKV_BF16 ? run(__nv_bfloat16()) : run(float());
}

// =====================================================================================================
// K/V merge-compaction (the cache of a layer shrinks together with its tokens: appendix "Method overview").
// The stage's merge map is applied per KV head; contiguous (strided) or paged (block-table) addressing
// on either side.  One CTA per output token, five CTAs per SM; every thread resolves the token's group
// itself (uniform, cached loads) and works on two 16-byte units and two group members at a time, i.e.
// four loads in flight whatever the group's size (four units on the copy path).  Groups of one are
// copied; larger groups are summed in fp32 in member order.
// =====================================================================================================
struct KvAddr {
  int64_t batch_stride, head_stride, row_stride, page_stride;
  const int* table;       // nullptr = contiguous
  int page_size, max_blocks;
  const int* seq_start;   // first token of each sample (packed caches) or nullptr
  unsigned magic_page;    // ceil(2^32 / page_size) where that divides every row of a table exactly, else 0
  __device__ inline int page_of(int n) const { return magic_page ? (int)__umulhi((unsigned)n, magic_page) : n / page_size; }
  __device__ inline int64_t token(int b, int n) const {
    if (seq_start) n += seq_start[b];
    if (!table) return int64_t(b) * batch_stride + int64_t(n) * row_stride;
    const int in_table = page_of(n), page = table[size_t(b) * max_blocks + in_table];
    return int64_t(page) * page_stride + int64_t(n - in_table * page_size) * row_stride;
  }
};

// THREADS per CTA, MB members of a group in flight.  ONE: heads of a single 16-byte piece, which there is no division for.  (A
// division that also does for one piece, by a test or with twice the number and half the multiplier, costs more than the form:
// 32 x 640 rows x 40 heads x 128 119.0 or 118.8 against 116.9 us, 8 x 3008 x 32 105.8 or 105.4 against 104.0; with the test the
// kernel spills.)
template <typename T, int THREADS, int MB, bool ONE>
__global__ void __launch_bounds__(THREADS, (THREADS > 256 ? 2 : (sizeof(T) == 2 ? 5 : 4)) - ONE)
kv_compact_kernel(const T* __restrict__ k_src, const T* __restrict__ v_src, T* __restrict__ k_dst,
                  T* __restrict__ v_dst, KvAddr sa, KvAddr da, int n_kv_heads, int dh, int vis_begin,
                  int n_text_after, int cap_in, int cap_out, int gather, int merge_at_survivor, unsigned magic_ch,
                  const int* __restrict__ n_vis, const int* __restrict__ n_vis_out,
                  const int* __restrict__ grp_off, const int* __restrict__ grp_src,
                  const float* __restrict__ weight) {
  grid_dependency_sync();
  constexpr int V = Vec<T>::n;
  const int b = blockIdx.y, row = blockIdx.x;
  const int n_in = n_vis ? min(n_vis[b], cap_in) : cap_in;
  const int n_out = n_vis_out[b];
  if (row >= vis_begin + n_out + n_text_after) return;
  const int ch = ONE ? 1 : dh / V, per_kv = n_kv_heads * ch, units = 2 * per_kv;
  auto head_of = [&](int piece) { return ONE ? piece : div_magic(piece, magic_ch); };
  int64_t d_tok = da.token(b, row);
  const bool text = row < vis_begin || row >= vis_begin + n_out;
  const int* gs = grp_src + size_t(b) * cap_in;
  const float* wt = weight + size_t(b) * cap_in;
  int g0 = 0, g1 = 1;
  if (!text) {
    const int* go = grp_off + size_t(b) * (cap_out + 1);
    g0 = go[row - vis_begin];
    g1 = gather ? g0 + 1 : go[row - vis_begin + 1];
  }
  if (merge_at_survivor) {
    // first phase of the in-place form: a merged group is written over its surviving token's own row (no other
    // group reads that row); rows that are only moved wait for the second phase
    if (text || g1 - g0 == 1) return;
    d_tok = da.token(b, vis_begin + gs[g0]);
  }
  if (text || g1 - g0 == 1) {                                       // copy: text, lone survivor, gather mode
    const int64_t s_tok = text ? sa.token(b, row < vis_begin ? row : row - n_out + n_in)
                               : sa.token(b, vis_begin + gs[g0]);
    for (int u0 = threadIdx.x; u0 < units; u0 += 4 * blockDim.x) {   // four units' loads in flight per thread
      uint4 v[4];
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int u = u0 + q * blockDim.x;
        if (u < units) {
          const int kv = u >= per_kv ? 1 : 0, rem = u - kv * per_kv, h = head_of(rem), c = rem - h * ch;
          v[q] = ld_stream16((kv ? v_src : k_src) + s_tok + int64_t(h) * sa.head_stride + c * V);
        }
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int u = u0 + q * blockDim.x;
        if (u < units) {
          const int kv = u >= per_kv ? 1 : 0, rem = u - kv * per_kv, h = head_of(rem), c = rem - h * ch;
          st_stream16((kv ? v_dst : k_dst) + d_tok + int64_t(h) * da.head_stride + c * V, v[q]);
        }
      }
    }
    return;
  }
  // merge: two units per thread and MB members at a time.  The lanes of a warp hold the members' addresses and weights
  // (one lookup each, 32 at a time), so that a round of loads waits for nothing but the round before.
  const int lane = threadIdx.x & 31, count = g1 - g0;
  int64_t m_tok = 0;
  float m_w = 0.f;
  auto members = [&](int first) {
    if (first + lane < count) {
      const int i = gs[g0 + first + lane];
      m_w = wt[i];
      m_tok = sa.token(b, vis_begin + i);
    }
  };
  members(0);
  for (int base = 0; base < units; base += 2 * blockDim.x) {
    const int u0 = base + threadIdx.x, u1 = u0 + blockDim.x;
    const bool one = u0 < units, two = u1 < units;
    const int kv0 = u0 >= per_kv ? 1 : 0, rem0 = u0 - kv0 * per_kv, h0 = head_of(rem0), c0 = rem0 - h0 * ch;
    const int ub = two ? u1 : u0;
    const int kv1 = ub >= per_kv ? 1 : 0, rem1 = ub - kv1 * per_kv, h1 = head_of(rem1), c1 = rem1 - h1 * ch;
    const T* sp0 = (kv0 ? v_src : k_src) + int64_t(h0) * sa.head_stride + c0 * V;
    const T* sp1 = (kv1 ? v_src : k_src) + int64_t(h1) * sa.head_stride + c1 * V;
    float acc0[V], acc1[V];
#pragma unroll
    for (int j = 0; j < V; ++j) { acc0[j] = 0.f; acc1[j] = 0.f; }
    for (int g = 0; g < count; g += MB) {
      if (count > 32 && (g & 31) == 0) members(g);
      uint4 va[MB], vb[MB];
#pragma unroll
      for (int m = 0; m < MB; ++m) {
        if (g + m < count) {
          const int64_t tok = __shfl_sync(0xffffffffu, m_tok, (g + m) & 31);
          if (one) va[m] = ld_stream16(sp0 + tok);
          if (two) vb[m] = ld_stream16(sp1 + tok);
        }
      }
#pragma unroll
      for (int m = 0; m < MB; ++m) {
        if (g + m < count) {
          const float w = __shfl_sync(0xffffffffu, m_w, (g + m) & 31);
          float f[V];
          unpack16(va[m], f, T());
#pragma unroll
          for (int j = 0; j < V; ++j) acc0[j] = fmaf(w, f[j], acc0[j]);
          if (two) {
            unpack16(vb[m], f, T());
#pragma unroll
            for (int j = 0; j < V; ++j) acc1[j] = fmaf(w, f[j], acc1[j]);
          }
        }
      }
    }
    if (one) st_stream16((kv0 ? v_dst : k_dst) + d_tok + int64_t(h0) * da.head_stride + c0 * V, pack16(acc0, T()));
    if (two) st_stream16((kv1 ? v_dst : k_dst) + d_tok + int64_t(h1) * da.head_stride + c1 * V, pack16(acc1, T()));
  }
}

// =====================================================================================================
// In place, where a plane fits on chip: one CTA owns a plane -- one (sample, K or V, head, column part) --, copies ALL of
// its rows from the first vision row on into shared memory, synchronises, and stores the merged and moved rows: no other
// CTA touches these bytes, so nothing is overwritten before it has been read, and one kernel does what the two below
// need a pass over memory more for.
// Bound by latency: the rows' addresses need no group lists (only a block table's part of the sample), so rows and lists
// are asked for at once (cp.async) and a plane is three round trips: counts and table, rows, stores.  In gather mode, where
// only the survivors' rows are read, the lists are a round trip of their own.  Columns are cut so that the launch has
// two CTAs per SM, in parts of at least 64 bytes (less where the rows would not fit otherwise).  A plane that leaves room
// for a second CTA on the SM gets 512 threads, one that does not 1024.
// us a call in a row of them, against gathering the merged rows into shared memory through the staged lists (which took
// up to ten round trips for the largest groups): 4 samples x 652 tokens, 8 KV heads x 128, pages of 16 15.4 -> 8.9; up
// to 16 x 624 x 8 x 64 packed 19.5 -> 12.4; 576 x 32 x 128 13.5 -> 8.2; 2304 x 8 x 128 24 -> 15; 5328 x 8 x 128 40 -> 18;
// 8 x 3008 x 32 x 128 351 -> 207 (with 512 threads 289).  The two kernels below take 21.3, 22.8, 20.6, 24.5, 25 and 238.
// 256 threads 12, 1024 13 in the first, where two CTAs of 512 fit.
// =====================================================================================================
struct KvPlaneSmem {
  int staged, n_in, n_out, blocks;             // capacities: rows in shared memory, vision tokens in / out, pages of the moving rows
  __host__ __device__ size_t wgt() const { return size_t(n_in) * 4; }                    // (the member list comes first)
  __host__ __device__ size_t off() const { return wgt() + size_t(n_in) * 4; }
  __host__ __device__ size_t blk() const { return off() + size_t(n_out + 1) * 4; }
  __host__ __device__ size_t rows() const { return (blk() + size_t(blocks) * 4 + 15) & ~size_t(15); }
  __host__ __device__ size_t bytes(int pieces) const { return rows() + size_t(staged) * pieces * 16; }
};

// ONE: rows of a single piece, as above
template <typename T, int THREADS, bool ONE>
__global__ void __launch_bounds__(THREADS)
kv_plane_kernel(T* __restrict__ k_buf, T* __restrict__ v_buf, KvAddr ad, KvPlaneSmem sm, int n_kv_heads, int ch, int parts,
                unsigned magic_ch, int vis_begin, int n_text_after, int gather, const int* __restrict__ n_vis,
                const int* __restrict__ n_vis_out, const int* __restrict__ grp_off, const int* __restrict__ grp_src,
                const float* __restrict__ weight) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int V = Vec<T>::n;
  int* mem = reinterpret_cast<int*>(smem_raw);                          // group members, survivor first
  float* wgt = reinterpret_cast<float*>(smem_raw + sm.wgt());           // weights of the tokens
  int* off = reinterpret_cast<int*>(smem_raw + sm.off());               // first member of every output row
  int* blk = reinterpret_cast<int*>(smem_raw + sm.blk());               // pages of the moving rows
  const uint4* rows = reinterpret_cast<const uint4*>(smem_raw + sm.rows());
  const uint32_t s_rows = tc::smem_u32(rows);
  const int tid = threadIdx.x;
  int plane = blockIdx.x;
  const int part = plane % parts; plane /= parts;
  const int h = plane % n_kv_heads; plane /= n_kv_heads;
  const int kv = plane & 1, b = plane >> 1;
  const int row0 = vis_begin + (ad.seq_start ? ad.seq_start[b] : 0), page0 = ad.table ? ad.page_of(row0) : 0;
  const int n_out = n_vis_out[b], n_in = n_vis ? min(n_vis[b], sm.n_in) : sm.n_in;
  if (ad.table)
    for (int j = tid; j < sm.blocks; j += THREADS)
      if (page0 + j < ad.max_blocks) tc::cp_async4(tc::smem_u32(blk + j), ad.table + size_t(b) * ad.max_blocks + page0 + j);
  tc::cp_async_commit();
  for (int o = tid; o <= sm.n_out; o += THREADS) tc::cp_async4(tc::smem_u32(off + o), grp_off + size_t(b) * (sm.n_out + 1) + o);
  for (int k = tid; k < sm.n_in; k += THREADS) {       // (lists that a short sample does not fill are never read)
    tc::cp_async4(tc::smem_u32(mem + k), grp_src + size_t(b) * sm.n_in + k);
    if (!gather) tc::cp_async4(tc::smem_u32(wgt + k), weight + size_t(b) * sm.n_in + k);
  }
  tc::cp_async_commit();
  T* buf = (kv ? v_buf : k_buf) + int64_t(h) * ad.head_stride + part * ch * V;
  auto at = [&](int l) -> T* {                             // the plane's part of row l behind the first vision row
    const int n = row0 + l;
    if (!ad.table) return buf + int64_t(b) * ad.batch_stride + int64_t(n) * ad.row_stride;
    const int page = ad.page_of(n);
    return buf + int64_t(blk[page - page0]) * ad.page_stride + int64_t(n - page * ad.page_size) * ad.row_stride;
  };
  if (ad.table || gather) {
    if (gather) tc::cp_async_wait<0>(); else tc::cp_async_wait<1>();
    __syncthreads();
  }
  auto member = [&](int k) { return (int)min((unsigned)mem[k], (unsigned)(n_in - 1)); };
  if (n_out >= n_in) {                                     // nothing was merged away: every row is where it belongs
    tc::cp_async_wait<0>();
    return;
  }
  const int total = (n_out + n_text_after) * ch, staged = gather ? total : (n_in + n_text_after) * ch;
#pragma unroll 4
  for (int idx = tid; idx < staged; idx += THREADS) {
    const int r = ONE ? idx : div_magic(idx, magic_ch), c = ONE ? 0 : idx - r * ch;
    const int l = !gather ? r : r < n_out ? member(off[r]) : r - n_out + n_in;
    tc::cp_async16(s_rows + uint32_t(idx) * 16, at(l) + c * V, 16);
  }
  tc::cp_async_commit();
  tc::cp_async_wait<0>();
  __syncthreads();                                         // every source of the plane has been read
#pragma unroll 2
  for (int idx = tid; idx < total; idx += THREADS) {
    const int r = ONE ? idx : div_magic(idx, magic_ch), c = ONE ? 0 : idx - r * ch;
    uint4 v;
    if (gather || r >= n_out) {
      v = rows[gather ? idx : idx + (n_in - n_out) * ch];
    } else {
      const int g0 = off[r], count = off[r + 1] - g0, first = member(g0);
      v = rows[first * ch + c];
      if (count > 1) {
        float acc[V], f[V];
        unpack16(v, f, T());
        float w = wgt[first];
#pragma unroll
        for (int j = 0; j < V; ++j) acc[j] = fmaf(w, f[j], 0.f);
        for (int g = 1; g < count; ++g) {
          const int i = member(g0 + g);
          unpack16(rows[i * ch + c], f, T());
          w = wgt[i];
#pragma unroll
          for (int j = 0; j < V; ++j) acc[j] = fmaf(w, f[j], acc[j]);
        }
        v = pack16(acc, T());
        // the merged group also replaces its survivor's row where that lies behind the new end, as the two-phase form leaves it
        if (first >= n_out + n_text_after) st_stream16(at(first) + c * V, v);
      }
    }
    st_stream16(at(r) + c * V, v);
  }
}

// =====================================================================================================
// Second phase of the in-place form for planes that do not fit on chip: every output row moves from its surviving token's row (which holds the
// merged group after the first phase) to its slot.  A slot never lies behind its source (o <= i), so rows only
// move towards the front.  One CTA owns a plane -- one (sample, K or V, head, column part) -- and sweeps its
// output rows in ascending chunks: the sources of a chunk are gathered into shared memory, the CTA
// synchronises, the chunk is stored.  The sources of chunk k + 1 lie at or behind its first slot, i.e. behind
// everything chunk k writes, so its gather is issued before chunk k is stored; and a chunk's own sources are in
// shared memory before any of its slots is written.  Rows before the vision block do not move.
// =====================================================================================================
constexpr int KVM_THREADS = 256, KVM_CHUNK_BYTES = 40 * 1024;

template <typename T>
__global__ void __launch_bounds__(KVM_THREADS)
kv_move_kernel(T* __restrict__ k_buf, T* __restrict__ v_buf, KvAddr ad, int n_kv_heads, int dh, int parts,
               int vis_begin, int n_text_after, int cap_in, const int* __restrict__ n_vis,
               const int* __restrict__ n_vis_out, const int* __restrict__ grp_off, const int* __restrict__ grp_src,
               int cap_out) {
  grid_dependency_sync();
  extern __shared__ __align__(16) unsigned char smem_raw[];
  constexpr int V = Vec<T>::n;
  int plane = blockIdx.x;
  const int part = plane % parts; plane /= parts;
  const int h = plane % n_kv_heads; plane /= n_kv_heads;
  const int kv = plane & 1, b = plane >> 1;
  const int n_in = n_vis ? min(n_vis[b], cap_in) : cap_in;
  const int n_out = n_vis_out[b];
  if (n_out >= n_in) return;                               // nothing was merged away: every row is where it belongs
  T* buf = (kv ? v_buf : k_buf) + int64_t(h) * ad.head_stride;
  const int ch_all = dh / V, ch0 = part * ch_all / parts, ch = (part + 1) * ch_all / parts - ch0;   // 16-byte pieces of this plane
  const int rows_per_chunk = KVM_CHUNK_BYTES / (ch * 16);
  const int* go = grp_off + size_t(b) * (cap_out + 1);
  const int* gs = grp_src + size_t(b) * cap_in;
  const int row_end = vis_begin + n_out + n_text_after;
  const uint32_t sbase = tc::smem_u32(smem_raw);
  auto source = [&](int row) {                            // row of the buffer that holds output row `row`
    return row < vis_begin + n_out ? vis_begin + gs[go[row - vis_begin]] : row - n_out + n_in;
  };
  auto gather = [&](int r0, uint32_t sm) {                // output rows r0 .. of one chunk -> shared memory
    const int nr = min(rows_per_chunk, row_end - r0);
    for (int idx = threadIdx.x; idx < nr * ch; idx += blockDim.x) {
      const int rr = idx / ch, c = idx - rr * ch;
      tc::cp_async16(sm + uint32_t(idx) * 16, buf + ad.token(b, source(r0 + rr)) + (ch0 + c) * V, 16);
    }
  };
  int r0 = vis_begin, k = 0;
  gather(r0, sbase);
  tc::cp_async_commit();
  for (; r0 < row_end; r0 += rows_per_chunk, ++k) {
    const int next = r0 + rows_per_chunk;
    if (next < row_end) gather(next, sbase + ((k + 1) & 1) * KVM_CHUNK_BYTES);
    tc::cp_async_commit();
    tc::cp_async_wait<1>();                               // this thread's pieces of chunk k have landed
    __syncthreads();                                      // ... and everybody else's: all sources of chunk k are on chip
    const int nr = min(rows_per_chunk, row_end - r0);
    const unsigned char* sm = smem_raw + (k & 1) * KVM_CHUNK_BYTES;
    for (int idx = threadIdx.x; idx < nr * ch; idx += blockDim.x) {
      const int rr = idx / ch, c = idx - rr * ch;
      const uint4 v = *reinterpret_cast<const uint4*>(sm + size_t(idx) * 16);
      st_stream16(buf + ad.token(b, r0 + rr) + (ch0 + c) * V, v);
    }
    __syncthreads();                                      // the buffer may be refilled two chunks on
  }
  tc::cp_async_wait<0>();
}

cudaError_t launch_kv_compact(const KvLaunch& K) {
  const lightkv_kv_args_t* a = K.a;
  // n * ceil(2^32 / d) >> 32 is n / d while n * d < 2^32 (the multiplier is less than 1 / d too large); d = 1: 2^32 does not fit
  const long long page = a->page_size;
  const unsigned magic_page = page > 1 && page < 65536 && a->max_blocks * page * page < (1ll << 32) ? (unsigned)(((1ull << 32) + page - 1) / page) : 0;
  KvAddr sa{a->src_batch_stride, a->src_head_stride, a->src_row_stride, a->src_page_stride,
            a->page_size > 0 ? a->src_block_table : nullptr, a->page_size, a->max_blocks, a->src_seq_start, magic_page};
  KvAddr da{a->dst_batch_stride, a->dst_head_stride, a->dst_row_stride, a->dst_page_stride,
            a->page_size > 0 ? a->dst_block_table : nullptr, a->page_size, a->max_blocks, a->dst_seq_start, magic_page};
  const int ch_host = K.head_dim * (K.dtype == LIGHTKV_BF16 ? 2 : 4) / 16;
  if (2 * K.n_kv_heads * ch_host >= 65536) return cudaErrorInvalidValue;      // range of the unit decode
  const dim3 grid(a->vis_begin + K.cap_out + a->n_text_after, K.batch);
  const int units = 2 * K.n_kv_heads * ch_host;
  // two units per thread (both in flight); narrow caches (GQA) get narrow CTAs
  const bool few = few_rows((long long)grid.x * grid.y);
  const int threads = std::min(few ? 512 : 256, ((units + 1) / 2 + 31) / 32 * 32);
  const int gather = a->mode == LIGHTKV_KV_GATHER;
  const int sms = sm_count();
  const bool in_place = a->k_src == a->k_dst;             // (the API checked that V and the addressing agree)
  auto run = [&](auto tag) -> cudaError_t {
    using T = decltype(tag);
    cudaError_t e = cudaSuccess;
    if (in_place) {
      // planes: (sample, K / V, head, column part); see kv_plane_kernel for the cut.  A gather stages the survivors' rows alone:
      // with room for all, samples of 5120 tokens or more took kv_move_kernel and fewer CTAs shared an SM (us a call, 8 heads x
      // 128, room for all / for these: 1 x 6400 tokens 14.4 / 9.4, 4 x 6400 57 / 35.6, 2 x 5776 24.9 / 16.6, 8 x 2304 22.4 / 15.7).
      // Cut as if all rows were staged: wider parts leave fewer CTAs (1 x 5328 8.4 -> 10.8).
      const int moving = K.cap_in + a->n_text_after, staged = gather ? K.cap_out + a->n_text_after : moving;
      const KvPlaneSmem all{moving, K.cap_in, K.cap_out, a->page_size > 0 ? (moving + a->page_size - 1) / a->page_size + 1 : 0};
      const KvPlaneSmem sm{staged, all.n_in, all.n_out, all.blocks};
      const long long planes = 2ll * K.batch * K.n_kv_heads;
      int p = 1;
      while (ch_host % (2 * p) == 0 && ch_host / p >= 4 &&
             (all.bytes(ch_host / p) > 220 * 1024 || (planes * p < 2 * sms && ch_host / p >= 8))) p *= 2;
      const int ch = ch_host / p;
      const bool two = all.bytes(ch) <= 110 * 1024 || (sm.bytes(ch) <= 110 * 1024 && planes * p > sms);   // CTAs share an SM
      if (sm.bytes(ch) <= 220 * 1024 && (long long)staged * ch < 65536) {
        auto launch = [&](auto kernel, int threads) -> cudaError_t {
          const cudaError_t rc = ensure_dynamic_smem(kernel, 220 * 1024);
          if (rc != cudaSuccess) return rc;
          return launch_kernel(kernel, dim3((unsigned)(planes * p)), threads, sm.bytes(ch), K.stream, 1,
              static_cast<T*>(a->k_dst), static_cast<T*>(a->v_dst), da, sm, K.n_kv_heads, ch, p,
              div_multiplier(ch), a->vis_begin, a->n_text_after, gather, a->n_vis, a->n_vis_out,
              a->grp_off, a->grp_src, a->weight);
        };
        if constexpr (sizeof(T) == 2)                     // (fp32 heads have two pieces or more, and planes are not cut to one)
          if (ch == 1) return two ? launch(kv_plane_kernel<T, 512, true>, 512) : launch(kv_plane_kernel<T, 1024, true>, 1024);
        return two ? launch(kv_plane_kernel<T, 512, false>, 512) : launch(kv_plane_kernel<T, 1024, false>, 1024);
      }
    }
    if (!(in_place && gather)) {                          // in place, gather mode has nothing to merge
      auto launch = [&](auto kernel) -> cudaError_t {
        return launch_kernel(kernel, grid, threads, 0, K.stream, 1,
            static_cast<const T*>(a->k_src), static_cast<const T*>(a->v_src), static_cast<T*>(a->k_dst),
            static_cast<T*>(a->v_dst), sa, da, K.n_kv_heads, K.head_dim, a->vis_begin, a->n_text_after, K.cap_in,
            K.cap_out, gather, in_place ? 1 : 0, div_multiplier(ch_host), a->n_vis, a->n_vis_out, a->grp_off, a->grp_src, a->weight);
      };
      bool one = false;
      if constexpr (sizeof(T) == 2) {
        one = ch_host == 1;
        if (one) e = few ? launch(kv_compact_kernel<T, 512, 4, true>) : launch(kv_compact_kernel<T, 256, 2, true>);
      }
      if (!one) e = few ? launch(kv_compact_kernel<T, 512, 4, false>) : launch(kv_compact_kernel<T, 256, 2, false>);
    }
    if (e != cudaSuccess || !in_place) return e;
    // planes: (sample, K / V, head), cut along head_dim while there are fewer of them than CTAs that fit
    int parts = 1;
    while (parts < ch_host && K.batch * 2 * K.n_kv_heads * parts < 4 * sms && ch_host % (2 * parts) == 0) parts *= 2;
    const size_t smem = 2 * size_t(KVM_CHUNK_BYTES);
    if ((e = ensure_dynamic_smem(kv_move_kernel<T>, (int)smem)) != cudaSuccess) return e;
    return launch_kernel(kv_move_kernel<T>, dim3(K.batch * 2 * K.n_kv_heads * parts), KVM_THREADS, smem, K.stream, 1,
        static_cast<T*>(a->k_dst), static_cast<T*>(a->v_dst), da, K.n_kv_heads, K.head_dim, parts, a->vis_begin,
        a->n_text_after, K.cap_in, a->n_vis, a->n_vis_out, a->grp_off, a->grp_src, K.cap_out);
  };
  return K.dtype == LIGHTKV_BF16 ? run(__nv_bfloat16()) : run(float());
}

}  // namespace lkv
