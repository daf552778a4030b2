// liblightkv kernels, part 3: FD + best partner for small windows, one pass over the hidden states.
#include <algorithm>

#include "launch.h"
#include "tc_common.cuh"
#include "windows.cuh"

namespace lkv {

// ======================================================================================================
// FD + best partner for windows of up to 8 * O source and 8 * O destination nodes (Eq. "similarity", Step 2).
//
// With windows this small the contraction has a few flops per byte and the kernel is bound by reading the vision
// rows once from HBM.  So the rows go straight from global memory into the fragments of mma.sync m16n8k16: no
// shared-memory staging, no swizzle, no barrier per chunk.  One CTA takes one window; its warps split the hidden
// dimension (contiguous column ranges, about 1 KB of every row per warp at eight warps).  Lane (g, t) of a warp
// loads 16 bytes of row g of every group of eight rows: four lanes cover 64 contiguous bytes.  The k order inside
// an MMA is free as long as both operands agree, so the eight bf16 of a 16-byte piece serve as the lane's k
// elements of two MMA steps, for the row's role as an A operand and as a B operand alike.  The squared norms
// accumulate from the same registers (exact products, fp32 sums).  Partial inner products of the warps meet in
// shared memory in warp order, then 8 to 32 lanes per source row take the minimum over the destinations (ties: lowest
// index).  A window with more nodes than the template holds is walked in blocks of 8 * O by 8 * O.
// Since the CTA has its whole window, it also finds the window's tokens (from the positions; no list has to be built
// before) and makes the selection of Steps 2 and 4; what is left for the map kernel is one prefix sum per sample.
// A lane's pieces wait in shared memory (cp.async, a ring of S chunks per warp that only this lane writes and reads,
// so no barrier): loads in flight then cost no registers.  Between events, search and selection included, against the
// tcgen05 kernel with its gathered 128-row tiles alone (which had a window build of 11 to 17 us in front of it): 8 samples
// x 2880 tokens x 4096 in windows of 16: 59 -> 42 us over the whole grid (189 MB: 4.5 TB/s), 49 where positions are given
// and searched; windows of 18: 41 -> 35, of 36: 39 -> 27; 32 x 576 x 5120 in windows of 36: 76 -> 48, of 72: 59 -> 31.
// The contraction alone took 37, 27, 23, 45 and 29 us; a CTA loads nothing while it searches and selects.
// ======================================================================================================
struct FdStreamArgs {
  const void* x;                       // first vision row of sample 0
  const int* seq_start;                // first row of each sample (packed batches) or nullptr
  int64_t batch_stride, row_stride;    // elements
  int d, metric;
  double keep;
  Geometry g;
  const int* n_vis;                    // tokens of each sample, nullptr = cap_in
  const int* pos;                      // grid positions, nullptr = identity
  int cap_in, max_cell;                // max_cell: most tokens a window can hold
  int* partner;                        // [B, cap_in] out, see Workspace
  int* place;                          // [B, cap_in] out
};

__device__ __forceinline__ void mma_m16n8k16(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3,
                                             uint32_t b0, uint32_t b1) {
  asm volatile("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};"
               : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
               : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ void st_shared16(uint32_t addr, const uint4& v) {
  asm volatile("st.shared.v4.u32 [%0], {%1,%2,%3,%4};" ::"r"(addr), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}
__device__ __forceinline__ float4 ld_shared_f4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0,%1,%2,%3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
// the quad of lanes takes 64 bytes of a row: ask L2 for the whole 128-byte line at once
__device__ __forceinline__ void cp_async16_l2(uint32_t smem_dst, const void* gmem_src, uint32_t src_bytes) {
  asm volatile("cp.async.cg.shared.global.L2::128B [%0], [%1], 16, %2;" ::"r"(smem_dst), "l"(gmem_src), "r"(src_bytes) : "memory");
}
// O: groups of eight rows a side; S: 32-column chunks in flight per warp; WARPS: warps of a CTA
template <int O, int S, int WARPS>
struct FdStreamSmem {
  static constexpr int R = 8 * O, PITCH = R + 2;
  static constexpr int RING = WARPS * S * 2 * O * 512;                              // bytes
  static constexpr int PART = (WARPS * R * PITCH + WARPS * 2 * R) * 4;              // over the drained ring
  static constexpr int FIXED = RING > PART ? RING : PART;
  // + the window's lists and the match masks of the search
  static size_t bytes(int max_cell, int cap_in) {
    return FIXED + WindowLists::bytes(max_cell) + window_search_bytes(cap_in);
  }
};

// CTAs an SM holds at least, which bounds the registers (0: as the compiler likes).  Eight warps, bf16: without the bound the
// compiler takes 156 registers for O = 5, one CTA per SM: 128 CTAs in clusters of eight then take two turns (4 x 345 tokens x
// 4096 in windows of 72: 22.5 -> 16.0 us).  O = 3 takes 94 by itself; it may have what nine warps leave, 112: with more the
// CTAs do not fit beside those of the kernel in front (one image, one layer: 27.5 us a pass with up to 112, 30.0 with 120).
// Two warps, where the SM is to hold as many CTAs as the shared memory of their rings allows: 24 samples x 547 tokens x 512 in
// windows of 16 16.6 us with 78 registers, 14.9 with 64; 40 x 576 x 256 in windows of 25 14.6 us with 64 and spills, 13.1 with
// 72; fp32, 24 x 576 x 384 in windows of 16 16.5 us with 80 and spills, 14.9 with 96.
__host__ __device__ constexpr int fd_min_ctas(bool bf16, int o, int warps) {
  if (warps == 8) return !bf16 || o == 4 ? 0 : o <= 2 ? 4 : 2;
  return o == 1 ? (bf16 ? 16 : 10) : o == 2 && bf16 ? 14 : 0;
}
__host__ __device__ constexpr int fd_max_threads(bool bf16, int o, int warps) { return 32 * (bf16 && o == 3 && warps == 8 ? 9 : warps); }

template <typename T, int O, int S, int WARPS>
__global__ void __launch_bounds__(fd_max_threads(sizeof(T) == 2, O, WARPS), fd_min_ctas(sizeof(T) == 2, O, WARPS))
fd_stream_kernel(const __grid_constant__ FdStreamArgs a) {
  grid_dependency_wait();
  grid_launch_dependents();                              // in this order: see grid_dependency_sync
  using M = FdStreamSmem<O, S, WARPS>;
  constexpr int R = M::R, MT = (O + 1) / 2, PITCH = M::PITCH, nwarps = WARPS, NT = 32 * WARPS;
  constexpr bool F32 = sizeof(T) == 4;
  constexpr int EL = 16 / sizeof(T), CH = 4 * EL;         // elements of a 16-byte piece and of a chunk of a row
  extern __shared__ __align__(16) unsigned char smem_raw[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  float* part = reinterpret_cast<float*>(smem_raw);      // [WARPS][R][PITCH] partial inner products
  float* nrm = part + WARPS * R * PITCH;                 // [WARPS][2 R] partial squared norms, row 0: the norms
  const WindowLists lists = WindowLists::at(smem_raw + M::FIXED, a.max_cell);
  unsigned int* match = reinterpret_cast<unsigned int*>(smem_raw + M::FIXED + WindowLists::bytes(a.max_cell));
  __shared__ int warp_sum[WARPS];
  // a cluster of ks CTAs shares a window: CTA `rank` contracts its part of the hidden dimension and finishes every ks-th row
  const int ks = (int)tc::cluster_nctarank(), rank = (int)tc::cluster_ctarank();
  const int w = blockIdx.x / ks, b = blockIdx.y;
  int* partner = a.partner + size_t(b) * a.cap_in;
  int* place = a.place + size_t(b) * a.cap_in;

  const int n = a.n_vis ? max(0, min(a.n_vis[b], a.cap_in)) : a.cap_in;
  const int nw = min(a.max_cell, window_tokens<WARPS>(a.g, a.pos ? a.pos + size_t(b) * a.cap_in : nullptr, n, w, match, warp_sum, [&](int l, int i) {
    if (l < a.max_cell) {
      lists.tok[l] = i;
    } else {                                             // only if positions repeat or lie outside the grid: survives
      partner[i] = -1;
      place[i] = 0;
    }
  }));
  if (nw == 0) return;
  const int par = a.g.src_par;
  const int na_all = (nw + 1 - par) >> 1, nb_all = nw - na_all;   // sources: local ranks of parity `par`
  const int removed = nb_all > 0 ? removal_count(nw, a.keep, par) : 0;
  for (int e = tid; e < na_all; e += NT) { lists.key[e] = 0xffffffffu; lists.best[e] = -1; }
  __syncthreads();

  const int g = lane >> 2, t = lane & 3;
  const int nc = (a.d + CH - 1) / CH, part_id = rank * WARPS + warp, parts = ks * WARPS;
  const int c_lo = part_id * nc / parts, nk = (part_id + 1) * nc / parts - c_lo;
  const T* base = static_cast<const T*>(a.x) + size_t(b) * a.batch_stride +
                  size_t(a.seq_start ? a.seq_start[b] : 0) * a.row_stride + c_lo * CH + t * EL;
  const uint32_t row16 = uint32_t(a.row_stride / EL);    // row pitch in 16-byte units
  // fp32 pieces are read by the whole warp: a row's four pieces are swizzled against bank conflicts
  const uint32_t warp_ring = tc::smem_u32(smem_raw) + warp * S * 2 * O * 512;
  const uint32_t ring = warp_ring + (F32 ? g * 64 + ((t ^ ((g >> 1) & 3)) << 4) : lane * 16);

  for (int a0 = 0; removed > 0 && a0 < na_all; a0 += R) {     // nothing to remove: no scores needed
    const int na = min(R, na_all - a0);
    for (int b0 = 0; b0 < nb_all; b0 += R) {
      const int nb = min(R, nb_all - b0);
      uint32_t off[2 * O];                               // row offsets in 16-byte units, A rows first; all ones: no such row
#pragma unroll
      for (int i = 0; i < O; ++i) {
        off[i] = 8 * i + g < na ? uint32_t(lists.tok[2 * (a0 + 8 * i + g) + par]) * row16 : 0xffffffffu;
        off[O + i] = 8 * i + g < nb ? uint32_t(lists.tok[2 * (b0 + 8 * i + g) + 1 - par]) * row16 : 0xffffffffu;
      }
      // rows the block does not have stay zero in every stage
#pragma unroll
      for (int i = 0; i < 2 * O; ++i)
        if (off[i] == 0xffffffffu)
#pragma unroll
          for (int st = 0; st < S; ++st) st_shared16(ring + (st * 2 * O + i) * 512, make_uint4(0, 0, 0, 0));
      auto issue = [&](int k, int st) {
        if (k < nk) {
          const uint32_t bytes = (c_lo + k) * CH + t * EL < a.d ? 16u : 0u;   // d is a multiple of 8
          const T* p = base + (bytes ? k * CH : 0);
#pragma unroll
          for (int i = 0; i < 2 * O; ++i)
            if (off[i] != 0xffffffffu) cp_async16_l2(ring + (st * 2 * O + i) * 512, p + size_t(off[i]) * EL, bytes);
        }
        tc::cp_async_commit();
      };
      float acc[F32 ? 1 : MT][O][4], accf[F32 ? O : 1][2 * O];
      float ss[2 * O];
#pragma unroll
      for (int i = 0; i < 2 * O; ++i) ss[i] = 0.f;
#pragma unroll
      for (int j = 0; j < O; ++j) {
#pragma unroll
        for (int i = 0; i < (F32 ? 1 : MT); ++i)
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.f;
      }
#pragma unroll
      for (int i = 0; i < (F32 ? O : 1); ++i)
#pragma unroll
        for (int j = 0; j < 2 * O; ++j) accf[i][j] = 0.f;

#pragma unroll
      for (int st = 0; st < S; ++st) issue(st, st);
      for (int k = 0, st = 0; k < nk; ++k) {
        tc::cp_async_wait<S - 1>();                      // this lane's pieces of chunk k
        if constexpr (!F32) {                            // nobody else reads them
          uint4 v[2 * O];
#pragma unroll
          for (int i = 0; i < 2 * O; ++i) v[i] = tc::ld_shared16(ring + (st * 2 * O + i) * 512);
#pragma unroll
          for (int i = 0; i < 2 * O; ++i) ss[i] = sumsq16(v[i], ss[i]);
#pragma unroll
          for (int i = 0; i < MT; ++i) {
            const uint4 lo = v[2 * i], hi = 2 * i + 1 < O ? v[2 * i + 1] : make_uint4(0, 0, 0, 0);
#pragma unroll
            for (int j = 0; j < O; ++j) {
              mma_m16n8k16(acc[i][j], lo.x, hi.x, lo.y, hi.y, v[O + j].x, v[O + j].y);
              mma_m16n8k16(acc[i][j], lo.z, hi.z, lo.w, hi.w, v[O + j].z, v[O + j].w);
            }
          }
        } else {
          // fp32: the warp's lanes hold the pairs (g + 8 i, t + 4 j) and read the chunk's rows from the ring
          __syncwarp();
          const uint32_t chunk = warp_ring + st * 2 * O * 512;
#pragma unroll
          for (int i = 0; i < 2 * O; ++i) {
            const float4 v = ld_shared_f4(ring + (st * 2 * O + i) * 512);
            ss[i] = fmaf(v.w, v.w, fmaf(v.z, v.z, fmaf(v.y, v.y, fmaf(v.x, v.x, ss[i]))));
          }
#pragma unroll
          for (int piece = 0; piece < 4; ++piece) {
            float4 va[O];
#pragma unroll
            for (int i = 0; i < O; ++i) va[i] = ld_shared_f4(chunk + i * 512 + g * 64 + ((piece ^ ((g >> 1) & 3)) << 4));
#pragma unroll
            for (int j = 0; j < 2 * O; ++j) {
              const int rr = t + 4 * (j & 1);
              const float4 vb = ld_shared_f4(chunk + (O + (j >> 1)) * 512 + rr * 64 + ((piece ^ ((rr >> 1) & 3)) << 4));
#pragma unroll
              for (int i = 0; i < O; ++i)
                accf[i][j] = fmaf(va[i].w, vb.w, fmaf(va[i].z, vb.z, fmaf(va[i].y, vb.y, fmaf(va[i].x, vb.x, accf[i][j]))));
            }
          }
          __syncwarp();                                  // everybody has read the stage before it is filled again
        }
        issue(k + S, st);
        st = st + 1 == S ? 0 : st + 1;
      }
      tc::cp_async_wait<0>();
      __syncthreads();                                   // every warp's ring is drained: the partial results go over it
      // ---- partial results of this warp
      float* pw = part + warp * R * PITCH;
      if constexpr (F32) {
#pragma unroll
        for (int i = 0; i < O; ++i)
#pragma unroll
          for (int j = 0; j < 2 * O; ++j) pw[(8 * i + g) * PITCH + t + 4 * j] = accf[i][j];
      } else {
#pragma unroll
        for (int i = 0; i < MT; ++i)
#pragma unroll
          for (int j = 0; j < O; ++j) {
            const int r = 16 * i + g, col = 8 * j + 2 * t;
            *reinterpret_cast<float2*>(pw + r * PITCH + col) = make_float2(acc[i][j][0], acc[i][j][1]);
            if (2 * i + 1 < O) *reinterpret_cast<float2*>(pw + (r + 8) * PITCH + col) = make_float2(acc[i][j][2], acc[i][j][3]);
          }
      }
#pragma unroll
      for (int i = 0; i < 2 * O; ++i) {
#pragma unroll
        for (int o = 1; o < 4; o <<= 1) ss[i] += __shfl_xor_sync(0xffffffffu, ss[i], o);
        if (t == 0) nrm[warp * 2 * R + 8 * i + g] = ss[i];
      }
      __syncthreads();
      // ---- norms and inner products over the warps (and the CTAs of the cluster), in that order
      if (ks == 1) {
        for (int i = tid; i < 2 * R; i += NT) {
          float s = nrm[i];
          for (int k = 1; k < nwarps; ++k) s += nrm[k * 2 * R + i];
          nrm[i] = a.metric == LIGHTKV_FD_COSINE ? sqrtf(s) : s;
        }
        __syncthreads();
      } else {
        for (int i = tid; i < 2 * R; i += NT) {
          float s = nrm[i];
          for (int k = 1; k < nwarps; ++k) s += nrm[k * 2 * R + i];
          nrm[2 * R + i] = s;                            // (row 0 takes the sum over the cluster)
        }
        for (int i = tid; i < na * R; i += NT) {
          const int r = i / R, col = i - r * R;
          if (col >= nb) continue;
          float s = part[r * PITCH + col];
          for (int k = 1; k < nwarps; ++k) s += part[(k * R + r) * PITCH + col];
          part[r * PITCH + col] = s;
        }
        tc::cluster_sync();
        for (int i = tid; i < 2 * R; i += NT) {
          float s = 0.f;
          for (int j = 0; j < ks; ++j) s += tc::ld_cluster_f32(tc::map_to_cta(tc::smem_u32(nrm + 2 * R + i), j));
          nrm[i] = a.metric == LIGHTKV_FD_COSINE ? sqrtf(s) : s;
        }
        __syncthreads();
      }
      // ---- the rows this CTA finishes (every ks-th), each by as many lanes as leave a lane for every row, at least eight
      const int nr = rank < na ? (na - rank + ks - 1) / ks : 0;
      int width = 8;
      while (width < 32 && width < nb && 2 * width * nr <= NT) width *= 2;
      for (int i0 = 0; i0 < nr; i0 += NT / width) {
        const int i = i0 + tid / width, r = rank + i * ks;
        float lowest = 3.0e38f;
        int col_min = -1;
        for (int col = tid & (width - 1); i < nr && col < nb; col += width) {
          float v[8], s = 0.f;
          if (ks == 1) {
#pragma unroll
            for (int k = 0; k < nwarps; ++k) v[k] = part[(k * R + r) * PITCH + col];
#pragma unroll
            for (int k = 0; k < nwarps; ++k) s += v[k];
          } else {
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] = j < ks ? tc::ld_cluster_f32(tc::map_to_cta(tc::smem_u32(part + r * PITCH + col), j)) : 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) s += v[j];
          }
          const float fd = pair_score(a.metric, s, nrm[r], nrm[R + col]);
          if (fd < lowest) { lowest = fd; col_min = col; }
        }
        for (int o = width >> 1; o > 0; o >>= 1) {       // minimum over the lanes, ties to the lower column
          const float of = __shfl_xor_sync(0xffffffffu, lowest, o);
          const int oc = __shfl_xor_sync(0xffffffffu, col_min, o);
          if (oc >= 0 && (col_min < 0 || of < lowest || (of == lowest && oc < col_min))) { lowest = of; col_min = oc; }
        }
        // later blocks of destinations hold higher indices: an equal score keeps the earlier one
        if (i < nr && (tid & (width - 1)) == 0 && col_min >= 0 && orderable(lowest) < lists.key[a0 + r]) {
          lists.key[a0 + r] = orderable(lowest);
          lists.best[a0 + r] = b0 + col_min;
          if (rank > 0) {                                // CTA 0 selects
            tc::st_cluster_u32(tc::map_to_cta(tc::smem_u32(lists.key + a0 + r), 0), orderable(lowest));
            tc::st_cluster_u32(tc::map_to_cta(tc::smem_u32(lists.best + a0 + r), 0), uint32_t(b0 + col_min));
          }
        }
      }
      if (ks == 1) __syncthreads(); else tc::cluster_sync();   // the partial results are overwritten by the next block
    }
  }
  if (rank == 0) select_window(lists, nw, removed, par, partner, place);
}

template <typename T, int O, int S, int WARPS>
static cudaError_t launch_fd_stream_o(const LayerLaunch& L, const FdStreamArgs& f) {
  const size_t smem = FdStreamSmem<O, S, WARPS>::bytes(f.max_cell, f.cap_in);
  const cudaError_t e = ensure_dynamic_smem(fd_stream_kernel<T, O, S, WARPS>, (int)smem);
  if (e != cudaSuccess) return e;
  // few windows: clusters of 2, 4 or 8 CTAs split the hidden dimension further, while that fills no SM twice and leaves a
  // CTA 32 KB to read (fp32, bound by its FMAs: 8 KB) beside the two cluster barriers it costs
  const long long window_bytes = 2ll * L.fd_side * L.hidden * (long long)sizeof(T) * (sizeof(T) == 4 ? 4 : 1);
  const int sms = sm_count();
  int ks = 1;
  while (ks < 8 && (long long)L.geo.n_windows * L.batch * 2 * ks <= sms && window_bytes >= 2 * ks * (32ll << 10)) ks *= 2;
  return launch_kernel(fd_stream_kernel<T, O, S, WARPS>, dim3(L.geo.n_windows * ks, L.batch), 32 * WARPS, smem, L.stream, ks, f);
}

// Eight warps split the hidden dimension where each still gets a few chunks of it (rows of more than 1.5 KB) or the
// windows are too few to fill the SMs; a large batch of a narrow model gets CTAs of two, so that the fixed cost of a
// window (its lists, the meeting of the warps) is paid by fewer threads.
template <int O, int S>
static cudaError_t launch_fd_stream_w(const LayerLaunch& L, const FdStreamArgs& f) {
  const bool wide = L.hidden * (L.dtype == LIGHTKV_FP32 ? 4 : 2) > 1536 || (long long)L.geo.n_windows * L.batch <= sm_count();
  // (fp32, two warps, O = 2: a fourth chunk in flight is worth more than a CTA; 24 x 576 x 384 in windows of 25 20.3 -> 18.9 us)
  constexpr int NARROW32 = O == 2 ? 4 : S;
  if (L.dtype == LIGHTKV_FP32) return wide ? launch_fd_stream_o<float, O, S, 8>(L, f) : launch_fd_stream_o<float, O, NARROW32, 2>(L, f);
  return wide ? launch_fd_stream_o<__nv_bfloat16, O, S, 8>(L, f) : launch_fd_stream_o<__nv_bfloat16, O, S, 2>(L, f);
}

// Five groups of eight rows a side is what the fragments of a thread hold at two CTAs per SM; beyond that the tcgen05
// kernel shares the rows between more pairs (in fp32, where the FMAs bound the work, windows of two blocks a side still
// gain).
bool fd_stream_supported(int dtype, int fd_side) { return fd_side > 0 && fd_side <= (dtype == LIGHTKV_FP32 ? 80 : 40); }

cudaError_t launch_fd_stream(const LayerLaunch& L) {
  const lightkv_layer_args_t* a = L.a;
  FdStreamArgs f;
  f.x = static_cast<const char*>(a->hidden) + size_t(a->vis_begin) * a->hidden_row_stride * (L.dtype == LIGHTKV_FP32 ? 4 : 2);
  f.seq_start = a->seq_start;
  f.batch_stride = a->hidden_batch_stride; f.row_stride = a->hidden_row_stride;
  f.d = L.hidden; f.metric = L.divergence; f.keep = L.keep; f.g = L.geo; f.n_vis = a->n_vis; f.pos = a->pos;
  f.cap_in = L.ws.cap_in; f.max_cell = L.max_cell; f.partner = L.ws.partner; f.place = L.ws.slot;
  // chunks in flight per warp (S): as few as still leave enough CTAs on an SM; with more, fewer CTAs fit and the
  // start and end of a window are less covered (contraction alone: S = 8, 6, 4 39 / 33 / 25 us, 6, 4, 3 37 / 27 / 23; O = 2
  // with S = 4 and three CTAs per SM 1 to 3 us more a pass of 8 x 2880 tokens than S = 3 and four)
  switch ((L.fd_side + 7) / 8) {
    case 1: return launch_fd_stream_w<1, 6>(L, f);
    case 2: return launch_fd_stream_w<2, 3>(L, f);
    case 3: return launch_fd_stream_w<3, 3>(L, f);
    case 4: return launch_fd_stream_w<4, 2>(L, f);
    default: return launch_fd_stream_w<5, 2>(L, f);
  }
}

}  // namespace lkv
