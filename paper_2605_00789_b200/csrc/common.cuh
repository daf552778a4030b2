// Shared device/host helpers of liblightkv (sm_100a only).
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "lightkv.h"

namespace lkv {

constexpr int kMaxTiles = 32;          // image tiles / frames per sample
constexpr int kFdTile = 128;           // sources (and destinations) per tile of the tensor-core FD kernel
constexpr int kMaxWindows = 2048;      // windows per sample (window-build kernel keeps 32 x n_windows u16 counters in smem)
constexpr int kMaxWindowTokens = 65535;  // tokens of one window (range of those counters)

// Grid geometry of one stage, passed by value to the kernels.
struct Geometry {
  int n_tiles;
  int w;                               // windows per axis, per tile
  int n_windows;                       // n_tiles * w * w
  int src_par;                         // parity of the local rank of the source nodes (0: A -> B, 1: B -> A)
  int tile_off[kMaxTiles + 1];         // first flat position of each tile
  int rows[kMaxTiles];
  int cols[kMaxTiles];
};

// Per-stage views into the caller's workspace (all DEVICE pointers, per-sample row strides in elements).
struct Workspace {
  int* win_off;    // [B, n_windows + 1]  first window-sorted slot of each window
  int* a_off;      // [B, n_windows + 1]  first A entry of each window (B entry offset = win_off - a_off)
  int* tok_win;    // [B, cap_in]         window of each token
  int* tok_l;      // [B, cap_in]         local index inside its window (even = A, odd = B)
  int* a_tok;      // [B, cap_a]          token index of each A entry (entries grouped by window)
  int* a_win;      // [B, cap_a]          window of each A entry
  int* b_tok;      // [B, cap_b]          token index of each B entry
  unsigned long long* a_key;  // [B, cap_a]  (orderable(lowest FD) << 32) | B entry index of the best partner;
                              //             all ones while no partner is known (set by the window build)
  // tiled FD kernel without window lists (these two lie over the arrays of the list form)
  unsigned long long* tile_key;  // [B, fd blocks, cap_in]  such keys by block of destinations and token, see fd_tc_kernel
  int* win_tok;    // [B, n_windows, max_cell + 1]  tiled FD kernel: the number of tokens of a window, then the tokens
  float* xi_h;     // [B, cap_in, H]      per-head attention mass on the prompt (ATTN modes): a token's heads in one line
  float* xi;       // [B, cap_in]
  int* partner;    // [B, cap_in]         token a source is merged into; negative: survives (-2: a source that was not
                   //                     selected, where the streaming FD kernel wrote it)
  int* slot;       // [B, cap_in]         output slot of surviving tokens; from the streaming FD kernel: a merged
                   //                     token's rank among its partner's, or the number of tokens merged into this one
  int* a_partner;  // [B, cap_a]          per A entry: token it is merged into, -1 = survives
  int* xi_redo;    // [ceil(cap_in / 128) * H * B]  links between the work items of the tensor-core xi kernel that a
                   //                               CTA has to repeat with a running maximum
  int cap_in, cap_out, cap_a, cap_b, n_windows;
};

// Prompt-token set J: up to LIGHTKV_MAX_TEXT_RANGES ascending, disjoint ranges of sequence indices in front of
// the vision block.  begin / end bound the whole set.
struct TextSet {
  int n;
  int begin, end;
  int lo[LIGHTKV_MAX_TEXT_RANGES], hi[LIGHTKV_MAX_TEXT_RANGES];
  __host__ __device__ inline bool holds(int j) const {
    for (int i = 0; i < n; ++i)
      if (j >= lo[i] && j < hi[i]) return true;
    return false;
  }
  // bit c set <=> key j0 + c belongs to J (c < 32)
  __device__ inline unsigned int mask32(int j0) const {
    if (n != 1) return (unsigned int)mask64(j0);
    const int a = begin > j0 ? begin - j0 : 0, b = end - j0 < 32 ? end - j0 : 32;
    return a >= b ? 0u : (0xffffffffu >> (32 - b)) & (0xffffffffu << a);
  }
  // bit c set <=> key j0 + c belongs to J (c < 64)
  __host__ __device__ inline unsigned long long mask64(int j0) const {
    unsigned long long m = 0;
    for (int i = 0; i < n; ++i) {
      const int a = (lo[i] > j0 ? lo[i] : j0) - j0, b = (hi[i] < j0 + 64 ? hi[i] : j0 + 64) - j0;
      if (b > a) m |= (b - a >= 64 ? ~0ull : ((1ull << (b - a)) - 1ull)) << a;
    }
    return m;
  }
};

// Tokens removed from a window of n tokens when a fraction `keep` must remain:
// floor((1 - keep) n) evaluated as n - ceil(keep n - 1e-9), at most the number of source nodes (the tokens
// of local rank parity `src_par`: ceil(n / 2) A nodes, or floor(n / 2) B nodes in the reverse direction), none
// from a window of one token.
__host__ __device__ inline int removal_count(int n, double keep, int src_par = 0) {
  if (n < 2) return 0;
#ifdef __CUDA_ARCH__
  double t = __dadd_rn(__dmul_rn(keep, (double)n), -1e-9);
#else
  volatile double prod = keep * (double)n;   // no fused multiply-add on the host either
  double t = prod - 1e-9;
#endif
  int r = n - (int)ceil(t);
  int na = (n + 1 - src_par) >> 1;
  return r < 0 ? 0 : (r > na ? na : r);
}

// Window id of a flat grid position; -1 when the position lies outside every tile.
__host__ __device__ inline int window_of(const Geometry& g, int pos) {
  int t = -1;
  for (int i = 0; i < g.n_tiles; ++i)
    if (pos >= g.tile_off[i] && pos < g.tile_off[i + 1]) { t = i; break; }
  if (t < 0) return -1;
  int local = pos - g.tile_off[t];
  int r = local / g.cols[t], c = local - r * g.cols[t];
  return t * g.w * g.w + (r * g.w / g.rows[t]) * g.w + (c * g.w / g.cols[t]);
}

// floor(n / d) for n < 65536, 2 <= d < 65536 by one multiplication with m = ceil(2^32 / d): n * m / 2^32 is more than n / d by
// less than n / 2^32 < 1 / d.  (For d = 1 the multiplier does not fit; the kernels have forms of their own for that.)
inline unsigned int div_multiplier(int d) { return (unsigned int)(((1ull << 32) + d - 1) / d); }
__host__ __device__ inline int div_magic(int n, unsigned int m) {
#ifdef __CUDA_ARCH__
  return (int)__umulhi((unsigned int)n, m);
#else
  return (int)((unsigned long long)(unsigned int)n * m >> 32);
#endif
}

// ---- 16-byte vector access and element conversion -----------------------------------------------
template <typename T> struct Vec;                      // elements per 16 bytes
template <> struct Vec<__nv_bfloat16> { static constexpr int n = 8; };
template <> struct Vec<float> { static constexpr int n = 4; };

__device__ inline void unpack16(const uint4& v, float (&f)[8], __nv_bfloat16) {
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    f[2 * i] = __uint_as_float(u[i] << 16);
    f[2 * i + 1] = __uint_as_float(u[i] & 0xffff0000u);
  }
}
__device__ inline void unpack16(const uint4& v, float (&f)[4], float) {
  f[0] = __uint_as_float(v.x); f[1] = __uint_as_float(v.y);
  f[2] = __uint_as_float(v.z); f[3] = __uint_as_float(v.w);
}
__device__ inline uint4 pack16(const float (&f)[8], __nv_bfloat16) {
  uint32_t u[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    __nv_bfloat162 p = __floats2bfloat162_rn(f[2 * i], f[2 * i + 1]);   // round to nearest even
    u[i] = *reinterpret_cast<uint32_t*>(&p);
  }
  return make_uint4(u[0], u[1], u[2], u[3]);
}
__device__ inline uint4 pack16(const float (&f)[4], float) {
  return make_uint4(__float_as_uint(f[0]), __float_as_uint(f[1]), __float_as_uint(f[2]), __float_as_uint(f[3]));
}
__device__ inline float to_float(__nv_bfloat16 v) { return __bfloat162float(v); }
__device__ inline float to_float(float v) { return v; }

// acc += lo^2 + hi^2 over the four bf16 pairs of v; every product is exact in fp32
__device__ __forceinline__ float sumsq16(const uint4& v, float acc) {
  const uint32_t u[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
  for (int j = 0; j < 4; ++j)
    asm("{\n\t.reg .b16 lo, hi;\n\tmov.b32 {lo, hi}, %1;\n\t"
        "fma.rn.f32.bf16 %0, lo, lo, %0;\n\tfma.rn.f32.bf16 %0, hi, hi, %0;\n\t}" : "+f"(acc) : "r"(u[j]));
  return acc;
}

// streaming 16-byte load / store (read-once data: do not keep in L1)
__device__ inline uint4 ld_stream16(const void* p) {
  uint4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.u32 {%0,%1,%2,%3}, [%4];"
               : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "l"(p));
  return v;
}
__device__ inline void st_stream16(void* p, const uint4& v) {
  asm volatile("st.global.L1::no_allocate.v4.u32 [%0], {%1,%2,%3,%4};"
               :: "l"(p), "r"(v.x), "r"(v.y), "r"(v.z), "r"(v.w) : "memory");
}

__device__ __forceinline__ void prefetch_l2(const void* p) { asm volatile("prefetch.global.L2 [%0];" ::"l"(p)); }

// monotone map float -> uint32 (ascending floats give ascending integers)
__device__ inline uint32_t orderable(float f) {
  uint32_t u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// pair score from the inner product g and the norms of the two rows: the norms themselves for FD = 1 - cosine,
// the squared norms for the Euclidean scores |a|^2 + |b|^2 - 2 g
__device__ __forceinline__ float pair_score(int metric, float g, float na, float nb) {
  if (metric == LIGHTKV_FD_COSINE) {
    const float den = na * nb;
    return 1.0f - (den > 0.f ? g / den : 0.f);
  }
  const float sq = fmaxf(fmaf(-2.0f, g, na + nb), 0.f);
  return metric == LIGHTKV_FD_L2 ? sqrtf(sq) : sq;
}

// Programmatic dependent launch.  Every kernel of the library is launched with programmatic stream serialization:
// it may start once every CTA of the kernel before it has called grid_launch_dependents() or exited, and
// grid_dependency_wait() returns when that kernel has completed and its writes are visible.  Every kernel waits
// before it exits, so a kernel's completion implies that of all before it.  Most wait before they touch global memory
// (grid_dependency_sync: a launch's latency then hides behind its predecessor).  Two use the order further: the first
// kernel of a call (window build or FD) lets the next start only after its own wait, so everything before the call is
// complete when any later kernel of the call starts; and the xi kernels, which read nothing the window build, FD or the
// map write, wait only at their end, i.e. run beside them.  Launched without the attribute, the instructions do nothing.
__device__ __forceinline__ void grid_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void grid_dependency_sync() {
  grid_launch_dependents();
  grid_dependency_wait();
}

}  // namespace lkv
