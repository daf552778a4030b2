// Host-side launch interface between the C ABI (lightkv_api.cu) and the kernel files.
#pragma once
#include <atomic>
#include <mutex>

#include "common.cuh"

namespace lkv {

// Launch with programmatic stream serialization (see grid_dependency_sync) and, for cluster > 1, a cluster
// of that many CTAs along x.
template <typename... P, typename... A>
inline cudaError_t launch_kernel(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                 unsigned cluster, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  unsigned n = 0;
  attr[n].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[n].val.programmaticStreamSerializationAllowed = 1;
  ++n;
  if (cluster > 1) {
    attr[n].id = cudaLaunchAttributeClusterDimension;
    attr[n].val.clusterDim.x = cluster; attr[n].val.clusterDim.y = 1; attr[n].val.clusterDim.z = 1;
    ++n;
  }
  cfg.attrs = attr;
  cfg.numAttrs = n;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// SMs of the current device (looked up once per device).  The launches choose variants and splits by it; results do not
// depend on it.
inline int sm_count() {
  constexpr int kB200 = 148, kDevices = 64;
  static std::atomic<int> known[kDevices];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kDevices) return kB200;
  int n = known[dev].load(std::memory_order_relaxed);
  if (n == 0) {
    if (cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || n <= 0) n = kB200;
    known[dev].store(n, std::memory_order_relaxed);
  }
  return n;
}

struct LayerLaunch {
  int batch, hidden, n_q_heads, n_kv_heads, head_dim;
  int dtype, xi_mode, divergence;
  double keep;
  int fd_side;                       // estimate of the larger side (A or B nodes) of a window: picks the FD kernel
  int fd_blocks;                     // tiles of kFdTile nodes a side the largest window may have
  int max_cell;                      // most tokens a window can hold
  int n_grid;                        // grid positions of all tiles
  Geometry geo;
  Workspace ws;
  TextSet text;                      // prompt-token set J of this call
  const lightkv_layer_args_t* a;
  cudaStream_t stream;
};

// How much dynamic shared memory every kernel has been allowed on every device, so that the attribute is set once and not
// before every launch.  Looked up without a lock (a hash table per device whose entries only ever appear and grow).
class SmemLimits {
 public:
  static constexpr int kDevices = 64, kSlots = 256;       // about 40 kernel instances a device
  // `set(bytes)` raises the limit of `kernel` on the current device, which is `dev`
  template <typename Set>
  cudaError_t ensure(const void* kernel, int dev, int bytes, Set set) {
    if (dev < 0 || dev >= kDevices) return set(bytes);
    Slot* s = find(kernel, dev);
    if (s && s->kernel.load(std::memory_order_acquire) == kernel && s->bytes.load(std::memory_order_acquire) >= bytes)
      return cudaSuccess;
    std::lock_guard<std::mutex> lock(mu_);
    s = find(kernel, dev);
    if (s && s->kernel.load(std::memory_order_relaxed) == kernel && s->bytes.load(std::memory_order_relaxed) >= bytes)
      return cudaSuccess;                                 // another thread was here first
    const cudaError_t rc = set(bytes);
    if (rc == cudaSuccess && s) {                         // (a full table forgets: the attribute is set again)
      s->bytes.store(bytes, std::memory_order_release);
      s->kernel.store(kernel, std::memory_order_release);
    }
    return rc;
  }

 private:
  struct Slot { std::atomic<const void*> kernel; std::atomic<int> bytes; };
  // the kernel's slot or the first empty one on its way, nullptr: neither
  Slot* find(const void* kernel, int dev) {
    const uint32_t start = uint32_t((reinterpret_cast<uintptr_t>(kernel) >> 4) * 0x9e3779b97f4a7c15ull >> 32);
    for (int i = 0; i < kSlots; ++i) {
      Slot* s = &slot_[dev][(start + i) % kSlots];
      const void* k = s->kernel.load(std::memory_order_acquire);
      if (k == kernel || !k) return s;
    }
    return nullptr;
  }
  std::mutex mu_;
  Slot slot_[kDevices][kSlots] = {};
};
inline cudaError_t ensure_dynamic_smem_ptr(const void* kernel, int bytes) {
  static SmemLimits limits;
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return cudaErrorInvalidDevice;
  return limits.ensure(kernel, dev, bytes, [&](int n) {
    return cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, n);
  });
}
template <typename... P>
inline cudaError_t ensure_dynamic_smem(void (*kernel)(P...), int bytes) {
  return ensure_dynamic_smem_ptr(reinterpret_cast<const void*>(kernel), bytes);
}

// window build (Step 1 and "Window partitioning")
cudaError_t launch_window_build(const LayerLaunch& L);
// FD + best partner per A node (Step 2), fp32 FMA path
cudaError_t launch_fd_simt(const LayerLaunch& L);
// windows, FD and selection for windows of at most 40 nodes a side (fp32: 80) in one kernel (Steps 1, 2 and 4): leaves every token's partner
// and its place for launch_map
bool fd_stream_supported(int dtype, int fd_side);
cudaError_t launch_fd_stream(const LayerLaunch& L);
// merge map from the partners (Steps 4, 5), with `select` from the keys of launch_fd_tc, and the weights where xi is given or
// uniform, or complete because the launch stands behind the xi kernel; at most kMapMaxTokens per sample
constexpr int kMapMaxTokens = 16384;
cudaError_t launch_map(const LayerLaunch& L, bool select, bool behind_xi = false);
// whether, with xi from attention, the map stands behind the xi kernel and not beside it
bool map_behind_xi(const LayerLaunch& L);
// xi per head (Eq. "attention-factor"), fp32 FMA path; handles ATTN_FULL and ATTN_LSE.  wait_first: the stream's last kernel
// is not one of the same call that lets the next start behind its own wait (FD, or the map behind it)
cudaError_t launch_xi_simt(const LayerLaunch& L, bool wait_first);
// head sum of xi, ranking, merge map, weights (Steps 2-5)
cudaError_t launch_select_map(const LayerLaunch& L);
// head sum of xi and weights behind launch_map and the xi kernel
cudaError_t launch_weights(const LayerLaunch& L);
// weighted merge of the hidden states (Eq. "message-passing"); `weights`: with the head sum of xi and the weights, for
// the launches that are faster so
bool merge_takes_weights(const LayerLaunch& L);
cudaError_t launch_merge_rows(const LayerLaunch& L, bool weights);

struct KvLaunch {
  int batch, n_kv_heads, head_dim, dtype, cap_in, cap_out;
  const lightkv_kv_args_t* a;
  cudaStream_t stream;
};
cudaError_t launch_kv_compact(const KvLaunch& K);

// tcgen05 paths (lightkv_tc.cu).  `supported` queries are host-only.
bool tc_fd_supported(int hidden);
bool tc_xi_supported(int head_dim);
// lists: windows from launch_window_build, keys by source entry for launch_select_map; else by token for launch_map
cudaError_t launch_fd_tc(const LayerLaunch& L, bool lists);
// wait_first: as for launch_xi_simt
cudaError_t launch_xi_tc(const LayerLaunch& L, bool wait_first);

// lightkv_compress_layer.  `least`: a workspace of least_workspace() bytes will do; where the tiled FD kernel's keys do not
// fit it, the call takes the list form.
size_t least_workspace(const lightkv_plan_t* p, int stage);
int compress_layer(const lightkv_plan_t* p, const lightkv_layer_args_t* a, bool least);

}  // namespace lkv
