"""Small functions of the kernels and their launches, and single launches, called from programs compiled with nvcc."""
import os
import subprocess

import pytest

import __graft_entry__ as entry

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2605_00789_b200", "csrc")


def _run(tmp_path, body, *link):
    """Compile `body` (a main file that includes the kernels' headers), run it and return what it prints."""
    src, exe = tmp_path / "unit.cu", tmp_path / "unit"
    src.write_text(body)
    nvcc = os.environ.get("NVCC", "/usr/local/cuda/bin/nvcc")
    subprocess.run([nvcc, "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC,
                    "-I", os.path.join(ROOT, "include"), "-o", str(exe), str(src), *link], check=True)
    return subprocess.check_output([str(exe)]).decode().split()


def test_a_key_that_was_never_written_names_no_destination_outside_the_window(tmp_path):
    """The map kernel turns the low word of a key into an index; a tile whose waits expired leaves whatever the workspace
    held.  Only ranks of destinations the window has may come out, and those of written keys unchanged."""
    out = _run(tmp_path, r"""
#include <stdio.h>
#include "windows.cuh"
int main() {
  const int sizes[] = {0, 1, 7, 128, 2048};
  unsigned long long x = 88172645463325252ull;
  int bad = 0, kept = 0;
  for (int nb : sizes) {
    auto check = [&](unsigned long long key) { const int to = lkv::key_partner(key, nb); bad += to < -1 || to >= nb; };
    for (int i = 0; i < 100000; ++i) {
      x ^= x << 13; x ^= x >> 7; x ^= x << 17;
      check(x); check(x >> 16); check(x >> 32); check(x >> 48);
    }
    check(0); check(~0ull); check(0x80000000ull); check(0x7fffffffull); check(0xffffffff00000000ull | (unsigned)nb);
    for (int to = 0; to < nb; ++to) kept += lkv::key_partner(0x3f80000000000000ull | (unsigned)to, nb) != to;
    bad += lkv::key_partner(~0ull, nb) != -1;
  }
  printf("%d %d\n", bad, kept);
}
""")
    assert out == ["0", "0"]


def test_division_by_a_multiplier_is_exact(tmp_path):
    """Every quotient of the range at small divisors, the numbers around every multiple at all of them."""
    out = _run(tmp_path, r"""
#include <stdio.h>
#include "common.cuh"
int main() {
  int bad = 0;
  for (int d = 2; d < 65536; ++d) {
    const unsigned m = lkv::div_multiplier(d);
    if (d <= 64) for (int n = 0; n < 65536; ++n) bad += lkv::div_magic(n, m) != n / d;
    for (int k = d; k < 65536; k += d) bad += lkv::div_magic(k, m) != k / d || lkv::div_magic(k - 1, m) != (k - 1) / d;
    bad += lkv::div_magic(65535, m) != 65535 / d;
  }
  printf("%d\n", bad);
}
""")
    assert out == ["0"]


def test_the_shared_memory_limit_is_set_once_per_kernel_and_device(tmp_path):
    """Sixty kernels on eight devices, launched in turn with growing and shrinking sizes by two threads: a limit is only ever
    set to raise it, and a set that failed is tried again."""
    out = _run(tmp_path, r"""
#include <stdio.h>
#include <string.h>
#include <atomic>
#include <thread>
#include "launch.h"
static lkv::SmemLimits limits;
int main() {
  static char code[60 * 64];
  static std::atomic<int> calls, limit[8][60];
  auto launches = [&](int bytes) {
    for (int dev = 0; dev < 8; ++dev)
      for (int k = 0; k < 60; ++k) {
        limits.ensure(code + 64 * k, dev, bytes, [&](int n) { ++calls; limit[dev][k] = n; return cudaSuccess; });
        if (limit[dev][k] < bytes) calls += 1000000;
      }
  };
  const int sizes[] = {1000, 1000, 500, 2000, 1000, 2000};             // two raises
  for (int n : sizes) { std::thread other([&] { launches(n); }); launches(n); other.join(); }
  int failed = 0;
  for (int i = 0; i < 2; ++i)
    failed += limits.ensure(code, 1, 9000, [](int) { return cudaErrorInvalidValue; }) == cudaErrorInvalidValue;
  int far = 0;
  for (int i = 0; i < 2; ++i) limits.ensure(code, 64, 10, [&](int) { ++far; return cudaSuccess; });   // beyond the table
  printf("%d %d %d\n", calls.load(), failed, far);
}
""")
    assert out == [str(2 * 8 * 60), "2", "2"]


def test_the_map_waits_for_xi_where_the_counts_are_replaced_in_place(tmp_path):
    """The xi kernel reads the counts item by item, so a map that replaces them stands behind it, however long the launch; one
    with counts of its own runs beside it unless the caller waits for the map of a short launch of few heads or tokens."""
    entry.build()
    out = _run(tmp_path, r"""
#include <stdio.h>
#include "launch.h"
int main() {
  int in[4], out[4], event;
  const int sizes[][3] = {{16, 4000, 3000}, {16, 4000, 100000}, {17, 500, 300}, {17, 501, 300}, {17, 2000, 300}, {17, 2001, 300}};
  for (int mode : {LIGHTKV_XI_ATTN_FULL, LIGHTKV_XI_ATTN_LSE})
    for (const auto& size : sizes)
      for (bool waits : {false, true})
        for (const int* counts : {(const int*)in, (const int*)out, (const int*)nullptr}) {
          lightkv_layer_args_t a = {};
          a.n_vis = counts; a.n_vis_out = out; a.map_event = waits ? &event : nullptr;
          lkv::LayerLaunch L = {};
          L.batch = 1; L.hidden = 4096; L.dtype = LIGHTKV_BF16; L.xi_mode = mode; L.a = &a;
          L.n_q_heads = size[0]; L.ws.cap_in = size[1]; L.ws.cap_out = size[2];
          printf("%d ", lkv::map_behind_xi(L));
        }
}
""", "-L", os.path.dirname(CSRC), "-l:liblightkv.so", "-Xlinker", "-rpath=" + os.path.dirname(CSRC))
    behind, beside = "0 1 0  1 1 1", "0 1 0  0 1 0"
    assert out == " ".join([behind, beside, behind, beside, beside, beside] + [behind, beside, behind, behind, behind, beside]).split()


@pytest.mark.gpu
def test_the_map_of_keys_that_were_never_written_is_a_partition(tmp_path):
    """What the map kernel makes of a workspace whose tiled FD kernel stored no key (its waits expired): the windows' tokens
    are there, the keys are random words.  Whatever is merged, every token ends up in exactly one group."""
    entry.build()
    out = _run(tmp_path, r"""
#include <stdio.h>
#include <vector>
#include "launch.h"
using namespace lkv;
template <typename T> T* device(const std::vector<T>& v) {
  T* p = nullptr;
  cudaMalloc(&p, v.size() * sizeof(T));
  cudaMemcpy(p, v.data(), v.size() * sizeof(T), cudaMemcpyHostToDevice);
  return p;
}
template <typename T> std::vector<T> host(const T* p, size_t n) {
  std::vector<T> v(n);
  cudaMemcpy(v.data(), p, n * sizeof(T), cudaMemcpyDeviceToHost);
  return v;
}
int main() {
  const int sizes[][2] = {{4, 130}, {3, 300}, {1, 2049}};              // windows, tokens of each (windows are stored in turn)
  unsigned long long x = 88172645463325252ull;
  for (const auto& size : sizes) {
    const int B = 2, W = size[0], cell = size[1], n = W * cell, blocks = ((cell + 1) / 2 + kFdTile - 1) / kFdTile;
    std::vector<unsigned long long> key(size_t(B) * blocks * n);
    for (size_t i = 0; i < key.size(); ++i) {
      x ^= x << 13; x ^= x >> 7; x ^= x << 17;
      key[i] = i % 3 ? x : x & 0xffffffff00000fffull;                  // some low words look like destinations
    }
    std::vector<int> tok(size_t(B) * W * (cell + 1));
    for (size_t k = 0; k < size_t(B) * W; ++k) {
      tok[k * (cell + 1)] = cell;
      for (int l = 0; l < cell; ++l) tok[k * (cell + 1) + 1 + l] = int(k % W) * cell + l;
    }
    std::vector<int> ints(size_t(B) * (n + 1), 0);
    std::vector<float> floats(size_t(B) * n, 0.f);
    lightkv_layer_args_t a = {};
    a.n_vis_out = device(ints); a.pos_out = device(ints); a.dst = device(ints); a.grp_off = device(ints);
    a.grp_src = device(ints); a.weight = device(floats); a.status = reinterpret_cast<uint32_t*>(device(ints));
    LayerLaunch L = {};
    L.batch = B; L.xi_mode = LIGHTKV_XI_UNIFORM; L.keep = 0.6; L.fd_blocks = blocks; L.max_cell = cell; L.n_grid = n;
    L.geo.n_windows = W;
    L.ws.tile_key = device(key); L.ws.win_tok = device(tok); L.ws.partner = device(ints); L.ws.slot = device(ints);
    L.ws.cap_in = L.ws.cap_out = L.ws.cap_a = L.ws.cap_b = n; L.ws.n_windows = W;
    L.a = &a;
    const cudaError_t launched = launch_map(L, true), ended = cudaDeviceSynchronize();
    int wrong = launched != cudaSuccess || ended != cudaSuccess, merged = 0;
    const auto n_out = host(a.n_vis_out, B), off = host(a.grp_off, size_t(B) * (n + 1)), src = host(a.grp_src, size_t(B) * n),
               dst = host(a.dst, size_t(B) * n);
    for (int b = 0; b < B && !wrong; ++b) {
      const int* o = &off[size_t(b) * (n + 1)];
      std::vector<int> seen(n, 0);
      wrong += n_out[b] < 0 || n_out[b] > n || o[0] != 0 || o[n_out[b]] != n;
      for (int g = 0; g < n_out[b] && !wrong; ++g)
        for (int c = o[g]; c < o[g + 1] && !wrong; ++c) {
          const int i = src[size_t(b) * n + c];
          wrong += i < 0 || i >= n || seen[i]++ || dst[size_t(b) * n + i] != g;
        }
      merged += n - n_out[b];
    }
    printf("%d %d\n", wrong, merged > 0);
  }
}
""", "-L", os.path.dirname(CSRC), "-l:liblightkv.so", "-Xlinker", "-rpath=" + os.path.dirname(CSRC))
    assert out == ["0", "1"] * 3
