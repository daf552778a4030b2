// liblightkv kernels, part 2: tcgen05 tensor-core contractions fed by TMA (sm_100a).
#include <algorithm>

#include "launch.h"
#include "tc_common.cuh"
#include "windows.cuh"

namespace lkv {

using namespace tc;

// ------------------------------------------------------------------------------------------------------
// Host: tensor maps.  cuTensorMapEncodeTiled is fetched through the runtime so that the library does not
// link against libcuda.
// ------------------------------------------------------------------------------------------------------
typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                                  CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

static EncodeTiledFn encode_fn() {
  static EncodeTiledFn fn = nullptr;
  if (!fn) {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &p, cudaEnableDefault, &q) != cudaSuccess ||
        q != cudaDriverEntryPointSuccess)
      return nullptr;
    fn = reinterpret_cast<EncodeTiledFn>(p);
  }
  return fn;
}

// bf16 tensor [batch, heads, rows, width] with element strides (width contiguous); box = 64 x box_rows
// elements, 128-byte swizzle.
static bool make_map_bhnd(CUtensorMap* map, const void* base, int width, int rows, int heads, int batch,
                          int64_t row_stride, int64_t head_stride, int64_t batch_stride, int box_rows) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return false;
  const cuuint64_t dims[4] = {(cuuint64_t)width, (cuuint64_t)rows, (cuuint64_t)heads, (cuuint64_t)batch};
  const cuuint64_t strides[3] = {(cuuint64_t)row_stride * 2, (cuuint64_t)head_stride * 2,
                                 (cuuint64_t)(batch > 1 ? batch_stride : head_stride * heads) * 2};
  const cuuint32_t box[4] = {64, (cuuint32_t)box_rows, 1, 1};
  const cuuint32_t estr[4] = {1, 1, 1, 1};
  return fn(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(base), dims, strides, box, estr,
            CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
            CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// ======================================================================================================
// xi per head on tensor cores (Eq. "attention-factor" over the softmax rows of Eq. "attention-matrix").
//
// A work item is (tile of 128 vision queries, head, sample).  The grid has one CTA per item, in an order that
// interleaves groups of 64 (sample, head) pairs whose K stays in L2 together, longest rows first inside a group;
// the CTAs that are resident (two per SM) take over the items of CTAs that have not started yet
// (clusterlaunchcontrol.try_cancel), so a CTA is set up once, the next item's loads hide behind the current item's
// last tiles, and no counter in global memory has to be cleared first.  Warp 0 is the scheduler and the TMA
// producer: it decodes an item once, publishes it to the other roles through a two-slot ring in shared memory,
// streams the item's Q tile once and its K tiles (128 keys) through a 2-stage ring; the next item's Q and first K
// tiles are requested as soon as the MMAs of the current item have drained.  Warp 1 issues S = Q K^T
// (128 x 128 x dh, bf16 -> fp32) into one of two TMEM accumulators.  Warps 2-9 are the softmax warps, two threads
// per query row (= TMEM lane): a thread pulls 32 of the 64 logits of a half of the accumulator into registers (the
// warp that takes the last piece releases the accumulator) and adds exp(logit - reference) to two sums (all
// visible keys / prompt keys J); the two threads of a row combine their references and sums once per item through
// shared memory.  Output per head: sum_J / sum_all.
//
// One exponential per logit on the special-function unit (16 per clock per SM) against one MMA per tile; at full load
// the SM clock drops to about 1.6 GHz (power), so what counts is instructions per logit (8 samples x 3008 keys x 32
// heads: 11.0 clocks and 7.3 instructions per warp and logit before the points below, 8.5 and 5.9 with them, 422 -> 330 us):
//   * the reference subtracted before the exponential is the thread's maximum over its FIRST 32 keys only
//     (softmax is invariant to the reference; fp32 holds exp of any later logit up to 88 above it), so the
//     other tiles need no maximum and no rescaling;
//   * runs of whole tiles that need no mask (all rows of the warp see every key; all or none are prompt keys) have a
//     loop of their own: sharing one with the masked tiles cost a register move per logit and more;
//   * scaling and summing take two logits per instruction (fma / add .f32x2: the same time on the FMA pipe, half the
//     issue slots);
//   * XT_POLY_PAIRS of every 16 pairs of exponentials are evaluated on the FMA pipe instead (range reduction + a
//     polynomial of degree four, relative error 2.7e-6): 0 pairs 360 us, 2: 340, 3: 335, 4: 329, 5: 331;
//   * an item is decoded once, by the scheduler, and masks are built only where the prompt set or the diagonal ends.
// Tried and slower: the second half's TMEM load in flight behind the first half's arithmetic (350), the polynomial
// on packed pairs (338).
// A row whose sum left the fp32 range (a later logit more than 88 above the first keys' maximum) is found at
// the end of its item; the CTA puts the item on its own list (links in global memory) and repeats it, once it has
// run out of new ones, with a running maximum and rescaling on every half as an ordinary online softmax does.
// With the caller's row log-sum-exp (LSE) only the prompt key tiles are visited.
// ======================================================================================================
__device__ __forceinline__ float ex2(float x) {          // one MUFU op, flush-to-zero
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// two fp32 values in one 64-bit register, and arithmetic on both
typedef unsigned long long f32x2;
__device__ __forceinline__ f32x2 pack2(float lo, float hi) {
  f32x2 r;
  asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack2(f32x2 v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f32x2 fma2(f32x2 a, f32x2 b, f32x2 c) {
  f32x2 r;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
  return r;
}
__device__ __forceinline__ f32x2 add2(f32x2 a, f32x2 b) {
  f32x2 r;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
  return r;
}
__device__ __forceinline__ float fma_sat(float a, float b, float c) {    // clamped to [0, 1] at no extra cost
  float r;
  asm("fma.rn.sat.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

// What the exponentials of a thread need: logits are scaled to log2 units, x = v * sc - ms.
struct ExpRef {
  f32x2 sc2, nms2;                   // {sc, sc}, {-ms, -ms}
  float sc_y, c_y;                   // y = (x + 126) / 254 = v * sc_y + c_y, clamped to [0, 1] by the fma
  __device__ __forceinline__ void set(float sc, float ms) {
    sc2 = pack2(sc, sc);
    nms2 = pack2(-ms, -ms);
    sc_y = sc * (1.0f / 254.0f);
    c_y = (126.0f - ms) * (1.0f / 254.0f);
  }
};
// 2^x of two logits on the FMA pipe: x is clamped to [-126, 128] (as y in [0, 1]), split into the nearest integer j
// (magic-number add) and r in [-0.5, 0.5]; 2^r by a minimax polynomial of degree four; j is added to the exponent
// field.  x = 128 gives a value of 3.4e38 or more, which the overflow check at the end of the item sees.
__device__ __forceinline__ float ex2_fma(float v, const ExpRef& e) {
  constexpr float kMagic = 12582912.f - 126.f;            // 1.5 * 2^23: the integer lands in the low mantissa bits
  const float y = fma_sat(v, e.sc_y, e.c_y);
  const float t = fmaf(y, 254.f, kMagic);                 // bits: 0x4b400000 + j
  const float r = fmaf(y, 254.f, kMagic - t);
  float p = fmaf(r, 0.009570102207f, 0.05591785908f);
  p = fmaf(p, r, 0.2402474433f);
  p = fmaf(p, r, 0.6931217909f);
  p = fmaf(p, r, 0.9999992847f);
  return __int_as_float(__float_as_int(p) + (__float_as_int(t) << 23));
}

struct XiTcArgs {
  const int* n_vis;
  const int* seq_start;              // first row of each sample in q, k, lse, lse_out (packed batches) or nullptr
  float* xi_h;
  uint32_t* status;
  const float* lse;                  // [B, H, N] row log-sum-exp (natural log) from the caller, or nullptr
  int64_t lse_bs, lse_hs;
  float* lse_out;                    // [B, H, N] receives the row log-sum-exp of the vision rows, or nullptr
  int64_t lse_out_bs, lse_out_hs;
  TextSet text;                      // prompt-token set J
  int n_text_after, bidirectional;   // bidirectional: every query sees all keys of its sample
  int cap_in, vis_begin, n_q_heads, group;
  int batch, n_qt;                   // samples, query tiles of 128 rows per (sample, head)
  float scale2;                      // log2(e) / sqrt(dh)
  int wait_first;                    // 1: the window build is not the kernel in front (see below)
  int* redo_next;                    // [n_qt * H * B] links of the CTAs' lists of items whose sums left the fp32 range
};

constexpr int XT_STAGES = 2;         // K tiles in the shared-memory ring
constexpr int XT_SBUF = 2;           // S accumulators in tensor memory
constexpr int XT_CTAS = 2;           // CTAs per SM
constexpr int XT_KEY_TILE = 128;     // keys per K tile and per MMA (the softmax warps read it as two halves of 64)
constexpr int XT_SUB = 64;           // keys per half
constexpr int XT_THREADS = 320;      // TMA / scheduler warp, MMA warp, eight softmax warps
constexpr int XT_HEAD_GROUP = 64;    // (sample, head) pairs whose work items are interleaved (their K: 64 x ~1 MB)
constexpr int XT_POLY_PAIRS = 4;     // of 16 pairs of exponentials: on the FMA pipe

// adds exp over 32 logits of a thread to two pairs of sums (masked logits are -inf and add nothing that counts)
__device__ __forceinline__ void exp_add32(const float (&v)[32], const ExpRef& e, f32x2 (&part)[2]) {
#pragma unroll
  for (int i = 0; i < 16; ++i) {
    f32x2 p;
    if ((i * XT_POLY_PAIRS) % 16 < XT_POLY_PAIRS) {
      p = pack2(ex2_fma(v[2 * i], e), ex2_fma(v[2 * i + 1], e));
    } else {
      float x0, x1;
      unpack2(fma2(pack2(v[2 * i], v[2 * i + 1]), e.sc2, e.nms2), x0, x1);
      p = pack2(ex2(x0), ex2(x1));
    }
    part[i & 1] = add2(part[i & 1], p);
  }
}
__device__ __forceinline__ float sum_pairs(const f32x2 (&part)[2]) {
  float s0, s1;
  unpack2(add2(part[0], part[1]), s0, s1);
  return s0 + s1;
}

// LSE: the caller supplied the row log-sum-exp (a.lse != nullptr).
template <int DH, bool LSE>
__global__ void __launch_bounds__(XT_THREADS, XT_CTAS)
xi_tc_kernel(const __grid_constant__ CUtensorMap q_map, const __grid_constant__ CUtensorMap k_map, XiTcArgs a) {
  constexpr int BK = XT_KEY_TILE;
  static_assert(BK == 2 * XT_SUB && XT_SUB == 64, "a K tile is two halves of 64 keys; the prompt mask of a half is one 64-bit word");
  constexpr int HALVES = DH / 64;
  constexpr uint32_t TILE_BYTES = HALVES * 16384;          // Q tile: 128 rows x DH bf16
  constexpr uint32_t KHALF_BYTES = BK * 128;               // BK key rows x 64 columns
  constexpr uint32_t KT_BYTES = HALVES * KHALF_BYTES;      // K tile: BK rows x DH bf16
  // With the caller's normaliser an item is one or two key tiles and the kernel is bound by reading Q from HBM:
  // then the Q tile is double buffered (two items' Q in flight per CTA) and one K stage is enough.
  constexpr int QBUF = LSE ? 2 : 1, KSTAGES = LSE ? 1 : XT_STAGES;

  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* q_s = base;                   // [QBUF] Q tiles
  unsigned char* k_s = base + QBUF * TILE_BYTES;
  unsigned char* ctl = base + QBUF * TILE_BYTES + KT_BYTES * KSTAGES;
  int4* item_slot = reinterpret_cast<int4*>(ctl);          // [2][2] published items
  uint4* clc_slot = reinterpret_cast<uint4*>(ctl + 64);    // answer to the request for another CTA's item
  uint64_t* bars = reinterpret_cast<uint64_t*>(ctl + 80);
  uint64_t* q_full = bars;                     // [2]
  uint64_t* q_empty = bars + 2;                // [2] every MMA that reads the Q tile has completed
  uint64_t* k_full = bars + 4;                 // [XT_STAGES]
  uint64_t* k_empty = k_full + XT_STAGES;      // [XT_STAGES]
  uint64_t* s_full = k_empty + XT_STAGES;      // [XT_SBUF]
  uint64_t* s_empty = s_full + XT_SBUF;        // [XT_SBUF]
  uint64_t* item_full = s_empty + XT_SBUF;     // [2] the scheduler published an item
  uint64_t* item_empty = item_full + 2;        // [2] the MMA thread has read it, the eight softmax warps are done with it
  uint64_t* pair_full = item_empty + 2;        // the upper column group has stored its partial sums of an item
  uint64_t* pair_empty = pair_full + 1;        // the lower column group has read them
  uint64_t* clc_full = pair_empty + 1;         // clc_slot has been written
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(clc_full + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  int* redo_mark = const_cast<int*>(abort_flag) + 1;       // last item this CTA put on its list
  int* redo_head = redo_mark + 1;                          // first item of the list, -1: empty
  float* pair_m = reinterpret_cast<float*>(ctl + 384);     // [128] each
  float* pair_all = pair_m + 128;
  float* pair_txt = pair_all + 128;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // key tiles to visit: all tiles up to the last query's own key, or, when the caller supplies the row
  // log-sum-exp, only the tiles that hold prompt keys (J lies before the vision block, so it is visible)
  const int kt_lo = LSE ? a.text.begin / BK : 0;
  const int nsub_lse = a.text.end > a.text.begin ? (a.text.end - 1) / XT_SUB + 1 - 2 * kt_lo : 0;

  if (threadIdx.x == 0) {
    for (int i = 0; i < 2; ++i) { mbar_init(&q_full[i], 1); mbar_init(&q_empty[i], 1); }
    for (int i = 0; i < XT_STAGES; ++i) { mbar_init(&k_full[i], 1); mbar_init(&k_empty[i], 1); }
    for (int i = 0; i < XT_SBUF; ++i) { mbar_init(&s_full[i], 1); mbar_init(&s_empty[i], 8); }
    for (int i = 0; i < 2; ++i) { mbar_init(&item_full[i], 1); mbar_init(&item_empty[i], 9); }
    mbar_init(pair_full, 4);
    mbar_init(pair_empty, 4);
    mbar_init(clc_full, 1);
    *abort_flag = 0;
    *redo_mark = -1;
    *redo_head = -1;
    fence_barrier_init();
    prefetch_tensormap(&q_map);
    prefetch_tensormap(&k_map);
  }
  if (warp == 1) { tmem_alloc(tmem_slot, XT_SBUF * BK); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem_base = *tmem_slot;
  // Behind the window build and FD of the same call everything this kernel reads is complete, and nothing reads what
  // it writes before it has completed: it runs beside them and waits for them at its end (grid_dependency_sync).
  grid_launch_dependents();
  if (a.wait_first) grid_dependency_wait();

  if (warp == 0) {
    if (lane == 0) {
      // ---- scheduler + TMA producer
      struct Item { int h, b, t0, nq, n_seq, nsub, row0; };
      // item -> (query tile, head, sample).  The (sample, head) pairs are taken in groups of XT_HEAD_GROUP whose
      // keys stay in L2 together; inside a group the list runs over the query tiles from the longest rows to the
      // shortest, all pairs of the group for each, so that the work left for the last items is short.
      auto decode = [&](int item, Item& it) -> bool {
        const int n_hb = a.n_q_heads * a.batch, per_group = XT_HEAD_GROUP * a.n_qt;
        const int grp = item / per_group, within = item - grp * per_group;
        const int gsize = min(XT_HEAD_GROUP, n_hb - grp * XT_HEAD_GROUP);
        const int qi = within / gsize, hb = grp * XT_HEAD_GROUP + within - qi * gsize;
        it.b = hb / a.n_q_heads; it.h = hb - it.b * a.n_q_heads;
        const int n = a.n_vis ? min(a.n_vis[it.b], a.cap_in) : a.cap_in;
        it.t0 = (a.n_qt - 1 - qi) * 128;
        if (it.t0 >= n) return false;
        it.nq = min(128, n - it.t0);
        it.n_seq = a.vis_begin + n + a.n_text_after;
        // halves of 64 keys the item visits
        it.nsub = LSE ? nsub_lse : ((a.bidirectional ? it.n_seq : a.vis_begin + it.t0 + it.nq) - 1) / XT_SUB + 1;
        it.row0 = a.seq_start ? a.seq_start[it.b] : 0;     // packed batch: one long row axis, batch coordinate 0
        return true;
      };
      uint32_t kf = 0, n = 0, nq_loaded = 0, n_clc = 0;    // K tiles fetched / items published / Q tiles loaded / requests
      auto publish = [&](int item, const Item& it, int safe) -> bool {
        const uint32_t slot = n & 1;
        if (!mbar_wait(&item_empty[slot], ((n >> 1) & 1) ^ 1, abort_flag)) return false;
        item_slot[2 * slot] = make_int4(item, it.h, it.b, it.t0 + safe);       // t0 is a multiple of 128
        item_slot[2 * slot + 1] = make_int4(it.nq, it.n_seq, it.nsub, it.row0);
        mbar_arrive(&item_full[slot]);                     // release: the slot is written before the arrival is seen
        ++n;
        return true;
      };
      bool asked = false;                                  // a request for another CTA's item is on its way
      auto ask = [&]() {
        if (asked) return;
        mbar_expect_tx(clc_full, 16);
        clc_try_cancel(clc_slot, clc_full);
        asked = true;
      };
      auto feed = [&](const Item& it, bool last_asks) -> bool {    // the item's Q and K tiles
        const int nkt = (it.nsub + 1) / 2;
        if (nkt == 0) return true;
        // a Q buffer is free once every MMA of the item that used it last has completed
        const uint32_t qb = nq_loaded % QBUF, q_use = nq_loaded / QBUF;
        const int bc = a.seq_start ? 0 : it.b;
        if (q_use > 0 && !mbar_wait(&q_empty[qb], (q_use - 1) & 1, abort_flag)) return false;
        mbar_expect_tx(&q_full[qb], TILE_BYTES);
        // Q is read once; what stays in L2 instead is read again: K here and by the compaction, the hidden states by the merge
        // (us a pass with a given log-sum-exp: 8 x 2880 tokens 507 -> 500, 4 x 576 104.6 -> 102.2)
#pragma unroll
        for (int hf = 0; hf < HALVES; ++hf)
          tma_load_4d_once(q_s + qb * TILE_BYTES + hf * 16384, &q_map, &q_full[qb], hf * 64, it.row0 + a.vis_begin + it.t0, it.h, bc);
        ++nq_loaded;
        const int hk = it.h / a.group;
        for (int kt = 0; kt < nkt; ++kt, ++kf) {
          const uint32_t s = kf % KSTAGES;
          if (last_asks && kt == nkt - 1) ask();           // late, so that no CTA sits on an item others could start
          if (!mbar_wait(&k_empty[s], ((kf / KSTAGES) & 1) ^ 1, abort_flag)) return false;
          mbar_expect_tx(&k_full[s], KT_BYTES);
#pragma unroll
          for (int hf = 0; hf < HALVES; ++hf)
            tma_load_4d(k_s + s * KT_BYTES + hf * KHALF_BYTES, &k_map, &k_full[s], hf * 64, it.row0 + (kt_lo + kt) * BK, hk, bc);
        }
        return true;
      };
      bool ok = true;
      Item it;
      for (int item = blockIdx.x; ok && item >= 0;) {
        if (decode(item, it)) ok = publish(item, it, 0) && feed(it, true);
        ask();
        ok = mbar_wait(clc_full, n_clc & 1, abort_flag) && ok;   // the answer is awaited even when the item failed
        ++n_clc;
        asked = false;
        item = clc_canceled_cta(clc_slot);
        fence_proxy_async();                               // the slot has been read before the next answer is written
      }
      if (!LSE && ok) {
        // all items handed out: once the softmax warps are done with the last two, the list of this CTA is complete
        ok = mbar_wait(&item_empty[n & 1], ((n >> 1) & 1) ^ 1, abort_flag) &&
             mbar_wait(&item_empty[(n + 1) & 1], (((n + 1) >> 1) & 1) ^ 1, abort_flag);
        int item = ok ? *const_cast<volatile int*>(redo_head) : -1;
        while (ok && item >= 0) {
          const int next = __ldcg(a.redo_next + item);     // read before the item runs again
          ok = decode(item, it) && publish(item, it, 1) && feed(it, false);
          item = next;
        }
      }
      it.h = it.b = it.t0 = it.nq = it.n_seq = it.nsub = it.row0 = 0;
      if (ok) publish(-1, it, 0);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---- MMA issue
      constexpr uint32_t idesc_full = idesc_bf16(128, BK), idesc_half = idesc_bf16(128, XT_SUB);
      // the operand descriptors are built once (Q: one per 16-column step; K: those of ring stage 0, a stage
      // adds a constant to the address field)
      uint64_t q_desc[DH / 16], k_desc[DH / 16];
#pragma unroll
      for (int kk = 0; kk < DH / 16; ++kk) {
        q_desc[kk] = smem_desc_sw128(smem_u32(q_s) + (kk >> 2) * 16384 + (kk & 3) * 32);
        k_desc[kk] = smem_desc_sw128(smem_u32(k_s) + (kk >> 2) * KHALF_BYTES + (kk & 3) * 32);
      }
      uint32_t kc = 0, n = 0, nq_used = 0;             // K tiles consumed / items read / Q tiles used
      for (;;) {
        const uint32_t slot = n & 1;
        if (!mbar_wait(&item_full[slot], (n >> 1) & 1, abort_flag)) break;
        const int item = item_slot[2 * slot].x, nsub = item_slot[2 * slot + 1].z, nkt = (nsub + 1) / 2;
        mbar_arrive(&item_empty[slot]);
        ++n;
        if (item < 0) break;
        if (nkt == 0) continue;
        const uint32_t qb = nq_used % QBUF;
        if (!mbar_wait(&q_full[qb], (nq_used / QBUF) & 1, abort_flag)) break;
        const uint64_t q_off = uint64_t(qb * (TILE_BYTES >> 4));
        bool ok = true;
        for (int kt = 0; kt < nkt; ++kt, ++kc) {
          const uint32_t s = kc % KSTAGES, buf = kc % XT_SBUF;
          if (!mbar_wait(&s_empty[buf], ((kc / XT_SBUF) & 1) ^ 1, abort_flag) ||
              !mbar_wait(&k_full[s], (kc / KSTAGES) & 1, abort_flag)) { ok = false; break; }
          tc_fence_after();
          const uint64_t stage_off = uint64_t(s * (KT_BYTES >> 4));     // the address field counts 16-byte units
          const uint32_t d_addr = tmem_base + buf * BK;
          // the last tile of an odd number of halves needs its first 64 keys only
          const uint32_t idesc = (2 * kt + 2 > nsub) ? idesc_half : idesc_full;
#pragma unroll
          for (int kk = 0; kk < DH / 16; ++kk) umma_bf16(d_addr, q_desc[kk] + q_off, k_desc[kk] + stage_off, idesc, kk > 0);
          umma_commit(&k_empty[s]);
          umma_commit(&s_full[buf]);
        }
        if (!ok) break;
        umma_commit(&q_empty[qb]);
        ++nq_used;
      }
    }
  } else {
    // ---- softmax warps: two threads per query row.  Warps 2-5 take the lower 32 columns of every half of 64
    //      keys, warps 6-9 the upper 32; warp w may read the TMEM lanes of quadrant w % 4.  Each thread keeps
    //      its own reference and sums; the two partial results of a row are combined once per item.
    const int sw = warp - 2, quad = warp & 3, cg = sw >> 2;   // softmax warp 0..7, lane quadrant, column group
    const int r = quad * 32 + lane;                     // query row of this thread
    const uint32_t lane_addr = tmem_base + (uint32_t(quad * 32) << 16) + cg * 32;
    const float sc = a.scale2;
    uint32_t kc = 0, n = 0, np = 0;                     // key tiles consumed / items read / exchanges done by this CTA
    bool alive = true;
    while (alive) {
      const uint32_t slot = n & 1;
      const bool published = mbar_wait(&item_full[slot], (n >> 1) & 1, abort_flag);
      if (!__all_sync(0xffffffffu, published)) break;
      const int4 i0 = item_slot[2 * slot], i1 = item_slot[2 * slot + 1];
      ++n;
      const int item = i0.x, h = i0.y, b = i0.z, t0 = i0.w & ~1, nq = i1.x, nsub = i1.z, row0 = i1.w;
      if (item < 0) break;
      const bool safe = i0.w & 1;
      const int s_first = a.vis_begin + t0;
      // last key seen by the first row of this warp / by this thread's row
      const int lim_lo = a.bidirectional ? i1.y - 1 : s_first + quad * 32;
      const int lim_own = a.bidirectional ? i1.y - 1 : s_first + r;
      float m_run = -INFINITY, l_all = 0.f, l_txt = 0.f;
      bool need_ref = !LSE;                             // some row of the warp has no reference yet
      ExpRef er;
      er.set(sc, 0.f);
      // the caller's normaliser of this row, in log2 units (fetched before the first wait: its latency hides there)
      if (LSE) {
        float l2 = 0.f;
        if (r < nq) l2 = a.lse[size_t(b) * a.lse_bs + size_t(h) * a.lse_hs + row0 + s_first + r] * 1.4426950408889634f;
        er.set(sc, l2);
      }
      const int nkt = (nsub + 1) / 2;
      int kt = 0;
      while (kt < nkt) {
        if (!LSE && !need_ref) {
          // The bulk: a run of whole tiles whose keys are visible to every row of the warp and all of which, or none of
          // which, are prompt keys.  A loop of its own, without masks: two thirds and more of the logits pass here.
          const int jt = kt * BK + cg * 32;             // first key of this thread's columns
          const bool inside = a.text.n == 1 && jt >= a.text.begin;
          const int end_key = min(inside && jt < a.text.end ? a.text.end : 0x7fffffff, lim_lo + 1);
          const bool uniform = jt >= a.text.end || (inside && jt + XT_SUB + 32 <= a.text.end);
          const int run_end = uniform ? min((end_key - cg * 32 - XT_SUB - 32 + BK) / BK, nsub / 2) : 0;
          if (kt < run_end) {
            const bool count = jt < a.text.end;
            f32x2 part[2] = {0ull, 0ull};
            do {
              const uint32_t buf = kc % XT_SBUF;
              const bool landed = mbar_wait(&s_full[buf], (kc / XT_SBUF) & 1, abort_flag);
              if (!__all_sync(0xffffffffu, landed)) { alive = false; break; }   // the TMEM loads below are warp-wide
              tc_fence_after();
              float va[32], vb[32];
              tmem_ld32(lane_addr + buf * BK, va);
              tmem_ld_wait();
              exp_add32(va, er, part);
              tmem_ld32(lane_addr + buf * BK + XT_SUB, vb);
              tmem_ld_wait();
              tc_fence_before();
              __syncwarp();
              if (lane == 0) mbar_arrive(&s_empty[buf]);   // the accumulator is in registers: hand it back
              exp_add32(vb, er, part);
              ++kc;
            } while (++kt < run_end);
            if (!alive) break;
            const float s = sum_pairs(part);
            l_all += s;
            if (count) l_txt += s;
            continue;
          }
        }
        const uint32_t buf = kc % XT_SBUF;
        const bool landed = mbar_wait(&s_full[buf], (kc / XT_SBUF) & 1, abort_flag);
        if (!__all_sync(0xffffffffu, landed)) { alive = false; break; }
        tc_fence_after();
        const int n_half = min(2, nsub - 2 * kt);       // halves of this tile the item needs
        for (int half = 0; half < n_half; ++half) {
          const int j0 = (kt_lo + kt) * BK + half * XT_SUB + cg * 32;      // first key of this thread's 32 columns
          float v[32];
          tmem_ld32(lane_addr + buf * BK + half * XT_SUB, v);
          tmem_ld_wait();
          if (half == n_half - 1) {
            tc_fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(&s_empty[buf]);
          }
          // prompt keys among the 32 (warp-uniform)
          const unsigned int tm = j0 < a.text.end && j0 + 32 > a.text.begin ? a.text.mask32(j0) : 0u;
          if (LSE && tm == 0u) continue;
          const int lim = lim_own - j0;                 // last visible column of this row
          if (!LSE) {
            if (j0 > lim_lo + (a.bidirectional ? 0 : 31)) continue;         // no row of this warp sees any of these keys
            if (j0 + 31 > lim_lo) {                     // some row does not: the diagonal, or the end of the sample
#pragma unroll
              for (int i = 0; i < 32; ++i)
                if (i > lim) v[i] = -INFINITY;
            }
            if (need_ref) {
              // reference of the thread: maximum of the first 32 columns of its own in which it sees a key (the
              // first 64 keys of the row, unless the row is among the first 32 of a sequence), of every half when
              // safe.  While some row of the warp has no reference yet the others update theirs, which is exact.
              float mx[4] = {v[0], v[1], v[2], v[3]};
#pragma unroll
              for (int i = 4; i < 32; ++i) mx[i & 3] = fmaxf(mx[i & 3], v[i]);
              const float m_new = fmaxf(fmaxf(fmaxf(mx[0], mx[1]), fmaxf(mx[2], mx[3])), m_run);
              if (m_new > -INFINITY) {                  // (a thread whose 32 columns are all masked keeps none)
                const float resc = ex2((m_run - m_new) * sc);   // 0 on the first half
                l_all *= resc;
                l_txt *= resc;
                m_run = m_new;
                er.set(sc, m_run * sc);
              }
              need_ref = safe || __any_sync(0xffffffffu, m_run == -INFINITY);
            }
          }
          if (tm == 0u || tm == 0xffffffffu) {
            f32x2 part[2] = {0ull, 0ull};
            exp_add32(v, er, part);
            const float s = sum_pairs(part);
            l_all += s;
            if (tm) l_txt += s;
          } else {                                      // the prompt set begins or ends among these keys
            float sa = 0.f, st = 0.f;
#pragma unroll
            for (int i = 0; i < 16; ++i) {
              float x0, x1;
              unpack2(fma2(pack2(v[2 * i], v[2 * i + 1]), er.sc2, er.nms2), x0, x1);
              const float p0 = ex2(x0), p1 = ex2(x1);   // exp2(-inf) = 0 on masked columns
              sa += p0 + p1;
              if ((tm >> (2 * i)) & 1u) st += p0;
              if ((tm >> (2 * i + 1)) & 1u) st += p1;
            }
            l_all += sa;
            l_txt += st;
          }
        }  // halves
        ++kt;
        ++kc;
      }  // key tiles
      // ---- the two threads of a row meet: the upper column group hands its reference and sums over.  Every warp
      //      that entered the item takes part, also after a failed wait (the flag is raised, nothing is stored).
      if (cg == 1) {
        const bool free_again = np == 0 || mbar_wait(pair_empty, (np - 1) & 1, abort_flag);
        if (!__all_sync(0xffffffffu, free_again)) alive = false;
        if (alive) { pair_m[r] = m_run; pair_all[r] = l_all; pair_txt[r] = l_txt; }
        __syncwarp();
        if (lane == 0) { mbar_arrive(pair_full); mbar_arrive(&item_empty[slot]); }
        ++np;
        continue;
      }
      {
        const bool handed = mbar_wait(pair_full, np & 1, abort_flag);
        if (!__all_sync(0xffffffffu, handed)) alive = false;
        ++np;
        if (!alive) break;
        if (!LSE) {
          const float m_o = pair_m[r], all_o = pair_all[r], m_new = fmaxf(m_run, m_o);
          // a sum at the end of the fp32 range means some logit lay more than 88 above the reference: the item goes on
          // the CTA's list, once (before the exchange buffers are handed back: no warp can be an item ahead here)
          const bool bad = r < nq && !safe && !(l_all <= 3.0e38f && all_o <= 3.0e38f);
          if (__any_sync(0xffffffffu, bad) && lane == 0 && atomicExch(redo_mark, item) != item)
            a.redo_next[item] = atomicExch(redo_head, item);
          const float f_own = ex2((m_run - m_new) * sc), f_o = m_o > -INFINITY ? ex2((m_o - m_new) * sc) : 0.f;
          l_all = fmaf(l_all, f_own, all_o * f_o);
          l_txt = fmaf(l_txt, f_own, pair_txt[r] * f_o);
          m_run = m_new;
        } else {
          l_txt += pair_txt[r];
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(pair_empty);             // the exchange buffers are free for the next item
      }
      if (r < nq && !*abort_flag) {
        a.xi_h[(size_t(b) * a.cap_in + t0 + r) * a.n_q_heads + h] = LSE ? l_txt : l_txt / l_all;
        if (!LSE && a.lse_out)
          a.lse_out[size_t(b) * a.lse_out_bs + size_t(h) * a.lse_out_hs + row0 + s_first + r] =
              fmaf(m_run, sc, log2f(l_all)) * 0.6931471805599453f;
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&item_empty[slot]);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem_base, XT_SBUF * BK);
  }
  if (threadIdx.x == 0 && *abort_flag && a.status) atomicOr(a.status, LIGHTKV_STATUS_TIMEOUT);
  grid_dependency_wait();
}

// A head of up to 64 (128) columns takes the kernel for 64 (128): the TMA loads fill the columns it lacks with zeros.
bool tc_xi_supported(int head_dim) { return head_dim <= 128; }

cudaError_t launch_xi_tc(const LayerLaunch& L, bool wait_first) {
  const lightkv_layer_args_t* a = L.a;
  const int rows = a->seq_rows > 0 ? a->seq_rows : a->vis_begin + L.ws.cap_in + a->n_text_after;
  CUtensorMap qm, km;
  const int map_batch = a->seq_start ? 1 : L.batch;       // packed batch: every sample lives on one row axis
  if (!make_map_bhnd(&qm, a->q, L.head_dim, rows, L.n_q_heads, map_batch, a->q_row_stride, a->q_head_stride,
                     a->q_batch_stride, 128) ||
      !make_map_bhnd(&km, a->k, L.head_dim, rows, L.n_kv_heads, map_batch, a->k_row_stride, a->k_head_stride,
                     a->k_batch_stride, XT_KEY_TILE))
    return cudaErrorInvalidValue;
  XiTcArgs x;
  x.n_vis = a->n_vis; x.seq_start = a->seq_start; x.xi_h = L.ws.xi_h; x.status = a->status; x.cap_in = L.ws.cap_in;
  x.lse = L.xi_mode == LIGHTKV_XI_ATTN_LSE ? a->lse : nullptr; x.lse_bs = a->lse_batch_stride; x.lse_hs = a->lse_head_stride;
  x.lse_out = L.xi_mode == LIGHTKV_XI_ATTN_FULL ? a->lse_out : nullptr;
  x.lse_out_bs = a->lse_out_batch_stride; x.lse_out_hs = a->lse_out_head_stride;
  x.text = L.text; x.n_text_after = a->n_text_after; x.bidirectional = a->bidirectional;
  x.vis_begin = a->vis_begin;
  x.n_q_heads = L.n_q_heads; x.group = L.n_q_heads / L.n_kv_heads;
  x.scale2 = 1.4426950408889634f / sqrtf((float)L.head_dim);
  x.batch = L.batch; x.n_qt = (L.ws.cap_in + 127) / 128;
  x.redo_next = L.ws.xi_redo; x.wait_first = wait_first ? 1 : 0;
  const long long n_items = (long long)x.n_qt * L.n_q_heads * L.batch;
  if (n_items > 0x7fffffffLL) return cudaErrorInvalidValue;
  // One CTA per item, taken over by the resident ones (with the caller's log-sum-exp, too, whose items are alike: FD and
  // the map may hold some SMs for a while, and a fixed share of the items would wait for them)
  const dim3 grid((unsigned)n_items);
  // Q tiles + K ring (LSE: two Q tiles, one K stage; otherwise one Q tile, XT_STAGES K stages) + control block + exchange
  const int halves = L.head_dim <= 64 ? 1 : 2;
  const size_t smem = size_t(halves) * (x.lse ? 2 * 16384 + XT_KEY_TILE * 128
                                                        : 16384 + size_t(XT_STAGES) * XT_KEY_TILE * 128) + 1024 + 384 + 1536;
  auto launch = [&](auto kernel) -> cudaError_t {
    const cudaError_t rc = ensure_dynamic_smem(kernel, (int)smem);
    if (rc != cudaSuccess) return rc;
    return launch_kernel(kernel, grid, XT_THREADS, smem, L.stream, 1, qm, km, x);
  };
  if (x.lse) return halves == 2 ? launch(xi_tc_kernel<128, true>) : launch(xi_tc_kernel<64, true>);
  return halves == 2 ? launch(xi_tc_kernel<128, false>) : launch(xi_tc_kernel<64, false>);
}

// ======================================================================================================
// FD + best partner for larger windows on tensor cores (Eq. "similarity", Step 2).
//
// A CTA (or a cluster of ks CTAs that split the hidden dimension, where there are few tiles) takes one tile of up to
// 128 sources x 128 destinations of one window.  The rows of a tile are scattered over the sequence; the CTA finds them
// from the positions (window_tokens) or, in the list form, in the lists the window build left.  Eight warps gather them
// with 16-byte cp.async copies, eight threads per 128-byte row segment, straight into the 128-byte-swizzled K-major layout tcgen05 reads, through a ring of stages of 32 KB (64 columns
// of both operands), and re-read their pieces to accumulate the squared norms.  A ninth warp issues
// G += X_A X_B^T (128 x N x 64 per chunk, bf16 -> fp32 in TMEM).  The MMA always reads 128 A
// rows: rows the tile does not have are never written and only feed accumulator rows nobody reads.  After the last chunk
// the loader warps turn into the epilogue: minimum over the destinations (ties: lowest index) of every source, one key
// per (source, block of destinations), of which the map kernel takes the lowest.
//
// Every tile reads its rows again, so the kernel is bound by the way from L2 through shared memory (a chunk: 32 KB
// written, read by the norms and read by the MMA), not by HBM or the tensor pipe.  Tiles of 256 x 256 halve that, but the
// four CTAs they then leave per SM's worth of work have to exchange partial products, and distributed shared memory gave
// 10 bytes per nanosecond and SM (13 us per 128 rows of 256): 62, with the exchange vectorised 56 us, where tiles of 128
// with a six-stage ring take 44, and 35 with the scores compared by reciprocals (two samples of 8192 tokens x 3584 in windows of
// 512; list-driven tiles that met in atomics took 77; windows of 1024 and 2048: 76 -> 45 and 76 -> 43 before the reciprocals).  The launch has as many tiles as windows of the expected
// size need; a CTA goes on with the blocks of a window that has grown beyond that.
// ======================================================================================================
struct FdTcArgs {
  const __nv_bfloat16* x;              // first vision row of sample 0
  const int* seq_start;                // first row of each sample (packed batches) or nullptr
  int64_t batch_stride, row_stride;    // elements
  int d;
  int metric;                          // LIGHTKV_FD_*
  double keep;
  Geometry g;
  const int* n_vis;
  const int* pos;
  int cap_in, max_cell;
  int blocks;                          // blocks a side the largest window may have (row pitch of key)
  int grid_blocks;                     // ... a window of the expected size has (the launch)
  int lists;                           // 1: windows from ws (window build), keys by source entry through atomics
  Workspace ws;
  uint32_t* status;
};

constexpr int FT_LOADERS = 256, FT_WARPS = 9;
constexpr int BLK = kFdTile;

template <int STAGES>
struct FdTcSmem {
  static constexpr int PITCH = BLK + 4;                   // row pitch (floats) of a partial G: 16-byte pieces of eight rows
                                                          // in a row of lanes meet no bank conflict
  static constexpr uint32_t STAGE = BLK * 256;            // BLK A rows | BLK B rows of 64 columns
  static constexpr uint32_t CTL = 128 + 6 * BLK * 4 + 2 * 128 * 4 + 2 * BLK * 4 + 16 * 4;
  static_assert(BLK * PITCH * 4 <= STAGES * STAGE, "a partial G fits over the drained ring");
  static size_t bytes(int cap_in, bool lists) {
    return 1024 /* alignment */ + STAGES * STAGE + CTL + (lists ? 0 : window_search_bytes(cap_in));
  }
};

// the best destination of source `row` of tile (ia, ib) of a window of sample b
__device__ __forceinline__ void store_key(const FdTcArgs& a, int b, int ia, int ib, int row, const int* row_a, int a_first,
                                          int b_first, float best, int best_c) {
  unsigned long long key = ~0ull;
  if (best_c >= 0)
    key = ((unsigned long long)orderable(best) << 32) | (unsigned)((a.lists ? b_first : 0) + ib * BLK + best_c);
  if (a.lists) atomicMin(a.ws.a_key + size_t(b) * a.ws.cap_a + a_first + ia * BLK + row, key);
  else a.ws.tile_key[(size_t(b) * a.blocks + ib) * a.cap_in + row_a[row]] = key;
}

// CLUSTER = false is the plain launch (ks = 1) with the cluster code compiled out.
template <bool CLUSTER, int FT_STAGES>
__global__ void __launch_bounds__(FT_LOADERS + 32, FT_STAGES > 3 ? 1 : 2) fd_tc_kernel(const __grid_constant__ FdTcArgs a) {
  using M = FdTcSmem<FT_STAGES>;
  constexpr int FT_AHEAD = FT_STAGES - 1;       // fills in flight beside the one being consumed
  constexpr int NR = BLK / 32;                  // rows of an operand per loader thread
  constexpr int PITCH = M::PITCH;
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = reinterpret_cast<unsigned char*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  unsigned char* ctl = base + FT_STAGES * M::STAGE;
  uint64_t* full = reinterpret_cast<uint64_t*>(ctl);   // [FT_STAGES] fill landed (one arrival per loader warp)
  uint64_t* empty = full + FT_STAGES;           // [FT_STAGES] fill consumed (MMA commit)
  uint64_t* acc_full = empty + FT_STAGES;       // accumulator complete
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(acc_full + 1);
  volatile int* abort_flag = reinterpret_cast<volatile int*>(tmem_slot + 1);
  float* sq = reinterpret_cast<float*>(ctl + 128);     // [2 BLK] squared norms of A, B rows over this CTA's columns
  float* nrm = sq + 2 * BLK;                           // [2 BLK] whole norms
  float* inv = nrm + 2 * BLK;                          // [2 BLK] their reciprocals (0 for 0)
  float* red_f = inv + 2 * BLK;                        // [128]
  int* red_c = reinterpret_cast<int*>(red_f + 128);    // [128]
  int* row_a = red_c + 128;                            // [BLK] token index of the tile's rows
  int* row_b = row_a + BLK;                            // [BLK]
  int* warp_sum = row_b + BLK;                         // [FT_WARPS]
  unsigned int* match = reinterpret_cast<unsigned int*>(warp_sum + 16);

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < FT_STAGES; ++i) { mbar_init(&full[i], FT_LOADERS / 32); mbar_init(&empty[i], 1); }
    mbar_init(acc_full, 1);
    *abort_flag = 0;
    fence_barrier_init();
  }
  if (warp == 8) { tmem_alloc(tmem_slot, BLK); tmem_relinquish(); }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // barriers and tensor memory are set up while the kernel before this one may still be running; from here on
  // global memory is read (and written), so that kernel must have completed
  grid_dependency_wait();
  grid_launch_dependents();                     // in this order: see grid_dependency_sync
  const uint32_t tmem_base = *tmem_slot;
  const uint32_t ring = smem_u32(base);
  const int ks = CLUSTER ? (int)cluster_nctarank() : 1, rank = CLUSTER ? (int)cluster_ctarank() : 0;
  const int b = blockIdx.y, tile = blockIdx.x / ks, per_window = a.grid_blocks * a.grid_blocks;
  const int w = tile / per_window, rem = tile - w * per_window, ia0 = rem / a.grid_blocks, ib0 = rem - ia0 * a.grid_blocks;
  const int par = a.g.src_par;
  const int n = a.n_vis ? max(0, min(a.n_vis[b], a.cap_in)) : a.cap_in;
  const int nk_all = (a.d + 63) >> 6;           // 64-column chunks of the whole hidden dimension
  const int c_lo = rank * nk_all / ks, nk = (rank + 1) * nk_all / ks - c_lo;
  int* win_tok = a.lists ? nullptr : a.ws.win_tok + (size_t(b) * a.g.n_windows + w) * (a.max_cell + 1);

  uint32_t done = 0, tiles = 0;                 // fills and tiles completed (phases of the barriers)
  for (int ia = ia0;; ia += a.grid_blocks) {
  bool more_a = false;
  for (int ib = ib0;; ib += a.grid_blocks) {
    // ---- the tile's rows
    int na, nb, a_first = 0, b_first = 0;       // sources and destinations of the whole window; list mode: first entries
    bool wanted = true;                         // the window loses tokens at all
    if (a.lists) {
      const int nW = a.ws.n_windows;
      const int* win_off = a.ws.win_off + size_t(b) * (nW + 1) + w;
      const int* a_off = a.ws.a_off + size_t(b) * (nW + 1) + w;
      a_first = a_off[0];
      b_first = win_off[0] - a_first;
      na = a_off[1] - a_first;
      nb = win_off[1] - win_off[0] - na;
      for (int r = tid; r < 2 * BLK; r += FT_LOADERS + 32) {
        const int e = r < BLK ? ia * BLK + r : ib * BLK + r - BLK;
        if (r < BLK) { if (e < na) row_a[r] = a.ws.a_tok[size_t(b) * a.ws.cap_a + a_first + e]; }
        else if (e < nb) row_b[r - BLK] = a.ws.b_tok[size_t(b) * a.ws.cap_b + b_first + e];
      }
    } else {
      const bool publish = rank == 0 && ia == 0 && ib == 0;   // the map kernel reads the window's tokens
      const int nw = min(a.max_cell, window_tokens<FT_WARPS>(a.g, a.pos ? a.pos + size_t(b) * a.cap_in : nullptr, n, w, match, warp_sum, [&](int l, int i) {
        if (l < a.max_cell) {
          const bool src = (l & 1) == par;
          const int r = (l >> 1) - (src ? ia : ib) * BLK;
          if (r >= 0 && r < BLK) (src ? row_a : row_b)[r] = i;
          if (publish) win_tok[1 + l] = i;
        } else if (publish) {                   // only if positions repeat or lie outside the grid: survives
          a.ws.partner[size_t(b) * a.cap_in + i] = -1;
          a.ws.slot[size_t(b) * a.cap_in + i] = 0;
        }
      }));
      if (publish && tid == 0) win_tok[0] = nw;
      na = (nw + 1 - par) >> 1;
      nb = nw - na;
      wanted = nb > 0 && removal_count(nw, a.keep, par) > 0;
    }
    const bool more_b = wanted && nb > (ib + a.grid_blocks) * BLK;
    more_a = wanted && na > (ia + a.grid_blocks) * BLK;
    wanted = wanted && na > ia * BLK && nb > ib * BLK;
    __syncthreads();
    if (wanted) {                               // the same for every thread of the CTA and of its cluster
      na = min(na - ia * BLK, BLK);
      nb = min(nb - ib * BLK, BLK);
      if (warp < 8) {
        // ---- gather: thread = 16-byte piece c of rows g + 32 i of both operands
        const int c = tid & 7, g = tid >> 3;
        const __nv_bfloat16* xb = a.x + size_t(b) * a.batch_stride + size_t(a.seq_start ? a.seq_start[b] : 0) * a.row_stride +
                                  c_lo * 64 + c * 8;
        const uint32_t row16 = uint32_t(a.row_stride >> 3);                   // row pitch in 16-byte units
        uint32_t off[2 * NR];                                                 // A rows, B rows; all ones: no such row
#pragma unroll
        for (int i = 0; i < NR; ++i) {
          off[i] = g + 32 * i < na ? uint32_t(row_a[g + 32 * i]) * row16 : 0xffffffffu;
          off[NR + i] = g + 32 * i < nb ? uint32_t(row_b[g + 32 * i]) * row16 : 0xffffffffu;
        }
        const uint32_t slot0 = uint32_t(g) * 128 + (uint32_t(c ^ (g & 7)) << 4);   // swizzled offset of row g; row g + 32 i is 4096 i further
        float ss[2 * NR];
#pragma unroll
        for (int i = 0; i < 2 * NR; ++i) ss[i] = 0.f;
        auto issue = [&](int k) {
          const uint32_t F = done + k, sb = ring + (F % FT_STAGES) * M::STAGE + slot0;
          const uint32_t bytes = (c_lo + k) * 64 + c * 8 < a.d ? 16u : 0u;    // d is a multiple of 8
          const __nv_bfloat16* p = xb + (bytes ? k * 64 : 0);
#pragma unroll
          for (int i = 0; i < 2 * NR; ++i)
            if (off[i] != 0xffffffffu) cp_async16(sb + i * 4096, p + size_t(off[i]) * 8, bytes);
        };
        bool ok = true;
        auto fill = [&](int k) {                            // once the MMAs that read the stage before have completed
          if (ok && k < nk) {
            const uint32_t F = done + k;
            ok = F < FT_STAGES || mbar_wait(&empty[F % FT_STAGES], ((F / FT_STAGES) & 1) ^ 1, abort_flag);
            if (ok) issue(k);
          }
          cp_async_commit();
        };
#pragma unroll
        for (int k = 0; k < FT_AHEAD; ++k) fill(k);
        for (int k = 0; ok && k < nk; ++k) {
          cp_async_wait<FT_AHEAD - 1>();                    // this thread's pieces of chunk k have landed
          const uint32_t s = (done + k) % FT_STAGES, sb = ring + s * M::STAGE + slot0;
          __syncwarp();
          if (lane == 0) mbar_arrive(&full[s]);             // the MMA warp fences the proxies after its wait
          // (rows the tile does not have hold whatever is there: their norms are not used.  Eight loads in flight and no test:
          // row after row the norms took 1.4 us a chunk, twice the MMAs)
#pragma unroll
          for (int i0 = 0; i0 < 2 * NR; i0 += 8) {
            uint4 v[8];
#pragma unroll
            for (int i = 0; i < 8; ++i) v[i] = ld_shared16(sb + (i0 + i) * 4096);
#pragma unroll
            for (int i = 0; i < 8; ++i) ss[i0 + i] = sumsq16(v[i], ss[i0 + i]);
          }
          fill(k + FT_AHEAD);                               // the stage of chunk k - 1, whose MMAs ran beside the norms
        }
        cp_async_wait<0>();

        // ---- squared norms of the rows (this CTA's columns)
#pragma unroll
        for (int i = 0; i < 2 * NR; ++i) {
#pragma unroll
          for (int o = 1; o < 8; o <<= 1) ss[i] += __shfl_xor_sync(0xffffffffu, ss[i], o);
          if (c == 0) sq[(i < NR ? 0 : BLK) + g + 32 * (i % NR)] = ss[i];
        }
        named_barrier(1, FT_LOADERS);
        ok = ok && mbar_wait(acc_full, tiles & 1, abort_flag);
        ok = __all_sync(0xffffffffu, ok);                   // the TMEM loads below are warp-wide
        tc_fence_after();
        const int q = warp & 3, half = warp >> 2;
        // Cosine scores of a row are compared as inner product / |destination| (the row's own norm scales them all), with a
        // reciprocal per destination instead of a division per pair; the lowest one's score is then computed as any other
        // (128 x 128 pairs: 6.0 -> 1.6 us).  Only where every norm of the tile is zero or far from the ends of the range.
        static_assert(2 * BLK == FT_LOADERS, "a norm per thread");
        auto set_norm = [&](float sum) {
          const float n = a.metric == LIGHTKV_FD_COSINE ? sqrtf(sum) : sum;
          const bool exists = tid < BLK ? tid < na : tid - BLK < nb;
          const bool plain = a.metric == LIGHTKV_FD_COSINE && (!exists || n == 0.f || (n >= 1e-15f && n <= 1e15f));
          nrm[tid] = n;
          inv[tid] = n > 0.f ? 1.f / n : 0.f;
          const bool all = __all_sync(0xffffffffu, plain);
          if (lane == 0) warp_sum[warp] = all;
        };
        auto all_plain = [&]() {
          const int4 v0 = *reinterpret_cast<const int4*>(warp_sum), v1 = *reinterpret_cast<const int4*>(warp_sum + 4);
          return (v0.x & v0.y & v0.z & v0.w & v1.x & v1.y & v1.z & v1.w) != 0;
        };
        if (!CLUSTER) {
          set_norm(sq[tid]);
          named_barrier(1, FT_LOADERS);
          const bool plain = all_plain();
          // ---- thread = A row (TMEM lane); warps 0-3 scan columns 0-63, warps 4-7 columns 64-127
          const int row = q * 32 + lane, col0 = half * 64;
          float best = 3.0e38f;
          int best_c = -1;
          if (ok && row - lane < na) {
            const float na_row = nrm[row];
            float best_r = -3.0e38f, best_g = 0.f;
            for (int c0 = col0; c0 < min(nb, col0 + 64); c0 += 32) {   // warp-uniform
              float v[32];
              tmem_ld32(tmem_base + (uint32_t(q * 32) << 16) + c0, v);
              tmem_ld_wait();
              if (plain) {
#pragma unroll
                for (int i = 0; i < 32; i += 4) {
                  const float4 w = *reinterpret_cast<const float4*>(inv + BLK + c0 + i);
                  const float r4[4] = {v[i] * w.x, v[i + 1] * w.y, v[i + 2] * w.z, v[i + 3] * w.w};
#pragma unroll
                  for (int k = 0; k < 4; ++k)
                    if (r4[k] > best_r && c0 + i + k < nb) { best_r = r4[k]; best_g = v[i + k]; best_c = c0 + i + k; }
                }
              } else {
#pragma unroll
                for (int i = 0; i < 32; ++i) {
                  if (c0 + i < nb) {                        // warp-uniform
                    const float fd = pair_score(a.metric, v[i], na_row, nrm[BLK + c0 + i]);
                    if (fd < best) { best = fd; best_c = c0 + i; }
                  }
                }
              }
            }
            if (plain && best_c >= 0) best = pair_score(a.metric, best_g, na_row, nrm[BLK + best_c]);
          }
          if (half == 1) { red_f[row] = best; red_c[row] = best_c; }
          named_barrier(1, FT_LOADERS);
          if (half == 0 && row < na && ok) {
            if (red_f[row] < best) { best = red_f[row]; best_c = red_c[row]; }   // ties stay with the lower column
            store_key(a, b, ia, ib, row, row_a, a_first, b_first, best, best_c);
          }
        } else {
          // ---- cluster: every CTA puts its partial G into shared memory (float [128][PITCH], over the drained ring), then CTA
          //      `rank` finishes every ks-th row.  All threads of every CTA pass both barriers, whatever happened before (an
          //      aborted CTA contributes garbage and the status bit, never a hang); the MMA warp joins them below.
          if (ok && q * 32 < na) {
            for (int c0 = half * 32; c0 < nb; c0 += 64) {
              float v[32];
              tmem_ld32(tmem_base + (uint32_t(q * 32) << 16) + c0, v);
              tmem_ld_wait();
              float4* prow = reinterpret_cast<float4*>(reinterpret_cast<float*>(base) + (q * 32 + lane) * PITCH + c0);
#pragma unroll
              for (int i = 0; i < 8; ++i) prow[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
            }
          }
          __syncwarp();
          cluster_sync();                                   // all partial G and squared norms are in shared memory
          {
            const uint32_t src = smem_u32(sq + tid);
            float part[8], sum = 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) part[j] = j < ks ? ld_cluster_f32(map_to_cta(src, j)) : 0.f;
#pragma unroll
            for (int j = 0; j < 8; ++j) sum += part[j];
            set_norm(sum);
          }
          named_barrier(1, FT_LOADERS);
          const bool plain = all_plain();
          // a warp per row, two rows at a time, four columns per lane, all of their remote reads in flight; the CTAs start
          // with different peers (rank ^ j).  The parts are added as a balanced tree: its pairs are the same peers in every
          // CTA, whatever the rank, so equal rows get equal scores bit for bit wherever they are finished (the tie rule
          // needs that; added from the CTA's own part on they differed in the last digit).
          for (int r = rank + warp * ks; r < na; r += 16 * ks) {
            float4 v[2][8];
#pragma unroll
            for (int t = 0; t < 2; ++t)
#pragma unroll
              for (int j = 0; j < 8; ++j) {
                const int rr = r + t * 8 * ks;
                v[t][j] = make_float4(0.f, 0.f, 0.f, 0.f);
                if (j < ks && rr < na && 4 * lane < nb)
                  v[t][j] = ld_cluster_f32x4(map_to_cta(ring + uint32_t(rr * PITCH + 4 * lane) * 4, rank ^ j));
              }
#pragma unroll
            for (int t = 0; t < 2; ++t) {
              const int rr = r + t * 8 * ks;
              if (rr >= na) break;                          // warp-uniform
              float best = 3.0e38f;
              int best_c = -1;
#pragma unroll
              for (int step = 1; step < 8; step *= 2)
#pragma unroll
                for (int j = 0; j < 8; j += 2 * step) {
                  v[t][j].x += v[t][j + step].x; v[t][j].y += v[t][j + step].y;
                  v[t][j].z += v[t][j + step].z; v[t][j].w += v[t][j + step].w;
                }
              const float g4[4] = {v[t][0].x, v[t][0].y, v[t][0].z, v[t][0].w};
              if (plain) {
                const float4 w = *reinterpret_cast<const float4*>(inv + BLK + 4 * lane);
                const float w4[4] = {w.x, w.y, w.z, w.w};
                float best_r = -3.0e38f, best_g = 0.f;
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  const float r = g4[k] * w4[k];
                  if (r > best_r && 4 * lane + k < nb) { best_r = r; best_g = g4[k]; best_c = 4 * lane + k; }
                }
                if (best_c >= 0) best = pair_score(a.metric, best_g, nrm[rr], nrm[BLK + best_c]);
              } else {
#pragma unroll
                for (int k = 0; k < 4; ++k) {
                  const int col = 4 * lane + k;
                  if (col < nb) {
                    const float fd = pair_score(a.metric, g4[k], nrm[rr], nrm[BLK + col]);
                    if (fd < best) { best = fd; best_c = col; }
                  }
                }
              }
              // minimum over the lanes, ties to the lower lane, i.e. column
              const unsigned int key = best_c >= 0 ? orderable(best) : 0xffffffffu, low = __reduce_min_sync(0xffffffffu, key);
              if (low != 0xffffffffu) {
                const int from = __ffs(__ballot_sync(0xffffffffu, key == low)) - 1;
                best = __shfl_sync(0xffffffffu, best, from);
                best_c = __shfl_sync(0xffffffffu, best_c, from);
              }
              if (lane == 0 && !*abort_flag) store_key(a, b, ia, ib, rr, row_a, a_first, b_first, best, best_c);
            }
          }
          __syncwarp();
          cluster_sync();                                   // nobody reads this CTA's shared memory any more
        }
        tc_fence_before();                                  // TMEM reads done before the next tile's MMAs
      } else {
        if (lane == 0) {
          // ---- MMA issue: one chunk = four K = 16 steps inside the 128-byte rows
          const uint32_t idesc = idesc_bf16(128, (nb + 15) & ~15);
          for (int k = 0; k < nk; ++k) {
            const uint32_t F = done + k, s = F % FT_STAGES, sa = ring + s * M::STAGE;
            if (!mbar_wait(&full[s], (F / FT_STAGES) & 1, abort_flag)) break;
            fence_proxy_async();                            // the loaders' cp.async writes -> visible to the tensor core
            tc_fence_after();
#pragma unroll
            for (int kk = 0; kk < 4; ++kk)
              umma_bf16(tmem_base, smem_desc_sw128(sa + kk * 32), smem_desc_sw128(sa + BLK * 128 + kk * 32), idesc, k > 0 || kk > 0);
            umma_commit(&empty[s]);
          }
          umma_commit(acc_full);
        }
        if (CLUSTER) {
          __syncwarp();
          cluster_sync();
          cluster_sync();
        }
      }
      done += nk;
      ++tiles;
      __syncthreads();                                      // the tile's lists and accumulators are free
    }
    if (!more_b || (!CLUSTER && *abort_flag)) break;     // (the CTAs of a cluster stay together)
  }
  if (!more_a || (!CLUSTER && *abort_flag)) break;
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 8) {
    tc_fence_after();
    tmem_dealloc(tmem_base, BLK);
  }
  if (tid == 0 && *abort_flag && a.status) atomicOr(a.status, LIGHTKV_STATUS_TIMEOUT);
}

bool tc_fd_supported(int hidden) { return hidden % 8 == 0; }

cudaError_t launch_fd_tc(const LayerLaunch& L, bool lists) {
  const lightkv_layer_args_t* a = L.a;
  FdTcArgs f;
  f.x = static_cast<const __nv_bfloat16*>(a->hidden) + size_t(a->vis_begin) * a->hidden_row_stride;
  f.seq_start = a->seq_start;
  f.batch_stride = a->hidden_batch_stride; f.row_stride = a->hidden_row_stride; f.d = L.hidden;
  f.metric = L.divergence; f.keep = L.keep; f.g = L.geo; f.n_vis = a->n_vis; f.pos = a->pos; f.cap_in = L.ws.cap_in;
  f.max_cell = L.max_cell; f.blocks = L.fd_blocks; f.lists = lists ? 1 : 0; f.ws = L.ws; f.status = a->status;
  f.grid_blocks = std::max(1, (L.fd_side + BLK - 1) / BLK);
  // While there are fewer tiles than CTAs that fit (two per SM), clusters of 2, 4 or 8 CTAs split the hidden dimension of
  // every tile.  Where every tile has an SM of its own without that, the ring takes all of its shared memory.
  const long long tiles = (long long)L.geo.n_windows * f.grid_blocks * f.grid_blocks, all = tiles * L.batch;
  const int sms = sm_count(), nk_all = (L.hidden + 63) / 64;
  const bool deep = all <= sms && 4 * all > 3 * sms;
  int ks = 1;
  while (!deep && ks < 8 && all * (2 * ks) <= 2 * sms && 4 * ks <= nk_all) ks *= 2;
  if (tiles * ks > 0x7fffffffLL) return cudaErrorInvalidValue;
  auto launch = [&](auto kernel, size_t smem) -> cudaError_t {
    const cudaError_t e = ensure_dynamic_smem(kernel, (int)smem);
    if (e != cudaSuccess) return e;
    return launch_kernel(kernel, dim3((unsigned)(tiles * ks), L.batch), FT_LOADERS + 32, smem, L.stream, ks, f);
  };
  if (deep) return launch(fd_tc_kernel<false, 6>, FdTcSmem<6>::bytes(f.cap_in, lists));
  const size_t smem = FdTcSmem<3>::bytes(f.cap_in, lists);
  return ks == 1 ? launch(fd_tc_kernel<false, 3>, smem) : launch(fd_tc_kernel<true, 3>, smem);
}

}  // namespace lkv
