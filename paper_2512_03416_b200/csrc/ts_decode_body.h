// Device code of the split-KV flash-decode path (sm_100a), shared by the stand-alone decode kernel
// and by the mixed kernel whose decode CTAs run it before they join the prefill work.
//
// The path is bound by HBM: every cached K/V byte is read once and used for 4*G flops.
//   * the work units (decode work item x KV head) sit in a global queue, longest first; a scheduler
//     warp per CTA takes one unit at a time, when the one before it is nearly fetched, and lays its
//     description into a small ring in shared memory. (Dealt out statically the CTAs of a mixed step
//     ended 132-152 us after its start, median 137: SMs do not pull on HBM at the same rate.) The
//     scheduler also touches the unit's queries and page ids, so that the eight streaming warps find
//     them in L1 instead of each paying a chain of L2 latencies at every unit change;
//   * K/V pages (16 tokens) arrive by TMA tensor copies, 128-byte swizzled, straight from the
//     paged pool; the page id is a TMA coordinate, so scattered pages cost nothing extra;
//   * every warp owns a private ring of page stages and issues its own copies: the pages of a
//     unit are dealt round-robin to the warps, and a warp's lookahead crosses unit boundaries;
//   * at the end of a unit a warp leaves its partial result in shared memory and goes on to its next
//     unit's pages; it adds up its eighth of the unit's results between two of those pages, once all
//     eight warps have left theirs: no warp waits for the others, the page streams do not stop;
//   * the tensor-core product is transposed, S^T = K Q^T and O^T = V^T P^T (mma.sync m16n8k16,
//     keys / head_dim as the M dimension, the G <= 8 query heads of the KV head as N), so no MMA
//     row is padding and the accumulators stay small; P^T is re-laid out with movmatrix;
//   * softmax is online in base 2 with fp32 state per head; a page without a new maximum costs no reduction.
// Measured (us, one static deal, a reduction and rescale per page, two copies per page, all warps
// meeting at every unit's end -> this): 64 rows of the 8B shape 127.9 -> 125.9; 203 rows of the 70B
// shape 237.4 -> 226.9; next to a 2048-token chunk 160.0 -> 155.9; 717 tokens next to 198 rows 281 -> 273.
// With the products left out (copies and waits only) 64 rows took 125 us where the whole took 127: what
// is left is the rate at which the page copies come in.
#pragma once
#include <cuda_bf16.h>
#include <math_constants.h>

#include "../../include/tokenscale.h"
#include "ts_internal.h"
#include "ts_ptx.h"
#include "ts_tma.h"

namespace ts {
namespace dec {


constexpr int kDecWarps = 8;
constexpr int kDecThreads = kDecWarps * 32;          // streaming threads; the scheduler warp comes on top
constexpr int kDecRing = 3;                          // units of a CTA that are described at a time
constexpr long long kDrainCycles = 20000000;         // about 10 ms: limit of the wait for copies in flight after a failure

// Barrier of the kDecThreads decode threads (id 1; id 0 stays with the whole block).
__device__ __forceinline__ void block_sync() { asm volatile("bar.sync 1, %0;\n" ::"n"(kDecThreads) : "memory"); }
// 2^x for x <= 0: a weight below 2^-126 of the head's largest one becomes 0 (l, at least 1, would not change)
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ uint32_t movmatrix_t(uint32_t a) {
  uint32_t d;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(d) : "r"(a));
  return d;
}
// Shared-memory image of one page stage (written by TMA with the 128-byte swizzle):
//   [K: 64 head_dim columns of 16 rows (16x128B), D = 128: the other 64][V: the same]   (one copy)
// Row r, 16-byte chunk c (of the 2*D-byte logical row) of K:
template <int D>
__device__ __forceinline__ uint32_t page_off(int kv, int r, int c) {
  return (uint32_t)(kv * (kPageSize * D * 2) + (c >> 3) * 2048 + r * 128 + (((c & 7) ^ (r & 7)) << 4));
}

// A work unit as the scheduler describes it: the pages [first_page, first_page + n_pg) of a table row
// and one KV head; page j is warp j % kDecWarps's.
struct UnitInfo {
  int first_page, n_pg;   // n_pg < 0: there are no more units
  int head;               // KV head
  int k_begin, k_end;     // keys at positions >= k_end are not visible (ctx + 1 or split end)
  int partial_slot;
  int tok, new_pos;       // token of the row in the step's tensors, position of the row's new token
  const int32_t* table_row;
  int combine;            // of a split row: its CombineItem, and what that says
  CombineItem merge;
  int pad;
};
static_assert(sizeof(UnitInfo) == 64, "UnitInfo is four 16-byte chunks");

// Shared memory: page stages, partial results of the warps, unit descriptions, mbarriers, failure flag.
template <int D, int STAGES>
struct DecSmem {
  static constexpr int kStageBytes = 2 * kPageSize * D * 2;   // K + V of one page and KV head
  static constexpr int kOffMerge = kDecWarps * STAGES * kStageBytes;
  __host__ __device__ static constexpr int off_units(int G) { return kOffMerge + kDecWarps * G * (D + 2) * 4; }
  __host__ __device__ static constexpr int off_bars(int G) { return off_units(G) + kDecRing * (int)sizeof(UnitInfo); }
  // barriers: page stages [kDecWarps][STAGES], unit described [kDecRing], unit done with [kDecRing],
  // partial results written, partial results added up, unit nearly fetched
  static constexpr int kBarDesc = kDecWarps * STAGES, kBarDone = kBarDesc + kDecRing, kBarWritten = kBarDone + kDecRing,
                       kBarAdded = kBarWritten + 1, kBarNear = kBarAdded + 1, kBars = kBarNear + 1;
  __host__ __device__ static constexpr int off_merges(int G) { return off_bars(G) + kBars * 8; }   // entries of the ring for merge_by_all
  __host__ __device__ static constexpr int off_failed(int G) { return off_merges(G) + kDecRing * 4; }
};
template <int D, int STAGES>
__host__ __device__ constexpr size_t decode_smem_bytes(int G) {
  return (size_t)DecSmem<D, STAGES>::off_failed(G) + 4;
}
// The streaming threads and the scheduler warp meet when the barriers are set up and before they are given back.
__device__ __forceinline__ void decode_meet() { asm volatile("bar.sync 3, %0;\n" ::"n"(kDecThreads + 32) : "memory"); }

// Every wait of the path is bounded. The copy of a page has the step's limit; a wait for other warps of the
// CTA may span many of their pages and has a limit of its own (unit_wait_cycles). A wait that runs out raises
// the CTA's failure flag, which ends the other waits and with them the path.
// Called by whole warps; true, for all lanes, when the phase has completed.
__device__ __forceinline__ bool wait_for_warps(uint32_t bar, uint32_t parity, const volatile int* failed, long long limit) {
  if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
  const long long t0 = clock64();
  for (;;) {
    if (__all_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if (__any_sync(0xffffffffu, *failed != 0 || clock64() - t0 > limit)) return false;
  }
}
__device__ __forceinline__ void give_up(const StepDevice& s, volatile int* failed) {
  if ((threadIdx.x & 31) == 0) {
    atomicOr(s.status, TS_DEV_TIMEOUT);
    *failed = 1;
  }
  __syncwarp();
}

// Merge of a row's splits, by one warp: the merge of merge_splits, bit for bit, for `n_heads` heads from head0 on, 32 * E of
// their columns from col0 on. The loads of HEADS heads x GROUPS groups of splits fly at a time. Lane i takes the weight of
// split i of these and the others get it from there: this is the end of a launch, whose code comes in cold, and a weight per
// lane and split is most of merge_group's.
template <int D, int E, int HEADS, int GROUPS>
__device__ __forceinline__ void merge_heads(const StepDevice& s, const CombineItem& c, int head0, int n_heads, int col0, int lane) {
  constexpr int kGroup = kMergeGroup, kSplits = GROUPS * kGroup;
  static_assert(kSplits <= 32, "a lane per split");
  const int col = col0 + lane * E;
  const float* ml = s.part_ml + ((size_t)c.first_partial * s.Hq + head0) * 2;
  const float* pa = s.part_acc + ((size_t)c.first_partial * s.Hq + head0) * D + col;
  const size_t ml_stride = (size_t)s.Hq * 2, pa_stride = (size_t)s.Hq * D;
#pragma unroll 1
  for (int h0 = 0; h0 < n_heads; h0 += HEADS) {
    float m[HEADS], l[HEADS], acc[HEADS][E];
#pragma unroll
    for (int h = 0; h < HEADS; ++h) {
      m[h] = -CUDART_INF_F;
      l[h] = 0.f;
#pragma unroll
      for (int e = 0; e < E; ++e) acc[h][e] = 0.f;
    }
#pragma unroll 1
    for (int b0 = 0; b0 < c.n_splits; b0 += kSplits) {
      float2 st[HEADS];                                // lane i: maximum and sum of split b0 + i
      float a[HEADS][kSplits][E];
#pragma unroll
      for (int h = 0; h < HEADS; ++h) {
        const bool head = h0 + h < n_heads;
        st[h] = make_float2(-CUDART_INF_F, 0.f);
        if (head && lane < kSplits && b0 + lane < c.n_splits)
          st[h] = __ldcg(reinterpret_cast<const float2*>(ml + (b0 + lane) * ml_stride + (h0 + h) * 2));
#pragma unroll
        for (int j = 0; j < kSplits; ++j) {
          const bool on = head && b0 + j < c.n_splits;
          const float* src = pa + (b0 + j) * pa_stride + (h0 + h) * D;
          if constexpr (E == 4) {
            const float4 v = on ? __ldcg(reinterpret_cast<const float4*>(src)) : make_float4(0.f, 0.f, 0.f, 0.f);
            a[h][j][0] = v.x; a[h][j][1] = v.y; a[h][j][2] = v.z; a[h][j][3] = v.w;
          } else {
            const float2 v = on ? __ldcg(reinterpret_cast<const float2*>(src)) : make_float2(0.f, 0.f);
            a[h][j][0] = v.x; a[h][j][1] = v.y;
          }
        }
      }
#pragma unroll
      for (int h = 0; h < HEADS; ++h) {
        float top = st[h].x;                           // the largest maximum of the lane's group
#pragma unroll
        for (int sh = 1; sh < kGroup; sh <<= 1) top = fmaxf(top, __shfl_xor_sync(0xffffffffu, top, sh));
        float mn[GROUPS], keep[GROUPS], mine = 0.f;
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) {
          const float before = g > 0 ? mn[g - 1] : m[h];
          mn[g] = fmaxf(before, __shfl_sync(0xffffffffu, top, g * kGroup));
          keep[g] = exp2f(before - mn[g]);             // 0 on the first group (m = -inf)
          if (lane / kGroup == g) mine = mn[g];
        }
        const float w = exp2f(st[h].x - mine);         // absent split: exp2(-inf) = 0
#pragma unroll
        for (int g = 0; g < GROUPS; ++g) {
          if (b0 + g * kGroup >= c.n_splits) break;
#pragma unroll
          for (int j = 0; j < kGroup; ++j) {
            const int i = g * kGroup + j;
            const float wj = __shfl_sync(0xffffffffu, w, i), lj = __shfl_sync(0xffffffffu, st[h].y, i);
            l[h] = j == 0 ? __fmaf_rn(l[h], keep[g], __fmul_rn(wj, lj)) : __fmaf_rn(wj, lj, l[h]);
#pragma unroll
            for (int e = 0; e < E; ++e)
              acc[h][e] = j == 0 ? __fmaf_rn(acc[h][e], keep[g], __fmul_rn(wj, a[h][i][e])) : __fmaf_rn(wj, a[h][i][e], acc[h][e]);
          }
        }
        m[h] = mn[GROUPS - 1];
      }
    }
#pragma unroll
    for (int h = 0; h < HEADS; ++h) {
      if (h0 + h >= n_heads) continue;
      uint32_t* dst = reinterpret_cast<uint32_t*>(s.out + ((size_t)c.token * s.Hq + head0 + h0 + h) * D + col);
#pragma unroll
      for (int e = 0; e < E; e += 2) dst[e / 2] = pack_bf16(acc[h][e] / l[h], acc[h][e + 1] / l[h]);
    }
  }
}
// Rows that were split. A unit whose eight warps have all written their shares is counted by the scheduler warp; whoever
// counts the last split of a (row, KV head) merges it: the scheduler warp itself while its CTA still streams, all
// streaming warps for the CTA's last units, where the merge is what the launch ends with. (Counted and merged by the
// streaming warps, the fence and the counter's round trip stopped the page stream.) A launch of few units leaves the
// merge to a launch of its own, whose blocks merge a head each (merge_here, decided on the host).
// True, for the whole warp, when this was the last split.
__device__ __forceinline__ bool count_split(const StepDevice& s, int combine, int n_splits, int kv_head, int lane) {
  int last = 0;
  if (lane == 0) {
    int32_t* count = s.merge_count + (size_t)combine * s.Hkv + kv_head;
    int before;
    // releases the unit's results, which this warp has seen through the unit's barrier, and acquires the other splits'
    asm volatile("atom.acq_rel.gpu.global.add.s32 %0, [%1], 1;\n" : "=r"(before) : "l"(count) : "memory");
    last = before == n_splits - 1;
    if (last) *count = 0;                              // for the next launch
  }
  last = __shfl_sync(0xffffffffu, last, 0);
  __syncwarp();                                        // what lane 0 acquired holds for the lanes that read the splits (a shuffle orders no memory)
  return last;
}
template <int D>
__device__ __forceinline__ void merge_by_scheduler(const StepDevice& s, const CombineItem& c, int kv_head, int lane) {
  const int G = s.Hq / s.Hkv;
  merge_heads<D, D / 32, 2, 1>(s, c, kv_head * G, G, 0, lane);
}
// Warp `warp` of the kDecWarps streaming warps: a head or half a head at a time, so that all have something to do.
template <int D>
__device__ __forceinline__ void merge_by_all(const StepDevice& s, const CombineItem& c, int kv_head, int warp, int lane) {
  const int G = s.Hq / s.Hkv;
  if (D == 64 || G <= kDecWarps / 2) {
    for (int i = warp; i < G * (D / 64); i += kDecWarps)
      merge_heads<D, 2, 1, 2>(s, c, kv_head * G + i / (D / 64), 1, i % (D / 64) * 64, lane);
  } else {
    for (int i = warp; i < G; i += kDecWarps) merge_heads<D, D / 32, 1, 1>(s, c, kv_head * G + i, 1, 0, lane);
  }
}

// Scheduler warp of CTA `cta` of `n_ctas`: its first unit is unit `cta`, the others come off the queue
// s.pf_queue[3], which the launch leaves at zero.
// `ready` waits for the launch in front of this one: called once the first unit is described. MERGE: the warp also merges
// the rows that were split (count_split), a unit once the entry of the ring it was described in is free.
template <int D, int STAGES, bool MERGE, typename Ready>
__device__ __forceinline__ void decode_schedule(const StepDevice& s, unsigned char* smem, uint32_t base, int cta, int n_ctas, Ready&& ready) {
  using L = DecSmem<D, STAGES>;
  const int lane = threadIdx.x & 31, G = s.Hq / s.Hkv;
  const uint32_t bars = base + L::off_bars(G);
  UnitInfo* ring = reinterpret_cast<UnitInfo*>(smem + L::off_units(G));
  const int n_units = (s.n_items - s.n_prefill_items) * s.Hkv;
  volatile int* failed = reinterpret_cast<volatile int*>(smem + L::off_failed(G));
  decode_meet();
  bool ok = true;
  const bool merging = MERGE && s.merge_here != 0;
  int n_described = 0, n_finished = 0;
  for (int k = 0;; ++k) {
    const int e = k % kDecRing;
    int unit = cta;
    if (k > 0) {
      // not earlier: units taken ahead of need are units that a faster CTA cannot take
      ok = wait_for_warps(bars + L::kBarNear * 8, (k - 1) & 1, failed, s.unit_wait_cycles);
      if (!ok) break;
      if (lane == 0) unit = n_ctas + atomicAdd(s.pf_queue + 3, 1);
      unit = __shfl_sync(0xffffffffu, unit, 0);
    }
    UnitInfo u = {};
    u.n_pg = -1;
    if (unit < n_units) {
      const WorkItem it = s.item(s.n_prefill_items + unit / s.Hkv);
      u.head = unit % s.Hkv;
      u.k_begin = it.k_begin;
      u.k_end = it.k_end;
      u.partial_slot = it.partial_slot;
      if (merging && it.partial_slot >= 0) {
        u.combine = it.combine;
        u.merge = s.combine(it.combine);
      }
      u.first_page = it.k_begin >> 4;
      u.n_pg = (it.k_end - it.k_begin + kPageSize - 1) >> 4;
      u.tok = s.row_tok0(it.row);
      u.new_pos = s.row_ctx(it.row);
      u.table_row = s.table + (size_t)s.row_slot(it.row) * s.max_pages_per_req;
    }
    if (k >= kDecRing) ok = wait_for_warps(bars + (L::kBarDone + e) * 8, ((k / kDecRing) & 1) ^ 1, failed, s.unit_wait_cycles);
    if (!ok) break;              // the entry may still be read: the streaming warps end by the failure flag
    bool split_done = false;                           // the unit whose entry this is going to be was a split: it is counted below
    int done_combine = 0, done_head = 0;
    CombineItem done_merge = {};
    if (merging && k >= kDecRing) {
      split_done = ring[e].partial_slot >= 0;
      done_combine = ring[e].combine;
      done_head = ring[e].head;
      done_merge = ring[e].merge;
      n_finished = k - kDecRing + 1;
    }
    __syncwarp();
    if (lane == 0) {
      ring[e] = u;
      mbar_arrive(bars + (L::kBarDesc + e) * 8);
    }
    __syncwarp();
    if (k == 0) ready();
    // one word of every 32-byte sector of the queries and of the page ids, for what it leaves in L1
    uint32_t touched = 0;
    if (u.n_pg > 0) {
      const uint32_t* q = reinterpret_cast<const uint32_t*>(s.q + ((size_t)u.tok * s.Hq + u.head * G) * D);
      for (int i = lane * 8; i < u.n_pg; i += 256) touched ^= __ldca(reinterpret_cast<const uint32_t*>(u.table_row) + u.first_page + i);
      for (int i = lane * 8; i < G * D / 2; i += 256) touched ^= __ldca(q + i);
    }
    asm volatile("" ::"r"(touched));
    if (split_done && count_split(s, done_combine, done_merge.n_splits, done_head, lane))
      merge_by_scheduler<D>(s, done_merge, done_head, lane);
    if (u.n_pg < 0) break;
    n_described = k + 1;
  }
  if (merging) {
    int* merges = reinterpret_cast<int*>(smem + L::off_merges(G));
    if (lane < kDecRing) merges[lane] = -1;
    __syncwarp();
    for (int k = n_finished; ok && k < n_described; ++k) {
      const int e = k % kDecRing;
      ok = wait_for_warps(bars + (L::kBarDone + e) * 8, (k / kDecRing) & 1, failed, s.unit_wait_cycles);
      if (ok && ring[e].partial_slot >= 0 && count_split(s, ring[e].combine, ring[e].merge.n_splits, ring[e].head, lane))
        merges[k - n_finished] = e;
    }
  }
  if (!ok) give_up(s, failed);
  decode_meet();                 // from here on nobody looks at a barrier of the path
}

// Streams the units that decode_schedule describes, on the first kDecThreads threads of the block
// (the scheduler runs on another warp at the same time). `smem` is the 1024-byte-aligned shared-memory
// window (decode_smem_bytes<D, STAGES>(G) bytes), `base` its shared-space address. `ready` waits for the launch
// in front of this one, once the barriers are set up. The function leaves no copy in flight when it returns.
template <int D, int NH, int STAGES, bool MERGE, typename Ready>
__device__ __forceinline__ void decode_units(const StepDevice& s, const CUtensorMap* kv_map, unsigned char* smem,
                                             uint32_t base, Ready&& ready) {
  using L = DecSmem<D, STAGES>;
  constexpr int W = kDecWarps;
  constexpr int STAGE_BYTES = L::kStageBytes;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int g = lane >> 2, t = lane & 3;
  const int G = s.Hq / s.Hkv;

  const uint32_t ring = base + warp * STAGES * STAGE_BYTES;
  float* merge_o = reinterpret_cast<float*>(smem + L::kOffMerge);         // [W][G][D]
  float* merge_ml = merge_o + W * G * D;                                  // [W][G][2]
  const UnitInfo* units = reinterpret_cast<const UnitInfo*>(smem + L::off_units(G));
  const uint32_t bars = base + L::off_bars(G);
  auto bar = [&](int i) { return bars + (uint32_t)i * 8u; };
  const uint32_t my_bars = bars + warp * STAGES * 8;
  volatile int* failed = reinterpret_cast<volatile int*>(smem + L::off_failed(G));

  if (tid == 0) {
    for (int i = 0; i < L::kBars; ++i) mbar_init(bar(i), i >= L::kBarDone && i != L::kBarNear ? W : 1);
    *failed = 0;
    mbar_init_fence();
  }
  decode_meet();
  ready();

  bool dead = false;           // a wait of this warp ran out (all lanes agree): it starts no copy and no page any more
  auto wait = [&](int i, uint32_t parity) {
    dead = dead || !wait_for_warps(bar(i), parity, failed, s.unit_wait_cycles);
  };
  // ---------------------------------------------------------------- producer side (this warp)
  // Never blocks: where the next unit is not described yet, the free stages stay free until the next call.
  UnitInfo pu;
  int pk = 0;                  // unit sequence number the producer is in
  int pj = warp;               // next local page of this warp in that unit
  bool p_have = false;         // pu describes unit pk
  int p_pages = -1;            // lane i holds the page id of local page warp + (p_chunk*32 + i)*W
  int p_chunk = -1;
  int n_issued = 0, n_consumed = 0;
  bool near_sent = false;      // warp 0 tells the scheduler when it has three pages of the unit left to fetch
  auto fill = [&]() {
#pragma unroll 1
    while (n_issued - n_consumed < STAGES && !dead) {
      if (!p_have) {
        const int e = pk % kDecRing;
        if (!__all_sync(0xffffffffu, mbar_test(bar(L::kBarDesc + e), (pk / kDecRing) & 1))) return;
        pu = units[e];
        p_have = true;
        pj = warp;
        p_chunk = -1;
        near_sent = false;
      }
      if (pu.n_pg < 0) return;                       // no more units
      if (warp == 0 && !near_sent && pj + 3 * W >= pu.n_pg) {
        near_sent = true;
        if (lane == 0) mbar_arrive(bar(L::kBarNear));
      }
      if (pj >= pu.n_pg) {
        ++pk;
        p_have = false;
        continue;
      }
      const int idx = (pj - warp) / W;
      if ((idx >> 5) != p_chunk) {
        p_chunk = idx >> 5;
        const int j = warp + ((p_chunk << 5) + lane) * W;
        p_pages = j < pu.n_pg ? pu.table_row[pu.first_page + j] : 0;
      }
      int page = __shfl_sync(0xffffffffu, p_pages, idx & 31);
      if (lane == 0) {
        if ((unsigned)page >= (unsigned)s.n_pages) {
          atomicOr(s.status, TS_DEV_BAD_PAGE);
          page = s.n_pages;    // out of range on purpose: the copy then delivers zeros
        }
        const int stage = n_issued % STAGES;
        const uint32_t b = my_bars + stage * 8;
        const uint32_t dst = ring + stage * STAGE_BYTES;
        fence_proxy_async();
        mbar_expect_tx(b, STAGE_BYTES);
        tma_load_5d(dst, kv_map, b, 0, pu.head * kPageSize, 0, 0, page);
      }
      ++n_issued;
      pj += W;
    }
  };

  // ------------------------------------------------------------------ sum over the warps of a unit
  // (they saw disjoint pages of it): this warp's eighth of unit k's results
  auto add_up = [&](int k) {
    const UnitInfo& u = units[k % kDecRing];
    for (int idx = tid; idx < G * D; idx += kDecThreads) {
      const int hh = idx / D, d = idx % D;
      float mm = -CUDART_INF_F;
#pragma unroll
      for (int w = 0; w < W; ++w) mm = fmaxf(mm, merge_ml[(w * G + hh) * 2]);
      float ll = 0.f, acc = 0.f;
#pragma unroll
      for (int w = 0; w < W; ++w) {
        const float wgt = exp2f(merge_ml[(w * G + hh) * 2] - mm);   // a warp without pages: exp2(-inf) = 0
        ll += wgt * merge_ml[(w * G + hh) * 2 + 1];
        acc += wgt * merge_o[((size_t)w * G + hh) * D + d];
      }
      const int head = u.head * G + hh;
      if (u.partial_slot < 0) {
        s.out[((size_t)u.tok * s.Hq + head) * D + d] = __bfloat16_as_ushort(__float2bfloat16_rn(acc / ll));
      } else {
        const size_t ph = (size_t)u.partial_slot * s.Hq + head;
        s.part_acc[ph * D + d] = acc;
        if (d == 0) {
          s.part_ml[ph * 2] = mm;
          s.part_ml[ph * 2 + 1] = ll;
        }
      }
    }
    __syncwarp();
    if (lane == 0) {
      mbar_arrive(bar(L::kBarAdded));
      mbar_arrive(bar(L::kBarDone + k % kDecRing));
    }
  };

  // ---------------------------------------------------------------------------- consumer side
  int ck = 0;
  bool owe = false;            // unit ck - 1 has not been added up by this warp yet
#pragma unroll 1
  for (;; ++ck) {
    wait(L::kBarDesc + ck % kDecRing, (ck / kDecRing) & 1);
    if (dead) break;           // what the ring holds is not known to be this unit
    const UnitInfo cu = units[ck % kDecRing];
    if (cu.n_pg < 0) break;
    fill();
    const int tok = cu.tok;
    const int n = cu.k_end;
    const int new_pos = cu.new_pos;
    // Q^T fragments: lane (g, t) holds head g (and g + 8), head_dim pairs 2t, 2t+1 (+8)
    uint32_t qf[NH][D / 16][2];
#pragma unroll
    for (int nh = 0; nh < NH; ++nh) {
      const int hh = nh * 8 + g;
      const uint16_t* qp = s.q + ((size_t)tok * s.Hq + cu.head * G + hh) * D + 2 * t;
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) {
        qf[nh][ks][0] = hh < G ? *reinterpret_cast<const uint32_t*>(qp + ks * 16) : 0u;
        qf[nh][ks][1] = hh < G ? *reinterpret_cast<const uint32_t*>(qp + ks * 16 + 8) : 0u;
      }
    }
    float o[NH][D / 16][4];
    float m[NH][2], l[NH][2];
#pragma unroll
    for (int nh = 0; nh < NH; ++nh) {
      m[nh][0] = m[nh][1] = -CUDART_INF_F;
      l[nh][0] = l[nh][1] = 0.f;
#pragma unroll
      for (int dt = 0; dt < D / 16; ++dt) o[nh][dt][0] = o[nh][dt][1] = o[nh][dt][2] = o[nh][dt][3] = 0.f;
    }

#pragma unroll 1
    for (int j = warp; j < cu.n_pg; j += W) {
      const int stage = n_consumed % STAGES;
      const uint32_t sp = ring + stage * STAGE_BYTES;
      dead = !__all_sync(0xffffffffu, mbar_wait(my_bars + stage * 8, (n_consumed / STAGES) & 1, s.wait_cycles));
      if (dead) break;
      const int pos0 = cu.k_begin + j * kPageSize;   // position of the page's first slot
      if (new_pos >= pos0 && new_pos < pos0 + kPageSize) {
        // KV append (Sec. 2.1) without a launch of its own: this page holds the row's new token,
        // which is not in the pool yet. Lay its K and V over the page image in shared memory and
        // write them to the pool page; a lane moves one 16-byte chunk of K or V.
        constexpr int CH = D / 8;
        const int r = new_pos - pos0;
        const int page = cu.table_row[cu.first_page + j];
        unsigned char* pg = smem + (sp - base);
        for (int i = lane; i < 2 * CH; i += 32) {
          const int kv = i / CH, c = i % CH;
          const uint4 val = *reinterpret_cast<const uint4*>((kv ? s.v_new : s.k_new) + ((size_t)tok * s.Hkv + cu.head) * D + c * 8);
          *reinterpret_cast<uint4*>(pg + page_off<D>(kv, r, c)) = val;
          if ((unsigned)page < (unsigned)s.n_pages)
            *reinterpret_cast<uint4*>(s.pool + ((((size_t)page * 2 + kv) * s.Hkv + cu.head) * kPageSize + r) * D + c * 8) = val;
        }
        __syncwarp();
      }
      const bool ragged = pos0 + kPageSize > n;
      if (ragged) {
        // slots past the last token hold whatever was there before: clear their V rows so
        // that a zero weight times stale bits cannot produce NaN
        const int valid = n - pos0;
        unsigned char* pg = smem + (sp - base);
        for (int i = lane; i < kPageSize * 8 * (D / 64); i += 32) {
          const int half = i / (kPageSize * 8), r = (i / 8) % kPageSize, c = i % 8;
          if (r >= valid)
            *reinterpret_cast<uint4*>(pg + kPageSize * D * 2 + half * 2048 + r * 128 + c * 16) = make_uint4(0, 0, 0, 0);
        }
        __syncwarp();
      }
      // ---- S^T = K Q^T : 16 keys x 8 heads per n-tile
      // (two accumulators per n-tile, even and odd k-steps: half the dependent MMA chain)
      float sc[NH][4], sc_odd[NH][4];
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        sc[nh][0] = sc[nh][1] = sc[nh][2] = sc[nh][3] = 0.f;
        sc_odd[nh][0] = sc_odd[nh][1] = sc_odd[nh][2] = sc_odd[nh][3] = 0.f;
      }
#pragma unroll
      for (int ks = 0; ks < D / 16; ++ks) {
        uint32_t a[4];
        const int mi = lane >> 3;
        ldmatrix_x4(a, sp + page_off<D>(0, (mi & 1) * 8 + (lane & 7), 2 * ks + (mi >> 1)));
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) mma_bf16((ks & 1) ? sc_odd[nh] : sc[nh], a, qf[nh][ks][0], qf[nh][ks][1]);
      }
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        sc[nh][0] += sc_odd[nh][0];
        sc[nh][1] += sc_odd[nh][1];
        sc[nh][2] += sc_odd[nh][2];
        sc[nh][3] += sc_odd[nh][3];
      }
      // ---- online softmax per head (this lane: heads 2t, 2t+1 of each n-tile; keys g, g+8)
      uint32_t pb[NH][2];
#pragma unroll
      for (int nh = 0; nh < NH; ++nh) {
        const bool v0 = !ragged || pos0 + g < n, v1 = !ragged || pos0 + g + 8 < n;
        float s0 = v0 ? sc[nh][0] * s.scale_log2 : -CUDART_INF_F;
        float s1 = v0 ? sc[nh][1] * s.scale_log2 : -CUDART_INF_F;
        float s2 = v1 ? sc[nh][2] * s.scale_log2 : -CUDART_INF_F;
        float s3 = v1 ? sc[nh][3] * s.scale_log2 : -CUDART_INF_F;
        // The reference of a head is the largest score so far, so that its largest weight is 1: exact in
        // bf16, where the weights that go into the second product are rounded (l adds them up unrounded, so
        // nothing cancels). A reference allowed to lag behind by 2^8 rounded the largest weight too: 2.1e-3
        // relative error became 2.3e-3 on N(0,1) keys. A page without a new maximum needs no reduction over the
        // lanes and no rescaling; the others come ever more seldom along a row.
        float al0 = 1.f, al1 = 1.f;
        const bool move = fmaxf(s0, s2) > m[nh][0] || fmaxf(s1, s3) > m[nh][1];
        if (__any_sync(0xffffffffu, move)) {
          float mx0 = fmaxf(s0, s2), mx1 = fmaxf(s1, s3);
#pragma unroll
          for (int sh = 4; sh < 32; sh <<= 1) {
            mx0 = fmaxf(mx0, __shfl_xor_sync(0xffffffffu, mx0, sh));
            mx1 = fmaxf(mx1, __shfl_xor_sync(0xffffffffu, mx1, sh));
          }
          const float mn0 = fmaxf(m[nh][0], mx0), mn1 = fmaxf(m[nh][1], mx1);
          al0 = exp2f(m[nh][0] - mn0);                    // first page: 2^(-inf) = 0
          al1 = exp2f(m[nh][1] - mn1);
          m[nh][0] = mn0;
          m[nh][1] = mn1;
#pragma unroll
          for (int dt = 0; dt < D / 16; ++dt) {
            o[nh][dt][0] *= al0;
            o[nh][dt][1] *= al1;
            o[nh][dt][2] *= al0;
            o[nh][dt][3] *= al1;
          }
        }
        s0 = ex2(s0 - m[nh][0]);
        s1 = ex2(s1 - m[nh][1]);
        s2 = ex2(s2 - m[nh][0]);
        s3 = ex2(s3 - m[nh][1]);
        l[nh][0] = l[nh][0] * al0 + s0 + s2;
        l[nh][1] = l[nh][1] * al1 + s1 + s3;
        // P^T as the B operand: transpose the two 8x8 (key x head) blocks across the warp
        pb[nh][0] = movmatrix_t(pack_bf16(s0, s1));
        pb[nh][1] = movmatrix_t(pack_bf16(s2, s3));
      }
      // ---- O^T += V^T P^T : 16 head_dim rows per m-tile
#pragma unroll
      for (int dt = 0; dt < D / 16; ++dt) {
        uint32_t a[4];
        const int mi = lane >> 3;
        ldmatrix_x4_trans(a, sp + page_off<D>(1, (mi >> 1) * 8 + (lane & 7), 2 * dt + (mi & 1)));
#pragma unroll
        for (int nh = 0; nh < NH; ++nh) mma_bf16(o[nh][dt], a, pb[nh][0], pb[nh][1]);
      }
      __syncwarp();
      ++n_consumed;
      fill();
      if (owe && __all_sync(0xffffffffu, mbar_test(bar(L::kBarWritten), (ck - 1) & 1))) {
        add_up(ck - 1);
        owe = false;
      }
    }

    // ---- leave this warp's partial result, once everyone is done with the previous unit's
    if (owe) {
      wait(L::kBarWritten, (ck - 1) & 1);
      if (dead) break;
      add_up(ck - 1);
      owe = false;
    }
    if (ck > 0) wait(L::kBarAdded, (ck - 1) & 1);
    if (dead) break;
#pragma unroll
    for (int nh = 0; nh < NH; ++nh) {
#pragma unroll
      for (int sh = 4; sh < 32; sh <<= 1) {
        l[nh][0] += __shfl_xor_sync(0xffffffffu, l[nh][0], sh);
        l[nh][1] += __shfl_xor_sync(0xffffffffu, l[nh][1], sh);
      }
      const int h0 = nh * 8 + 2 * t, h1 = h0 + 1;
      float* wo = merge_o + (size_t)warp * G * D;
#pragma unroll
      for (int dt = 0; dt < D / 16; ++dt) {
        const int d = dt * 16 + g;
        if (h0 < G) {
          wo[h0 * D + d] = o[nh][dt][0];
          wo[h0 * D + d + 8] = o[nh][dt][2];
        }
        if (h1 < G) {
          wo[h1 * D + d] = o[nh][dt][1];
          wo[h1 * D + d + 8] = o[nh][dt][3];
        }
      }
      if (g == 0) {
        if (h0 < G) {
          merge_ml[(warp * G + h0) * 2] = m[nh][0];
          merge_ml[(warp * G + h0) * 2 + 1] = l[nh][0];
        }
        if (h1 < G) {
          merge_ml[(warp * G + h1) * 2] = m[nh][1];
          merge_ml[(warp * G + h1) * 2 + 1] = l[nh][1];
        }
      }
    }
    __syncwarp();
    if (lane == 0) mbar_arrive(bar(L::kBarWritten));
    owe = true;
  }
  if (owe) {
    wait(L::kBarWritten, (ck - 1) & 1);
    if (!dead) add_up(ck - 1);
  }
  // no copy stays in flight (only after a failure are there any left)
  if (dead) give_up(s, failed);
  for (; n_consumed < n_issued; ++n_consumed) mbar_wait(my_bars + (n_consumed % STAGES) * 8, (n_consumed / STAGES) & 1, kDrainCycles);
  decode_meet();               // the scheduler included: then the barriers' shared memory can be given back
  if (MERGE && s.merge_here != 0) {
    const int* merges = reinterpret_cast<const int*>(smem + L::off_merges(G));
    for (int i = 0; i < kDecRing; ++i)
      if (merges[i] >= 0) merge_by_all<D>(s, units[merges[i]].merge, units[merges[i]].head, warp, lane);
  }
  if (tid == 0) {
    for (int i = 0; i < L::kBars; ++i) asm volatile("mbarrier.inval.shared::cta.b64 [%0];\n" ::"r"(bar(i)) : "memory");
  }
}

}  // namespace dec
}  // namespace ts
