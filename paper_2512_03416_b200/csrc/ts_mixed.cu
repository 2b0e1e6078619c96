// The attention kernel of a mixed step (sm_100a, head_dim 128): causal prefill-chunk tiles on the
// 5th-generation tensor cores and, in the same launch, the split-KV decode units.
//
// One persistent CTA per SM. The first n_prefill_ctas CTAs take prefill work units (prefill work
// item x KV head) from a global queue, heaviest first. The remaining CTAs first run the decode units
// (dec::decode_units: a queue of its own, TMA page copies, bound by HBM bandwidth) and then join the
// prefill queue, so that the HBM-bound and the tensor-bound halves of a step overlap
// instead of running back to back, and whichever CTAs finish first pick up what is left.
//
// A prefill work unit = two query tiles A and B of 128 packed rows each (128/G consecutive tokens
// x the G query heads of one KV head per tile) against all keys they may see, 128 keys per block.
// Per tile and block:
//     S = Q K^T   (tcgen05.mma, operands in 128B-swizzled shared memory, fp32 accumulator in TMEM)
//     online softmax by two warpgroups, two threads per query row, half a score row in registers each
//     O += P V    (tcgen05.mma, P read from TMEM as bf16, V from shared memory, O accumulates in TMEM)
// The two tiles share every K/V block (half the shared-memory fill per flop) and run out of phase:
// while one tile's warpgroups are in their softmax, the tensor pipe works for the other tile.
// TMEM (512 columns): S_A, S_B, O_A, O_B, 128 columns each; the P of the keys in a 64-column half
// of S overwrites the first 32 columns of that half.
// Warp roles: warps 0-3 / 8-11 softmax and epilogue of tile A (keys 0-63 / 64-127 of each block,
// head_dim columns 0-63 / 64-127 of O), warps 4-7 / 12-15 the same for tile B (thread = TMEM lane =
// query row; a warp can only reach the 32 lanes its index modulo 4 selects, so a row is split by
// columns). The two threads of a row agree on a new row maximum by a vote of their two warps per block. Two softmax warps per tile and SM sub-partition hide each
// other's instruction latencies: one warp per row quarter left the tensor pipe idle more than
// half of the time although no unit was saturated. Warp 16 K loader, warp 17 V loader (TMA copies of
// pages and of the chunk's own tokens; the K loader's first thread also claims the work units), warp 18 MMA issuer and TMEM owner, warp 19 Q loader (TMA).
// All barrier phases follow running block counters, so the roles flow from one work unit into the
// next without a CTA-wide stop: the loaders run ahead into the next unit's K/V, its Q tiles land
// as soon as the last Q K^T of the current unit has been issued, and its first Q K^T overlaps
// the epilogue of the current unit.
// The O rescale is lazy: a row's reference maximum only moves when a block's maximum exceeds it by
// more than 2^8, so most blocks never touch O.
// The kernel appends the step's new K/V to the pages itself, which saves a launch in front of it:
// every CTA copies a share of the prefill rows' tokens next to its other work, and nothing waits for
// the copies, because the tiles take a chunk's own tokens from the step's tensors; the decode units
// write their rows' own tokens.
// Every wait is bounded (the hardware barriers are not, but all who meet on one do so equally often); a wait
// that runs out raises TS_DEV_TIMEOUT and the CTA drains: nothing new is
// started, the other waits end early, and before the CTA leaves, the copies and MMAs it did start are
// waited for (with a limit of their own).
#include <cuda_bf16.h>
#include <math_constants.h>

#include "../../include/tokenscale.h"
#include "ts_decode_body.h"
#include "ts_internal.h"
#include "ts_ptx.h"
#include "ts_tc.h"
#include "ts_tma.h"
#include "ts_units.h"

namespace ts {
namespace {

constexpr int kPfThreads = 640;                 // 16 softmax warps + K loader, V loader, MMA and Q-loader warps
constexpr int kSoftmaxWarps = 16;
// Register split (setmaxnreg works on whole warpgroups): the block is launched with 96 registers
// per thread; the four softmax warpgroups grow to hold their half score row, the fifth warpgroup
// (loaders, MMA issuer) shrinks. In a CTA that runs decode units first, the two warpgroups that run
// them take the registers the other two softmax warpgroups do not need yet.
constexpr int kRegsLaunch = 96, kRegsSoftmax = 104, kRegsAux = 64, kRegsDecode = 168, kRegsParked = 24;
static_assert(4 * 128 * kRegsSoftmax + 128 * kRegsAux <= kPfThreads * kRegsLaunch,
              "register split exceeds the launch's total");
static_assert(2 * 128 * kRegsDecode + 2 * 128 * kRegsParked + 128 * kRegsAux <= kPfThreads * kRegsLaunch,
              "register split of the decode phase exceeds the launch's total");
constexpr int kWarpLoader0 = 16, kWarpMma = 18, kWarpSched = 19;
constexpr int kD = 128;
constexpr int kTileBytes = 128 * kD * 2;        // one 128 x 128 bf16 operand tile: 32 KB
constexpr int kHalfBytes = kTileBytes / 2;      // 64 head_dim columns of it
constexpr int kKStages = 2, kVStages = 3;       // measured: a third V stage is worth more than a third K stage (3%)
constexpr long long kDrainCycles = 20000000;    // about 10 ms: limit of the waits for copies and MMAs in flight after a failure
// Keys of each half row whose P is announced, and multiplied by V, before the other ones' exponentials are taken: the
// P V of these 48 and the exponentials of the last 16 take about the same time (six MMAs 384 cycles, 16 exponentials
// of two warps 256 and the announcement), so that only two MMAs and the next Q K^T are left behind the last P.
// 8192 tokens alone, 70B shape / 2048 tokens alone, 8B shape (us, launches too short for the power cap): all 64 at once 879 / 40.0,
// 32 and 32 856 / 39.4, 48 and 16 837 / 38.4, three parts (32, 16, 16) no better than one; back to back, at the power cap
// 1023 / 41.6, 993 / 41.2, 979 / 40.7.
constexpr int kFirst = 48;
constexpr float kRescaleThreshold = 8.0f;       // log2 units

// shared-memory map (offsets from the 1024-aligned base)
constexpr int kOffQ = 0;                                    // Q_A, Q_B
constexpr int kOffK = kOffQ + 2 * kTileBytes;
constexpr int kOffV = kOffK + kKStages * kTileBytes;
constexpr int kOffBar = kOffV + kVStages * kTileBytes;
enum {
  BAR_Q = 0,
  BAR_K_FULL = 1,                         // [kKStages]
  BAR_K_EMPTY = BAR_K_FULL + kKStages,    // [kKStages]
  BAR_V_FULL = BAR_K_EMPTY + kKStages,    // [kVStages]
  BAR_V_EMPTY = BAR_V_FULL + kVStages,    // [kVStages]
  BAR_S_FULL = BAR_V_EMPTY + kVStages,    // [2] per tile
  BAR_P_FULL = BAR_S_FULL + 2,            // [2][2] per tile: the first kFirst keys of both halves of P, the others
  BAR_O_FULL = BAR_P_FULL + 4,            // [2] per tile: the last P V of a work unit has landed in O
  BAR_Q_EMPTY = BAR_O_FULL + 2,           // the last Q K^T of a work unit has consumed the Q tiles
  BAR_V_LANDED = BAR_Q_EMPTY + 1,         // [kVStages] the copies of a V tile are in shared memory
  BAR_K_LANDED = BAR_V_LANDED + kVStages, // the same for a K tile that needs a touch-up before it is announced
  BAR_DRAIN = BAR_K_LANDED + 1,           // after a failure: the MMAs issued before it are done
  BAR_COUNT = BAR_DRAIN + 1
};
// misc words: [0] TMEM base address, [1] failure flag, [2] work units published so far;
// then a ring of the published units' records (8 words each)
constexpr int kOffMisc = kOffBar + BAR_COUNT * 8;
constexpr int kOffRing = kOffMisc + 16;
// row statistics the two threads of a query row exchange: [tile][half][row] floats
constexpr int kOffXchg = kOffRing + kSchedRing * 32;
constexpr int kSmemBytes = kOffXchg + 2 * 2 * 128 * 4;
// The operand tiles need a 1024-byte-aligned base. The kernel has no static shared memory, so its
// dynamic window starts on such a boundary; the kernel checks that and refuses to run otherwise
// (there is no room left for alignment slack).
static_assert(kSmemBytes <= 232448, "exceeds the shared memory one CTA can opt into");

template <int N>
__device__ __forceinline__ void reg_inc() { asm volatile("setmaxnreg.inc.sync.aligned.u32 %0;\n" ::"n"(N)); }
template <int N>
__device__ __forceinline__ void reg_dec() { asm volatile("setmaxnreg.dec.sync.aligned.u32 %0;\n" ::"n"(N)); }
__device__ __forceinline__ float max3(float a, float b, float c) {
  float d;
  asm("max.f32 %0, %1, %2, %3;\n" : "=f"(d) : "f"(a), "f"(b), "f"(c));
  return d;
}
// Packed pairs of fp32 (sm_100 has two-wide fp32 add/fma): half the issue slots of scalar code.
__device__ __forceinline__ uint64_t pack_f2(float lo, float hi) {
  uint64_t r;
  asm("mov.b64 %0, {%1, %2};\n" : "=l"(r) : "f"(lo), "f"(hi));
  return r;
}
__device__ __forceinline__ void unpack_f2(uint64_t v, float& lo, float& hi) {
  asm("mov.b64 {%0, %1}, %2;\n" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ uint64_t fma2(uint64_t a, uint64_t b, uint64_t c) {
  uint64_t d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;\n" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ uint64_t add2(uint64_t a, uint64_t b) {
  uint64_t d;
  asm("add.rn.f32x2 %0, %1, %2;\n" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ float ex2(float x) {
  float y;
  asm("ex2.approx.ftz.f32 %0, %1;\n" : "=f"(y) : "f"(x));
  return y;
}

// N scores of a row: p_i = 2^(v_i * scale + neg_m) as bf16 pairs in pk (the scores are not needed
// afterwards, so their registers come free as the loop advances); adds the unrounded p_i to sum. The largest of
// these and of the NW scores in w rides along, in issue slots the exponentials leave free.
template <int N, int NW = 0>
__device__ __forceinline__ void exp_pack(const float* v, const float* w, uint64_t scale2, uint64_t negm2, uint32_t* pk, uint64_t (&sum)[2], float (&mx)[2]) {
#pragma unroll
  for (int i = 0; i < N / 2; ++i) {
    float x0, x1, p0, p1;
    unpack_f2(fma2(pack_f2(v[2 * i], v[2 * i + 1]), scale2, negm2), x0, x1);
    if (NW > 0) mx[0] = max3(mx[0], v[2 * i], v[2 * i + 1]);
    if (i < NW / 2) mx[1] = max3(mx[1], w[2 * i], w[2 * i + 1]);
    p0 = ex2(x0);
    p1 = ex2(x1);
    sum[i & 1] = add2(sum[i & 1], pack_f2(p0, p1));
    pk[i] = pack_bf16(p0, p1);
  }
}
// `mine` of any of the 64 threads of two warps, which meet on barrier `id`.
__device__ __forceinline__ bool pair_any(int id, bool mine) {
  int r;
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.s32 p, %2, 0;\nbarrier.cta.red.or.pred q, %1, 64, p;\nselp.s32 %0, 1, 0, q;\n}\n"
      : "=r"(r)
      : "r"(id), "r"((int)mine)
      : "memory");
  return r != 0;
}
// Largest of the 64 raw scores of a half row.
__device__ __forceinline__ float max64(const float (&v)[64]) {
  float m0 = max3(v[0], v[1], v[2]), m1 = max3(v[3], v[4], v[5]);
  float m2 = max3(v[6], v[7], v[8]), m3 = max3(v[9], v[10], v[11]);
#pragma unroll
  for (int i = 12; i < 60; i += 8) {
    m0 = max3(m0, v[i], v[i + 1]);
    m1 = max3(m1, v[i + 2], v[i + 3]);
    m2 = max3(m2, v[i + 4], v[i + 5]);
    m3 = max3(m3, v[i + 6], v[i + 7]);
  }
  m0 = max3(m0, v[60], v[61]);
  m1 = max3(m1, v[62], v[63]);
  return fmaxf(fmaxf(m0, m1), fmaxf(m2, m3));
}
// The append of the prefill rows' new tokens (Sec. 2.1). The prefill work items cover those tokens
// exactly once, `per_item` at most each; warp i of n appends tokens i, i + n, ... of that list. A lane
// looks up one of the warp's next 32 tokens (item -> row -> block table: three dependent loads, paid
// once per 32 tokens instead of once per token, 5 us each), then the warp copies them one by one, U
// 16-byte loads in flight per lane.
struct AppendCursor {
  __device__ __forceinline__ AppendCursor(int first, int n, int warps) : next(first), end(n), stride(warps) {}
  int next, end, stride;       // list position of the next token, end of the list, warps that share it
  int left = 0, at = 0;        // looked-up tokens not yet copied, lane that holds the next one
  int tok = -1;                // this lane's token in the step's tensors (-1: nothing to copy)
  uint32_t dst = 0;            // its page * 16 + slot

  __device__ __forceinline__ bool done() const { return left == 0 && next >= end; }
  __device__ __forceinline__ void look_up(const StepDevice& s, int per_item, int lane) {
    const int w = next + lane * stride;
    tok = -1;
    if (w < end) {
      const WorkItem it = s.item(w / per_item);
      const int j = w % per_item;
      if (j < it.q_count) {
        const int slot = s.row_slot(it.row), t = it.k_end - it.q_count + j;
        if ((unsigned)slot >= (unsigned)s.max_requests || (unsigned)(t >> 4) >= (unsigned)s.max_pages_per_req) {
          atomicOr(s.status, TS_DEV_BAD_INDEX);
        } else {
          const int page = s.table[(size_t)slot * s.max_pages_per_req + (t >> 4)];
          if ((unsigned)page >= (unsigned)s.n_pages) {
            atomicOr(s.status, TS_DEV_BAD_PAGE);
          } else {
            tok = s.row_tok0(it.row) + it.q_begin + j;
            dst = (uint32_t)page * kPageSize + (uint32_t)(t & 15);
          }
        }
      }
    }
    left = min(32, (end - next + stride - 1) / stride);
    at = 0;
    next += 32 * stride;
  }
  // Copies one token (call only while !done()).
  template <int U>
  __device__ __forceinline__ void step(const StepDevice& s, int per_item, int lane) {
    if (left == 0) look_up(s, per_item, lane);
    const int token = __shfl_sync(0xffffffffu, tok, at);
    const uint32_t d = __shfl_sync(0xffffffffu, dst, at);
    ++at;
    --left;
    if (token < 0) return;
    const int half = s.Hkv * (kD / 8);             // 16-byte chunks of the token's K (and of its V)
    const size_t src = (size_t)token * s.Hkv * kD, page0 = (size_t)(d / kPageSize) * 2 * s.Hkv;
#pragma unroll 1
    for (int c0 = lane; c0 < 2 * half; c0 += U * 32) {
      uint4 v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int c = c0 + u * 32;
        if (c < 2 * half) v[u] = *reinterpret_cast<const uint4*>(c < half ? s.k_new + src + c * 8 : s.v_new + src + (c - half) * 8);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {                // chunk c: K|V and head = c / 16 counted through, c % 16 of that head's row
        const int c = c0 + u * 32;
        if (c < 2 * half)
          *reinterpret_cast<uint4*>(s.pool + ((page0 + c / 16) * kPageSize + d % kPageSize) * kD + (c & 15) * 8) = v[u];
      }
    }
  }
  template <int U>
  __device__ __forceinline__ void run(const StepDevice& s, int per_item, int lane) {
    while (!done()) step<U>(s, per_item, lane);
  }
};

__device__ __forceinline__ void cta_sync() { asm volatile("bar.sync 0;\n" ::: "memory"); }

template <int W>
__global__ void __launch_bounds__(kPfThreads, 1)
mixed_kernel(const __grid_constant__ StepParams<W> params, const __grid_constant__ CUtensorMap q_map,
             const __grid_constant__ CUtensorMap kv_map, const __grid_constant__ CUtensorMap kv_tile_map,
             const __grid_constant__ NewKvMaps new_maps, const int n_prefill_ctas) {
  const StepDevice& s = params.s;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - smem_u32(smem_raw));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_launch_dependents();
  if (base != smem_u32(smem_raw)) {          // never expected, see kSmemBytes
    if (tid == 0) atomicOr(s.status, TS_DEV_BAD_INDEX);
    return;
  }
  const uint32_t bar0 = base + kOffBar;
  auto bar = [&](int i) { return bar0 + (uint32_t)i * 8u; };
  volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);
  const int G = s.Hq / s.Hkv;
  const int tile_tokens = 128 / G;
  const int n_units = s.n_prefill_items * s.Hkv;
  const bool decode_first = (int)blockIdx.x >= n_prefill_ctas;

  auto give_up = [&]() {
    if (misc[1] == 0) {
      atomicOr(s.status, TS_DEV_TIMEOUT);
      misc[1] = 1;
    }
  };
  auto wait = [&](int i, uint32_t parity) {
    if (!mbar_wait(bar(i), parity, misc[1] ? 2000 : s.wait_cycles)) give_up();
  };
  // k-th work unit of this CTA (w = -1 after the last one), published by the K loader. An entry of the
  // ring stays while it is read: the K loader is at most three units in front of the softmax warps (it is
  // two key blocks in front of the MMAs, and those need the P of all blocks before), and after a failure,
  // when its waits end early, it publishes no further unit. (A tile without rows in a unit is not waited
  // for; its warps only read the record, and have the whole unit's time for it.)
  volatile int4* ring = reinterpret_cast<volatile int4*>(smem + kOffRing);
  auto read_unit = [&](int k, PfUnit& u) -> bool {           // of a published unit
    UnitRec r;
    const int e = (k & (kSchedRing - 1)) * 2;
    const int4 lo = make_int4(ring[e].x, ring[e].y, ring[e].z, ring[e].w);
    const int4 hi = make_int4(ring[e + 1].x, ring[e + 1].y, ring[e + 1].z, ring[e + 1].w);
    r.w = lo.x; r.table_slot = lo.y; r.kv_head = lo.z; r.q_begin = lo.w;
    r.q_count = hi.x; r.ctx = hi.y; r.tok0 = hi.z;
    if (r.w < 0) return false;
    u = unit_shape(r, tile_tokens);
    return true;
  };
  // Called by whole warps; all lanes get the same answer (a warp that left its loop in part would never
  // meet its partner, or itself, again).
  auto get_work = [&](int k, PfUnit& u) -> bool {
    if (__any_sync(0xffffffffu, (int)misc[2] <= k)) {
      const long long t0 = clock64();
      while (__any_sync(0xffffffffu, (int)misc[2] <= k)) {
        if (__any_sync(0xffffffffu, clock64() - t0 > (misc[1] ? 2000 : s.wait_cycles))) {
          give_up();
          return false;
        }
      }
    }
    return read_unit(k, u);
  };
  auto ready = []() { pdl_wait(); };
  // The set-up every warp class runs between the decode phase and the prefill phase.
  auto prefill_setup = [&]() {
    if (tid == 0) {
      misc[1] = 0;
      misc[2] = 0;
      for (int i = 0; i < BAR_COUNT; ++i) {
        mbar_init(bar(i), i >= BAR_P_FULL && i < BAR_P_FULL + 4 ? kSoftmaxWarps / 2 : 1);
      }
      mbar_init_fence();
    }
    if (warp == kWarpMma) tmem_alloc(base + kOffMisc, 512);
    // When G does not divide 128 a query tile holds tile_tokens * G < 128 packed rows and the Q
    // copies never write the rest: clear those rows once, so that the MMA reads zeros there and
    // not whatever the shared memory held before.
    const int used_rows = tile_tokens * G;
    if (used_rows < 128) {
      const int n16 = (128 - used_rows) * 8;                 // 16-byte chunks per 64-column half tile
      for (int i = tid; i < 4 * n16; i += kPfThreads) {
        const int half = i / n16, c = i % n16;
        *reinterpret_cast<uint4*>(smem + kOffQ + half * kHalfBytes + used_rows * 128 + c * 16) = make_uint4(0, 0, 0, 0);
      }
      fence_proxy_async();
    }
    tc_fence_before();
    cta_sync();
    tc_fence_after();
  };
  // ---------------------------------------------------------------- KV append (Sec. 2.1)
  // The new tokens of the prefill rows are copied into their pages straight from the prefill work
  // items (which cover those tokens exactly once), and nothing in this launch waits for the copies:
  // the K/V loaders read a chunk's own tokens from the step's tensors. In a CTA that streams decode
  // rows first three warps of the fifth warpgroup copy a share while warps 0-7 are on their decode units. In a CTA
  // that takes prefill units from the start the Q loader copies one between its Q tiles; where the
  // units are too short to hide that (s.append_wide, decided on the host) the sixteen softmax warps
  // copy before their first scores arrive. The new token of a decode row is written by the decode
  // unit that reads the row's last page.
  constexpr int kWarpsAux = 3;                                    // warps 17-19; warp 16 schedules the decode units
  const int warps_first = s.append_wide ? kSoftmaxWarps : 1;     // appending warps of a CTA that starts on prefill units
  const int append_end = s.n_prefill_items * 2 * tile_tokens;
  const int append_warps = n_prefill_ctas * warps_first + ((int)gridDim.x - n_prefill_ctas) * kWarpsAux;
  // The fifth warpgroup (loaders, MMA issuer, Q loader): gives registers to the softmax warpgroups
  // and, in a decode-first CTA, appends and schedules while warps 0-7 run decode units.
  auto aux_setup = [&]() {
    reg_dec<kRegsAux>();
    if (decode_first) {
      if (warp == kSoftmaxWarps)
        dec::decode_schedule<128, 3, false>(s, smem, base, (int)blockIdx.x - n_prefill_ctas, (int)gridDim.x - n_prefill_ctas, ready);
      else {
        ready();
        AppendCursor{n_prefill_ctas * warps_first + ((int)blockIdx.x - n_prefill_ctas) * kWarpsAux + (warp - kSoftmaxWarps - 1),
                     append_end, append_warps}
            .run<8>(s, 2 * tile_tokens, lane);
      }
      cta_sync();
    }
    prefill_setup();
  };

  // The launch in front of this one (the previous step's kernels, which must be done with the pool and the counters) is
  // waited for as late as can be: a CTA's barriers, TMEM and, where the step's metadata are launch parameters, its
  // first decode unit are set up before.
  if (decode_first && s.meta) ready();
  if (tid == kSoftmaxWarps * 32) {
    tma_prefetch_desc(&q_map);
    tma_prefetch_desc(&kv_tile_map);
    tma_prefetch_desc(&new_maps.k);
    tma_prefetch_desc(&new_maps.v);
  }

  if (warp < kSoftmaxWarps) {
    // ------------------ softmax + epilogue: thread = half of a query row of tile x (64 of the 128
    // keys of every block, 64 of the 128 head_dim columns of O)
    if (decode_first) {
      if (warp < 8) {
        reg_inc<kRegsDecode>();       // waits until the parked warpgroups have given their registers up
        dec::decode_units<128, 1, 3, false>(s, &kv_map, smem, base, ready);
        if (tid == 0) {          // this CTA's split partials are written: count it as done
          __threadfence();
          atomicAdd(s.pf_queue + 1, 1);
        }
        fence_proxy_async();     // the prefill phase reuses this shared memory through other proxies
        reg_dec<kRegsSoftmax>();
        cta_sync();
      } else {
        reg_dec<kRegsParked>();
        cta_sync();
        reg_inc<kRegsSoftmax>();
      }
    } else {
      reg_inc<kRegsSoftmax>();
    }
    prefill_setup();
    ready();
    if (!decode_first && s.append_wide)
      AppendCursor{(int)blockIdx.x * kSoftmaxWarps + warp, append_end, append_warps}.run<8>(s, 2 * tile_tokens, lane);
    const uint32_t tmem = misc[0];
    const int x = (warp >> 2) & 1;          // tile
    const int hf = warp >> 3;               // which half of the keys / of the head_dim columns
    const int row = (warp & 3) * 32 + lane;
    const uint32_t lane_addr = (uint32_t)((warp & 3) * 32) << 16;
    const uint32_t tS = tmem + x * 128 + hf * 64 + lane_addr;         // my 64 score columns; P goes to the first 32
    const uint32_t tO = tmem + 256 + x * 128 + hf * 64 + lane_addr;   // my 64 columns of O
    // The two warps that share a quarter of a tile's rows meet on a hardware barrier (ids 4-11): around
    // each exchange through shared memory, and for the vote on a block's maxima; it wakes them sooner than an mbarrier (together with
    // the other changes to the unit loop that came with it: 8192-token chunk next to 190 rows 1272 -> 1263 us,
    // 2048 tokens alone 49.5 -> 46.3 us). It has no time limit, so
    // the two must never disagree about how often they meet: all their other waits are limited and end
    // in the same control flow, and how many blocks of a unit the tile has (-1: there is no further unit)
    // is for the first of them to say, one number for all lanes of both.
    auto pair_sync = [&]() { asm volatile("bar.sync %0, 64;\n" ::"r"(4 + x * 4 + (warp & 3)) : "memory"); };
    float* xchg = reinterpret_cast<float*>(smem + kOffXchg) + x * 256;   // [half][row] of my tile
    float* xchg_mine = xchg + hf * 128 + row;
    float* xchg_other = xchg + (hf ^ 1) * 128 + row;
    int row_g = row / G, row_h = row % G;   // token of the tile and query head of this row
    const float scale = s.scale_log2;
    const uint64_t scale2 = pack_f2(scale, scale);
    int sx = 0;                 // blocks of this tile in earlier work units: barrier phases follow it
    int n_o = 0;                // earlier work units in which the tile had rows (O_FULL phases)
    for (int k = 0;; ++k) {
      PfUnit u = {};
      int nbx = -1;
      if (hf == 0) {
        nbx = __shfl_sync(0xffffffffu, posted_blocks(get_work(k, u), u, x), 0);
        *xchg_other = __int_as_float(nbx);   // the other thread's own slot: it reads it before it writes it again
      }
      pair_sync();
      if (hf == 1) nbx = __shfl_sync(0xffffffffu, __float_as_int(*xchg_mine), 0);
      if (nbx < 0) break;
      if (hf == 1) read_unit(k, u);
      const int cnt = x ? u.cnt_b : u.cnt_a;
      const int tok = u.q_begin + x * tile_tokens + row_g;     // token inside the request row
      const bool real = row_g < cnt && row < tile_tokens * G;
      const int lim = real ? u.ctx + tok + 1 : (x ? u.k_end_b : u.k_end_a);   // keys at positions >= lim are masked
      // the row's place in the output (counted in rows of head_dim), none for a row that is padding
      const uint32_t orow = real ? (uint32_t)(u.tok0 + tok) * s.Hq + u.kv_head * G + row_h : 0xffffffffu;
      const int lim_min = (int)__reduce_min_sync(0xffffffffu, (unsigned)lim);
      float m_ref = -CUDART_INF_F, l = 0.f;
      for (int j = 0; j < nbx; ++j) {
        wait(BAR_S_FULL + x, (sx + j) & 1);
        tc_fence_after();
        // my half of the score row comes into registers: one trip to TMEM per block
        float v[64];
        const int nvalid = lim - j * kBlockKeys - hf * 64;     // keys of my half the row may see
        tmem_ld32(&v[0], tS);
        tmem_ld32(&v[32], tS + 32);
        tmem_ld_wait();
        if (lim_min - j * kBlockKeys - hf * 64 < 64) {         // only the blocks on the diagonal
#pragma unroll
          for (int i = 0; i < 64; ++i)
            if (i >= nvalid) v[i] = -CUDART_INF_F;             // 2^(-inf) = 0 exactly
        }
        // p = 2^(s*scale - m_ref) as bf16, to go over the first 32 columns of my half of S. Any
        // common reference is exact; p <= 2^threshold keeps the bf16 P and the fp32 sums
        // comfortable, so the reference only moves (and O is only rescaled) when the block maximum
        // exceeds it by more than the threshold. After the first block of a unit the first exponentials are
        // taken at once against the reference the row already has, and the maximum of all 64 scores rides along
        // with them: that is nearly always the final answer, and one vote of the two warps says so. Where some
        // row has to move, the two threads of each row post the maxima of their halves (the scale is positive, so it
        // commutes with max) and see the same two numbers, so they take the same decision; no P has been stored by then,
        // so the scores are still in TMEM and are fetched once more. A row of the last, diagonal block may be masked
        // completely; it keeps its reference (block 0 always holds key 0, which every row sees).
        uint32_t pk[32];
        float mx[2] = {-CUDART_INF_F, -CUDART_INF_F};
        uint64_t sum[2] = {0, 0};
        uint64_t negm2;
        if (j == 0) {
          *xchg_mine = max64(v) * scale;
          pair_sync();
          m_ref = fmaxf(*xchg_mine, *xchg_other);
          negm2 = pack_f2(-m_ref, -m_ref);
          exp_pack<kFirst>(&v[0], nullptr, scale2, negm2, pk, sum, mx);
        } else {
          negm2 = pack_f2(-m_ref, -m_ref);
          exp_pack<kFirst, 64 - kFirst>(&v[0], &v[kFirst], scale2, negm2, pk, sum, mx);
          const float mine = fmaxf(mx[0], mx[1]) * scale;
          if (pair_any(4 + x * 4 + (warp & 3), mine > m_ref + kRescaleThreshold)) {
            *xchg_mine = mine;
            pair_sync();
            const float m_blk = fmaxf(mine, *xchg_other);
            const bool move = m_blk > m_ref + kRescaleThreshold;
            float alpha = 1.f;
            if (move) {
              alpha = ex2(m_ref - m_blk);
              m_ref = m_blk;
              l *= alpha;
            }
            // O is complete up to block j-1: that P V was issued in front of these scores' Q K^T
#pragma unroll 1
            for (int c = 0; c < 4; ++c) {
              float ov[16];
              tmem_ld16(ov, tO + c * 16);
              tmem_ld_wait();
#pragma unroll
              for (int i = 0; i < 16; ++i) ov[i] *= alpha;
              tmem_st16(tO + c * 16, *reinterpret_cast<const uint32_t(*)[16]>(ov));
            }
            tmem_ld32(&v[0], tS);
            if (kFirst > 32) tmem_ld16(&v[32], tS + 32);
            tmem_ld_wait();
#pragma unroll
            for (int i = 0; i < kFirst; ++i)
              if (i >= nvalid) v[i] = -CUDART_INF_F;
            negm2 = pack_f2(-m_ref, -m_ref);
            sum[0] = sum[1] = 0;
            exp_pack<kFirst>(&v[0], nullptr, scale2, negm2, pk, sum, mx);
          }
        }
        // The exponentials of half of the rest hide the time the stores of the first part take.
        auto announce = [&](int part) {
          tmem_st_wait();
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(BAR_P_FULL + x * 2 + part));
        };
        constexpr int kHalfRest = (64 - kFirst) / 2;
        tmem_st16(tS, *reinterpret_cast<const uint32_t(*)[16]>(&pk[0]));
        if (kFirst > 32) tmem_st8(tS + 16, &pk[16]);
        exp_pack<kHalfRest>(&v[kFirst], nullptr, scale2, negm2, pk + kFirst / 2, sum, mx);
        announce(0);
        exp_pack<kHalfRest>(&v[kFirst + kHalfRest], nullptr, scale2, negm2, pk + kFirst / 2 + kHalfRest / 2, sum, mx);
        if (kFirst > 32) tmem_st8(tS + 24, &pk[24]);
        else tmem_st16(tS + 16, *reinterpret_cast<const uint32_t(*)[16]>(&pk[16]));
        float s0, s1;
        unpack_f2(add2(sum[0], sum[1]), s0, s1);
        l += s0 + s1;
        announce(1);
      }
      if (nbx > 0) {
        // epilogue: O / l -> bf16 -> global; l is the sum over both halves of the keys. (The last
        // P V has been issued, so the partner has arrived for the last block and is done with
        // that block's exchange slots.)
        wait(BAR_O_FULL + x, n_o++ & 1);
        tc_fence_after();
        *xchg_mine = l;
        pair_sync();
        const float inv = 1.f / (l + *xchg_other);
        pair_sync();                      // both have read: the slots may be written again
        // A row's 64 columns are one thread's; stored as they are, every 16-byte store of a warp would touch
        // 32 rows. The four lanes of a quad swap 16-byte chunks first, so that they write 64 bytes of a
        // row together.
#pragma unroll 1
        for (int c = 0; c < 2; ++c) {
          float ov[32];
          tmem_ld32(ov, tO + c * 32);
          tmem_ld_wait();
          uint32_t w[4][4];                      // [chunk of 8 columns][bf16 pair]
#pragma unroll
          for (int i = 0; i < 4; ++i)
#pragma unroll
            for (int e = 0; e < 4; ++e) w[i][e] = pack_bf16(ov[8 * i + 2 * e] * inv, ov[8 * i + 2 * e + 1] * inv);
#pragma unroll
          for (int bit = 1; bit < 4; bit <<= 1) {          // 4 x 4 transpose over the quad: w[i] becomes chunk lane % 4 of row i
            const bool up = lane & bit;
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              if (i & bit) continue;
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const uint32_t got = __shfl_xor_sync(0xffffffffu, up ? w[i][e] : w[i | bit][e], bit);
                if (up) w[i][e] = got; else w[i | bit][e] = got;
              }
            }
          }
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const uint32_t r = __shfl_sync(0xffffffffu, orow, (lane & ~3) + i);
            if (r != 0xffffffffu)
              *reinterpret_cast<uint4*>(s.out + (size_t)r * kD + hf * 64 + c * 32 + (lane & 3) * 8) =
                  make_uint4(w[i][0], w[i][1], w[i][2], w[i][3]);
          }
        }
      }
      if (nbx == 0) pair_sync();             // hf 1 has read the slot
      sx += nbx;
    }
    // -------------------------------------------------------------- merge of the decode splits
    // By now the decode CTAs are normally long done; once all of them have counted themselves,
    // the first eight warps of every CTA merge the split rows between them.
    const int n_decode_ctas = (int)gridDim.x - n_prefill_ctas;
    if (warp < 8 && s.n_combines > 0 && n_decode_ctas > 0) {
      if (tid == 0) {
        const volatile int32_t* done = s.pf_queue + 1;
        const long long t0 = clock64();
        while (*done < n_decode_ctas + s.debug_arrivals) {
          if (clock64() - t0 > (misc[1] ? 2000 : s.wait_cycles)) {
            give_up();
            break;
          }
        }
        __threadfence();
      }
      dec::block_sync();
      // one warp per (split row, query head), dealt round-robin over all warps of the launch;
      // a lane merges four head_dim elements
      const int n_pairs = s.n_combines * s.Hq;
      for (int pi = (int)blockIdx.x * 8 + warp; pi < n_pairs; pi += (int)gridDim.x * 8) {
        const CombineItem c = s.combine(pi / s.Hq);
        const int h = pi % s.Hq;
        const float* ml = s.part_ml + ((size_t)c.first_partial * s.Hq + h) * 2;
        const float* pa = s.part_acc + ((size_t)c.first_partial * s.Hq + h) * kD + lane * 4;
        const size_t ml_stride = (size_t)s.Hq * 2, pa_stride = (size_t)s.Hq * kD;
        float m = -CUDART_INF_F, l = 0.f;
        float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
        for (int b0 = 0; b0 < c.n_splits; b0 += 8) {
          float mi[8], li[8];
          float4 ai[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const bool on = b0 + j < c.n_splits;
            mi[j] = on ? __ldcg(ml + (b0 + j) * ml_stride) : -CUDART_INF_F;
            li[j] = on ? __ldcg(ml + (b0 + j) * ml_stride + 1) : 0.f;
            ai[j] = on ? __ldcg(reinterpret_cast<const float4*>(pa + (b0 + j) * pa_stride)) : make_float4(0.f, 0.f, 0.f, 0.f);
          }
          float mn = m;
#pragma unroll
          for (int j = 0; j < 8; ++j) mn = fmaxf(mn, mi[j]);
          const float keep = exp2f(m - mn);          // 0 on the first group (m = -inf)
          l *= keep;
          acc.x *= keep; acc.y *= keep; acc.z *= keep; acc.w *= keep;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const float wgt = exp2f(mi[j] - mn);     // absent split: exp2(-inf) = 0
            l += wgt * li[j];
            acc.x += wgt * ai[j].x; acc.y += wgt * ai[j].y; acc.z += wgt * ai[j].z; acc.w += wgt * ai[j].w;
          }
          m = mn;
        }
        const float inv = 1.f / l;
        uint2 o;
        o.x = pack_bf16(acc.x * inv, acc.y * inv);
        o.y = pack_bf16(acc.z * inv, acc.w * inv);
        *reinterpret_cast<uint2*>(s.out + ((size_t)c.token * s.Hq + h) * kD + lane * 4) = o;
      }
    }
  } else {
    // warps 16-19 are one warpgroup: they change their register count with one instruction
    aux_setup();
    if (warp < kWarpLoader0 + 2) {
      // ------------------------------------------------------------------ K/V loaders
      // One warp per operand. A 128-key tile of cached tokens is sixteen tensor copies of 2 KB (one
      // page of one KV head, 64 head_dim columns each; the page id is a coordinate of the copy, so
      // scattered pages cost nothing extra), issued by sixteen lanes at once and landing in the
      // 128-byte-swizzled operand layout the MMA reads. The tokens of the chunk itself come from the
      // step's K/V tensors, sixteen at a time, not from the pages they are appended to; where the
      // chunk starts inside a page the cached rows of that page are laid over the copy by plain
      // loads. (Reading the chunk back from its pages meant that every CTA waited for the whole
      // launch's append: 11 us in front of the first tile on a 2048-token chunk alone, ~30 us next
      // to decode streams. 2048-token chunk alone, 8B shape: 54.3 -> 52.0 us with the step's tensors
      // cold, 52.5 -> 48.6 us repeated. One copy of 128 tokens instead of eight measured the same.)
      // K tiles complete their "full" barrier by transaction bytes. V tiles complete a "landed"
      // barrier first: the warp then clears, in shared memory, the V rows past the unit's last key
      // (they may hold anything, and 0 * NaN would poison O; the same rows of K only produce scores
      // that are masked) and announces the tile. A K tile with cached rows to lay over does the same.
      // The loaders run up to a ring of stages ahead of the tensor pipe.
      const int kv = warp - kWarpLoader0;                      // 0: K, 1: V
      const int stages = kv ? kVStages : kKStages;
      const int lag = stages - 1;                              // V tiles in flight besides the announced one
      const int full = kv ? BAR_V_FULL : BAR_K_FULL, empty = kv ? BAR_V_EMPTY : BAR_K_EMPTY;
      const uint32_t tile0 = base + (kv ? kOffV : kOffK);
      const CUtensorMap* new_map = kv ? &new_maps.v : &new_maps.k;
      int n_touched = 0;                                       // K tiles that went through BAR_K_LANDED
      // The K loader's first thread takes work units off the global queue, one at a time and only
      // when the K loader is ready for it (it runs a few key blocks ahead of the tensor pipe, which
      // hides the round trip), and publishes each to the other roles through a small ring.
      int fetched = 0;
      auto fetch_one = [&]() {
        // a CTA that starts on prefill work has its first unit without asking; the queue hands out the rest
        const int w = next_unit(misc[1] != 0, fetched == 0 && !decode_first, (int)blockIdx.x, n_units,
                                [&]() { return n_prefill_ctas + atomicAdd(s.pf_queue, 1); });
        UnitRec r = {};
        r.w = -1;
        if (w < n_units) {
          const WorkItem it = s.item(w / s.Hkv);
          r.w = w;
          r.table_slot = s.row_slot(it.row);
          r.kv_head = w % s.Hkv;
          r.q_begin = it.q_begin;
          r.q_count = it.q_count;
          r.ctx = it.k_end - it.q_begin - it.q_count;
          r.tok0 = s.row_tok0(it.row);
          if ((unsigned)r.table_slot >= (unsigned)s.max_requests) {
            atomicOr(s.status, TS_DEV_BAD_INDEX);
            r.w = -1;
          }
        }
        const int e = (fetched & (kSchedRing - 1)) * 2;
        ring[e].x = r.w; ring[e].y = r.table_slot; ring[e].z = r.kv_head; ring[e].w = r.q_begin;
        ring[e + 1].x = r.q_count; ring[e + 1].y = r.ctx; ring[e + 1].z = r.tok0; ring[e + 1].w = 0;
        __threadfence_block();
        misc[2] = (uint32_t)++fetched;
      };
      // A first unit that the launch parameters tell is published before the wait: the reads that describe it
      // are a chain, and cold (1.1 us in front of the first copies of 2048 tokens alone).
      const bool first_early = !decode_first && !s.meta;
      if (first_early && kv == 0 && lane == 0) fetch_one();
      ready();
      int g0 = 0;                                              // key blocks of earlier work units
      int n_copied = 0;                                        // tiles whose copies were started: the first n_copied ones
      for (int k = 0;; ++k) {
        if (kv == 0 && lane == 0 && !(first_early && k == 0)) fetch_one();
        __syncwarp();
        PfUnit u;
        if (!get_work(k, u)) break;
        const int32_t* table_row = s.table + (size_t)u.table_slot * s.max_pages_per_req;
        // lane i < 16 copies page i / 2 of the tile, head_dim columns [64 (i % 2), +64): page id of a
        // page that only holds cached tokens (others: not needed)
        auto fetch_page = [&](int j) {
          const int key = j * kBlockKeys + (lane >> 1) * kPageSize;
          int page = s.n_pages;                                // out of range on purpose: the copy delivers zeros
          if (lane < 16 && key < u.k_end && key + kPageSize <= u.ctx) {
            page = table_row[key >> 4];
            if ((unsigned)page >= (unsigned)s.n_pages) {
              atomicOr(s.status, TS_DEV_BAD_PAGE);
              page = s.n_pages;
            }
          }
          return page;
        };
        // does the chunk start inside a page of this tile?
        const int start_tile = (u.ctx & 15) ? u.ctx / kBlockKeys : -1;
        // ... then the page's cached rows are laid over the copy of the new tokens
        auto lay_cached = [&](unsigned char* tile_smem) {
          const int r0 = (u.ctx & ~15) % kBlockKeys, n_rows = u.ctx & 15;
          const int page = table_row[u.ctx >> 4];
          const bool ok = (unsigned)page < (unsigned)s.n_pages;
          if (!ok && lane == 0) atomicOr(s.status, TS_DEV_BAD_PAGE);
          const uint16_t* src = s.pool + (((size_t)(ok ? page : 0) * 2 + kv) * s.Hkv + u.kv_head) * kPageSize * kD;
          for (int i = lane; i < n_rows * 16; i += 32) {
            const int r = i >> 4, c = i & 15;                  // a row is 8 chunks of 16 bytes in each 64-column half
            const uint4 val = ok ? *reinterpret_cast<const uint4*>(src + r * kD + c * 8) : make_uint4(0, 0, 0, 0);
            *reinterpret_cast<uint4*>(tile_smem + (c >> 3) * kHalfBytes + (r0 + r) * 128 + (((c ^ r) & 7) << 4)) = val;
          }
        };
        auto announce = [&](int tile) {                        // V only; tile = block index within the unit
          const int gt = g0 + tile, st = gt % stages;
          wait(BAR_V_LANDED + st, (gt / stages) & 1);
          unsigned char* vt = smem + kOffV + st * kTileBytes;
          const int first_bad = u.k_end - tile * kBlockKeys;   // rows from here on hold no key of the unit
          if (tile == start_tile) lay_cached(vt);
          if (first_bad < kBlockKeys) {
            for (int i = lane; i < (kBlockKeys - first_bad) * 16; i += 32) {
              const int r = first_bad + (i >> 4), c = i & 15;
              *reinterpret_cast<uint4*>(vt + (c >> 3) * kHalfBytes + r * 128 + ((c & 7) << 4)) = make_uint4(0, 0, 0, 0);
            }
          }
          if (tile == start_tile || first_bad < kBlockKeys) fence_proxy_async();
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(full + st));
        };
        int page = fetch_page(0);
        for (int j = 0; j < u.nb; ++j) {
          const int g = g0 + j;
          const int st = g % stages;
          if (kv && j >= lag) announce(j - lag);
          const int page_next = j + 1 < u.nb ? fetch_page(j + 1) : 0;   // the table load flies while this tile is issued
          if (g >= stages) wait(empty + st, ((g / stages) & 1) ^ 1);
          const bool touch = kv == 0 && j == start_tile;
          const uint32_t landed = bar(kv ? BAR_V_LANDED + st : touch ? BAR_K_LANDED : full + st);
          if (__all_sync(0xffffffffu, misc[1] == 0)) {         // after a failure no new copies are started
            n_copied = g + 1;
            if (lane == 0) mbar_expect_tx(landed, kTileBytes);
            __syncwarp();
            const uint32_t dst = tile0 + st * kTileBytes;
            const int first_tok = u.tok0 + j * kBlockKeys - u.ctx;      // token of the tile's first key, if it is a new one
            if (lane < 16) {
              const int key = j * kBlockKeys + (lane >> 1) * kPageSize;
              const uint32_t page_dst = dst + (lane & 1) * kHalfBytes + (lane >> 1) * 2048;
              if (key + kPageSize > u.ctx && key < u.k_end)
                tma_load_3d(page_dst, new_map, landed, (lane & 1) * 64, u.kv_head, first_tok + (lane >> 1) * kPageSize);
              else
                tma_load_5d(page_dst, &kv_tile_map, landed, (lane & 1) * 64, 0, u.kv_head, kv, page);
            }
            if (touch) {
              __syncwarp();
              wait(BAR_K_LANDED, n_touched & 1);
              lay_cached(smem + kOffK + st * kTileBytes);
              fence_proxy_async();
              __syncwarp();
              if (lane == 0) mbar_arrive(bar(full + st));
              ++n_touched;
            }
          }
          page = page_next;
        }
        // the last `lag` V tiles (fewer when the unit is short) have not been announced yet
        if (kv)
          for (int tile = max(0, u.nb - lag); tile < u.nb; ++tile) announce(tile);
        g0 += u.nb;
      }
      if (misc[1]) {
        if (n_touched > 0) mbar_wait(bar(BAR_K_LANDED), (n_touched - 1) & 1, kDrainCycles);
        for (int g = max(0, n_copied - stages); g < n_copied; ++g)
          mbar_wait(bar((kv ? BAR_V_LANDED : full) + g % stages), (g / stages) & 1, kDrainCycles);
      }
    } else {
      // ------------------------------------------------------------------- MMA issuer
      if (warp == kWarpMma) {
        if (s.meta) ready();       // the first unit is published behind the launch in front
        const uint32_t tmem = misc[0];
        const uint32_t issue = elect_one();
        // the warp keeps its own failure flag in a register: nothing on its path reads shared memory
        bool dead = false;
        auto iwait = [&](int i, uint32_t parity) {
          if (!mbar_wait(bar(i), parity, dead ? 2000 : s.wait_cycles)) {
            dead = true;
            give_up();
          }
        };
        constexpr uint32_t idesc_qk = instr_desc(false), idesc_pv = instr_desc(true);
        // descriptors differ only in their start-address field (16-byte units in the low bits)
        const uint64_t q_desc0 = smem_desc(base + kOffQ, 0, 1024);
        const uint64_t k_desc0 = smem_desc(base + kOffK, 0, 1024);
        const uint64_t v_desc0 = smem_desc(base + kOffV, kHalfBytes, 1024);
        auto issue_qk = [&](int x, int stage) {      // S_x = Q_x K^T
          const uint64_t q_desc = q_desc0 + (uint64_t)((x * kTileBytes) >> 4);
          const uint64_t k_desc = k_desc0 + (uint64_t)((stage * kTileBytes) >> 4);
#pragma unroll
          for (int ks = 0; ks < kD / 16; ++ks) {
            const uint64_t off = (uint64_t)(((ks >> 2) * kHalfBytes + (ks & 3) * 32) >> 4);
            mma_ss(tmem + x * 128, q_desc + off, k_desc + off, idesc_qk, ks > 0, issue);
          }
          tc_commit(bar(BAR_S_FULL + x), issue);
        };
        auto issue_pv = [&](int x, int stage, int part, bool first) {   // O_x (+)= P_x V, half of the keys
          const uint64_t v_desc = v_desc0 + (uint64_t)((stage * kTileBytes) >> 4);
#pragma unroll
          for (int kk = 0; kk < kBlockKeys / 16; ++kk) {       // P of keys 0-63 sits in columns 0-31 of S, of keys 64-127 in 64-95
            if (((kk & 3) < kFirst / 16) != (part == 0)) continue;
            mma_ts(tmem + 256 + x * 128, tmem + x * 128 + (kk >> 2) * 64 + (kk & 3) * 8,
                   v_desc + (uint64_t)((kk * 2048) >> 4), idesc_pv, (!first || kk > 0) ? 1u : 0u, issue);
          }
        };
        int ks = 0, vs = 0;          // ring stages of the next K tile to be multiplied and of the next V tile
        uint32_t kph = 0, vph = 0;   // and the parities of their "full" phases
        int sxb[2] = {0, 0};         // blocks per tile in earlier work units (P phases)
        for (int k = 0;; ++k) {
          PfUnit u;
          if (!get_work(k, u)) break;
          // Order: both Q K^T of block 0; then per block, for tile A then tile B: P V of block j and,
          // at once behind it, Q K^T of block j+1 of the same tile, so that the tile's warpgroup gets its
          // next scores while the pipe turns to the other tile. Whatever else the two need (V of block j,
          // K of block j+1) is waited for in front of P: from P to the next scores is the tile's critical
          // path, and this warp shares its scheduler with four softmax warps. P comes in two parts, the first of which
          // is multiplied while the softmax warps take the exponentials of the second. One commit tells of both products,
          // and the warp parks while it waits: the launch runs at the chip's power limit. (Looks at barriers between
          // the products, a commit for each, polling, and arrivals by all lanes of the softmax warps, all together: 8192-token
          // chunk next to 190 rows 1250 us instead of 1237; 2048 tokens alone 45.4 instead of 44.4.)
          // The loaders start behind the launch in front, and the limit is for this launch: if it has run out before the first
          // tiles are there, it runs again from the end of that launch on. (A ready() in front of the loop: 64 rows
          // and 2048 tokens 144.0 us instead of 143.8, 30 rows and 700 tokens 39.5 instead of 39.3.)
          if (k == 0 && !mbar_wait(bar(BAR_Q), 0, s.wait_cycles)) ready();
          iwait(BAR_Q, k & 1);
          iwait(BAR_K_FULL + ks, kph);
          tc_fence_after();
          if (!dead) {
            if (u.nb_a > 0) issue_qk(0, ks);
            if (u.nb_b > 0) issue_qk(1, ks);
            tc_commit(bar(BAR_K_EMPTY + ks), issue);
            if (u.nb == 1) tc_commit(bar(BAR_Q_EMPTY), issue);
          }
          if (++ks == kKStages) { ks = 0; kph ^= 1; }
          for (int j = 0; j < u.nb; ++j) {
            const bool next = j + 1 < u.nb;
            iwait(BAR_V_FULL + vs, vph);
            if (next) iwait(BAR_K_FULL + ks, kph);
#pragma unroll
            for (int x = 0; x < 2; ++x) {
              const int nbx = x ? u.nb_b : u.nb_a;
              if (j >= nbx) continue;
              // P of a unit's first block also says that O is free: the warps that arrive have read the
              // previous unit's O before.
              iwait(BAR_P_FULL + x * 2, (sxb[x] + j) & 1);
              tc_fence_after();
              if (!dead) issue_pv(x, vs, 0, j == 0);
              iwait(BAR_P_FULL + x * 2 + 1, (sxb[x] + j) & 1);
              tc_fence_after();
              if (dead) continue;
              issue_pv(x, vs, 1, j == 0);
              if (j + 1 < nbx) issue_qk(x, ks);
              else tc_commit(bar(BAR_O_FULL + x), issue);
            }
            if (!dead) {                                      // both tiles are done with V(j) and K(j+1)
              tc_commit(bar(BAR_V_EMPTY + vs), issue);
              if (next) tc_commit(bar(BAR_K_EMPTY + ks), issue);
              if (j + 2 == u.nb) tc_commit(bar(BAR_Q_EMPTY), issue);   // that was the unit's last Q K^T
            }
            if (++vs == kVStages) { vs = 0; vph ^= 1; }
            if (next && ++ks == kKStages) { ks = 0; kph ^= 1; }
          }
          sxb[0] += u.nb_a;
          sxb[1] += u.nb_b;
        }
        if (__any_sync(0xffffffffu, misc[1] != 0)) {
          tc_commit(bar(BAR_DRAIN), issue);
          mbar_wait(bar(BAR_DRAIN), 0, kDrainCycles);
        }
      }
      if (warp == kWarpSched) {
        // ------------------------------------------------------------------ Q loader
        // Brings in each work unit's Q tiles by TMA once the previous unit's last Q K^T is done.
        // Between two units it appends, a token at a time, this CTA's share of the new K/V.
        ready();
        AppendCursor app{decode_first || s.append_wide ? append_end : (int)blockIdx.x, append_end, append_warps};
        auto append_until = [&](auto&& ready) {
          while (!app.done() && !__any_sync(0xffffffffu, ready())) app.step<4>(s, 2 * tile_tokens, lane);   // 4: 64 registers here
        };
        int n_loaded = 0;
        for (int k = 0;; ++k) {
          PfUnit u;
          if (k > 0) append_until([&]() { return (int)misc[2] > k; });   // the first Q tiles wait for nothing
          if (!get_work(k, u)) break;
          const int ta = u.tok0 + u.q_begin;
          if (k > 0) {
            append_until([&]() { return mbar_test(bar(BAR_Q_EMPTY), (k - 1) & 1); });
            wait(BAR_Q_EMPTY, (k - 1) & 1);
          }
          if (__any_sync(0xffffffffu, misc[1] != 0)) break;    // after a failure no new copies are started
          n_loaded = k + 1;
          // a box delivers 64 columns of tile_tokens * G packed rows (all 128 only when G divides 128)
          if (lane == 0) {
            mbar_expect_tx(bar(BAR_Q), (u.cnt_b > 0 ? 2 : 1) * 2 * (tile_tokens * G * 128));
            tma_load_4d(base + kOffQ, &q_map, bar(BAR_Q), 0, 0, u.kv_head, ta);
            tma_load_4d(base + kOffQ + kHalfBytes, &q_map, bar(BAR_Q), 64, 0, u.kv_head, ta);
            if (u.cnt_b > 0) {
              tma_load_4d(base + kOffQ + kTileBytes, &q_map, bar(BAR_Q), 0, 0, u.kv_head, ta + tile_tokens);
              tma_load_4d(base + kOffQ + kTileBytes + kHalfBytes, &q_map, bar(BAR_Q), 64, 0, u.kv_head, ta + tile_tokens);
            }
          }
          __syncwarp();
        }
        append_until([]() { return false; });
        if (misc[1] && n_loaded > 0) mbar_wait(bar(BAR_Q), (n_loaded - 1) & 1, kDrainCycles);
      }
      __syncwarp();
    }
  }
  tc_fence_before();
  cta_sync();
  if (warp == kWarpMma) tmem_dealloc(misc[0], 512);
  if (tid == 0) {
    // the last CTA to leave puts the launch's counters back to zero for the next launch
    __threadfence();
    if (atomicAdd(s.pf_queue + 2, 1) == (int)gridDim.x - 1) {
      s.pf_queue[0] = 0;
      s.pf_queue[1] = 0;
      s.pf_queue[2] = 0;
      s.pf_queue[3] = 0;
    }
  }
}

template <int W>
cudaError_t launch_mixed_w(const StepDevice& s, const CUtensorMap& q_map, const CUtensorMap& kv_map,
                           const CUtensorMap& kv_tile_map, const NewKvMaps& new_maps, int n_ctas, int n_prefill_ctas, cudaStream_t stream) {
  if (s.n_prefill_items <= 0 || n_ctas <= 0) return cudaSuccess;
  const int G = s.Hq / s.Hkv;
  size_t smem = kSmemBytes;
  if (n_prefill_ctas < n_ctas) {
    const size_t dec_smem = 1024 + dec::decode_smem_bytes<128, 3>(G);
    if (dec_smem > smem) smem = dec_smem;
  }
  cudaError_t e = cudaFuncSetAttribute(mixed_kernel<W>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  StepParams<W> params;
  fill_params(s, &params);
  return launch_pdl(mixed_kernel<W>, dim3(n_ctas), dim3(kPfThreads), smem, stream, params, q_map, kv_map, kv_tile_map, new_maps, n_prefill_ctas);
}

}  // namespace

cudaError_t launch_mixed(const StepDevice& s, const CUtensorMap& q_map, const CUtensorMap& kv_map,
                         const CUtensorMap& kv_tile_map, const NewKvMaps& new_maps, int n_ctas, int n_prefill_ctas, cudaStream_t stream) {
  const auto launch = s.n_words <= kInlineWords      ? launch_mixed_w<kInlineWords>
                      : s.n_words <= kInlineWordsMid ? launch_mixed_w<kInlineWordsMid>
                                                     : launch_mixed_w<kInlineWordsMax>;
  return launch(s, q_map, kv_map, kv_tile_map, new_maps, n_ctas, n_prefill_ctas, stream);
}

}  // namespace ts
