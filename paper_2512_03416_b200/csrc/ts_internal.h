// Internal interface between the host scheduler (ts_host.cpp) and the kernels (ts_kernels.cu).
// Nothing here is part of the public ABI.
#pragma once
#include <cuda.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include "../../include/tokenscale.h"

#include <cstddef>
#include <cstring>
#include <utility>

namespace ts {

constexpr int kPageSize = 16;
constexpr int kKeysPerTile = 64;     // keys staged per pipeline stage of the attention kernel
constexpr int kPackedRowsPerTile = 64;  // (token, head) rows of a prefill tile, head_dim 64 path
constexpr int kPackedRowsTc = 128;      // (token, head) rows of a prefill tile, tcgen05 path (head_dim 128)
constexpr long long kWaitCycles = 2000000000LL;  // default limit of a bounded wait: about one second at boost clock
constexpr int kMaxGroup = 16;        // query heads per KV head a decode work item can hold

// One unit of attention work; the KV head comes from the grid.
// Inside a kernel the (token, head-in-group) pairs of an item are "packed rows":
//   packed row pr -> token q_begin + pr / G, query head kv_head*G + pr % G.
struct WorkItem {
  int32_t row;          // index into the step's rows
  int32_t kind;         // 0: decode split, 1: prefill tile
  int32_t q_begin;      // first new token of the row this item covers (decode: 0)
  int32_t q_count;      // tokens in this item (decode: 1; prefill: tile_rows / G at most)
  int32_t k_begin;      // first key position (multiple of kKeysPerTile)
  int32_t k_end;        // one past the last key position any row of the item may see
  int32_t partial_slot; // >= 0: write (m, l, acc) partials there; -1: write out directly
  int32_t combine;      // of a partial_slot >= 0, as the kernels get it: index of the token's CombineItem
};
static_assert(sizeof(WorkItem) == 32, "WorkItem is 8 int32");

// One entry per token whose splits must be merged.
struct CombineItem {
  int32_t token;         // flat token index of the step
  int32_t first_partial; // first partial slot
  int32_t n_splits;
  int32_t reserved;
};

struct TableDelta {
  int32_t slot, index, page;
};

// Words of row arrays and work list that travel as launch parameters. Every kernel takes up to kInlineWords (3 KB: with
// its other parameters that stays within 4 KB), the mixed kernel and the decode kernel of head_dim 128 with up to eight
// heads per KV head are there for larger steps as well (parameters end at 32764 bytes). A launch with 3 KB of
// parameters costs the host 2.4 us, with 8 KB 2.7, 16 KB 3.7, 30 KB 5 to 11; an upload on the copy stream, its event and the
// wait for it 4.8 with the launch. The wait also ends the overlap with the launch in front: next to a 2048-token chunk a
// step's first thread blocks started 5.7 us after the last one of the step before had left, 1.7 without.
constexpr int kInlineWords = 768, kInlineWordsMid = 3072, kInlineWordsMax = 7680;
// One step as its kernels see it; device pointers lie in the caller's workspace unless noted.
struct StepDevice {
  // static
  uint16_t* pool;          // caller's KV pool
  int32_t* table;          // [max_requests][max_pages_per_req]
  int32_t* status;         // device status word
  int32_t* pf_queue;       // counters, all zero between launches (the last CTA to leave resets them):
                           // mixed kernel [0] next prefill work unit, [1] decode CTAs that have finished
                           // their units, [2] CTAs that have left; [3] decode units taken besides the
                           // CTAs' first ones; decode kernel [4] CTAs that are done
  int32_t* merge_count;    // [n_combines][Hkv] splits of a token that the decode kernel has finished, zero between launches
  int32_t merge_here;      // the decode kernel merges the rows it split itself (see count_split)
  float* part_acc;         // [max_partials][Hq][D]
  float* part_ml;          // [max_partials][Hq][2]  (running max in log2 units, sum)
  // step tensors
  const uint16_t* q;
  const uint16_t* k_new;
  const uint16_t* v_new;
  uint16_t* out;
  // shape
  int32_t n_rows, n_tokens, n_items, n_combines;
  int32_t n_prefill_items;  // items[0, n_prefill_items) are prefill tiles, the rest decode splits
  int32_t Hq, Hkv, D, n_pages, max_pages_per_req, max_requests;
  float scale_log2;        // softmax scale * log2(e)
  long long wait_cycles;   // limit of every bounded wait of the step's kernels, in clock cycles, but for those
                           // that may span the pages of a whole decode unit:
  long long unit_wait_cycles;
  int32_t append_wide;     // mixed kernel: CTAs that start on prefill units append with their softmax warps first
  int32_t debug_arrivals;  // decode CTAs besides the launch's own that the mixed kernel's merge waits for (TS_DEBUG_LOSE_APPEND_ARRIVAL)
  // The step's row arrays and work list: word offsets from `meta`, a device address, or, unless they
  // are large, from the words behind this struct in the launch parameters (StepParams): no upload of their own (a copy
  // on another stream, two event records and two waits: ~6 us of host time and a dependency per step).
  const int32_t* meta;     // null: the words behind this struct
  // Whether a launch behind the step's first reading one may read them before it waits for the launch in front: they are
  // launch parameters, or the stream waited for their upload before the first launch that reads them. Not where a kernel plans the step.
  int32_t meta_in_place;
  uint32_t o_slot, o_ctx, o_tok0, o_items, o_combines;
  int32_t n_words;             // for the launchers: words in host memory that travel with the launch (none where meta is set)
  const int32_t* host_words;
#ifdef __CUDACC__
  __device__ __forceinline__ const int32_t* at(uint32_t o) const { return (meta ? meta : reinterpret_cast<const int32_t*>(this + 1)) + o; }
  __device__ __forceinline__ int32_t row_slot(int r) const { return at(o_slot)[r]; }
  __device__ __forceinline__ int32_t row_ctx(int r) const { return at(o_ctx)[r]; }
  __device__ __forceinline__ int32_t row_tok0(int r) const { return at(o_tok0)[r]; }   // [n_rows + 1] prefix sums of the new tokens
  __device__ __forceinline__ WorkItem item(int i) const { return reinterpret_cast<const WorkItem*>(at(o_items))[i]; }
  __device__ __forceinline__ CombineItem combine(int i) const { return reinterpret_cast<const CombineItem*>(at(o_combines))[i]; }
#endif
};

// A step as a launch parameter.
template <int W>
struct StepParams {
  StepDevice s;
  int32_t words[W];
};
static_assert(offsetof(StepParams<kInlineWords>, words) == sizeof(StepDevice), "the words follow the step");
template <int W>
inline void fill_params(const StepDevice& s, StepParams<W>* p) {
  p->s = s;
  if (s.n_words > 0) std::memcpy(p->words, s.host_words, sizeof(int32_t) * (size_t)s.n_words);
}

// Launchers. Each enqueues on `stream` and returns the launch's cudaError_t.
cudaError_t launch_table_update(int32_t* table, int max_pages_per_req, int max_requests, int32_t* status,
                                const TableDelta* deltas, int n_deltas, cudaStream_t stream);
// The same for up to kInlineDeltas entries, which travel as launch parameters.
constexpr int kInlineDeltas = 64;
struct InlineDeltas {
  int32_t n;
  TableDelta d[kInlineDeltas];
};
cudaError_t launch_table_update(int32_t* table, int max_pages_per_req, int max_requests, int32_t* status,
                                const InlineDeltas& deltas, cudaStream_t stream);
cudaError_t launch_kv_append(const StepDevice& s, cudaStream_t stream);
// Work items [0, n_items); prefill items read their chunk's own K/V from the step's tensors and append them.
cudaError_t launch_attention(const StepDevice& s, cudaStream_t stream);
// Prefill items and decode splits of a head_dim 64 step in one launch, a block per (item, KV head): for steps that have
// both and no more of these than the device has SMs. Split rows are left to launch_combine.
cudaError_t launch_small_step(const StepDevice& s, const CUtensorMap& kv_map, cudaStream_t stream);
// Merges the splits that launch_attention left, or launch_decode without merge_here (launch_mixed merges its own).
cudaError_t launch_combine(const StepDevice& s, cudaStream_t stream);
// Decode splits items[n_prefill_items, n_items): persistent kernel, one CTA per SM, K/V pages by TMA
// through kv_map (5-D view of the pool: 64 columns, KV head x slot, half, K|V, page; box = one page of one head).
// Prefill tiles items[0, n_prefill_items), head_dim 128: persistent tcgen05/TMEM kernel of n_ctas
// CTAs. The first n_prefill_ctas CTAs work on the prefill queue only; the others first run all
// decode splits (as launch_decode would, needs G <= 8) and then join the prefill queue. The
// kernel also appends the step's new K/V itself (no launch_kv_append before it). With
// n_prefill_ctas == n_ctas the decode splits are left to launch_decode. When it runs the decode
// splits it also merges them (no launch_combine needed).
// q_map views q as (head_dim, G, KV head, token), box 64 x G x 1 x 128/G. kv_tile_map views
// the pool as (head_dim, slot, KV head, K|V, page), box 64 x 16 x 1 x 1 x 1: the prefill tiles' copies of
// cached K/V; new_maps view the step's own K/V.
struct NewKvMaps {          // k_new / v_new as (head_dim, KV head, token), box 64 x 1 x 16
  CUtensorMap k, v;
};
cudaError_t launch_mixed(const StepDevice& s, const CUtensorMap& q_map, const CUtensorMap& kv_map,
                         const CUtensorMap& kv_tile_map, const NewKvMaps& new_maps, int n_ctas, int n_prefill_ctas, cudaStream_t stream);
cudaError_t launch_decode(const StepDevice& s, const CUtensorMap& kv_map, int n_sms, cudaStream_t stream);

// ---- the decoder layer around the attention step: GEMMs and small kernels (ts_gemm.cu, ts_layer_kernels.cu)
enum { GEMM_EPI_STORE = 0, GEMM_EPI_ROPE = 1, GEMM_EPI_SILU_MUL = 2 };
// C = A . B^T (+ R), A [M][K], B [N][K] bf16 K-major (their tensor maps travel beside this struct).
struct GemmArgs {
  int32_t M, N, K;
  int32_t epi;              // GEMM_EPI_*
  const uint16_t* B;        // the weights themselves (prefetches)
  uint16_t* C;              // STORE: [M][ldc]; ROPE: the query heads [M][q_cols]; SILU_MUL: [M][ldc], ldc = N / 2
  const uint16_t* R;        // STORE: residual [M][ldc] added before rounding, or null
  int32_t ldc;
  // ROPE (fused QKV projection, head_dim 128): columns [0, q_cols) are query heads -> C, the next
  // kv_cols key heads -> C2, the last kv_cols value heads -> C3 (not rotated)
  int32_t q_cols, kv_cols;
  uint16_t* C2;
  uint16_t* C3;
  const int32_t* pos;       // [M] position of every token
  const float2* rope_table; // [max_position][64] (cos, sin) of pos * theta^(-2i/128)
  int32_t* status;          // device status word
  long long wait_cycles;    // limit of every bounded wait
};
// What the layer code needs to know of a context (ts_host.cpp fills it in; it also makes sure the
// context's CUDA set-up has run and its status word is cleared).
struct CtxView {
  const ts_config* cfg;
  int n_sms;
  void* encode_fn;          // cuTensorMapEncodeTiled
  int32_t* status;          // device status word of the context
  long long wait_cycles;
  int max_tokens;           // most tokens a step may hold
};
int ctx_view(ts_ctx* c, cudaStream_t stream, CtxView* out);
// How a product is laid over the chip. split = 0: 128 x 256 tiles, one CTA each, or (tile_m = 256)
// tiles of pair_tokens tokens x 256 features, a pair of CTAs each; split > 0: 128 x 128 tiles whose K range a
// cluster of `split` CTAs shares.
struct GemmPlan {
  int tile_m, split, pair_tokens;
};
// Smallest number of tokens, a multiple of 16, with which `tiles` tiles hold M tokens.
inline int pair_tokens(int M, int tiles) { return ((M + tiles - 1) / tiles + 15) / 16 * 16; }
// The plan for a product (M, N, K and epi are read). The device is the current one.
GemmPlan gemm_plan(const GemmArgs& g, int n_sms);
// Views of the operands as (K, row). x, w: boxes of 64 x 128. The pair kernel's: x_pair, a box of 64 x
// pair_tokens / 2; w_pair, for STORE the same as w, else boxes of 64 x 128 whose rows come in the order the epilogue
// pairs them in (make_paired_map). Those that the plan does not use may be null.
struct GemmMaps {
  const CUtensorMap *x, *x_pair, *w, *w_pair;
};
cudaError_t launch_gemm(const GemmArgs& g, const GemmMaps& maps, GemmPlan plan, int n_sms, cudaStream_t stream);
// out[row] = x[row] / sqrt(mean(x[row]^2) + eps) * gain, bf16 in and out, fp32 inside; width % 8 == 0
cudaError_t launch_rmsnorm(const uint16_t* x, const uint16_t* gain, uint16_t* out, int rows, int width, float eps,
                           cudaStream_t stream);
// The same, and pos[t] = position of token t: row r holds tokens tok0[r] .. tok0[r + 1] - 1 at positions
// from ctx[r] on.
constexpr int kPosRows = 400;           // 3.2 KB of launch parameters
template <bool POS>
struct PosRows {};
template <>
struct PosRows<true> {
  int32_t* pos;
  int32_t n_rows;
  int32_t tok0[kPosRows], ctx[kPosRows];
};
cudaError_t launch_rmsnorm_pos(const uint16_t* x, const uint16_t* gain, uint16_t* out, int rows, int width, float eps,
                               const PosRows<true>& pos, cudaStream_t stream);
// table[p][i] = (cos, sin)(p * theta^(-2 i / 128)), p < max_position, i < 64 (computed in fp64)
cudaError_t launch_rope_table(float2* table, int max_position, float theta, cudaStream_t stream);
// dst row 256 b + r = gate row 128 b + r, dst row 256 b + 128 + r = up row 128 b + r (r < 128)
cudaError_t launch_pack_gate_up(const uint16_t* gate, const uint16_t* up, uint16_t* dst, int intermediate, int width,
                                cudaStream_t stream);

// Programmatic dependent launch: every kernel of a step is launched with the attribute that lets
// it become resident while its predecessor in the stream is still draining. Each kernel runs its
// set-up (shared-memory barriers, TMEM allocation, descriptor prefetch), then executes
// griddepcontrol.wait before it touches anything an earlier kernel may have written or may still
// be reading; launch latency and set-up thus overlap the predecessor's tail.
template <typename... Params, typename... Args>
inline cudaError_t launch_pdl(void (*kernel)(Params...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                              Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}
#ifdef __CUDACC__
// Copies the K/V of the step's new tokens into their pages (Sec. 2.1): one warp per token at a time,
// warps `first_warp`, `first_warp + n_warps`, ... of the launch; a lane moves 16-byte chunks, eight
// loads in flight before the first store, and the source loads are issued before the block-table
// look-up they do not depend on. `rows` = a shared-memory copy of the step's row arrays made by
// stage_rows (the token -> row search and the row's slot and length then cost no global round trips).
// Slots and page ids are range checked; a bad one sets a status bit and skips the token.
__device__ __forceinline__ void stage_rows(const StepDevice& s, int32_t* rows, int tid, int n_threads) {
  const int n = s.n_rows + 1;                  // rows[0..n): first-token prefix sums, then ctx, then slot
  for (int i = tid; i < n; i += n_threads) {
    rows[i] = s.row_tok0(i);
    if (i < s.n_rows) {
      rows[n + i] = s.row_ctx(i);
      rows[2 * n + i] = s.row_slot(i);
    }
  }
}
__host__ __device__ inline size_t staged_rows_bytes(int n_rows) { return (size_t)3 * (n_rows + 1) * sizeof(int32_t); }
// One token: its K and V for all KV heads go to position t of the request in table row `slot`.
__device__ __forceinline__ void append_one(const StepDevice& s, int tok, int t, int slot, int lane) {
  const int cpr = s.D / 8;                      // chunks per (token, head) row
  const int per_tok = 2 * s.Hkv * cpr;
  const bool index_ok = (unsigned)slot < (unsigned)s.max_requests && (unsigned)(t >> 4) < (unsigned)s.max_pages_per_req;
  int page = -1;
  for (int base = 0; base < per_tok; base += 256) {
    uint4 v[8];
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int c = base + u * 32 + lane;
      if (c < per_tok) {
        const int kv = c / (s.Hkv * cpr);
        const int rem = c - kv * s.Hkv * cpr;
        const int head = rem / cpr, ch = rem % cpr;
        v[u] = *reinterpret_cast<const uint4*>((kv ? s.v_new : s.k_new) + ((size_t)tok * s.Hkv + head) * s.D + ch * 8);
      }
    }
    if (base == 0) {
      if (!index_ok) {
        if (lane == 0) atomicOr(s.status, TS_DEV_BAD_INDEX);
        break;
      }
      page = s.table[(size_t)slot * s.max_pages_per_req + (t >> 4)];
      if ((unsigned)page >= (unsigned)s.n_pages) {
        if (lane == 0) atomicOr(s.status, TS_DEV_BAD_PAGE);
        break;
      }
    }
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      const int c = base + u * 32 + lane;
      if (c < per_tok) {
        const int kv = c / (s.Hkv * cpr);
        const int rem = c - kv * s.Hkv * cpr;
        const int head = rem / cpr, ch = rem % cpr;
        uint16_t* dst = s.pool + ((((size_t)page * 2 + kv) * s.Hkv + head) * kPageSize + (t & 15)) * s.D + ch * 8;
        *reinterpret_cast<uint4*>(dst) = v[u];
      }
    }
  }
}
__device__ __forceinline__ void append_tokens(const StepDevice& s, const int32_t* rows, int first_warp, int n_warps,
                                              int lane) {
  const int n = s.n_rows + 1;
  const int32_t* row_start = rows;
  for (int tok = first_warp; tok < s.n_tokens; tok += n_warps) {
    int lo = 0, hi = s.n_rows;                  // row of this token: last r with row_start[r] <= tok
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (row_start[mid] <= tok) lo = mid; else hi = mid;
    }
    append_one(s, tok, rows[n + lo] + (tok - row_start[lo]), rows[2 * n + lo], lane);
  }
}
// Log-sum-exp merge of the splits of one (token, head),
//   m = max m_i,  l = sum l_i 2^(m_i - m),  O = sum acc_i 2^(m_i - m) / l,
// in groups of eight: one group added to the running (m, l, acc) of E head_dim elements. The groups and each rounding are
// the same for whoever merges (the combine launch, or inside the decode launch whichever warps come last), so that a row's
// result does not depend on the timing of its splits. Splits that are not there have m_i = -inf, l_i = acc_i = 0.
constexpr int kMergeGroup = 8;
template <int E>
__device__ __forceinline__ void merge_group(float& m, float& l, float (&acc)[E], const float (&mi)[kMergeGroup],
                                            const float (&li)[kMergeGroup], const float (&ai)[kMergeGroup][E]) {
  float mn = m;
#pragma unroll
  for (int j = 0; j < kMergeGroup; ++j) mn = fmaxf(mn, mi[j]);
  const float keep = exp2f(m - mn);            // 0 on the first group (m = -inf)
#pragma unroll
  for (int j = 0; j < kMergeGroup; ++j) {
    const float w = exp2f(mi[j] - mn);         // absent split: exp2(-inf) = 0
    l = j == 0 ? __fmaf_rn(l, keep, __fmul_rn(w, li[j])) : __fmaf_rn(w, li[j], l);
#pragma unroll
    for (int e = 0; e < E; ++e) acc[e] = j == 0 ? __fmaf_rn(acc[e], keep, __fmul_rn(w, ai[j][e])) : __fmaf_rn(w, ai[j][e], acc[e]);
  }
  m = mn;
}
// The merge for head_dim element d over the partial slots [first_partial, first_partial + n_splits). A group's
// loads are in flight at a time. Reads bypass L1 (another SM wrote the partials).
__device__ __forceinline__ float merge_splits(const StepDevice& s, int first_partial, int n_splits, int h, int d) {
  const float* ml = s.part_ml + ((size_t)first_partial * s.Hq + h) * 2;
  const float* pa = s.part_acc + ((size_t)first_partial * s.Hq + h) * s.D + d;
  const size_t ml_stride = (size_t)s.Hq * 2, pa_stride = (size_t)s.Hq * s.D;
  float m = -__int_as_float(0x7f800000), l = 0.f, acc[1] = {0.f};
  for (int base = 0; base < n_splits; base += kMergeGroup) {
    float mi[kMergeGroup], li[kMergeGroup], ai[kMergeGroup][1];
#pragma unroll
    for (int j = 0; j < kMergeGroup; ++j) {
      const bool on = base + j < n_splits;
      mi[j] = on ? __ldcg(ml + (base + j) * ml_stride) : -__int_as_float(0x7f800000);
      li[j] = on ? __ldcg(ml + (base + j) * ml_stride + 1) : 0.f;
      ai[j][0] = on ? __ldcg(pa + (base + j) * pa_stride) : 0.f;
    }
    merge_group<1>(m, l, acc, mi, li, ai);
  }
  return acc[0] / l;
}
__device__ __forceinline__ void pdl_launch_dependents() { asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory"); }
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;\n" ::: "memory"); }
#endif

}  // namespace ts
