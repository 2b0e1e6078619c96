// Work units of the prefill tiles as the roles of a CTA of the mixed kernel hand them on: plain C++, so
// that the rules the roles agree by can be run on the host as well.
#pragma once
#include <stdint.h>

#ifdef __CUDACC__
#define TS_HOST_DEVICE __host__ __device__ __forceinline__
#else
#define TS_HOST_DEVICE inline
#endif

namespace ts {

constexpr int kBlockKeys = 128;            // keys of a block of the tile path
// Published units that are kept: entry k % kSchedRing holds unit k of the CTA.
constexpr int kSchedRing = 8;

// One prefill work unit as the K loader publishes it in shared memory (8 words), and the shape
// every role derives from it.
struct UnitRec {
  int32_t w;                 // work unit index, -1 = there are no more
  int32_t table_slot;        // request slot: row of the block table
  int32_t kv_head, q_begin, q_count;
  int32_t ctx;               // tokens cached before the chunk
  int32_t tok0;              // first token of the request row in the step's tensors
  int32_t pad;
};
static_assert(sizeof(UnitRec) == 32, "UnitRec is 8 words");
struct PfUnit {
  int table_slot, kv_head, q_begin, ctx, tok0;
  int cnt_a, cnt_b;          // tokens of tile A / tile B (tile B may be empty)
  int k_end_a, k_end_b;      // one past the last key any row of the tile may see
  int nb_a, nb_b, nb;        // key blocks per tile, and of the unit
  int k_end;
};
TS_HOST_DEVICE PfUnit unit_shape(const UnitRec& r, int tile_tokens) {
  PfUnit u;
  u.table_slot = r.table_slot;
  u.kv_head = r.kv_head;
  u.q_begin = r.q_begin;
  u.ctx = r.ctx;
  u.tok0 = r.tok0;
  u.cnt_a = r.q_count < tile_tokens ? r.q_count : tile_tokens;
  u.cnt_b = r.q_count - u.cnt_a;
  u.k_end_a = u.ctx + r.q_begin + u.cnt_a;
  u.k_end_b = u.k_end_a + u.cnt_b;
  u.nb_a = (u.k_end_a + kBlockKeys - 1) / kBlockKeys;
  u.nb_b = u.cnt_b > 0 ? (u.k_end_b + kBlockKeys - 1) / kBlockKeys : 0;
  u.nb = u.nb_a > u.nb_b ? u.nb_a : u.nb_b;
  u.k_end = u.k_end_a > u.k_end_b ? u.k_end_a : u.k_end_b;
  return u;
}

// The unit the K loader publishes next; n_units or more: the end of the list. After a failure (a wait of
// the CTA has run out, the others end early) it is the end at once: with nothing to hold the K loader
// back, further units would overwrite entries that are still read.
template <typename Take>
TS_HOST_DEVICE int next_unit(bool failed, bool first_is_known, int first, int n_units, Take&& take) {
  return failed ? n_units : first_is_known ? first : take();
}
// What the first warp of a pair posts for both: the blocks that tile `x` has in the unit, -1: leave. The
// two warps of a pair meet on a barrier without a time limit, once per block and a fixed number of
// times per unit, so both must go by this one number, whatever either of them reads from the ring.
TS_HOST_DEVICE int posted_blocks(bool have, const PfUnit& u, int x) { return !have ? -1 : x ? u.nb_b : u.nb_a; }

}  // namespace ts
