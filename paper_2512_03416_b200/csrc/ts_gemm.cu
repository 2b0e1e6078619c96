// bf16 GEMM of the decoder layer around the attention step (sm_100a): C = A . B^T with fp32
// accumulation on the 5th-generation tensor cores.
//
//   A [M][K] bf16 (activations, one token per row), B [N][K] bf16 (weights, [out features][in
//   features]), C [M][N] bf16. Both operands are K-major, exactly as they sit in memory.
//
// Three kernels, chosen by gemm_plan from the shape:
//   gemm_kernel        one persistent CTA per SM walks 128 x 256 tiles (one tcgen05.mma M = 128, N = 256
//                      per 16 of K); two 256-column accumulators in TMEM alternate between tiles, so a
//                      tile's epilogue overlaps the next tile's main loop;
//   gemm_pair_kernel   many rows: a pair of CTAs (cta_group::2) walks tiles of 256 features x 16 to 256 tokens,
//                      each CTA fetches and holds half of both operand blocks; two accumulators as above;
//   gemm_split_kernel  few tiles: a cluster of 2 to 8 CTAs shares the K range of one 128 x 128 tile and adds
//                      its fp32 accumulators up through distributed shared memory.
// Tile index t -> column block t / m_tiles, row block t % m_tiles, so the CTAs that run at the same time
// share a few weight blocks through L2. Operands arrive by TMA in 64-wide K blocks (128-byte swizzle)
// through a ring of stages.
// Warp roles: warp 0 TMA producer, warp 1 MMA issuer and TMEM owner, warps 2-9 epilogue (thread = half an
// accumulator row: TMEM -> registers -> bf16 -> global; in the split kernel all warps add up and write).
// Epilogues: plain store, store + residual (C = R + A . B^T), rotary embedding of the query and key
// heads of a fused QKV projection, and SiLU-gated product of a fused gate/up projection.
// Every wait is bounded; a wait that runs out raises TS_DEV_TIMEOUT and the CTA drains.
#include <cuda_bf16.h>

#include <algorithm>
#include <atomic>

#include "../../include/tokenscale.h"
#include "ts_internal.h"
#include "ts_ptx.h"
#include "ts_tc.h"
#include "ts_tma.h"

namespace ts {
namespace {

constexpr int kGemmThreads = 320;               // producer warp, MMA warp, eight epilogue warps
constexpr int kBN = 256, kBK = 64;
constexpr int kTileStages = 4;                  // of gemm_kernel
constexpr int kMaxSplit = 8;                    // portable cluster size
constexpr int kABytes = 128 * kBK * 2;          // one 128-row operand block: 16 KB
constexpr int kBBytes = kBN * kBK * 2;          // the 256-row weight block: 32 KB

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
// Asks for `bytes` bytes of weight row `row`, from byte `at` on, in L2. The weights do not come from the
// kernel in front of this one, so a launch asks for the first part of what it will read before it waits
// for that kernel: HBM then works while the chip drains and refills, and it is asked for runs of
// kilobytes instead of the 128-byte pieces of a K block.
constexpr int kPrefetchBytes = 512;             // about what the stages hold; 2 KB or more per row got in the way of the copies themselves
__device__ __forceinline__ void prefetch_weights(const GemmArgs& g, int row, int k0, int k1) {
  if (row >= g.N) return;
  const int bytes = min(kPrefetchBytes, (min(k1, g.K) - k0) * 2);
  const uint16_t* src = g.B + (size_t)row * g.K + k0;
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(src), "r"(bytes) : "memory");
}
// bf16 x bf16 -> fp32, M = 128, N = 256, both operands K-major
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 3) << 17) | ((128u >> 4) << 24);

// After a time-out a role starts nothing any more, but the copies and MMAs of the last K blocks may still be
// under way. They are done within microseconds; the thread that calls this gives them a millisecond before
// its CTA leaves and gives shared memory and TMEM back.
__device__ __forceinline__ void settle(bool failed) {
  if (!failed) return;
  const long long t0 = clock64();
  while (clock64() - t0 < 2000000) {}
}

__device__ __forceinline__ uint4 pack8(const float* v) {
  uint4 w;
  w.x = pack_bf16(v[0], v[1]);
  w.y = pack_bf16(v[2], v[3]);
  w.z = pack_bf16(v[4], v[5]);
  w.w = pack_bf16(v[6], v[7]);
  return w;
}
__device__ __forceinline__ void unpack8(const uint4& w, float* v) {
  const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(u[i] << 16);
    v[2 * i + 1] = __uint_as_float(u[i] & 0xFFFF0000u);
  }
}

// Eight columns c .. c + 7 of a 128-column head that starts at column col0 of the fused projection,
// and their partners 64 further on: rotated by cs (query and key heads) and written to the head's tensor.
__device__ __forceinline__ void rope8(const GemmArgs& g, int row, int col0, int c, float (&lo)[8], float (&hi)[8], const float4 (&cs)[4]) {
  const bool rotate = col0 < g.q_cols + g.kv_cols;
  uint16_t* dst = col0 < g.q_cols ? g.C + (size_t)row * g.q_cols + col0
                  : rotate        ? g.C2 + (size_t)row * g.kv_cols + (col0 - g.q_cols)
                                  : g.C3 + (size_t)row * g.kv_cols + (col0 - g.q_cols - g.kv_cols);
  if (rotate) {
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float co = e & 1 ? cs[e / 2].z : cs[e / 2].x, si = e & 1 ? cs[e / 2].w : cs[e / 2].y;
      const float a = lo[e], b = hi[e];
      lo[e] = a * co - b * si;
      hi[e] = b * co + a * si;
    }
  }
  *reinterpret_cast<uint4*>(dst + c) = pack8(lo);
  *reinterpret_cast<uint4*>(dst + 64 + c) = pack8(hi);
}
// silu(gate) * up = gate / silu_den(gate) * up, of values rounded to bf16 first (they are bf16 tensors of the layer's
// definition)
__device__ __forceinline__ float silu_den(float gate) { return 1.f + __expf(-gate); }
__device__ __forceinline__ void silu_mul8(float* gate, const float* up) {
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const float a = __bfloat162float(__float2bfloat16_rn(gate[e])), b = __bfloat162float(__float2bfloat16_rn(up[e]));
    gate[e] = a / silu_den(a) * b;
  }
}

// Epilogue of one accumulator (TMEM lanes = 128 rows, 256 columns): half `hf` of this thread's row of
// the tile whose columns start at n0 (two warps share a quarter of the lanes; the epilogue of a
// launch's last tiles is not hidden behind anything). `release` is called once that half is in registers.
template <int EPI, typename Release>
__device__ __forceinline__ void epilogue_row(const GemmArgs& g, uint32_t tacc, int row, int n0, int hf, Release&& release) {
  const bool row_ok = row < g.M;
  if (EPI == GEMM_EPI_STORE) {
    uint16_t* crow = g.C + (size_t)row * g.ldc + n0;
    const uint16_t* rrow = g.R ? g.R + (size_t)row * g.ldc + n0 : nullptr;
#pragma unroll 1
    for (int c = hf * 4; c < hf * 4 + 4; ++c) {
      float v[32];
      uint4 r[4];
      const bool with_r = rrow && row_ok;
#pragma unroll
      for (int i = 0; i < 4; ++i)                          // the residual's loads fly while TMEM is read
        if (with_r && n0 + c * 32 + i * 8 < g.N) r[i] = *reinterpret_cast<const uint4*>(rrow + c * 32 + i * 8);
      tmem_ld32(v, tacc + c * 32);
      tmem_ld_wait();
      if (c == hf * 4 + 3) release();
      if (row_ok) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          if (n0 + c * 32 + i * 8 < g.N) {
            if (with_r) {
              float x[8];
              unpack8(r[i], x);
#pragma unroll
              for (int e = 0; e < 8; ++e) v[i * 8 + e] += x[e];
            }
            *reinterpret_cast<uint4*>(crow + c * 32 + i * 8) = pack8(v + i * 8);
          }
        }
      }
    }
  } else if (EPI == GEMM_EPI_ROPE) {
    // A tile holds two heads of 128 columns. Query and key heads are rotated: column i < 64 of a
    // head pairs with column i + 64, angle table[pos][i]. Each head goes to its own tensor.
    const float2* cs = g.rope_table + (size_t)(row_ok ? g.pos[row] : 0) * 64;
    const int col0 = n0 + hf * 128;
    const bool rotate = col0 < g.q_cols + g.kv_cols;
    uint16_t* dst = col0 < g.q_cols ? g.C + (size_t)row * g.q_cols + col0
                    : rotate        ? g.C2 + (size_t)row * g.kv_cols + (col0 - g.q_cols)
                                    : g.C3 + (size_t)row * g.kv_cols + (col0 - g.q_cols - g.kv_cols);
#pragma unroll 1
    for (int c = 0; c < 2; ++c) {
      float lo[32], hi[32];
      float2 t2[32];                                      // (cos, sin); the loads fly while TMEM is read
      if (rotate) {
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const float4 w = *reinterpret_cast<const float4*>(cs + c * 32 + i);
          t2[i] = make_float2(w.x, w.y);
          t2[i + 1] = make_float2(w.z, w.w);
        }
      }
      tmem_ld32(lo, tacc + hf * 128 + c * 32);
      tmem_ld32(hi, tacc + hf * 128 + 64 + c * 32);
      tmem_ld_wait();
      if (c == 1) release();
      if (row_ok && col0 < g.N) {
        if (rotate) {
#pragma unroll
          for (int i = 0; i < 32; ++i) {
            const float a = lo[i], b = hi[i];
            lo[i] = a * t2[i].x - b * t2[i].y;
            hi[i] = b * t2[i].x + a * t2[i].y;
          }
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          *reinterpret_cast<uint4*>(dst + c * 32 + i * 8) = pack8(lo + i * 8);
          *reinterpret_cast<uint4*>(dst + 64 + c * 32 + i * 8) = pack8(hi + i * 8);
        }
      }
    }
  } else {
    // GEMM_EPI_SILU_MUL: the weight rows of a tile are 128 gate rows followed by the 128 up rows of
    // the same intermediate features; out[row][n0 / 2 + i] = silu(gate_i) * up_i.
    uint16_t* crow = g.C + (size_t)row * g.ldc + n0 / 2;
#pragma unroll 1
    for (int c = hf * 2; c < hf * 2 + 2; ++c) {
      float gt[32], up[32];
      tmem_ld32(gt, tacc + c * 32);
      tmem_ld32(up, tacc + 128 + c * 32);
      tmem_ld_wait();
      if (c == hf * 2 + 1) release();
      if (row_ok && n0 < g.N) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          silu_mul8(gt + i * 8, up + i * 8);
          *reinterpret_cast<uint4*>(crow + c * 32 + i * 8) = pack8(gt + i * 8);
        }
      }
    }
  }
}

// One CTA per 128 x 256 tile, persistent; the two accumulators alternate between tiles.
template <int EPI>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_kernel(const GemmArgs g, const __grid_constant__ CUtensorMap a_map, const __grid_constant__ CUtensorMap b_map) {
  constexpr int kStages = kTileStages, kStageBytes = kABytes + kBBytes;
  constexpr int kOffBar = kStages * kStageBytes;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - smem_u32(smem_raw));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  pdl_launch_dependents();
  // barriers: full[kStages], empty[kStages], acc_full[2], acc_empty[2]
  auto bar = [&](int i) { return base + kOffBar + (uint32_t)i * 8u; };
  const int BAR_FULL = 0, BAR_EMPTY = kStages, BAR_ACC_FULL = 2 * kStages, BAR_ACC_EMPTY = 2 * kStages + 2;
  volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(smem + kOffBar + (2 * kStages + 4) * 8);   // [0] TMEM base, [1] failure flag
  if (tid == 0) {
    misc[1] = 0;
    for (int i = 0; i < 2 * kStages + 2; ++i) mbar_init(bar(i), 1);
    mbar_init(bar(BAR_ACC_EMPTY), 256);
    mbar_init(bar(BAR_ACC_EMPTY + 1), 256);
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(base + kOffBar + (2 * kStages + 4) * 8, 512);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = misc[0];
  auto give_up = [&]() {
    if (misc[1] == 0) {
      atomicOr(g.status, TS_DEV_TIMEOUT);
      misc[1] = 1;
    }
  };
  auto wait = [&](int i, uint32_t parity) {
    if (!mbar_wait(bar(i), parity, misc[1] ? 2000 : g.wait_cycles)) give_up();
  };
  const int m_tiles = (g.M + 127) / 128, n_tiles = (g.N + kBN - 1) / kBN;
  const int n_work = m_tiles * n_tiles;
  const int k_blocks = (g.K + kBK - 1) / kBK;

  if (warp == 0) {
    // ---------------------------------------------------------------------- TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&a_map);
      tma_prefetch_desc(&b_map);
      pdl_wait();                  // the activations come from the kernel in front of this one
      int it = 0;                                          // K blocks issued so far (ring position)
      for (int t = blockIdx.x; t < n_work; t += gridDim.x) {
        const int m0 = (t % m_tiles) * 128, n0 = (t / m_tiles) * kBN;
        for (int kb = 0; kb < k_blocks; ++kb, ++it) {
          const int st = it % kStages;
          if (it >= kStages) wait(BAR_EMPTY + st, ((it / kStages) & 1) ^ 1);
          if (misc[1]) continue;                           // after a failure no new copies are started
          const uint32_t dst = base + st * kStageBytes;
          mbar_expect_tx(bar(BAR_FULL + st), kStageBytes);
          tma_load_2d(dst, &a_map, bar(BAR_FULL + st), kb * kBK, m0);
          tma_load_2d(dst + kABytes, &b_map, bar(BAR_FULL + st), kb * kBK, n0);
          tma_load_2d(dst + kABytes + kBBytes / 2, &b_map, bar(BAR_FULL + st), kb * kBK, n0 + 128);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------------ MMA issuer
    pdl_wait();                    // the time limits of its waits are for this launch, not for what the one in front still has to do
    const uint32_t issue = elect_one();
    bool dead = false;
    auto iwait = [&](int i, uint32_t parity) {
      if (!mbar_poll(bar(i), parity, dead ? 2000 : g.wait_cycles)) {
        dead = true;
        give_up();
      }
    };
    int it = 0, n_done = 0;                                // K blocks consumed, tiles issued
    for (int t = blockIdx.x; t < n_work; t += gridDim.x, ++n_done) {
      const int buf = n_done & 1, uses = n_done >> 1;      // accumulator, earlier tiles that used it
      if (uses > 0) iwait(BAR_ACC_EMPTY + buf, (uses - 1) & 1);
      tc_fence_after();
      for (int kb = 0; kb < k_blocks; ++kb, ++it) {
        const int st = it % kStages;
        iwait(BAR_FULL + st, (it / kStages) & 1);
        tc_fence_after();
        if (!dead) {
          const uint64_t a_desc = smem_desc(base + st * kStageBytes, 0, 1024);
          const uint64_t b_desc = smem_desc(base + st * kStageBytes + kABytes, 0, 1024);
#pragma unroll
          for (int ks = 0; ks < kBK / 16; ++ks)            // 16 of K = 32 bytes along the swizzled row
            mma_ss(tmem + buf * 256, a_desc + (uint64_t)(ks * 2), b_desc + (uint64_t)(ks * 2), kIdesc,
                   (kb > 0 || ks > 0) ? 1u : 0u, issue);
          tc_commit(bar(BAR_EMPTY + st), issue);           // the stage is free once these MMAs have read it
        }
      }
      if (!dead) tc_commit(bar(BAR_ACC_FULL + buf), issue);
    }
  } else {
    // --------------------------------------------------------------------------- epilogue
    const int q = warp & 3, hf = (warp - 2) >> 2;          // the TMEM lanes this warp can reach, its half of the columns
    prefetch_weights(g, ((int)blockIdx.x / m_tiles) * kBN + tid - 64, 0, g.K);
    pdl_wait();                    // the residual or the positions may come from the kernel in front of this one
    int n_done = 0;
    for (int t = blockIdx.x; t < n_work; t += gridDim.x, ++n_done) {
      const int m0 = (t % m_tiles) * 128, n0 = (t / m_tiles) * kBN;
      const int buf = n_done & 1;
      wait(BAR_ACC_FULL + buf, (n_done >> 1) & 1);
      tc_fence_after();
      epilogue_row<EPI>(g, tmem + buf * 256 + ((uint32_t)(q * 32) << 16), m0 + q * 32 + lane, n0, hf, [&]() {
        tc_fence_before();
        mbar_arrive(bar(BAR_ACC_EMPTY + buf));             // the accumulator is in registers
      });
    }
  }
  settle(misc[1] != 0);
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// ------------------------------------------------------------------------------------ pair kernel
// For products with many rows. Two CTAs of a cluster share a tile of 256 features x `nt` tokens
// (cta_group::2), computed transposed: the weights are the MMA's M (always 256), the tokens its N, which may be
// any multiple of 16 up to 256, so that the tokens divide into tiles of nearly equal size and little is
// computed for padding: 2112 of them are nine tiles of 240, 300 two of 160 (as M they would take 256 each). CTA r fetches 128 weight rows and nt / 2 token rows per 64 of K and holds the accumulator of its
// weight rows: TMEM lane = feature, column = token. One MMA reads the token halves of both CTAs. Per CTA and
// 64 of K that is at most 32 KB fetched and 32 KB read for 512 cycles of tensor work, where a CTA on its own moves
// 48 KB + 48 KB for a 128 x 256 tile (shared memory gives 128 bytes per clock: its limit, not the tensor pipe's).
// CTA 0 issues all MMAs. Every CTA's copies complete CTA 0's "full" barrier; the commits arrive at
// both CTAs' "empty" and "accumulator full" barriers; both epilogues release the accumulator to CTA 0.
// Features that the epilogue brings together (the two of a rotary pair, 64 apart; a gate and its up
// feature, 128 apart) sit sixteen lanes apart: the weights' tensor map has those rows as a dimension of its own.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}
// `bar` may lie in the other CTA of the pair
__device__ __forceinline__ void tma_load_2d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
__device__ __forceinline__ void tma_load_5d_pair(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1, int c2, int c3, int c4) {
  asm volatile(
      "cp.async.bulk.tensor.5d.cta_group::2.shared::cluster.global.tile.mbarrier::complete_tx::bytes "
      "[%0], [%1, {%3, %4, %5, %6, %7}], [%2];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1), "r"(c2), "r"(c3), "r"(c4)
      : "memory");
}
__device__ __forceinline__ void mma_ss_pair(uint32_t d, uint64_t a, uint64_t b, uint32_t idesc, uint32_t accumulate, uint32_t issue) {
  asm volatile(
      "{\n.reg .pred p, q;\nsetp.ne.u32 p, %4, 0;\nsetp.ne.u32 q, %5, 0;\n"
      "@q tcgen05.mma.cta_group::2.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(d),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate), "r"(issue)
      : "memory");
}
// Arrives at this barrier of both CTAs once the MMAs issued so far are done.
__device__ __forceinline__ void tc_commit_pair(uint32_t bar, uint32_t issue) {
  asm volatile(
      "{\n.reg .pred q;\nsetp.ne.u32 q, %1, 0;\n"
      "@q tcgen05.commit.cta_group::2.mbarrier::arrive::one.shared::cluster.multicast::cluster.b64 [%0], %2;\n}\n" ::"r"(bar),
      "r"(issue), "h"((uint16_t)3)
      : "memory");
}
__device__ __forceinline__ void mbar_arrive_cluster(uint32_t bar) {
  asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];\n" ::"r"(bar) : "memory");
}

constexpr int kPairStages = 6, kPairStageBytes = 2 * kABytes;
constexpr int kPairBars = 2 * kPairStages + 4;
constexpr int kPairSmem = kPairStages * kPairStageBytes + kPairBars * 8 + 16 + 1024;
constexpr uint32_t kIdescPair = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 4) << 24);   // M = 256; N is added

// One word of a token's row, read or written where at < n, by a predicate: with a branch around each, the sixteen
// stores of 32 tokens take a warp 1640 cycles instead of 1050, and the sixteen loads of their residual 1100 instead of
// 500, which the last tiles' epilogue adds to the launch.
// (Zero is in the word before: put there behind the load by the opposite predicate, it waits for every load, and 3000 x 8192 x
// 1024 with a residual takes 78.9 us instead of 48.5.)
__device__ __forceinline__ uint32_t ld_below(const uint16_t* p, int at, int n) {
  uint32_t w = 0;
  asm volatile("{\n.reg .pred p;\nsetp.lt.s32 p, %2, %3;\n@p ld.global.b32 %0, [%1];\n}\n" : "+r"(w) : "l"(p), "r"(at), "r"(n) : "memory");
  return w;
}
__device__ __forceinline__ void st_below(uint16_t* p, uint32_t w, int at, int n) {
  asm volatile("{\n.reg .pred p;\nsetp.lt.s32 p, %2, %3;\n@p st.global.b32 [%0], %1;\n}\n" ::"l"(p), "r"(w), "r"(at), "r"(n) : "memory");
}

// The residual's words of 32 tokens x a warp's 32 features, as epilogue_tokens<STORE> adds them: r[i] = features
// n0 + q * 32 + (lane & ~1) and the next one of token t0 + 2 i + (lane & 1). Zero outside the product.
__device__ __forceinline__ void load_residual(const GemmArgs& g, uint32_t (&r)[16], int t0, int end, int n0, int q, int lane) {
  const int col = n0 + q * 32 + (lane & ~1), n = col < g.N ? end - t0 - (lane & 1) : 0;
  const uint16_t* src = g.R + (size_t)(t0 + (lane & 1)) * g.ldc + col;
#pragma unroll
  for (int i = 0; i < 16; ++i) r[i] = ld_below(src + (size_t)(2 * i) * g.ldc, 2 * i, n);
}

// 32 tokens (t0 .. t0 + 31, those below `end`) of this lane's feature of a 128-feature accumulator: quarter q of
// the features, feature n0 + q * 32 + lane of the product (STORE) or the order of the permuted weight rows.
// Neighbouring lanes swap values first, so that a lane writes two features of one token: 64 bytes
// (STORE) or 32 bytes (the others) of a token's row together. r: the residual (STORE with g.R).
template <int EPI>
__device__ __forceinline__ void epilogue_tokens(const GemmArgs& g, float (&v)[32], const uint32_t (&r)[16], int t0, int end, int n0, int q, int lane) {
  const bool odd = lane & 1, upper = lane & 16;
  const int rest = end - t0 - odd;                         // tokens from this lane's first one on
  auto swap_pair = [&](float mine_even, float mine_odd, float& lo, float& hi) {   // even lanes keep the first token, odd ones the second
    const float got = __shfl_xor_sync(0xffffffffu, odd ? mine_even : mine_odd, 1);
    lo = odd ? got : mine_even;
    hi = odd ? mine_odd : got;
  };
  if (EPI == GEMM_EPI_STORE) {
    const int col = n0 + q * 32 + (lane & ~1), n = col < g.N ? rest : 0;
    uint16_t* dst = g.C + (size_t)(t0 + odd) * g.ldc + col;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      float lo, hi;
      swap_pair(v[2 * i], v[2 * i + 1], lo, hi);
      if (g.R) {
        lo += __uint_as_float(r[i] << 16);
        hi += __uint_as_float(r[i] & 0xFFFF0000u);
      }
      st_below(dst + (size_t)(2 * i) * g.ldc, pack_bf16(lo, hi), 2 * i, n);
    }
  } else if (EPI == GEMM_EPI_ROPE) {
    // lanes 0-15: features 16 q + lane of the head, lanes 16-31: their partners 64 further on
    if (n0 >= g.N) return;
    const bool rotate = n0 < g.q_cols + g.kv_cols;
    const int ld = n0 < g.q_cols ? g.q_cols : g.kv_cols, f = q * 16 + (lane & 15);
    uint16_t* dst = n0 < g.q_cols ? g.C + n0 : rotate ? g.C2 + (n0 - g.q_cols) : g.C3 + (n0 - g.q_cols - g.kv_cols);
    dst += (size_t)(t0 + odd) * ld + (upper ? 64 : 0) + (f & ~1);
    if (rotate) {
      const int pos = t0 + lane < end ? g.pos[t0 + lane] : 0;
#pragma unroll
      for (int i = 0; i < 32; ++i) {
        const float2 cs = g.rope_table[(size_t)__shfl_sync(0xffffffffu, pos, i) * 64 + f];   // (cos, sin)
        const float other = __shfl_xor_sync(0xffffffffu, v[i], 16);
        const float a = upper ? other : v[i], b = upper ? v[i] : other;
        v[i] = upper ? b * cs.x + a * cs.y : a * cs.x - b * cs.y;
      }
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      float lo, hi;
      swap_pair(v[2 * i], v[2 * i + 1], lo, hi);
      st_below(dst + (size_t)(2 * i) * ld, pack_bf16(lo, hi), 2 * i, rest);
    }
  } else {
    // lanes 0-15: gate features, lanes 16-31: the up features that belong to them. Of four tokens the lower lanes
    // take the first two, the upper ones the others: bf16 values of two tokens change lanes in one word (one fp32 value
    // of a token each: 1024 x 11264 x 2048 44.9 us instead of 42.0).
    // out[token][n0 / 2 + i] = silu(gate_i) * up_i. A division has a path of its own for rare operands and lets nothing move across
    // it, so exponentials, divisions and exchanges are taken sixteen at a time each (token by token a K of 2048 or less
    // does not hide the epilogue: 4096 x 16384 x 1024 117 us instead of 102).
    if (n0 >= g.N) return;
    const int first = odd + (upper ? 2 : 0);
    uint16_t* dst = g.C + (size_t)(t0 + first) * g.ldc + n0 / 2 + q * 16 + (lane & 14);
    float gate[16], up[16], z[16];
#pragma unroll
    for (int i = 0; i < 8; ++i) {                          // four tokens at a time
      const uint32_t front = pack_bf16(v[4 * i], v[4 * i + 1]), back = pack_bf16(v[4 * i + 2], v[4 * i + 3]);
      const uint32_t got = __shfl_xor_sync(0xffffffffu, upper ? front : back, 16);
      const uint32_t gates = upper ? got : front, ups = upper ? back : got;
      gate[2 * i] = __uint_as_float(gates << 16);
      gate[2 * i + 1] = __uint_as_float(gates & 0xFFFF0000u);
      up[2 * i] = __uint_as_float(ups << 16);
      up[2 * i + 1] = __uint_as_float(ups & 0xFFFF0000u);
      z[2 * i] = silu_den(gate[2 * i]);
      z[2 * i + 1] = silu_den(gate[2 * i + 1]);
    }
#pragma unroll
    for (int i = 0; i < 16; ++i) z[i] = gate[i] / z[i] * up[i];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      float lo, hi;
      swap_pair(z[2 * i], z[2 * i + 1], lo, hi);
      st_below(dst + (size_t)(4 * i) * g.ldc, pack_bf16(lo, hi), 4 * i, end - t0 - first);
    }
  }
}

template <int EPI>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_pair_kernel(const GemmArgs g, const __grid_constant__ CUtensorMap x_map, const __grid_constant__ CUtensorMap w_map, const int nt) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - smem_u32(smem_raw));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t rank = blockIdx.x & 1;                    // in the cluster
  constexpr int kOffBar = kPairStages * kPairStageBytes, kOffMisc = kOffBar + kPairBars * 8;
  pdl_launch_dependents();
  auto bar = [&](int i) { return base + kOffBar + (uint32_t)i * 8u; };
  constexpr int BAR_FULL = 0, BAR_EMPTY = kPairStages, BAR_ACC_FULL = 2 * kPairStages, BAR_ACC_EMPTY = 2 * kPairStages + 2;
  volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);   // [0] TMEM base, [1] failure flag
  if (tid == 0) {
    misc[1] = 0;
    for (int i = 0; i < BAR_ACC_EMPTY; ++i) mbar_init(bar(i), 1);
    mbar_init(bar(BAR_ACC_EMPTY), 16);                     // eight epilogue warps of each CTA (CTA 0's barrier is the one used)
    mbar_init(bar(BAR_ACC_EMPTY + 1), 16);
    mbar_init_fence();
  }
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], 512;\n" ::"r"(base + kOffMisc) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync();                  // the other CTA's barriers are initialised too
  tc_fence_after();
  const uint32_t tmem = misc[0];
  auto give_up = [&]() {
    if (misc[1] == 0) {
      atomicOr(g.status, TS_DEV_TIMEOUT);
      misc[1] = 1;
    }
  };
  auto wait = [&](int i, uint32_t parity) {
    if (!mbar_wait(bar(i), parity, misc[1] ? 2000 : g.wait_cycles)) give_up();
  };
  const int m_tiles = (g.M + nt - 1) / nt, n_tiles = (g.N + kBN - 1) / kBN;
  const int n_work = m_tiles * n_tiles, first = blockIdx.x >> 1, stride = gridDim.x >> 1;
  const int k_blocks = (g.K + kBK - 1) / kBK;

  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&x_map);
      tma_prefetch_desc(&w_map);
      pdl_wait();
      const uint32_t bytes = 2u * (kABytes + (uint32_t)nt * (kBK * 2 / 2));
      int it = 0;
      for (int t = first; t < n_work; t += stride) {
        const int m0 = (t % m_tiles) * nt + (int)rank * (nt / 2), nb = t / m_tiles;
        for (int kb = 0; kb < k_blocks; ++kb, ++it) {
          const int st = it % kPairStages;
          if (it >= kPairStages) wait(BAR_EMPTY + st, ((it / kPairStages) & 1) ^ 1);
          if (misc[1]) continue;                           // after a failure no new copies are started
          const uint32_t dst = base + st * kPairStageBytes, full = mapa(bar(BAR_FULL + st), 0);
          if (rank == 0) mbar_expect_tx(bar(BAR_FULL + st), bytes);
          if (EPI == GEMM_EPI_STORE)
            tma_load_2d_pair(dst, &w_map, full, kb * kBK, nb * kBN + (int)rank * 128);
          else if (EPI == GEMM_EPI_ROPE)                   // sixteen rows, half of a head, quarter of its half, head
            tma_load_5d_pair(dst, &w_map, full, kb * kBK, 0, 0, 0, nb * 2 + (int)rank);
          else                                             // sixteen rows, gate | up, sixteenth of the block, block of 256 rows
            tma_load_5d_pair(dst, &w_map, full, kb * kBK, 0, 0, (int)rank * 4, nb);
          tma_load_2d_pair(dst + kABytes, &x_map, full, kb * kBK, m0);
        }
      }
      // the commits that free the last stages arrive here too: they must have before this CTA may leave
      for (int i = max(0, it - kPairStages); i < it; ++i) wait(BAR_EMPTY + i % kPairStages, (i / kPairStages) & 1);
    }
  } else if (warp == 1) {
    if (rank == 0) {
      pdl_wait();                  // as in gemm_kernel
      const uint32_t issue = elect_one();
      bool dead = false;
      auto iwait = [&](int i, uint32_t parity) {
        if (!mbar_poll(bar(i), parity, dead ? 2000 : g.wait_cycles)) {
          dead = true;
          give_up();
        }
      };
      const uint32_t idesc = kIdescPair | ((uint32_t)(nt >> 3) << 17);
      int it = 0, n_done = 0;
      for (int t = first; t < n_work; t += stride, ++n_done) {
        const int buf = n_done & 1, uses = n_done >> 1;
        if (uses > 0) iwait(BAR_ACC_EMPTY + buf, (uses - 1) & 1);
        tc_fence_after();
        for (int kb = 0; kb < k_blocks; ++kb, ++it) {
          const int st = it % kPairStages;
          iwait(BAR_FULL + st, (it / kPairStages) & 1);
          tc_fence_after();
          if (!dead) {
            const uint64_t a_desc = smem_desc(base + st * kPairStageBytes, 0, 1024);
            const uint64_t b_desc = smem_desc(base + st * kPairStageBytes + kABytes, 0, 1024);
#pragma unroll
            for (int ks = 0; ks < kBK / 16; ++ks)
              mma_ss_pair(tmem + buf * 256, a_desc + (uint64_t)(ks * 2), b_desc + (uint64_t)(ks * 2), idesc,
                          (kb > 0 || ks > 0) ? 1u : 0u, issue);
            tc_commit_pair(bar(BAR_EMPTY + st), issue);
          }
        }
        if (!dead) tc_commit_pair(bar(BAR_ACC_FULL + buf), issue);
      }
    }
  } else {
    if (tid - 64 < 128) prefetch_weights(g, (first / m_tiles) * kBN + (int)rank * 128 + tid - 64, 0, g.K);
    pdl_wait();                    // the residual or the positions may come from the kernel in front of this one
    const int q = warp & 3, hf = (warp - 2) >> 2;
    int n_done = 0;
    for (int t = first; t < n_work; t += stride, ++n_done) {
      const int m0 = (t % m_tiles) * nt, end = min(g.M, m0 + nt);
      // first feature of this CTA's half of the tile; SILU_MUL: gate and up features of half a block
      const int n0 = (t / m_tiles) * kBN + (int)rank * 128;
      const int buf = n_done & 1;
      const int chunks = (nt + 31) / 32, last = ((chunks - 1 - hf) & ~1) + hf;   // this warp: chunks hf, hf + 2, ...
      // The residual is fetched a chunk ahead, the first one's before the sums are there: the epilogue of a launch's
      // last tiles is not hidden behind anything. (1024 x 4096 x 4096, both with branches around the stores: 33.2 us
      // with the residual fetched where it is added, 31.1 so.)
      const bool with_r = EPI == GEMM_EPI_STORE && g.R != nullptr;
      uint32_t next_r[16];
      if (with_r) load_residual(g, next_r, m0 + hf * 32, end, n0, q, lane);
      wait(BAR_ACC_FULL + buf, (n_done >> 1) & 1);
      tc_fence_after();
      for (int c = hf; c < chunks; c += 2) {
        float v[32];
        uint32_t r[16];
        tmem_ld32(v, tmem + buf * 256 + ((uint32_t)(q * 32) << 16) + c * 32);
        if (with_r) {
#pragma unroll
          for (int i = 0; i < 16; ++i) r[i] = next_r[i];
          load_residual(g, next_r, m0 + (c + 2) * 32, end, n0, q, lane);
        }
        tmem_ld_wait();
        if (c == last) {
          tc_fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster(mapa(bar(BAR_ACC_EMPTY + buf), 0));
        }
        if (m0 + c * 32 < end) epilogue_tokens<EPI>(g, v, r, m0 + c * 32, end, n0, q, lane);
      }
      if (hf >= chunks) {                                  // a narrow tile: nothing for this warp
        __syncwarp();
        if (lane == 0) mbar_arrive_cluster(mapa(bar(BAR_ACC_EMPTY + buf), 0));
      }
    }
  }
  settle(misc[1] != 0);
  tc_fence_before();
  __syncwarp();
  cluster_sync();                  // no CTA leaves while the other one's copies, commits or arrivals may still reach it
  if (warp == 1) asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, 512;\n" ::"r"(tmem) : "memory");
}

// ---------------------------------------------------------------------------------- split-K kernel
// For products with few tiles (a decode batch: one 128-row block of tokens). Such a product is bound
// by the HBM traffic of its weights, but with one CTA per 128 x 256 tile only 16-24 of the 148 SMs
// pull on HBM (hidden 4096: 37 us for the 50 MB of QKV weights, 1.35 TB/s). Here a cluster of S
// CTAs shares a 128 x 128 tile: CTA r multiplies K blocks [kb r / S, kb (r+1) / S), lays its fp32
// accumulator into its own shared memory (the operand stages are free by then), and after a cluster
// barrier the S CTAs add up the S accumulators, each a share of the elements, in the order r = 0 ..
// S-1 (through distributed shared memory: nothing goes to global memory, no workspace, and the
// result does not depend on timing), apply the epilogue and write it. The merge is bound by the
// distributed reads (~8 bytes per clock and SM); half the tile width with half the split halves them
// twice over: 128 x 256 tiles in clusters of 6-8 took 18.2 / 15.8 / 31.5 us at 64 rows (QKV / output /
// down), 128 x 128 tiles in clusters of 3-4 take
// 15.3 / 11.6 / 25.5 us.
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr));
  return v;
}
constexpr int kSplitN = 128;
constexpr int kSplitStages = 6, kSplitStageBytes = kABytes + kBBytes / 2;
constexpr int kSplitSmem = kSplitStages * kSplitStageBytes + (2 * kSplitStages + 1) * 8 + 16 + 1024;
static_assert(128 * kSplitN * 4 <= kSplitStages * kSplitStageBytes, "the accumulator image takes the place of the operand stages");
// 16-byte chunk `c` of row `row` of the accumulator image; the XOR spreads a column of rows over the banks
__device__ __forceinline__ uint32_t image_off(int row, int c) { return (uint32_t)(row * (kSplitN * 4) + ((c ^ (row & 7)) << 4)); }

template <int EPI>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_split_kernel(const GemmArgs g, const __grid_constant__ CUtensorMap a_map, const __grid_constant__ CUtensorMap b_map, const int split) {
  extern __shared__ unsigned char smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - smem_u32(smem_raw));
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  constexpr int kOffBar = kSplitStages * kSplitStageBytes;
  pdl_launch_dependents();
  // barriers: full[kSplitStages], empty[kSplitStages], accumulator full
  auto bar = [&](int i) { return base + kOffBar + (uint32_t)i * 8u; };
  constexpr int BAR_FULL = 0, BAR_EMPTY = kSplitStages, BAR_ACC = 2 * kSplitStages;
  constexpr int kOffMisc = kOffBar + (2 * kSplitStages + 1) * 8;
  volatile uint32_t* misc = reinterpret_cast<volatile uint32_t*>(smem + kOffMisc);   // [0] TMEM base, [1] failure flag
  if (tid == 0) {
    misc[1] = 0;
    for (int i = 0; i < 2 * kSplitStages + 1; ++i) mbar_init(bar(i), 1);
    mbar_init_fence();
  }
  if (warp == 1) tmem_alloc(base + kOffMisc, kSplitN);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = misc[0];
  auto give_up = [&]() {
    if (misc[1] == 0) {
      atomicOr(g.status, TS_DEV_TIMEOUT);
      misc[1] = 1;
    }
  };
  const int m_tiles = (g.M + 127) / 128;
  const int t = blockIdx.x / split, rank = blockIdx.x % split;     // the cluster's CTAs are consecutive blocks
  const int m0 = (t % m_tiles) * 128, n0 = (t / m_tiles) * kSplitN;
  const int rows = min(128, g.M - m0);
  const int k_blocks = (g.K + kBK - 1) / kBK;
  const int kb0 = k_blocks * rank / split, kb1 = k_blocks * (rank + 1) / split;   // never empty: split <= k_blocks

  // one item = 8 columns of a row, for ROPE with their partners 64 further on
  constexpr int kItems = EPI == GEMM_EPI_STORE ? 16 : 8;
  const int first_item = rank * kGemmThreads + tid, stride = split * kGemmThreads;
  // What an item adds to the product: the residual's columns, or the angles' (cos, sin).
  auto fetch = [&](int i, float4 (&extra)[EPI == GEMM_EPI_STORE ? 1 : 4]) {
    const int r = i / kItems, ch = i % kItems, row = m0 + r;
    if (i >= rows * kItems) return;
    if constexpr (EPI == GEMM_EPI_STORE) {
      if (g.R && n0 + ch * 8 < g.N) extra[0] = *reinterpret_cast<const float4*>(g.R + (size_t)row * g.ldc + n0 + ch * 8);
    } else if (n0 < g.q_cols + g.kv_cols) {
      const float4* cs = reinterpret_cast<const float4*>(g.rope_table + (size_t)g.pos[row] * 64 + ch * 8);
#pragma unroll
      for (int e = 0; e < 4; ++e) extra[e] = cs[e];
    }
  };
  // Each thread fetches its first item's (of a decode batch its only one) before the product: behind it, position and
  // angles are two round trips in a row.
  float4 extra[EPI == GEMM_EPI_STORE ? 1 : 4];
  if (warp >= 2 && tid - 64 < kSplitN) prefetch_weights(g, n0 + tid - 64, kb0 * kBK, kb1 * kBK);
  if (tid == 0) {
    tma_prefetch_desc(&a_map);
    tma_prefetch_desc(&b_map);
  }
  pdl_wait();                      // the activations, the residual and the positions come from the launches in front

  if (warp == 0) {
    if (lane == 0) {
      for (int kb = kb0, it = 0; kb < kb1; ++kb, ++it) {
        const int st = it % kSplitStages;
        if (it >= kSplitStages && !mbar_wait(bar(BAR_EMPTY + st), ((it / kSplitStages) & 1) ^ 1, misc[1] ? 2000 : g.wait_cycles)) give_up();
        if (misc[1]) continue;                             // after a failure no new copies are started
        const uint32_t dst = base + st * kSplitStageBytes;
        mbar_expect_tx(bar(BAR_FULL + st), kSplitStageBytes);
        tma_load_2d(dst + kABytes, &b_map, bar(BAR_FULL + st), kb * kBK, n0);
        tma_load_2d(dst, &a_map, bar(BAR_FULL + st), kb * kBK, m0);
      }
    }
  } else if (warp == 1) {
    const uint32_t issue = elect_one();
    bool dead = false;
    for (int kb = kb0, it = 0; kb < kb1; ++kb, ++it) {
      const int st = it % kSplitStages;
      if (!mbar_poll(bar(BAR_FULL + st), (it / kSplitStages) & 1, dead ? 2000 : g.wait_cycles)) {
        dead = true;
        give_up();
      }
      tc_fence_after();
      if (dead) continue;
      const uint64_t a_desc = smem_desc(base + st * kSplitStageBytes, 0, 1024);
      const uint64_t b_desc = smem_desc(base + st * kSplitStageBytes + kABytes, 0, 1024);
#pragma unroll
      for (int ks = 0; ks < kBK / 16; ++ks)
        mma_ss(tmem, a_desc + (uint64_t)(ks * 2), b_desc + (uint64_t)(ks * 2), instr_desc(false), (it > 0 || ks > 0) ? 1u : 0u, issue);
      tc_commit(bar(BAR_EMPTY + st), issue);
    }
    if (!dead) tc_commit(bar(BAR_ACC), issue);
  } else {
    fetch(first_item, extra);
    // accumulator -> image in shared memory; every operand stage has been read once the barrier completes
    if (!mbar_wait(bar(BAR_ACC), 0, misc[1] ? 2000 : g.wait_cycles)) give_up();
    tc_fence_after();
    const int q = warp & 3, hf = (warp - 2) >> 2;          // the TMEM lanes this warp can reach, its half of the columns
    const int row = q * 32 + lane;
    if (q * 32 < rows && misc[1] == 0) {
#pragma unroll 1
      for (int c = hf * 2; c < hf * 2 + 2; ++c) {
        float v[32];
        tmem_ld32(v, tmem + ((uint32_t)(q * 32) << 16) + c * 32);
        tmem_ld_wait();
        if (row < rows) {
#pragma unroll
          for (int i = 0; i < 8; ++i)
            *reinterpret_cast<float4*>(smem + image_off(row, c * 8 + i)) = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
        }
      }
    }
  }
  settle(misc[1] != 0);
  __syncwarp();
  if (warp < 2) fetch(first_item, extra);
  cluster_sync();                  // the images are complete
  auto sum8 = [&](int row, int col, float (&v)[8]) {
    float4 x[kMaxSplit], y[kMaxSplit];                     // all loads fly at once
#pragma unroll
    for (int r = 0; r < kMaxSplit; ++r) {
      x[r] = y[r] = make_float4(0.f, 0.f, 0.f, 0.f);
      if (r < split) {
        const uint32_t img = mapa(base, (uint32_t)r);
        x[r] = ld_cluster4(img + image_off(row, col / 4));
        y[r] = ld_cluster4(img + image_off(row, col / 4 + 1));
      }
    }
    v[0] = x[0].x; v[1] = x[0].y; v[2] = x[0].z; v[3] = x[0].w;
    v[4] = y[0].x; v[5] = y[0].y; v[6] = y[0].z; v[7] = y[0].w;
#pragma unroll
    for (int r = 1; r < kMaxSplit; ++r) {                  // a rank that is not there adds zeros
      v[0] += x[r].x; v[1] += x[r].y; v[2] += x[r].z; v[3] += x[r].w;
      v[4] += y[r].x; v[5] += y[r].y; v[6] += y[r].z; v[7] += y[r].w;
    }
  };
  for (int i = first_item; i < rows * kItems; i += stride) {
    const int r = i / kItems, ch = i % kItems, row = m0 + r;
    if (i != first_item) fetch(i, extra);
    if constexpr (EPI == GEMM_EPI_STORE) {
      const int col = n0 + ch * 8;
      if (col >= g.N) continue;
      float v[8];
      sum8(r, ch * 8, v);
      if (g.R) {
        float x[8];
        unpack8(*reinterpret_cast<const uint4*>(&extra[0]), x);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] += x[e];
      }
      *reinterpret_cast<uint4*>(g.C + (size_t)row * g.ldc + col) = pack8(v);
    } else {
      float lo[8], hi[8];
      sum8(r, ch * 8, lo);
      sum8(r, 64 + ch * 8, hi);
      rope8(g, row, n0, ch * 8, lo, hi, extra);
    }
  }
  tc_fence_before();
  cluster_sync();                  // no CTA leaves while another one reads its image
  if (warp == 1) tmem_dealloc(tmem, kSplitN);
}

// launch_pdl for a grid of clusters of `cluster` CTAs.
template <typename... Params, typename... Args>
cudaError_t launch_cluster(void (*kernel)(Params...), int ctas, int cluster, int smem, cudaStream_t stream, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(ctas);
  cfg.blockDim = dim3(kGemmThreads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<Args>(args)...);
}

template <int EPI>
cudaError_t launch_split_t(const GemmArgs& g, const CUtensorMap& a_map, const CUtensorMap& b_map, int split, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(gemm_split_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem);
  if (e != cudaSuccess) return e;
  const int tiles = ((g.M + 127) / 128) * ((g.N + kSplitN - 1) / kSplitN);
  return launch_cluster(gemm_split_kernel<EPI>, tiles * split, split, kSplitSmem, stream, g, a_map, b_map, split);
}

// CTAs of gemm_split_kernel that the device runs at once in clusters of `split` (a hardware figure;
// asked for once per device and size).
int split_slots(int split) {
  constexpr int kMaxDevices = 64;
  static std::atomic<int> known[kMaxDevices][kMaxSplit + 1];
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= kMaxDevices) return 0;
  const int have = known[dev][split].load(std::memory_order_relaxed);
  if (have > 0) return have - 1;
  if (cudaFuncSetAttribute(gemm_split_kernel<GEMM_EPI_STORE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem) != cudaSuccess) return 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(split);
  cfg.blockDim = dim3(kGemmThreads);
  cfg.dynamicSmemBytes = kSplitSmem;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = (unsigned)split;
  attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  int clusters = 0;
  if (cudaOccupancyMaxActiveClusters(&clusters, gemm_split_kernel<GEMM_EPI_STORE>, &cfg) != cudaSuccess) {
    cudaGetLastError();
    clusters = 0;
  }
  known[dev][split].store(clusters * split + 1, std::memory_order_relaxed);
  return clusters * split;
}

template <int EPI>
cudaError_t launch_tile_t(const GemmArgs& g, const CUtensorMap& a_map, const CUtensorMap& b_map, int n_sms, cudaStream_t stream) {
  const size_t smem = (size_t)kTileStages * (kABytes + kBBytes) + (2 * kTileStages + 4) * 8 + 16 + 1024;
  cudaError_t e = cudaFuncSetAttribute(gemm_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int tiles = ((g.M + 127) / 128) * ((g.N + kBN - 1) / kBN);
  return launch_pdl(gemm_kernel<EPI>, dim3(std::min(n_sms, tiles)), dim3(kGemmThreads), smem, stream, g, a_map, b_map);
}

template <int EPI>
cudaError_t launch_pair_t(const GemmArgs& g, const CUtensorMap& x_map, const CUtensorMap& w_map, int nt, int n_sms, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(gemm_pair_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, kPairSmem);
  if (e != cudaSuccess) return e;
  const int tiles = ((g.M + nt - 1) / nt) * ((g.N + kBN - 1) / kBN);
  return launch_cluster(gemm_pair_kernel<EPI>, 2 * std::min(n_sms / 2, tiles), 2, kPairSmem, stream, g, x_map, w_map, nt);
}

template <int EPI>
cudaError_t launch_epi(const GemmArgs& g, const GemmMaps& maps, GemmPlan plan, int n_sms, cudaStream_t stream) {
  if constexpr (EPI != GEMM_EPI_SILU_MUL)                // a gate and its up column are 128 columns apart: no tile of 128 holds both
    if (plan.split > 0) return launch_split_t<EPI>(g, *maps.x, *maps.w, plan.split, stream);
  if (plan.tile_m == 256) return launch_pair_t<EPI>(g, *maps.x_pair, *maps.w_pair, plan.pair_tokens, n_sms, stream);
  return launch_tile_t<EPI>(g, *maps.x, *maps.w, n_sms, stream);
}

}  // namespace

// Cost of a launch in us besides what every launch pays: waves x K blocks x the time of a K block, which
// is what the tensor pipe and shared memory take (0.45 us for a CTA's 128 x 256 tile, 0.2 us + 0.65 ns per token
// for a pair's tile, 0.33 us for a 128 x 128 tile), what an SM needs to get a pair's weights from HBM (0.285 us), or
// what HBM needs for the weight blocks in flight
// at that moment; for the split kernel also what its merge takes longer than another kernel's last epilogue, and only
// where all clusters run at once.
// Measured (bursts too short for the power cap, weights not in L2, us; 128 x 256 tile / pair / split kernel, the latter two
// with their best tokens and split): 64 rows QKV 32.3 / 21.5 / 15.9, output 29.7 / 20.6 / 12.2, gate/up 46.5 / 47.7, down 88.8 / 62.9 /
// 25.7; 256 rows output 32.3 / 22.2 / 17.8, down 92.4 / 66.9 / 42.0; gate/up with 130 rows 63.8 / 54.0, 300 86.4 / 84.5, 512 111 /
// 94.3, 800 161 / 150, 2112 342 / 319; 2112 rows QKV 94.9 / 76.8, output 60.6 / 50.6, down 192 / 160. 2048 x 2048, where a pair's main
// loop is short: 130 rows 19.7 / 12.5 / 10.7, 256 rows 19.8 / 12.7 / 11.0.
GemmPlan gemm_plan(const GemmArgs& g, int n_sms) {
  constexpr double kTileUs = 0.45, kPairUs = 0.2, kPairTokenUs = 0.00065, kPairMinUs = 0.285, kSplitUs = 0.33, kHbmBytesPerUs = 6.2e6;
  const double merge_us = 2.0 + 0.03 * std::min(g.M, 128);
  const int n_tiles = (g.N + kBN - 1) / kBN, m128 = (g.M + 127) / 128, m256 = (g.M + 255) / 256;
  const int kb = (g.K + kBK - 1) / kBK;
  // `at_once` workers on weight blocks of `width` rows, each on another one unless m_tiles row blocks share it
  auto cost_of = [&](double us, int tiles, int workers, int m_tiles, int width, int blocks) {
    const double hbm = (double)std::min(tiles, workers) / m_tiles * width * kBK * 2 / kHbmBytesPerUs;
    return (double)((tiles + workers - 1) / workers) * blocks * std::max(us, hbm);
  };
  GemmPlan best = {128, 0, 0};
  double cost = cost_of(kTileUs, m128 * n_tiles, n_sms, m128, kBN, kb);
  // tokens of a pair's tile: as many tiles as need be, or a few more where they fill the pairs' last wave better
  for (int m = m256; m <= m256 + 3; ++m) {
    const int nt = pair_tokens(g.M, m), tiles = (g.M + nt - 1) / nt;
    const double c = cost_of(std::max(kPairUs + kPairTokenUs * nt, kPairMinUs), tiles * n_tiles, n_sms / 2, tiles, kBN, kb);
    if (c < cost) {
      cost = c;
      best = {256, 0, nt};
    }
  }
  const int split_tiles = m128 * ((g.N + kSplitN - 1) / kSplitN);
  for (int s = 2; s <= std::min(kMaxSplit, kb) && g.epi != GEMM_EPI_SILU_MUL; ++s) {
    if (split_tiles * s > n_sms || split_tiles * s > split_slots(s)) break;
    const double c = cost_of(kSplitUs, split_tiles * s, split_tiles * s, m128, kSplitN, (kb + s - 1) / s) + merge_us;
    if (c < cost * 0.98) {
      cost = c;
      best = {128, s, 0};
    }
  }
  return best;
}

cudaError_t launch_gemm(const GemmArgs& g, const GemmMaps& maps, GemmPlan plan, int n_sms, cudaStream_t stream) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  switch (g.epi) {
    case GEMM_EPI_ROPE: return launch_epi<GEMM_EPI_ROPE>(g, maps, plan, n_sms, stream);
    case GEMM_EPI_SILU_MUL: return launch_epi<GEMM_EPI_SILU_MUL>(g, maps, plan, n_sms, stream);
    default: return launch_epi<GEMM_EPI_STORE>(g, maps, plan, n_sms, stream);
  }
}

}  // namespace ts
