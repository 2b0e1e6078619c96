// bf16 GEMM of the decoder layer around the attention step (sm_100a): C = A . B^T with fp32
// accumulation on the 5th-generation tensor cores.
//
//   A [M][K] bf16 (activations, one token per row), B [N][K] bf16 (weights, [out features][in
//   features]), C [M][N] bf16. Both operands are K-major, exactly as they sit in memory.
//
// One persistent CTA per SM walks the output tiles (tile index t -> column block t / m_tiles, row
// block t % m_tiles, so the CTAs that run at the same time share a few weight blocks through L2).
// A tile is TILE_M x 256: TILE_M = 128 (one tcgen05.mma M = 128, N = 256 per 16 of K) or 256 (two of
// them that share the weight block in shared memory, which cuts the bytes fetched per flop by a
// third). Operands arrive by TMA in 64-wide K blocks (128-byte swizzle) through a ring of stages;
// the accumulators live in TMEM (2 x 256 columns): with TILE_M = 128 they alternate between tiles,
// so the epilogue of a tile overlaps the main loop of the next one; with TILE_M = 256 a tile takes both.
// Warp roles: warp 0 TMA producer, warp 1 MMA issuer and TMEM owner, warps 2-5 epilogue
// (thread = accumulator row: TMEM -> registers -> bf16 -> global).
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

constexpr int kGemmThreads = 192;
constexpr int kBN = 256, kBK = 64;
constexpr int kMaxSplit = 8;                    // portable cluster size
constexpr int kABytes = 128 * kBK * 2;          // one 128-row operand block: 16 KB
constexpr int kBBytes = kBN * kBK * 2;          // the 256-row weight block: 32 KB

__device__ __forceinline__ void tma_load_2d(uint32_t dst, const CUtensorMap* map, uint32_t bar, int c0, int c1) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.tile.mbarrier::complete_tx::bytes [%0], [%1, {%3, %4}], [%2];\n" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(bar), "r"(c0), "r"(c1)
      : "memory");
}
// The box at (c0, c1) into L2.
__device__ __forceinline__ void tma_prefetch_2d(const CUtensorMap* map, int c0, int c1) {
  asm volatile("cp.async.bulk.prefetch.tensor.2d.L2.global.tile [%0, {%1, %2}];\n" ::"l"(reinterpret_cast<uint64_t>(map)), "r"(c0), "r"(c1)
               : "memory");
}
// bf16 x bf16 -> fp32, M = 128, N = 256, both operands K-major
constexpr uint32_t kIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((256u >> 3) << 17) | ((128u >> 4) << 24);

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
// and their partners 64 further on: rotated (query and key heads) and written to the head's tensor.
__device__ __forceinline__ void rope8(const GemmArgs& g, int row, int col0, int c, float (&lo)[8], float (&hi)[8]) {
  const bool rotate = col0 < g.q_cols + g.kv_cols;
  uint16_t* dst = col0 < g.q_cols ? g.C + (size_t)row * g.q_cols + col0
                  : rotate        ? g.C2 + (size_t)row * g.kv_cols + (col0 - g.q_cols)
                                  : g.C3 + (size_t)row * g.kv_cols + (col0 - g.q_cols - g.kv_cols);
  if (rotate) {
    const float2* cs = g.rope_table + (size_t)g.pos[row] * 64 + c;
#pragma unroll
    for (int e = 0; e < 8; ++e) {
      const float2 t2 = cs[e];                             // (cos, sin)
      const float a = lo[e], b = hi[e];
      lo[e] = a * t2.x - b * t2.y;
      hi[e] = b * t2.x + a * t2.y;
    }
  }
  *reinterpret_cast<uint4*>(dst + c) = pack8(lo);
  *reinterpret_cast<uint4*>(dst + 64 + c) = pack8(hi);
}
// gate <- silu(gate) * up, both rounded to bf16 first (they are bf16 tensors of the layer's definition)
__device__ __forceinline__ void silu_mul8(float* gate, const float* up) {
#pragma unroll
  for (int e = 0; e < 8; ++e) {
    const float a = __bfloat162float(__float2bfloat16_rn(gate[e])), b = __bfloat162float(__float2bfloat16_rn(up[e]));
    gate[e] = a / (1.f + __expf(-a)) * b;
  }
}

template <int TILE_M, int EPI>
__global__ void __launch_bounds__(kGemmThreads, 1)
gemm_kernel(const GemmArgs g, const __grid_constant__ CUtensorMap a_map, const __grid_constant__ CUtensorMap b_map) {
  constexpr int kMB = TILE_M / 128;                       // accumulators (and M = 128 MMAs per K step) of a tile
  constexpr int kStageBytes = kMB * kABytes + kBBytes;    // 48 KB or 64 KB
  constexpr int kStages = TILE_M == 128 ? 4 : 3;
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
    mbar_init(bar(BAR_ACC_EMPTY), 128);
    mbar_init(bar(BAR_ACC_EMPTY + 1), 128);
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
  const int m_tiles = (g.M + TILE_M - 1) / TILE_M, n_tiles = (g.N + kBN - 1) / kBN;
  const int n_work = m_tiles * n_tiles;
  const int k_blocks = (g.K + kBK - 1) / kBK;
  pdl_wait();                      // the operands may come from the kernel in front of this one

  if (warp == 0) {
    // ---------------------------------------------------------------------- TMA producer
    if (lane == 0) {
      tma_prefetch_desc(&a_map);
      tma_prefetch_desc(&b_map);
      int it = 0;                                          // K blocks issued so far (ring position)
      for (int t = blockIdx.x; t < n_work; t += gridDim.x) {
        const int m0 = (t % m_tiles) * TILE_M, n0 = (t / m_tiles) * kBN;
        for (int kb = 0; kb < k_blocks; ++kb, ++it) {
          const int st = it % kStages;
          if (it >= kStages) wait(BAR_EMPTY + st, ((it / kStages) & 1) ^ 1);
          if (misc[1]) continue;                           // after a failure no new copies are started
          const uint32_t dst = base + st * kStageBytes;
          mbar_expect_tx(bar(BAR_FULL + st), kStageBytes);
#pragma unroll
          for (int mb = 0; mb < kMB; ++mb) tma_load_2d(dst + mb * kABytes, &a_map, bar(BAR_FULL + st), kb * kBK, m0 + mb * 128);
          tma_load_2d(dst + kMB * kABytes, &b_map, bar(BAR_FULL + st), kb * kBK, n0);
        }
      }
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------------------ MMA issuer
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
      // TILE_M = 128: tile n uses accumulator n % 2; TILE_M = 256: both, so every tile waits for the epilogue
      const int buf = kMB == 1 ? (n_done & 1) : 0;
      const int uses = kMB == 1 ? (n_done >> 1) : n_done;  // earlier tiles that used this accumulator
      if (uses > 0) {
        iwait(BAR_ACC_EMPTY + buf, (uses - 1) & 1);
        if (kMB == 2) iwait(BAR_ACC_EMPTY + 1, (uses - 1) & 1);
      }
      tc_fence_after();
      for (int kb = 0; kb < k_blocks; ++kb, ++it) {
        const int st = it % kStages;
        iwait(BAR_FULL + st, (it / kStages) & 1);
        tc_fence_after();
        if (!dead) {
          const uint64_t b_desc = smem_desc(base + st * kStageBytes + kMB * kABytes, 0, 1024);
#pragma unroll
          for (int mb = 0; mb < kMB; ++mb) {
            const uint64_t a_desc = smem_desc(base + st * kStageBytes + mb * kABytes, 0, 1024);
#pragma unroll
            for (int ks = 0; ks < kBK / 16; ++ks)          // 16 of K = 32 bytes along the swizzled row
              mma_ss(tmem + (kMB == 1 ? buf : mb) * 256, a_desc + (uint64_t)(ks * 2), b_desc + (uint64_t)(ks * 2), kIdesc,
                     (kb > 0 || ks > 0) ? 1u : 0u, issue);
          }
          tc_commit(bar(BAR_EMPTY + st), issue);           // the stage is free once these MMAs have read it
        }
      }
      if (!dead) {
        tc_commit(bar(BAR_ACC_FULL + buf), issue);
        if (kMB == 2) tc_commit(bar(BAR_ACC_FULL + 1), issue);
      }
    }
  } else {
    // --------------------------------------------------------------------------- epilogue
    const int q = warp & 3;                                // the TMEM lanes this warp can reach
    const int row_in_blk = q * 32 + lane;
    int n_done = 0;
    for (int t = blockIdx.x; t < n_work; t += gridDim.x, ++n_done) {
      const int m0 = (t % m_tiles) * TILE_M, n0 = (t / m_tiles) * kBN;
#pragma unroll 1
      for (int mb = 0; mb < kMB; ++mb) {
        const int buf = kMB == 1 ? (n_done & 1) : mb;
        const int uses = kMB == 1 ? (n_done >> 1) : n_done;
        wait(BAR_ACC_FULL + buf, uses & 1);
        tc_fence_after();
        const int row = m0 + mb * 128 + row_in_blk;
        const bool row_ok = row < g.M;
        const uint32_t tacc = tmem + buf * 256 + ((uint32_t)(q * 32) << 16);
        if (EPI == GEMM_EPI_STORE) {
          uint16_t* crow = g.C + (size_t)row * g.ldc + n0;
          const uint16_t* rrow = g.R ? g.R + (size_t)row * g.ldc + n0 : nullptr;
#pragma unroll 1
          for (int c = 0; c < kBN / 32; ++c) {
            float v[32];
            tmem_ld32(v, tacc + c * 32);
            tmem_ld_wait();
            if (c == kBN / 32 - 1) {
              tc_fence_before();
              mbar_arrive(bar(BAR_ACC_EMPTY + buf));       // the accumulator is in registers
            }
            if (row_ok) {
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                const int col = n0 + c * 32 + i * 8;
                if (col < g.N) {
                  if (rrow) {
                    float r[8];
                    unpack8(*reinterpret_cast<const uint4*>(rrow + c * 32 + i * 8), r);
#pragma unroll
                    for (int e = 0; e < 8; ++e) v[i * 8 + e] += r[e];
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
#pragma unroll 1
          for (int h = 0; h < 2; ++h) {
            const int col0 = n0 + h * 128;
            const bool rotate = col0 < g.q_cols + g.kv_cols;
            uint16_t* dst = col0 < g.q_cols ? g.C + (size_t)row * g.q_cols + col0
                            : rotate        ? g.C2 + (size_t)row * g.kv_cols + (col0 - g.q_cols)
                                            : g.C3 + (size_t)row * g.kv_cols + (col0 - g.q_cols - g.kv_cols);
#pragma unroll 1
            for (int c = 0; c < 2; ++c) {
              float lo[32], hi[32];
              tmem_ld32(lo, tacc + h * 128 + c * 32);
              tmem_ld32(hi, tacc + h * 128 + 64 + c * 32);
              tmem_ld_wait();
              if (h == 1 && c == 1) {
                tc_fence_before();
                mbar_arrive(bar(BAR_ACC_EMPTY + buf));
              }
              if (row_ok && col0 < g.N) {
                if (rotate) {
#pragma unroll
                  for (int i = 0; i < 32; ++i) {
                    const float2 t2 = cs[c * 32 + i];     // (cos, sin)
                    const float a = lo[i], b = hi[i];
                    lo[i] = a * t2.x - b * t2.y;
                    hi[i] = b * t2.x + a * t2.y;
                  }
                }
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  *reinterpret_cast<uint4*>(dst + c * 32 + i * 8) = pack8(lo + i * 8);
                  *reinterpret_cast<uint4*>(dst + 64 + c * 32 + i * 8) = pack8(hi + i * 8);
                }
              }
            }
          }
        } else {
          // GEMM_EPI_SILU_MUL: the weight rows of a tile are 128 gate rows followed by the 128 up rows of
          // the same intermediate features; out[row][n0 / 2 + i] = silu(gate_i) * up_i, both
          // rounded to bf16 first (they are bf16 tensors of the layer's definition).
          uint16_t* crow = g.C + (size_t)row * g.ldc + n0 / 2;
#pragma unroll 1
          for (int c = 0; c < 4; ++c) {
            float gt[32], up[32];
            tmem_ld32(gt, tacc + c * 32);
            tmem_ld32(up, tacc + 128 + c * 32);
            tmem_ld_wait();
            if (c == 3) {
              tc_fence_before();
              mbar_arrive(bar(BAR_ACC_EMPTY + buf));
            }
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
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 1) tmem_dealloc(tmem, 512);
}

// ---------------------------------------------------------------------------------- split-K kernel
// For products with few tiles (a decode batch: one 128-row block of tokens). Such a product is bound
// by the HBM traffic of its weights, but with one CTA per 128 x 256 tile only 16-24 of the 148 SMs
// pull on HBM (hidden 4096: 37 us for the 50 MB of QKV weights, 1.35 TB/s). Here a cluster of S
// CTAs shares a tile: CTA r multiplies K blocks [kb r / S, kb (r+1) / S), lays its fp32 accumulator
// into its own shared memory (the operand stages are free by then), and after a cluster barrier the
// S CTAs add up the S accumulators, each a share of the elements, in the order r = 0 .. S-1
// (through distributed shared memory: nothing goes to global memory, no workspace, and the result
// does not depend on timing), apply the epilogue and write it.
__device__ __forceinline__ uint32_t mapa(uint32_t addr, uint32_t rank) {
  uint32_t r;
  asm volatile("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ float4 ld_cluster4(uint32_t addr) {
  float4 v;
  asm volatile("ld.shared::cluster.v4.f32 {%0,%1,%2,%3}, [%4];\n" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(addr) : "memory");
  return v;
}
__device__ __forceinline__ void cluster_sync() {
  asm volatile("barrier.cluster.arrive.release;\nbarrier.cluster.wait.acquire;\n" ::: "memory");
}

constexpr int kSplitStages = 4, kSplitStageBytes = kABytes + kBBytes;
constexpr int kSplitSmem = kSplitStages * kSplitStageBytes + (2 * kSplitStages + 1) * 8 + 16 + 1024;
static_assert(128 * kBN * 4 <= kSplitStages * kSplitStageBytes, "the accumulator image takes the place of the operand stages");
// 16-byte chunk `c` of row `row` of the accumulator image; the XOR spreads a column of rows over the banks
__device__ __forceinline__ uint32_t image_off(int row, int c) { return (uint32_t)(row * (kBN * 4) + ((c ^ (row & 7)) << 4)); }

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
  if (warp == 1) tmem_alloc(base + kOffMisc, 256);
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
  const int m0 = (t % m_tiles) * 128, n0 = (t / m_tiles) * kBN;
  const int rows = min(128, g.M - m0);
  const int k_blocks = (g.K + kBK - 1) / kBK;
  const int kb0 = k_blocks * rank / split, kb1 = k_blocks * (rank + 1) / split;   // never empty: split <= k_blocks

  if (warp == 0) {
    if (lane == 0) {
      tma_prefetch_desc(&a_map);
      tma_prefetch_desc(&b_map);
      // the weights do not come from the kernel in front of this one: bring the first of them into L2 meanwhile
      for (int kb = kb0; kb < min(kb1, kb0 + 2 * kSplitStages); ++kb) tma_prefetch_2d(&b_map, kb * kBK, n0);
      pdl_wait();
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
        mma_ss(tmem, a_desc + (uint64_t)(ks * 2), b_desc + (uint64_t)(ks * 2), kIdesc, (it > 0 || ks > 0) ? 1u : 0u, issue);
      tc_commit(bar(BAR_EMPTY + st), issue);
    }
    if (!dead) tc_commit(bar(BAR_ACC), issue);
  } else {
    // accumulator -> image in shared memory; every operand stage has been read once the barrier completes
    if (!mbar_wait(bar(BAR_ACC), 0, misc[1] ? 2000 : g.wait_cycles)) give_up();
    tc_fence_after();
    const int q = warp & 3;                                // the TMEM lanes this warp can reach
    const int row = q * 32 + lane;
    if (q * 32 < rows && misc[1] == 0) {
#pragma unroll 1
      for (int c = 0; c < kBN / 32; ++c) {
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
  __syncwarp();
  cluster_sync();                  // the images are complete
  pdl_wait();                      // every thread reads the residual or the positions below
  // one item = 8 columns of a row (STORE), or 8 columns and their partners 64 (ROPE) or 128 (SILU_MUL) further on
  constexpr int kItems = EPI == GEMM_EPI_STORE ? 32 : 16;
  auto sum8 = [&](int row, int col, float (&v)[8]) {
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = 0.f;
#pragma unroll 4
    for (int r = 0; r < split; ++r) {
      const uint32_t img = mapa(base, (uint32_t)r);
      const float4 x = ld_cluster4(img + image_off(row, col / 4)), y = ld_cluster4(img + image_off(row, col / 4 + 1));
      v[0] += x.x; v[1] += x.y; v[2] += x.z; v[3] += x.w;
      v[4] += y.x; v[5] += y.y; v[6] += y.z; v[7] += y.w;
    }
  };
  for (int i = rank * kGemmThreads + tid; i < rows * kItems; i += split * kGemmThreads) {
    const int r = i / kItems, ch = i % kItems, row = m0 + r;
    if (EPI == GEMM_EPI_STORE) {
      const int col = n0 + ch * 8;
      if (col >= g.N) continue;
      float v[8];
      sum8(r, ch * 8, v);
      if (g.R) {
        float x[8];
        unpack8(*reinterpret_cast<const uint4*>(g.R + (size_t)row * g.ldc + col), x);
#pragma unroll
        for (int e = 0; e < 8; ++e) v[e] += x[e];
      }
      *reinterpret_cast<uint4*>(g.C + (size_t)row * g.ldc + col) = pack8(v);
    } else if (EPI == GEMM_EPI_ROPE) {
      const int h = ch / 8, c = (ch % 8) * 8, col0 = n0 + h * 128;
      if (col0 >= g.N) continue;
      float lo[8], hi[8];
      sum8(r, h * 128 + c, lo);
      sum8(r, h * 128 + 64 + c, hi);
      rope8(g, row, col0, c, lo, hi);
    } else {
      if (n0 >= g.N) continue;
      float gt[8], up[8];
      sum8(r, ch * 8, gt);
      sum8(r, 128 + ch * 8, up);
      silu_mul8(gt, up);
      *reinterpret_cast<uint4*>(g.C + (size_t)row * g.ldc + n0 / 2 + ch * 8) = pack8(gt);
    }
  }
  tc_fence_before();
  cluster_sync();                  // no CTA leaves while another one reads its image
  if (warp == 1) tmem_dealloc(tmem, 256);
}

template <int EPI>
cudaError_t launch_split_t(const GemmArgs& g, const CUtensorMap& a_map, const CUtensorMap& b_map, int split, cudaStream_t stream) {
  cudaError_t e = cudaFuncSetAttribute(gemm_split_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSplitSmem);
  if (e != cudaSuccess) return e;
  const int tiles = ((g.M + 127) / 128) * ((g.N + kBN - 1) / kBN);
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(tiles * split);
  cfg.blockDim = dim3(kGemmThreads);
  cfg.dynamicSmemBytes = kSplitSmem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim = {(unsigned)split, 1, 1};
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, gemm_split_kernel<EPI>, g, a_map, b_map, split);
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
  attr[0].val.clusterDim = {(unsigned)split, 1, 1};
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

template <int TILE_M, int EPI>
cudaError_t launch_t(const GemmArgs& g, const CUtensorMap& a_map, const CUtensorMap& b_map, int n_sms, cudaStream_t stream) {
  constexpr int kStageBytes = (TILE_M / 128) * kABytes + kBBytes;
  constexpr int kStages = TILE_M == 128 ? 4 : 3;
  const size_t smem = (size_t)kStages * kStageBytes + (2 * kStages + 4) * 8 + 16 + 1024;
  cudaError_t e = cudaFuncSetAttribute(gemm_kernel<TILE_M, EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const int m_tiles = (g.M + TILE_M - 1) / TILE_M, n_tiles = (g.N + kBN - 1) / kBN;
  const int grid = std::min(n_sms, m_tiles * n_tiles);
  return launch_pdl(gemm_kernel<TILE_M, EPI>, dim3(grid), dim3(kGemmThreads), smem, stream, g, a_map, b_map);
}

}  // namespace

// Cost of a launch in us. Without a split: waves x K blocks, the 256-row tile being cheaper per flop
// (it fetches a third fewer operand bytes) but coarser in the wave count. With a split: the K blocks
// of the longest share and the merge; only where all clusters run at once. A K block takes a CTA
// kBlockUs, or as long as HBM needs for the weight blocks that are in flight at that moment. Measured
// (8B-shaped projections, weights not in L2, one CTA per tile -> split): 64 rows QKV 35.2 -> 18.5 us,
// output 34.6 -> 17.2, down 96.7 -> 35.2; 256 rows QKV 36.8 -> 32.9, output 35.5 -> 22.4, down 96.5
// -> 42.0; 512 rows output 35.3 -> 31.7, down 96.2 -> 66.9. The merge takes 2-3 us for one row and
// ~8 us for 128 rows. Gate/up (112 tiles) is not split: its tiles already fill three quarters of the SMs.
GemmPlan gemm_plan(int M, int N, int K, int n_sms, bool tall) {
  constexpr double kBlockUs = 0.42, kHbmBytesPerUs = 6.2e6;
  const double merge_us = 2.5 + 0.045 * std::min(M, 128);
  const int n_tiles = (N + kBN - 1) / kBN, m128 = (M + 127) / 128, m256 = (M + 255) / 256;
  const int kb = (K + kBK - 1) / kBK;
  auto block_us = [&](int ctas, int m_tiles, double tile_cost) {
    return std::max(kBlockUs * tile_cost, (double)std::min(ctas, n_sms) / m_tiles * kBBytes / kHbmBytesPerUs);
  };
  auto waves = [&](int tiles) { return (tiles + n_sms - 1) / n_sms; };
  GemmPlan best = {128, 1};
  double cost = (double)waves(m128 * n_tiles) * kb * block_us(m128 * n_tiles, m128, 1.0);
  if (tall) {
    const double c = (double)waves(m256 * n_tiles) * kb * block_us(m256 * n_tiles, m256, 2.0 * 0.9);
    if (c < cost) {
      cost = c;
      best = {256, 1};
    }
  }
  for (int s = 2; s <= std::min(kMaxSplit, kb); ++s) {
    if (m128 * n_tiles * s > n_sms || m128 * n_tiles * s > split_slots(s)) break;
    const double c = (double)((kb + s - 1) / s) * block_us(m128 * n_tiles * s, m128, 1.0) + merge_us;
    if (c < cost * 0.98) {
      cost = c;
      best = {128, s};
    }
  }
  return best;
}

cudaError_t launch_gemm(const GemmArgs& g, const CUtensorMap& a_map, const CUtensorMap& b_map, GemmPlan plan, int n_sms,
                        cudaStream_t stream) {
  if (g.M <= 0 || g.N <= 0) return cudaSuccess;
  if (plan.split > 1) {
    if (g.epi == GEMM_EPI_ROPE) return launch_split_t<GEMM_EPI_ROPE>(g, a_map, b_map, plan.split, stream);
    if (g.epi == GEMM_EPI_SILU_MUL) return launch_split_t<GEMM_EPI_SILU_MUL>(g, a_map, b_map, plan.split, stream);
    return launch_split_t<GEMM_EPI_STORE>(g, a_map, b_map, plan.split, stream);
  }
  if (g.epi == GEMM_EPI_ROPE) return launch_t<128, GEMM_EPI_ROPE>(g, a_map, b_map, n_sms, stream);
  if (g.epi == GEMM_EPI_SILU_MUL)
    return plan.tile_m == 256 ? launch_t<256, GEMM_EPI_SILU_MUL>(g, a_map, b_map, n_sms, stream)
                              : launch_t<128, GEMM_EPI_SILU_MUL>(g, a_map, b_map, n_sms, stream);
  return plan.tile_m == 256 ? launch_t<256, GEMM_EPI_STORE>(g, a_map, b_map, n_sms, stream)
                            : launch_t<128, GEMM_EPI_STORE>(g, a_map, b_map, n_sms, stream);
}

}  // namespace ts
