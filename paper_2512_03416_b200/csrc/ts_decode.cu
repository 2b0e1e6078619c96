// Stand-alone split-KV flash-decode kernel for the 1-token rows (sm_100a): one persistent CTA
// per SM running dec::decode_units and its scheduler (ts_decode_body.h) over all decode units of the step. The schedulers
// also merge the rows that were split.
// The units also append the rows' new K/V.
#include "ts_decode_body.h"

namespace ts {
namespace {

using dec::kDecThreads;

template <int D, int NH, int STAGES, int W>
__global__ void __launch_bounds__(kDecThreads + 32, 1)
decode_kernel(const __grid_constant__ StepParams<W> params, const __grid_constant__ CUtensorMap kv_map) {
  const StepDevice& s = params.s;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t base = (smem_u32(smem_raw) + 1023u) & ~1023u;
  unsigned char* smem = smem_raw + (base - smem_u32(smem_raw));
  pdl_launch_dependents();
  if (threadIdx.x == 0) tma_prefetch_desc(&kv_map);
  // Where the step's metadata are launch parameters, the barriers and each CTA's first unit are set up before the
  // wait, and only the pool, the tables and Q are read behind it. Uploaded metadata (larger steps) and those of
  // a planning kernel are read behind the wait, and all of the set-up stays there too.
  // (Device time of a step, prepared steps back to back, with everything behind the wait and so, us: four rows of ~1500
  // keys 10.50 / 9.74, one row of 4000 10.31 / 9.46, eight of ~1500 17.5 / 16.8, 64 rows 126.7 / 126.8. A call that
  // marshals its rows and waits is bound by the host for so few.)
  auto ready = [&]() { pdl_wait(); };
  if (s.meta) ready();
  if (threadIdx.x < kDecThreads) {
    dec::decode_units<D, NH, STAGES, true>(s, &kv_map, smem, base, ready);
  } else {
    dec::decode_schedule<D, STAGES, true>(s, smem, base, blockIdx.x, gridDim.x, ready);
    if (threadIdx.x == kDecThreads) {
      // the last scheduler to get here puts the queue back to zero for the next launch
      __threadfence();
      if (atomicAdd(s.pf_queue + 4, 1) == (int)gridDim.x - 1) {
        s.pf_queue[3] = 0;
        s.pf_queue[4] = 0;
      }
    }
  }
}

template <int D, int NH, int STAGES, int W>
cudaError_t launch_decode_w(const StepDevice& s, const CUtensorMap& map, int n_sms, cudaStream_t stream) {
  const int G = s.Hq / s.Hkv;
  const size_t smem = 1024 + dec::decode_smem_bytes<D, STAGES>(G);
  cudaError_t e = cudaFuncSetAttribute(decode_kernel<D, NH, STAGES, W>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long long units = (long long)(s.n_items - s.n_prefill_items) * s.Hkv;
  const int grid = (int)(units < n_sms ? units : n_sms);
  StepParams<W> params;
  fill_params(s, &params);
  return launch_pdl(decode_kernel<D, NH, STAGES, W>, dim3(grid), dim3(kDecThreads + 32), smem, stream, params, map);
}
template <int D, int NH, int STAGES>
cudaError_t launch_decode_t(const StepDevice& s, const CUtensorMap& map, int n_sms, cudaStream_t stream) {
  if (s.n_words <= kInlineWords) return launch_decode_w<D, NH, STAGES, kInlineWords>(s, map, n_sms, stream);
  if constexpr (D == 128 && NH == 1)
    return s.n_words <= kInlineWordsMid ? launch_decode_w<D, NH, STAGES, kInlineWordsMid>(s, map, n_sms, stream)
                                        : launch_decode_w<D, NH, STAGES, kInlineWordsMax>(s, map, n_sms, stream);
  return cudaErrorInvalidValue;
}

}  // namespace

cudaError_t launch_decode(const StepDevice& s, const CUtensorMap& kv_map, int n_sms, cudaStream_t stream) {
  if (s.n_items - s.n_prefill_items <= 0) return cudaSuccess;
  const int G = s.Hq / s.Hkv;
  if (s.D == 128) {
    return G <= 8 ? launch_decode_t<128, 1, 3>(s, kv_map, n_sms, stream)
                  : launch_decode_t<128, 2, 2>(s, kv_map, n_sms, stream);
  }
  return G <= 8 ? launch_decode_t<64, 1, 4>(s, kv_map, n_sms, stream)
                : launch_decode_t<64, 2, 4>(s, kv_map, n_sms, stream);
}

}  // namespace ts
