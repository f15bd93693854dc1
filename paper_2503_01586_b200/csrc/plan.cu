// Work plan for the split-K decode kernels: cuts every sequence's token range into pieces of
// near-equal size so that ragged batches keep all SMs busy.  Integer arithmetic only, on
// device-resident lengths, so a decode step never synchronises with the host.  (The paper
// leaves scheduling open; this is the library's load balancer.)
//
// With tiles_b = ceil(len_b / tile), total = sum tiles_b and budget = max_items - B:
//   target   = max(1, ceil(total / budget))            tiles per item
//   pieces_b = ceil(tiles_b / target)                  (sum <= budget + B = max_items)
//   piece j of sequence b covers tiles [tiles_b*j/pieces_b, tiles_b*(j+1)/pieces_b)
#include "plan.cuh"

namespace {

template <class T>
__global__ void __launch_bounds__(kPlanThreads) plan_kernel(const PlanArgs a) {
  __shared__ PlanShared<T> sh;
  plan_behind_wait<true>(a, sh);      // earlier kernels may still read the arrays written here
}

}  // namespace

int ekv_launch_plan(const PlanArgs& a, cudaStream_t st) {
  EKV_CUDA_OK(ekv_launch_pdl(plan_narrow(a) ? plan_kernel<int> : plan_kernel<long long>, dim3(1), dim3(kPlanThreads), 0, st, a));
  EKV_CUDA_OK(cudaGetLastError());
  return ELITEKV_OK;
}

extern "C" int elitekv_plan(const int32_t* seq_lens, int32_t B, int32_t tile_tokens,
                            int32_t max_items, int32_t* items, int32_t* seq_first_item,
                            elitekv_stream_t stream) {
  if (!seq_lens || !items || !seq_first_item || B <= 0 || tile_tokens <= 0 || max_items <= B)
    return ELITEKV_ERR_INVALID_ARG;
  if ((uintptr_t)items & 15) return ELITEKV_ERR_INVALID_ARG;
  return ekv_launch_plan(PlanArgs{seq_lens, B, tile_tokens, 0, max_items, items, seq_first_item, nullptr, nullptr, 0,
                                  0x7fffffffLL, nullptr, 0, nullptr}, (cudaStream_t)stream);
}

extern "C" int elitekv_plan_workers(const int32_t* seq_lens, int32_t B, int32_t tile_tokens,
                                    int32_t n_workers, int32_t item_overhead_tiles, int32_t max_items,
                                    int32_t* items, int32_t* seq_first_item, int32_t* worker_first,
                                    elitekv_stream_t stream) {
  if (!seq_lens || !items || !seq_first_item || !worker_first || B <= 0 || tile_tokens <= 0 ||
      n_workers <= 0 || max_items < B + n_workers || item_overhead_tiles < 0 || item_overhead_tiles > 64)
    return ELITEKV_ERR_INVALID_ARG;
  if ((uintptr_t)items & 15) return ELITEKV_ERR_INVALID_ARG;
  return ekv_launch_plan(PlanArgs{seq_lens, B, tile_tokens, n_workers, max_items, items, seq_first_item, worker_first,
                                  nullptr, 0, 0x7fffffffLL, nullptr, item_overhead_tiles, nullptr}, (cudaStream_t)stream);
}
