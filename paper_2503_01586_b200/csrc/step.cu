// Front end of a decode step in one launch: cache append, work plan and query preparation.
//
// The three depend on the step's inputs only, and each is a few microseconds of latency (dependent
// look-ups, one trip for the weights).  As separate launches on two streams they cost 13-20 us before
// the attention kernel could start, most of it launch gaps, and the events that joined the streams cut
// the chain of programmatic dependent launches.  Here they are blocks of one grid: block 0 the plan, then
// the appended tokens, the query RoPE of a head each, and the (head, 128 coordinates, sequences)
// blocks of the absorption, whose weight slabs are fetched before the dependency wait.
// From the release of the grid by the previous step's combine to its end: one sequence 2.8 us, 7B 75 % B16
// 3.0 (the plan; the query preparation 2.6 and 2.9); while the plan was a thread per sequence at every size 4.0 and 5.0,
// ragged B64 7.0, 13B B32 5.3, 50 % B32 9.5 (11 to 12 us for the last three while a single warp fetched
// the weights and registers kept blocks waiting for a second wave; the 50 % shape's 833 blocks still do not
// all fit).  As separate launches: 16 us at B16, 21 at ragged B64.
#include "absorb.cuh"
#include "append.cuh"
#include "plan.cuh"

namespace {

static_assert(kPlanThreads == kAbsorbThreads, "one block size for every part");

template <int MT>
__global__ void __launch_bounds__(kAbsorbThreads, MT == kAbsorbMaxTiles ? 4 : 5)     // what shared memory holds
step_prep_kernel(const AbsorbArgs q, const AppendArgs t, const PlanArgs p, int n_append, int vec, int slices) {
  extern __shared__ __align__(16) unsigned char smem_b[];
  ekv_pdl_trigger();      // the attention kernel waits for this grid's completion itself
  int blk = blockIdx.x;
  if (blk != 0) {      // (the plan last in the code: 7B 75 % 8 x 1500 30.7 us a step, 31.3 with it first)
    blk -= 1;
    if (blk < n_append) {
      ekv_pdl_wait();
      if (vec) append_tokens<true>(t, blk, n_append);
      else append_tokens<false>(t, blk, n_append);
      return;
    }
    blk -= n_append;
    if (blk < q.n_h) {
      absorb_rope(q, blk);
      return;
    }
    blk -= q.n_h;
    const int h = blk % q.n_h, s = blk / q.n_h;
    absorb_block<MT>(q, h, s % slices * kAbsorbCoords, s / slices * 16 * MT, smem_b);
    return;
  }
  plan_behind_wait<false>(p, *(PlanShared<int>*)smem_b);
}

}  // namespace

int ekv_launch_step_prep(const elitekv_layer* L, const elitekv_cache* cache, const CacheView& cv, const void* k_e,
                         const void* c, const int32_t* seq_id, const int32_t* pos, const void* q, int B, void* q_rope,
                         void* q_abs, const PlanArgs& plan, cudaStream_t st) {
  const AbsorbShape s = absorb_shape(L, B);
  if (!absorb_ok(L, s)) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  if (!plan_narrow(plan)) {      // (lengths that only pages shared by many sequences can have)
    int rc = ekv_launch_append(L, cache, cv, k_e, c, seq_id, pos, B, st);
    if (rc == ELITEKV_OK) rc = ekv_launch_absorb(L, q, pos, B, q_rope, q_abs, st);
    return rc == ELITEKV_OK ? ekv_launch_plan(plan, st) : rc;
  }
  const AbsorbArgs a = absorb_args(L, q, pos, 0, B, q_rope, q_abs);
  const AppendArgs t = append_args(L, cache, cv, k_e, c, seq_id, pos, B);
  const int n_append = B < L->sm_count ? B : L->sm_count;      // a block per token; more tokens go round
  const int grid = 1 + n_append + L->n_h * (1 + s.slices * s.groups);
  const size_t smem = s.smem > sizeof(PlanShared<int>) ? s.smem : sizeof(PlanShared<int>);
  auto launch = [&](auto kern) -> int {
    EKV_CUDA_OK(ekv_allow_smem(kern, smem));
    EKV_CUDA_OK(ekv_launch_pdl(kern, dim3((unsigned)grid), dim3(kAbsorbThreads), smem, st, a, t, plan, n_append,
                               (int)append_vec_ok(L), s.slices));
    EKV_CUDA_OK(cudaGetLastError());
    return ELITEKV_OK;
  };
  return s.mt == 1   ? launch(step_prep_kernel<1>)
         : s.mt == 2 ? launch(step_prep_kernel<2>)
                     : launch(step_prep_kernel<4>);
}
