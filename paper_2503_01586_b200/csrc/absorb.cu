// Query preparation: RoPE on the elite chunks of q and absorption of B^k into the query
// (score equation of Section 3.1; Section 5 on folding B^k into the neighbouring product).
//
//   q_rope[b,h,2j:2j+2] = q[b,h,chunk idx[h][j]] . R(q_pos[b] * theta_idx[h][j])
//   q_abs [b,h,k]       = sum_i q_nope[b,h,i] * W_uk[k][h*dn + i]
//
// Grid (n_h, ceil(kw/128) + 1, groups of up to 64 sequences).  A block of the first rows owns one
// head and 128 latent coordinates: it computes the [16..64 x d_h] . [d_h x 128] product with mma.sync
// (m16n8k16, bf16 in, fp32 accumulate; both operands are bf16 already, so the products are exact),
// one warp per 16 coordinates.  The weights come regrouped as [n_h][dn][kw] (kw contiguous); the
// block's slab is copied into shared memory asynchronously.  The blocks of the
// last grid row do the query RoPE (dependent look-ups), off the path of the others.  kw is the
// width of the latent the scores read: the whole latent row, or the key latent d_ck when keys and
// values have latents of their own (S-LRD, Section 3.2).
//
// Bound: latency, not its 11 MB of weights or 0.2 GFLOP.  Slab and dim table belong to the layer, so
// they are fetched before the dependency wait, while earlier kernels of the stream run; behind it
// there is one trip (the queries) before the product.  All rows of a block are taken at once: a
// loop over 16 sequences at a time, each a trip and a gather by dim, took 18 us at 64 rows; a
// two-byte gather of 64 rows straight from memory 28 us; this form 12-16 us.
#include "absorb.cuh"

namespace {

template <int MT>
__global__ void __launch_bounds__(kAbsorbThreads)
absorb_kernel(const AbsorbArgs a) {
  extern __shared__ __align__(16) unsigned char smem_b[];
  ekv_pdl_trigger();      // nothing later in the stream is held up by this kernel's start
  if (blockIdx.y == gridDim.y - 1) {       // last grid row: query RoPE only
    if (blockIdx.z == 0) absorb_rope(a, blockIdx.x);
    else ekv_pdl_wait();
    return;
  }
  absorb_block<MT>(a, blockIdx.x, blockIdx.y * kAbsorbCoords, blockIdx.z * 16 * MT, smem_b);
}

}  // namespace

int ekv_launch_absorb(const elitekv_layer* L, const void* q, const int32_t* q_pos, int B,
                      void* q_rope, void* q_abs, cudaStream_t st) {
  if (B == 0) return ELITEKV_OK;
  const AbsorbShape s = absorb_shape(L, B);
  if (!absorb_ok(L, s)) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  auto launch = [&](auto kern) -> int {
    EKV_CUDA_OK(ekv_allow_smem(kern, s.smem));
    // one launch up to four million rows (a loop over groups in the kernel costs 1024 rows 71 -> 90 us)
    for (int g0 = 0; g0 < s.groups; g0 += kGridZ) {
      const int groups = s.groups - g0 < kGridZ ? s.groups - g0 : kGridZ, b0 = g0 * 16 * s.mt;
      const AbsorbArgs a = absorb_args(L, q, q_pos, b0, B - b0 < groups * 16 * s.mt ? B - b0 : groups * 16 * s.mt, q_rope, q_abs);
      EKV_CUDA_OK(ekv_launch_pdl(kern, dim3(L->n_h, s.slices + 1, groups), dim3(kAbsorbThreads), s.smem, st, a));
    }
    EKV_CUDA_OK(cudaGetLastError());
    return ELITEKV_OK;
  };
  return s.mt == 1 ? launch(absorb_kernel<1>) : s.mt == 2 ? launch(absorb_kernel<2>) : launch(absorb_kernel<4>);
}
