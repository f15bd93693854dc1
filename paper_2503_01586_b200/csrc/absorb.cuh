// Query preparation (absorb.cu has the description): shared by the stand-alone kernel and by the
// kernel that prepares a whole decode step.
#pragma once

#include "common.cuh"

constexpr int kAbsorbThreads = 256;    // 8 warps x 16 coordinates
constexpr int kAbsorbCoords = 128;
constexpr int kAbsorbPitch = kAbsorbCoords + 8;   // slab row pitch: 16 bytes of padding keep ldmatrix free of bank conflicts
constexpr int kAbsorbMaxTiles = 4;     // 16-row query tiles per block

struct AbsorbArgs {
  const bf16* q;
  const int32_t* q_pos;
  int B;
  const bf16* WukT;
  const int32_t* qdims;
  const uint16_t* qkeep;
  const int32_t* idx;
  const float2* cs;
  bf16* q_rope;
  bf16* q_abs;
  int n_h, d_h, r, kw, max_pos;      // kw: width of the latent the scores read
  int row0;                          // the first row's index in the call, for reports
  int32_t* status;
};

// Query RoPE of one head (every sequence).
__device__ __forceinline__ void absorb_rope(const AbsorbArgs& a, int h) {
  const int32_t* dims = a.qdims + (size_t)h * a.d_h;
  ekv_pdl_wait();
  for (int e = threadIdx.x; e < a.B * a.r; e += blockDim.x) {
    const int b = e / a.r, j = e % a.r;
    int p = a.q_pos[b];
    if (p < 0 || p >= a.max_pos) {
      ekv_record(a.status, ELITEKV_ERR_BAD_POSITION, a.row0 + b, p);
      p = 0;
    }
    const float2 w = a.cs[(size_t)p * (a.d_h / 2) + a.idx[h * a.r + j]];
    const bf16* qq = a.q + ((size_t)b * a.n_h + h) * a.d_h;
    const float x0 = __bfloat162float(qq[dims[2 * j]]), x1 = __bfloat162float(qq[dims[2 * j + 1]]);
    const float y0 = __fsub_rn(__fmul_rn(x0, w.x), __fmul_rn(x1, w.y));
    const float y1 = __fadd_rn(__fmul_rn(x0, w.y), __fmul_rn(x1, w.x));
    bf162* dst = (bf162*)(a.q_rope + ((size_t)b * a.n_h + h) * 2 * a.r + 2 * j);
    *dst = __floats2bfloat162_rn(y0, y1);
  }
}

// Absorbed queries of one head, 128 latent coordinates from k0 on, sequences [b0, b0 + 16 MT).  The
// product runs over all d_h query dims in their own order: the weight row of a dim goes to the
// shared-memory row of that dim, and the rows of the rotated (elite) dims are zeros.  Those dims of the
// queries are zeros too (a zero weight alone would turn an infinite one into NaN).
template <int MT>
__device__ __forceinline__ void absorb_block(const AbsorbArgs& a, int h, int k0, int b0, unsigned char* smem_b) {
  const int dn = a.d_h - 2 * a.r;
  const int kpad = (a.d_h + 15) & ~15;               // K of the product, zero-padded to 16
  const int qpitch = kpad + 8;                       // row pitch of the query tile (bank spread)
  bf16* s_w = (bf16*)smem_b;                         // [kpad][128 + 8] weight slab
  bf16* s_q = s_w + (size_t)kpad * kAbsorbPitch;     // [16 MT][qpitch] queries; then [16 MT][128 + 8] results
  const int32_t* dims = a.qdims + (size_t)h * a.d_h;
  const uint16_t* keep = a.qkeep + (size_t)h * a.d_h;      // all ones at un-rotated dims
  const int kw = min(kAbsorbCoords, a.kw - k0);      // coordinates of this slab (a multiple of 8)
  const int nb = min(16 * MT, a.B - b0);
  // weights and tables belong to the layer: fetched while earlier kernels of the stream still run.
  // Sixteen threads copy a row, 128 rows are looked up at a time: 2.4 us from the block's start.  (One bulk
  // copy per row, issued by a single warp with a look-up in front of each, took 5.3 us.)
  {
    const bf16* src = a.WukT + (size_t)h * dn * a.kw + k0;
    const int v = threadIdx.x % 16 * 8;
    for (int i0 = threadIdx.x / 16; i0 < dn; i0 += 128) {
      int row[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) row[k] = i0 + 16 * k < dn && v < kw ? __ldg(dims + 2 * a.r + i0 + 16 * k) : -1;
#pragma unroll
      for (int k = 0; k < 8; ++k)
        if (row[k] >= 0) cp_async16(s_w + (size_t)row[k] * kAbsorbPitch + v, src + (size_t)(i0 + 16 * k) * a.kw + v);
    }
    cp_async_commit();
  }
  {
    // the elite dims' rows of the slab, and the rows past d_h (K padding)
    const int n_zero = 2 * a.r + kpad - a.d_h;
    for (int e = threadIdx.x; e < n_zero * (kAbsorbCoords / 8); e += kAbsorbThreads) {
      const int i = e / (kAbsorbCoords / 8);
      const int row = i < 2 * a.r ? __ldg(dims + i) : a.d_h + i - 2 * a.r;
      *(uint4*)(s_w + (size_t)row * kAbsorbPitch + (e % (kAbsorbCoords / 8)) * 8) = make_uint4(0, 0, 0, 0);
    }
  }
  // a thread's 16-byte units of the queries lie in one column of the rows: one mask for all of them
  const int v8 = kpad / 8, bb0 = threadIdx.x / v8, v = threadIdx.x - bb0 * v8, step = kAbsorbThreads / v8;
  const bool vec = (a.d_h & 7) == 0, in = vec && bb0 < step && v * 8 < a.d_h;
  const uint4 mask = in ? __ldg((const uint4*)keep + v) : make_uint4(0, 0, 0, 0);
  ekv_pdl_wait();
  // the queries, 16 bytes a load where rows are whole 16-byte units; padding and missing rows are zeros
  if (vec) {
    const bf16* src = a.q + ((size_t)b0 * a.n_h + h) * a.d_h + v * 8;
    for (int bb = bb0 < step ? bb0 : 16 * MT; bb < 16 * MT; bb += MT * step) {
      uint4 raw[MT];
#pragma unroll
      for (int k = 0; k < MT; ++k)
        raw[k] = in && bb + k * step < nb ? *(const uint4*)(src + (size_t)(bb + k * step) * a.n_h * a.d_h) : make_uint4(0, 0, 0, 0);
#pragma unroll
      for (int k = 0; k < MT; ++k)
        if (bb + k * step < 16 * MT)
          *(uint4*)(s_q + (bb + k * step) * qpitch + v * 8) =
              make_uint4(raw[k].x & mask.x, raw[k].y & mask.y, raw[k].z & mask.z, raw[k].w & mask.w);
    }
  } else {
    for (int e = threadIdx.x; e < 16 * MT * kpad; e += kAbsorbThreads) {
      const int bb = e / kpad, i = e - bb * kpad;
      const bool there = bb < nb && i < a.d_h;
      const uint16_t x = there ? ((const uint16_t*)a.q)[((size_t)(b0 + bb) * a.n_h + h) * a.d_h + i] : (uint16_t)0;
      ((uint16_t*)s_q)[bb * qpitch + i] = there ? (uint16_t)(x & __ldg(keep + i)) : (uint16_t)0;
    }
  }
  cp_async_wait<0>();
  __syncthreads();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = warp * 16;                          // first coordinate (inside the slab) of this warp
  float acc[MT][2][4] = {};
  if (n0 < kw) {
    for (int kk = 0; kk < kpad; kk += 16) {
      uint32_t w[4];
      ldmatrix_x4_trans(w, s_w + (size_t)(kk + (lane & 15)) * kAbsorbPitch + n0 + (lane >> 4) * 8);
#pragma unroll
      for (int mt = 0; mt < MT; ++mt) {
        uint32_t x[4];
        ldmatrix_x4(x, s_q + (16 * mt + (lane & 15)) * qpitch + kk + (lane >> 4) * 8);
        mma_bf16_16816(acc[mt][0], x, w[0], w[1]);
        mma_bf16_16816(acc[mt][1], x, w[2], w[3]);
      }
    }
  }
  __syncthreads();
  // through shared memory, so that whole rows of 256 bytes are written
  const int g = lane >> 2, t = lane & 3;
#pragma unroll
  for (int mt = 0; mt < MT; ++mt)
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      bf16* dst = s_q + (16 * mt + g) * kAbsorbPitch + n0 + nt * 8 + 2 * t;
      *(bf162*)dst = __floats2bfloat162_rn(acc[mt][nt][0], acc[mt][nt][1]);
      *(bf162*)(dst + 8 * kAbsorbPitch) = __floats2bfloat162_rn(acc[mt][nt][2], acc[mt][nt][3]);
    }
  __syncthreads();
#pragma unroll MT
  for (int e = threadIdx.x; e < 16 * MT * (kAbsorbCoords / 8); e += kAbsorbThreads) {
    const int bb = e / (kAbsorbCoords / 8), v = e % (kAbsorbCoords / 8);
    if (bb < nb && v * 8 < kw)
      *(uint4*)(a.q_abs + ((size_t)(b0 + bb) * a.n_h + h) * a.kw + k0 + v * 8) = *(const uint4*)(s_q + bb * kAbsorbPitch + v * 8);
  }
}

// 16-row tiles per block (1, 2 or 4), blocks along the latent and along the sequences, shared memory
struct AbsorbShape {
  int mt, slices, groups;
  size_t smem;
};
inline AbsorbShape absorb_shape(const elitekv_layer* L, int B) {
  AbsorbShape s;
  s.mt = B <= 16 ? 1 : B <= 32 ? 2 : kAbsorbMaxTiles;
  s.slices = (L->kw + kAbsorbCoords - 1) / kAbsorbCoords;
  s.groups = (B + 16 * s.mt - 1) / (16 * s.mt);
  const size_t kpad = (size_t)((L->d_h + 15) & ~15);
  const size_t pitch = kpad + 8 > (size_t)kAbsorbPitch ? kpad + 8 : kAbsorbPitch;
  s.smem = sizeof(bf16) * (kpad * kAbsorbPitch + 16 * s.mt * pitch) + 16;
  return s;
}
inline bool absorb_ok(const elitekv_layer* L, const AbsorbShape& s) {
  return (int)s.smem <= L->smem_optin && L->kw % 8 == 0;
}
// rows [b0, b0 + B) of the call's arrays
inline AbsorbArgs absorb_args(const elitekv_layer* L, const void* q, const int32_t* q_pos, int b0, int B, void* q_rope, void* q_abs) {
  const size_t at = (size_t)b0 * L->n_h;
  return AbsorbArgs{(const bf16*)q + at * L->d_h, q_pos + b0, B, L->d_WukT, L->d_qdims, L->d_qkeep, L->d_idx, L->d_cs,
                    (bf16*)q_rope + at * 2 * L->r, (bf16*)q_abs + at * L->kw, L->n_h, L->d_h, L->r, L->kw, L->max_pos, b0, L->d_status};
}
