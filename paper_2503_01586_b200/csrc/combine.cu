// Split combine + value up-projection.
//
// Each plan item left (m_s, l_s, acc_s[d_c]) per head, with m in base-2 log units.  For
// sequence b and head h (items s of b):
//   M = max_s m_s,  L = sum_s l_s 2^(m_s - M),  o_lat = sum_s acc_s 2^(m_s - M) / L
//   o[b,h,:] = o_lat . W_uv[:, h*d_h:(h+1)*d_h]        (B^v folded outwards, Section 5;
//                                                      V = c W_uv of Section 3.2)
//
// Fast kernel (d_h = 128, d_c % 128 == 0): grid (n_h, d_c/128, groups of 16 rows; a row is a
// sequence, or a query row of one).  A block stages W_uv's [128 x 128] sub-block of its head and
// latent slice in shared memory, merges the items' partial outputs of its slice (16-byte loads,
// weights 2^(m_s-M)/L) and multiplies.  The d_c/128 slice results of a head are written to
// scratch; the block that finishes last for that (head, group) adds them in a fixed order and
// writes bf16, so the result does not depend on scheduling.
//
// Bound: the latency of its dependent trips to L2 (a few MB to tens of MB move in ~10 us).  So
// groups are blocks of their own and not a loop (a [128 x 128] weight block read again from L2
// costs less than another round of trips), a warp takes its two rows from the statistics to the
// merged result without a block barrier, and the first partial results are requested together
// with the statistics.  Time from the end of the split-K kernel to the end of this one, against the
// form that looped over groups with a barrier per step: 7B 75 % B16 17 -> 11 us, ragged B64 61 -> 30,
// 13B B32 44 -> 26, 50 % B32 50 -> 35, 87.5 % B32 33 -> 12, four rows x B16 36 -> 27.
//
// Generic kernel: any even d_h <= 512, any d_c; block per (head, 8 sequences).
//
// With several query rows per sequence the partial results are [item][row][head]; every row uses
// its head's columns of W_uv.
//
// With separated latents (S-LRD) the partial outputs span the value latent only; `d_c` below is
// then d_cv and W_uv is B^v_S.
#include "common.cuh"

namespace {

// ------------------------------------------------------------------ fast path
constexpr int kFB = 16;          // rows (sequence, query row) per block
constexpr int kFK = 128;         // latent slice
constexpr int kFD = 128;         // head dim
constexpr int kFThreads = 256;
constexpr int kFPitch = kFD + 8; // shared-memory row pitch in bf16: 16 bytes of padding keep ldmatrix free of bank conflicts
// Slice results in flight when they are added.  Us a step with 4 / 6 / 8 / 12 / 24: 87.5 % 16 x 1500 (6 slices) 32.9 / 32.7 / 32.3 /
// 33.3 / 34.6, 7B 75 % 1 x 1999 (12) 23.6 / 23.1 / 23.3 / 23.1 / 23.6, 32 x 1000 58.9 / 58.6 / 58.6 / 58.8 / 59.2, 13B 8 x 1000 (15)
// 38.4 / 39.0 / 38.7 / 38.9 / 39.0, 50 % 8 x 1000 (24) 45.9 / 45.7 / 45.8 / 45.7 / 45.5.
constexpr int kFSum = 6;
constexpr int kFAhead = 4;       // partial results per row in flight beside the statistics

// kMore: blocks start at group g0 of n_groups (calls of more rows than one grid holds).  kOne: one query row per sequence
template <bool kShare, bool kMore, bool kOne>
__global__ void __launch_bounds__(kFThreads, kShare ? 3 : 4)
combine_fast_kernel(const float* part_acc, const float* part_ml,   // written by the split-K kernel while this
                                                                   // kernel may already be resident: read
                                                                   // with plain L2 loads, never ld.global.nc
                    const int32_t* seq_first, const bf16* __restrict__ Wuv,
                    float* __restrict__ slice_out /* [n_slices][B * rows][n_h][128] */,
                    int32_t* __restrict__ counters /* [n_h][groups], zeroed by the plan kernel */,
                    bf16* __restrict__ out, int B, int n_query, int n_h, int d_c, int g0, int n_groups) {
  const int rows = kOne ? 1 : n_query;
  __shared__ __align__(16) bf16 s_w[kFK][kFPitch];        // W_uv slice
  __shared__ __align__(16) bf16 s_o[2][kFB][kFPitch];     // merged latent outputs: bf16 head and remainder
  bf16 (*const s_hi)[kFPitch] = s_o[0];
  bf16 (*const s_lo)[kFPitch] = s_o[1];
  __shared__ int s_last;
  const int h = blockIdx.x, slice = blockIdx.y, n_slices = gridDim.y, g = kMore ? g0 + blockIdx.z : blockIdx.z;
  const int k0 = slice * kFK;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int n_rows = B * rows, r0 = g * kFB, nb = min(kFB, n_rows - r0);

  // W_uv[k0 + k][h*128 + d] -> shared, 16-byte asynchronous copies that land while the split-K
  // kernel drains and the partial results are merged
  for (int e = tid; e < kFK * (kFD / 8); e += kFThreads) {
    const int k = e / (kFD / 8), v = e % (kFD / 8);
    cp_async16(&s_w[k][v * 8], Wuv + (size_t)(k0 + k) * n_h * kFD + (size_t)h * kFD + v * 8);
  }
  cp_async_commit();
  // Row r = (sequence r / rows, query row r % rows).  A warp merges two rows; half a warp holds a row's
  // softmax statistics, lane j of the half those of its j-th item.  kShare: at most 8 rows, and 8 / 4 / 2
  // warps take turns at the items of a pair.  The plan was written before the split-K kernel started
  // computing (that kernel waited for it before it let this one be launched), so the item ranges are
  // fetched while the split-K kernel still runs.
  const int share = !kShare ? 1 : nb <= 2 ? 8 : nb <= 4 ? 4 : 2;
  const int row_w = 2 * (warp / share), sub = warp % share;
  const int half = lane >> 4, j = lane & 15;
  int i0[2], ni[2];
  size_t src0[2];                // first partial result of the row on this slice, in floats
#pragma unroll
  for (int e = 0; e < 2; ++e) {
    const int rr = row_w + e;
    i0[e] = ni[e] = 0;
    src0[e] = 0;
    if (rr < nb) {
      const int b = (r0 + rr) / rows, q = (r0 + rr) % rows;
      i0[e] = __ldcg(seq_first + b);
      ni[e] = __ldcg(seq_first + b + 1) - i0[e];
      src0[e] = (((size_t)i0[e] * rows + q) * n_h + h) * d_c + k0 + lane * 4;
    }
  }
  const size_t stride = (size_t)rows * n_h * d_c;                // from one item to the next
  const int my_i0 = half ? i0[1] : i0[0], my_ni = half ? ni[1] : ni[0];
  const int my_q = (r0 + row_w + half) % rows;
  auto item_ml = [&](int k) -> float2 {
    return __ldcg((const float2*)part_ml + ((size_t)(my_i0 + k) * rows + my_q) * n_h + h);
  };
  ekv_pdl_wait();         // everything below reads the split-K kernel's output
  ekv_pdl_trigger();

  // statistics and the first partial results of both rows are requested together
  float2 ml = make_float2(-INFINITY, 0.f), ml2 = ml;
  if (j < my_ni) ml = item_ml(j);
  if (kShare && j + 16 < my_ni) ml2 = item_ml(j + 16);
  const int first = kShare ? kFAhead * sub : 0;      // this warp's first item
  float4 p[2][kFAhead];
#pragma unroll
  for (int e = 0; e < 2; ++e)
#pragma unroll
    for (int k = 0; k < kFAhead; ++k)
      p[e][k] = first + k < ni[e] ? __ldcg((const float4*)(part_acc + src0[e] + (first + k) * stride)) : make_float4(0.f, 0.f, 0.f, 0.f);
  constexpr int kHeld = kShare ? 32 : 16;    // items whose statistics are in registers
  float M = kShare ? fmaxf(ml.x, ml2.x) : ml.x;
  for (int k = j + kHeld; k < my_ni; k += 16) M = fmaxf(M, item_ml(k).x);       // rare: more items
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) M = fmaxf(M, __shfl_xor_sync(0xffffffffu, M, o));
  float L = j < my_ni ? ml.y * exp2f(ml.x - M) : 0.f;
  if (kShare && j + 16 < my_ni) L = fmaf(ml2.y, exp2f(ml2.x - M), L);
  for (int k = j + kHeld; k < my_ni; k += 16) {
    const float2 x = item_ml(k);
    L += x.y * exp2f(x.x - M);
  }
#pragma unroll
  for (int o = 1; o < 16; o <<= 1) L += __shfl_xor_sync(0xffffffffu, L, o);
  const float invL = my_ni > 0 && L > 0.f ? 1.f / L : 0.f;
  // normalised weight of item j (shared rows: of the warp's first group of items)
  float wt = j < my_ni ? exp2f(ml.x - M) * invL : 0.f;
  const float wt2 = kShare && j + 16 < my_ni ? exp2f(ml2.x - M) * invL : 0.f;
  if (kShare && first >= 16) wt = wt2;
  float4 acc[2];
#pragma unroll
  for (int e = 0; e < 2; ++e) acc[e] = make_float4(0.f, 0.f, 0.f, 0.f);
  auto add = [](float4& x, float w, const float4& y) {
    x.x = fmaf(w, y.x, x.x); x.y = fmaf(w, y.y, x.y); x.z = fmaf(w, y.z, x.z); x.w = fmaf(w, y.w, x.w);
  };
#pragma unroll
  for (int e = 0; e < 2; ++e)
#pragma unroll
    for (int k = 0; k < kFAhead; ++k) add(acc[e], __shfl_sync(0xffffffffu, wt, 16 * e + ((first + k) & 15)), p[e][k]);
  const int n_most = max(ni[0], ni[1]);
  for (int k0b = first + kFAhead * share; k0b < n_most; k0b += kFAhead * share) {
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int k = 0; k < kFAhead; ++k)
        p[e][k] = k0b + k < ni[e] ? __ldcg((const float4*)(part_acc + src0[e] + (size_t)(k0b + k) * stride))
                                  : make_float4(0.f, 0.f, 0.f, 0.f);
    if (kShare) {
      const int kj = (k0b & ~15) + j;
      wt = k0b < 16 ? (j < my_ni ? exp2f(ml.x - M) * invL : 0.f) : k0b < 32 ? wt2 : kj < my_ni ? exp2f(item_ml(kj).x - M) * invL : 0.f;
    } else if ((k0b & 15) == 0) {
      wt = k0b + j < my_ni ? exp2f(item_ml(k0b + j).x - M) * invL : 0.f;
    }
#pragma unroll
    for (int e = 0; e < 2; ++e)
#pragma unroll
      for (int k = 0; k < kFAhead; ++k) add(acc[e], __shfl_sync(0xffffffffu, wt, 16 * e + ((k0b + k) & 15)), p[e][k]);
  }
  // the fp32 rows are fed to the product as a bf16 head plus a bf16 remainder, so nothing but the
  // last ~2^-17 of them is lost; W_uv is bf16 as stored
  auto store_row = [&](int rr, const float4& x) {
    const bf162 h0 = __floats2bfloat162_rn(x.x, x.y), h1 = __floats2bfloat162_rn(x.z, x.w);
    const float2 f0 = __bfloat1622float2(h0), f1 = __bfloat1622float2(h1);
    const bf162 l0 = __floats2bfloat162_rn(x.x - f0.x, x.y - f0.y);
    const bf162 l1 = __floats2bfloat162_rn(x.z - f1.x, x.w - f1.y);
    *(uint2*)&s_hi[rr][lane * 4] = make_uint2(*(const uint32_t*)&h0, *(const uint32_t*)&h1);
    *(uint2*)&s_lo[rr][lane * 4] = make_uint2(*(const uint32_t*)&l0, *(const uint32_t*)&l1);
  };
  if (!kShare) {
#pragma unroll
    for (int e = 0; e < 2; ++e) store_row(row_w + e, acc[e]);
  } else {
    // the sums of the warps that shared a pair, added in order by a warp per row; rows 8 to 15 hold
    // nothing that is stored
    static_assert(kFThreads / 32 * 2 * 32 * sizeof(float4) <= sizeof(s_o), "partial sums take the rows' place");
    float4* const s_part = (float4*)s_o;                   // [warp][2][32]
#pragma unroll
    for (int e = 0; e < 2; ++e) s_part[(2 * warp + e) * 32 + lane] = acc[e];
    __syncthreads();
    float4 x = make_float4(0.f, 0.f, 0.f, 0.f);
    if (warp < nb)
      for (int s = 0; s < share; ++s) add(x, 1.f, s_part[(2 * (warp / 2 * share + s) + (warp & 1)) * 32 + lane]);
    __syncthreads();
    store_row(warp, x);
    store_row(warp + 8, make_float4(0.f, 0.f, 0.f, 0.f));
  }
  cp_async_wait<0>();
  __syncthreads();
  // [16 x 128] . [128 x 128] on mma.sync (m16n8k16, bf16 in, fp32 accumulate): one warp per 16 output dims
  {
    const int n0 = warp * 16;
    float c[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
    for (int kk = 0; kk < kFK; kk += 16) {
      uint32_t ahi[4], alo[4], w[4];
      ldmatrix_x4(ahi, &s_hi[lane & 15][kk + (lane >> 4) * 8]);
      ldmatrix_x4(alo, &s_lo[lane & 15][kk + (lane >> 4) * 8]);
      ldmatrix_x4_trans(w, &s_w[kk + (lane & 15)][n0 + (lane >> 4) * 8]);
      mma_bf16_16816(c[0], ahi, w[0], w[1]);
      mma_bf16_16816(c[1], ahi, w[2], w[3]);
      mma_bf16_16816(c[0], alo, w[0], w[1]);
      mma_bf16_16816(c[1], alo, w[2], w[3]);
    }
    const int gr = lane >> 2, t = lane & 3;
    float* dst = slice_out + (((size_t)slice * n_rows + r0) * n_h + h) * kFD + n0 + 2 * t;
#pragma unroll
    for (int nt = 0; nt < 2; ++nt) {
      if (gr < nb) __stcg((float2*)(dst + (size_t)gr * n_h * kFD + nt * 8), make_float2(c[nt][0], c[nt][1]));
      if (gr + 8 < nb) __stcg((float2*)(dst + (size_t)(gr + 8) * n_h * kFD + nt * 8), make_float2(c[nt][2], c[nt][3]));
    }
  }
  // the block of a (head, group) that arrives last adds the slices in order
  __syncthreads();
  if (tid == 0) {
    int before;      // (the barrier in front orders the block's stores before the release, the one behind its loads after the acquire)
    asm volatile("atom.add.acq_rel.gpu.global.s32 %0, [%1], 1;"
                 : "=r"(before) : "l"(counters + h * (kMore ? n_groups : gridDim.z) + g) : "memory");
    s_last = before == n_slices - 1;
  }
  __syncthreads();
  if (s_last) {
    for (int e = tid; e < nb * (kFD / 4); e += kFThreads) {
      const int rr = e / (kFD / 4), d = (e % (kFD / 4)) * 4;
      const float* src = slice_out + ((size_t)(r0 + rr) * n_h + h) * kFD + d;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      for (int s0 = 0; s0 < n_slices; s0 += kFSum) {
        float4 y[kFSum];
#pragma unroll
        for (int s = 0; s < kFSum; ++s)
          y[s] = s0 + s < n_slices ? __ldcg((const float4*)(src + (size_t)(s0 + s) * n_rows * n_h * kFD)) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int s = 0; s < kFSum; ++s) { v.x += y[s].x; v.y += y[s].y; v.z += y[s].z; v.w += y[s].w; }
      }
      const bf162 o0 = __floats2bfloat162_rn(v.x, v.y), o1 = __floats2bfloat162_rn(v.z, v.w);
      bf162* dst = (bf162*)(out + ((size_t)(r0 + rr) * n_h + h) * kFD + d);      // the caller's `out` is 4-byte aligned
      dst[0] = o0;
      dst[1] = o1;
    }
  }
}

// ------------------------------------------------------------------ generic path
constexpr int kCombBatch = 8;
constexpr int kCombThreads = 256;
constexpr int kCombChunk = 128;

__global__ void __launch_bounds__(kCombThreads)
combine_upproj_kernel(const float* part_acc, const float* part_ml,      // (as above: never ld.global.nc)
                      const int32_t* seq_first, const bf16* __restrict__ Wuv,
                      bf16* __restrict__ out, int B, int n_h /* query rows x heads */, int n_phys /* heads */,
                      int d_h, int d_c) {
  __shared__ float s_olat[kCombBatch][kCombChunk];
  __shared__ float s_M[kCombBatch], s_invL[kCombBatch];
  __shared__ int s_first[kCombBatch + 1];
  extern __shared__ float s_red[];     // [kgroups][kCombBatch][d_h]
  const int h = blockIdx.x;
  const int b0 = blockIdx.y * kCombBatch;
  const int nb = min(kCombBatch, B - b0);
  const int npair = d_h >> 1;
  const int kgroups = max(1, kCombThreads / npair);
  const int pair = threadIdx.x % npair;
  const int kg = threadIdx.x / npair;
  const bool worker = kg < kgroups;

  ekv_pdl_wait();
  ekv_pdl_trigger();
  if (threadIdx.x <= nb) s_first[threadIdx.x] = seq_first[b0 + threadIdx.x];
  __syncthreads();
  {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    for (int bb = warp; bb < nb; bb += kCombThreads / 32) {
      const int i0 = s_first[bb], i1 = s_first[bb + 1];
      float M = -INFINITY;
      for (int i = i0 + lane; i < i1; i += 32) M = fmaxf(M, part_ml[((size_t)i * n_h + h) * 2]);
      M = warp_max(M);
      float Lsum = 0.f;
      for (int i = i0 + lane; i < i1; i += 32) {
        const float* ml = part_ml + ((size_t)i * n_h + h) * 2;
        Lsum += ml[1] * exp2f(ml[0] - M);
      }
      Lsum = warp_sum(Lsum);
      if (lane == 0) {
        s_M[bb] = M;
        s_invL[bb] = (i1 > i0 && Lsum > 0.f) ? 1.f / Lsum : 0.f;
      }
    }
  }
  __syncthreads();

  float acc0[kCombBatch], acc1[kCombBatch];
#pragma unroll
  for (int bb = 0; bb < kCombBatch; ++bb) acc0[bb] = acc1[bb] = 0.f;

  for (int k0 = 0; k0 < d_c; k0 += kCombChunk) {
    const int kc = min(kCombChunk, d_c - k0);
    for (int e = threadIdx.x; e < kCombBatch * kCombChunk; e += kCombThreads) {
      const int bb = e / kCombChunk, k = e % kCombChunk;
      float v = 0.f;
      if (bb < nb && k < kc) {
        const float M = s_M[bb];
#pragma unroll 4
        for (int i = s_first[bb]; i < s_first[bb + 1]; ++i) {
          const float w = exp2f(part_ml[((size_t)i * n_h + h) * 2] - M);
          v = fmaf(w, part_acc[((size_t)i * n_h + h) * d_c + k0 + k], v);
        }
        v *= s_invL[bb];
      }
      s_olat[bb][k] = v;
    }
    __syncthreads();
    if (worker) {
      for (int k = kg; k < kc; k += kgroups) {
        const float2 w = __bfloat1622float2(
            *(const bf162*)(Wuv + (size_t)(k0 + k) * n_phys * d_h + (size_t)(h % n_phys) * d_h + 2 * pair));
#pragma unroll
        for (int bb = 0; bb < kCombBatch; ++bb) {
          const float x = s_olat[bb][k];
          acc0[bb] = fmaf(x, w.x, acc0[bb]);
          acc1[bb] = fmaf(x, w.y, acc1[bb]);
        }
      }
    }
    __syncthreads();
  }

  if (worker) {
#pragma unroll
    for (int bb = 0; bb < kCombBatch; ++bb) {
      s_red[((size_t)kg * kCombBatch + bb) * d_h + 2 * pair] = acc0[bb];
      s_red[((size_t)kg * kCombBatch + bb) * d_h + 2 * pair + 1] = acc1[bb];
    }
  }
  __syncthreads();
  for (int e = threadIdx.x; e < nb * d_h; e += kCombThreads) {
    const int bb = e / d_h, d = e % d_h;
    float v = 0.f;
    for (int g = 0; g < kgroups; ++g) v += s_red[((size_t)g * kCombBatch + bb) * d_h + d];
    out[((size_t)(b0 + bb) * n_h + h) * d_h + d] = __float2bfloat16_rn(v);
  }
}

}  // namespace

int ekv_combine_fast_ok(const elitekv_layer* L) { return L->d_h == kFD && L->vw % kFK == 0; }

size_t ekv_combine_scratch_bytes(const elitekv_layer* L, int B) {
  if (!ekv_combine_fast_ok(L)) return 0;
  return sizeof(float) * (size_t)(L->vw / kFK) * B * L->n_h * kFD;
}

int ekv_combine_counters(const elitekv_layer* L, int B) {
  return ekv_combine_fast_ok(L) ? L->n_h * ((B + kFB - 1) / kFB) : 0;
}

int ekv_launch_combine(const elitekv_layer* L, int B, const DecodeScratch& ws, void* out,
                       cudaStream_t st) {
  // several query rows per sequence: row i, head h is "head" i * n_h + h of the partial results
  // and of the output; it uses head h's slice of W_uv
  const int nv = (ws.rows > 0 ? ws.rows : 1) * L->n_h;
  if (ekv_combine_fast_ok(L)) {
    const int rows = ws.rows > 0 ? ws.rows : 1;
    const int n_groups = (B * rows + kFB - 1) / kFB;
    // at most 8 rows: idle warps share the rows' items (a 7B step of one sequence: 34.8 -> 32.4 us at 32
    // items, 8 sequences 50.1 -> 49.4); from 9 rows on at least half of the warps have a pair of their own
    const auto kern = n_groups > kGridZ ? combine_fast_kernel<false, true, false>
                      : rows > 1        ? (B * rows <= 8 ? combine_fast_kernel<true, false, false> : combine_fast_kernel<false, false, false>)
                      : B <= 8          ? combine_fast_kernel<true, false, true>
                                        : combine_fast_kernel<false, false, true>;
    for (int g0 = 0; g0 < n_groups; g0 += kGridZ) {      // one launch up to a million rows
      const dim3 grid(L->n_h, L->vw / kFK, n_groups - g0 < kGridZ ? n_groups - g0 : kGridZ);
      EKV_CUDA_OK(ekv_launch_pdl(kern, grid, dim3(kFThreads), 0, st, (const float*)ws.part_acc, (const float*)ws.part_ml,
                                 (const int32_t*)ws.seq_first, (const bf16*)L->d_Wuv, ws.slice_out, ws.counters, (bf16*)out,
                                 B, rows, L->n_h, L->vw, g0, n_groups));
    }
    EKV_CUDA_OK(cudaGetLastError());
    return ELITEKV_OK;
  }
  const int npair = L->d_h / 2;
  if (npair > kCombThreads) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  const int kgroups = kCombThreads / npair > 0 ? kCombThreads / npair : 1;
  const size_t smem = sizeof(float) * (size_t)kgroups * kCombBatch * L->d_h;
  dim3 grid(nv, (B + kCombBatch - 1) / kCombBatch);
  EKV_CUDA_OK(ekv_allow_smem(combine_upproj_kernel, smem));
  EKV_CUDA_OK(ekv_launch_pdl(combine_upproj_kernel, grid, dim3(kCombThreads), smem, st, (const float*)ws.part_acc,
                             (const float*)ws.part_ml, (const int32_t*)ws.seq_first, (const bf16*)L->d_Wuv, (bf16*)out, B,
                             nv, L->n_h, L->d_h, L->vw));
  EKV_CUDA_OK(cudaGetLastError());
  return ELITEKV_OK;
}
