// Projection fused with the cache append (tcgen05 + TMEM + TMA).
//
// The cache row of a token is made from its hidden state x by two projections (Section 3.2):
// the elite key chunks k_e = x W^k_e (the columns of W^k that belong to the head's elite chunks,
// Eq. 2) and the shared latent c = x A^kv.  Both are one GEMM against the column-concatenated
// weight [W^k_e | A^kv], x [T x d] . [d x (2 r n_h + d_c)].  The append (Section 3.1: the elite
// chunks are rotated once, at the token's position) is the epilogue of that GEMM: accumulators
// leave TMEM with one thread per token, rope columns are rotated as (even, odd) pairs with the
// (cos, sin) of pos * theta_{idx[h][j]}, everything is rounded once to bf16 and written straight
// to the token's cache row (contiguous or paged).  k_e and c never touch memory.
//
// One block computes a [128 tokens x 128 output columns] tile (prefill-sized calls: 256 or 512
// x 256 per block pair, see further down): warp 0 streams the operand tiles
// ([128 x 64] of x and of the transposed weight, 128-byte swizzle) through a 4-stage ring, warp 1
// issues tcgen05.mma (M = 128, N = 128, K = 16, bf16 in, fp32 in TMEM), warps 2-5 run the epilogue.
// A 128-wide tile lies either in the rope part or in the latent part (both are multiples of 128 wide).
//
// Few tokens make few tiles: a decode step's batch has one token tile, so the grid above would be
// n_out / 128 blocks reading the 2 d n_out bytes of weights between them, 16 blocks for the 7B
// shape.  Such a call runs as clusters of 8, 4 or 2 blocks per tile, each block taking its share of
// the depth d.  The partial sums leave TMEM, cross distributed shared memory (block i of a cluster
// of s collects rows [128 i / s, 128 (i + 1) / s) from all of them) and are added in block order, so the
// result does not depend on scheduling; the collecting block rotates, rounds and stores.
// The weights of the first stages are requested before the dependency wait.
// Every wait is bounded (timeouts are recorded and the block leaves through the common exit).
#include "tc_ptx.cuh"

namespace {

constexpr int kPM = 128, kPN = 128, kPK = 64;     // tile: tokens, output columns, depth per stage
constexpr int kPStages = 4;
constexpr int kPStageBytes = (kPM + kPN) * kPK * 2;   // 32 KB
constexpr int kPThreads = 192;
constexpr int kRecvBytes = kPM * kPN * 4;         // 64 KB: [source block][row][column] fp32, rows of one block

struct ProjArgs {
  const int32_t* seq_id;
  const int32_t* pos;
  long long T;
  bf16* rope;
  bf16* latent;
  CacheView cv;
  const int32_t* idx;       // [n_h * r] chunk id of every cached pair
  const float2* cs;         // [max_pos][d_h/2]
  int rope_w, d_c, half, max_pos, nk;
  int32_t* status;
};

struct __align__(8) ProjBarriers {
  uint64_t full[kPStages], empty[kPStages], done;
};

// rotation, single rounding and the 16-byte stores of 8 consecutive output columns of one token
__device__ __forceinline__ void finish_columns(const ProjArgs& a, const float* v, long long row, int p, int g0) {
  uint32_t packed[4];
  if (g0 < a.rope_w) {
    const float2* csrow = a.cs + (long long)p * a.half;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float2 w = __ldg(csrow + __ldg(a.idx + (g0 >> 1) + j));
      const float y0 = __fsub_rn(__fmul_rn(v[2 * j], w.x), __fmul_rn(v[2 * j + 1], w.y));
      const float y1 = __fadd_rn(__fmul_rn(v[2 * j], w.y), __fmul_rn(v[2 * j + 1], w.x));
      const bf162 y = __floats2bfloat162_rn(y0, y1);
      packed[j] = *(const uint32_t*)&y;
    }
    *(uint4*)(a.rope + row * a.rope_w + g0) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
  } else {
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const bf162 y = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
      packed[j] = *(const uint32_t*)&y;
    }
    *(uint4*)(a.latent + row * a.d_c + (g0 - a.rope_w)) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
  }
}

// cache row of token t (-1 and a recorded error when its position or sequence is out of range)
__device__ __forceinline__ long long token_row(const ProjArgs& a, long long t, int* p_out) {
  const int s = a.seq_id[t];
  const int p = a.pos[t];
  *p_out = p;
  if (p < 0 || p >= a.max_pos) {
    ekv_record(a.status, ELITEKV_ERR_BAD_POSITION, s, p);
    return -1;
  }
  int code, detail;
  const long long row = ekv_token_row(a.cv, s, p, &code, &detail);
  if (row < 0) ekv_record(a.status, code, s, detail);
  return row;
}

template <int kSplit>                              // blocks per cluster that share the depth
__global__ void __launch_bounds__(kPThreads, 1)
project_append_kernel(const __grid_constant__ CUtensorMap map_x, const __grid_constant__ CUtensorMap map_w,
                      const ProjArgs a) {
  constexpr bool kSplitDepth = kSplit > 1;
  constexpr int kSplitRows = kPM / kSplit;         // token rows each block of a cluster finishes
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  float* s_recv = (float*)(base + kPStages * kPStageBytes);      // split-depth form only
  ProjBarriers* bars = (ProjBarriers*)(base + kPStages * kPStageBytes + (kSplitDepth ? kRecvBytes : 0));
  uint32_t* s_tmem = (uint32_t*)(bars + 1);
  volatile int* s_abort = (volatile int*)(s_tmem + 1);
  volatile int* s_lost = s_abort + 1;              // a block of the cluster gave up: no sum here is complete
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n0 = blockIdx.x * kPN;                 // first output column of the tile
  const long long t0 = (long long)blockIdx.y * kPM; // first token of the tile
  // depth steps of this block: all of them, or the cluster rank's share
  const int crank = kSplitDepth ? (int)cluster_ctarank() : 0;
  const int k_lo = kSplitDepth ? (int)((long long)a.nk * crank / kSplit) : 0;
  const int k_hi = kSplitDepth ? (int)((long long)a.nk * (crank + 1) / kSplit) : a.nk;

  if (threadIdx.x == 0) {
    for (int i = 0; i < kPStages; ++i) {
      mbar_init(smem_u32(&bars->full[i]), 1);
      mbar_init(smem_u32(&bars->empty[i]), 1);
    }
    mbar_init(smem_u32(&bars->done), 1);
    *s_abort = 0;
    *s_lost = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
  }
  ekv_pdl_trigger();      // whatever is launched behind waits for this grid itself
  constexpr uint32_t tmem_cols = 128;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  // a block's shared memory is written by its peers once they know that it has started: every warp waits
  // for that before its first remote store, behind the loads and products
  if (kSplitDepth) cluster_arrive();
  const uint32_t tmem_base = *s_tmem;

  if (warp == 0) {
    // ---- operand tiles: x rows [t0, t0+128) and weight rows [n0, n0+128), 64 of d per stage
    //      (rows past T come back as zeros: they are never stored)
    //      The first stages' weights belong to the layer: requested while earlier kernels still run.
    bool ok = true;
    const int early = min(k_hi - k_lo, kPStages);
    auto load = [&](int k, bool w, bool x) {
      if (elect_one()) {
        const uint32_t fb = smem_u32(&bars->full[k % kPStages]), dst = smem_u32(base + k % kPStages * kPStageBytes);
        if (w) {
          mbar_expect_tx(fb, (uint32_t)kPStageBytes);
          tma_load_2d(dst + kPM * kPK * 2, &map_w, (k_lo + k) * kPK, n0, fb);
        }
        if (x) tma_load_2d(dst, &map_x, (k_lo + k) * kPK, (int)t0, fb);
      }
      __syncwarp();
    };
    for (int k = 0; k < early; ++k) load(k, true, false);
    ekv_pdl_wait();
    for (int k = 0; k < early; ++k) load(k, false, true);
    for (int k = early; k < k_hi - k_lo && ok; ++k) {
      ok = warp_wait(smem_u32(&bars->empty[k % kPStages]), ((k / kPStages) & 1) ^ 1, s_abort, 1);
      if (!ok) break;
      load(k, true, true);
    }
  } else if (warp == 1) {
    constexpr uint32_t idesc = make_idesc(kPM, kPN, 0, 0);
    constexpr uint32_t hi_sw = desc_hi(1024, 2);
    const uint32_t base16 = (smem_u32(base) >> 4) & 0x3FFFu;
    bool ok = true;
    for (int k = 0; k < k_hi - k_lo && ok; ++k) {
      const int s = k % kPStages;
      ok = warp_wait(smem_u32(&bars->full[s]), (k / kPStages) & 1, s_abort, 2);
      if (!ok) break;
      const uint32_t la = (base16 + (uint32_t)s * (kPStageBytes >> 4)) | (1u << 16);
      const uint32_t lb = la + ((kPM * kPK * 2) >> 4);
      if (elect_one()) {
        tc_mma_w(tmem_base, la, hi_sw, lb, hi_sw, idesc, k != 0);
        tc_mma_w(tmem_base, la + 2, hi_sw, lb + 2, hi_sw, idesc, 1);
        tc_mma_w(tmem_base, la + 4, hi_sw, lb + 4, hi_sw, idesc, 1);
        tc_mma_w(tmem_base, la + 6, hi_sw, lb + 6, hi_sw, idesc, 1);
        tc_commit(smem_u32(&bars->empty[s]));
      }
      __syncwarp();
    }
    if (ok && elect_one()) tc_commit(smem_u32(&bars->done));
    __syncwarp();
  } else {
    // ---- epilogue: thread = token row of the tile
    ekv_pdl_wait();                                        // (tokens, and the cache that earlier kernels read)
    const int quarter = warp & 3;
    const int trow = quarter * 32 + lane;
    const long long t = t0 + trow;
    long long row = -1;
    int p = 0;
    if (!kSplitDepth && t < a.T) row = token_row(a, t, &p);
    // one outcome per warp: the TMEM loads below want all 32 lanes
    const bool ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->done), 0, s_abort, 3));
    tc_fence_after();
    if (kSplitDepth) cluster_wait();
    if (ok) {
      // split depth: this row's partial sums go to the block that finishes the row
      const uint32_t dst = kSplitDepth
          ? map_to_cta(smem_u32(s_recv + ((size_t)crank * kSplitRows + (trow % kSplitRows)) * kPN), (uint32_t)(trow / kSplitRows))
          : 0u;
      for (int cc = 0; cc < kPN / 32; ++cc) {
        float v[32];
        tc_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(cc * 32), v);
        tc_wait_ld();
        if (kSplitDepth) {
          if (t < a.T) {
#pragma unroll
            for (int q = 0; q < 8; ++q)
              st_cluster_f4(dst + (uint32_t)(cc * 32 + 4 * q) * 4u, make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]));
          }
        } else if (row >= 0) {
#pragma unroll
          for (int q = 0; q < 4; ++q) finish_columns(a, v + 8 * q, row, p, n0 + cc * 32 + 8 * q);
        }
      }
    }
  }

  if (kSplitDepth) {
    __syncwarp();
    if (warp < 2) cluster_wait();
    if (*s_abort && lane < kSplit) st_cluster_u32(map_to_cta(smem_u32((const void*)s_lost), (uint32_t)lane), 1u);
    __syncwarp();
    // every block of the cluster has delivered (or given up, and said so): the barrier orders the remote
    // stores above before the sums below, and nobody is written to after it
    cluster_sync_all();
    if (warp >= 2 && !*s_lost) {
      const int e = threadIdx.x - 64;                    // 128 threads: 16 rows x 8 column groups
      const int cg = e & 7;
      for (int rr = e >> 3; rr < kSplitRows; rr += 16) {
        const long long t = t0 + crank * kSplitRows + rr;
        if (t >= a.T) break;
        int p = 0;
        const long long row = token_row(a, t, &p);
        if (row >= 0) {
          float v[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) v[i] = 0.f;
          for (int src = 0; src < kSplit; ++src) {       // fixed order: the sum does not depend on timing
            const float4* pr = (const float4*)(s_recv + ((size_t)src * kSplitRows + rr) * kPN + cg * 16);
#pragma unroll
            for (int i = 0; i < 4; ++i) {
              const float4 x = pr[i];
              v[4 * i] += x.x; v[4 * i + 1] += x.y; v[4 * i + 2] += x.z; v[4 * i + 3] += x.w;
            }
          }
          finish_columns(a, v, row, p, n0 + cg * 16);
          finish_columns(a, v + 8, row, p, n0 + cg * 16 + 8);
        }
      }
    }
  }

  // ---- teardown
  tc_fence_before();
  __syncthreads();
  if (*s_abort) drain_after_abort();
  if (threadIdx.x == 0 && *s_abort) ekv_record(a.status, ELITEKV_ERR_TIMEOUT, (int)blockIdx.x | (*s_abort << 16), (int)blockIdx.y);
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// ------------------------------------------------------------------ prefill form: block pairs
// A 128 x 128 tile asks L2 for 32 KB of operands per 256 tensor-core clocks; at prefill size all
// SMs together ask for more than L2 delivers, and the tensor pipe idles more than half of the
// time.  Here a cluster of two blocks computes 256 H tokens x 256 columns with paired instructions
// (cta_group::2: M = 256 over both blocks, N = 256): a block keeps 128 H rows of x and HALF of the 256
// weight rows per 64 of depth, the other half of the weights is read out of its peer's shared memory
// by the tensor core.  H = 2: two accumulators (TMEM columns 0-255 and 256-511), 48 KB per 1024 clocks
// and block, which L2 can deliver to the whole chip.  H = 1: 32 KB per 512 clocks, for calls whose
// tiles of 512 tokens would leave half of the chip idle.
// The ring holds 14 units of 128 rows (weights and 128 tokens each in turn), not whole stages: a unit
// is refilled as soon as its own product has read it, and a load takes about 3000 clocks under this
// traffic, three stages' time.  Every block loads its own units, but onto the first block's barriers:
// its MMA warp issues for both.
// The epilogue of a rope tile reads the tokens' whole (cos, sin) rows into idle ring units while the
// last products run, rotates out of shared memory and writes 256-byte pieces of the cache rows.
// 4096 tokens of the 7B shape (68.7 GFLOP): 51 us, 1.34 PFLOP/s (82 us with 256 x 256 tiles of one
// block), 63 us back to back at the power cap; the main loop keeps the tensor cores busy (65.5 k
// clocks of products take 67.2 k), 10 k clocks of epilogue follow.  2048 tokens: 29 us (46 us with 128 x 128 tiles).
constexpr int kBN = 256;                 // columns per pair
constexpr int kUnits = 14;
constexpr int kUnitBytes = 128 * kPK * 2;                 // 16 KB
constexpr int kBThreads = 320;           // warp 0 loads, warp 1 MMA (first block), warps 2-9 epilogue

constexpr int kCsUnits = 8;              // units that take table rows for the epilogue, one per epilogue warp

struct __align__(8) PairBarriers {
  uint64_t full[kUnits], empty[kUnits], done;      // full: of the first block only, for both blocks' units
  uint64_t last[kCsUnits];                         // the last product of such a unit is done: one phase only
};

// Epilogue buffers lie in the operand ring, in the units read last.  Per warp of 32 tokens: the tokens'
// rows of the (cos, sin) table in one unit (512 bytes a row, entry e at e ^ row: equal columns of 32
// tokens are on different banks), which starts to fill as soon as that unit's last product is done;
// and 128 finished columns of the 32 cache rows in half a unit (16-byte pieces XORed with the row).
constexpr int kCsHalf = 64;              // table rows of up to 64 chunks
static_assert(32 * kCsHalf * 8 == kUnitBytes && 2 * 32 * 256 == kUnitBytes && kCsUnits + 4 <= kUnits, "epilogue buffers fit");

template <int H>
__global__ void __launch_bounds__(kBThreads, 1)
project_append_pair_kernel(const __grid_constant__ CUtensorMap map_t, const __grid_constant__ CUtensorMap map_w,
                           const ProjArgs a) {
  extern __shared__ unsigned char smem_raw[];
  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  PairBarriers* bars = (PairBarriers*)(base + kUnits * kUnitBytes);
  uint32_t* s_tmem = (uint32_t*)(bars + 1);
  volatile int* s_abort = (volatile int*)(s_tmem + 1);
  static_assert(sizeof(PairBarriers) % 16 == 8, "s_idx on 16 bytes");
  int* s_idx = (int*)(s_tmem + 2);                 // [128] chunk ids of the tile's rope columns
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_ctarank();
  const int n0 = (blockIdx.x >> 1) * kBN;
  const long long t0 = (long long)blockIdx.y * (256 * H) + rank * (128 * H);      // first token of this block

  if (threadIdx.x == 0) {
    for (int i = 0; i < kUnits; ++i) {
      mbar_init(smem_u32(&bars->full[i]), 1);
      mbar_init(smem_u32(&bars->empty[i]), 1);
    }
    mbar_init(smem_u32(&bars->done), 1);
    for (int i = 0; i < kCsUnits; ++i) mbar_init(smem_u32(&bars->last[i]), 1);
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
  }
  constexpr uint32_t tmem_cols = 512;      // the whole tensor memory: one block per SM (224 KB of shared memory)
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::2.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::2.sync.aligned;" ::: "memory");
  }
  if (threadIdx.x >= 64 && threadIdx.x < 192) {
    const int pr = (n0 >> 1) + (int)threadIdx.x - 64;
    s_idx[threadIdx.x - 64] = 2 * pr < a.rope_w ? __ldg(a.idx + pr) : 0;
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                      // both blocks' barriers and tensor memory exist
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;

  if (warp == 0) {
    // ---- per 64 of depth: this block's 128 weight rows and its H units of 128 token rows (zeros past
    //      the end).  (Prefetching later steps into L2 takes the same copy engine: 41 us instead of 33
    //      for 2048 tokens.)
    const int w0 = n0 + (int)rank * (kBN / 2);
    bool ok = true;
    int slot = 0;
    uint32_t turn = 1;                     // parity of `empty` before the first pass over the ring
    for (int k = 0; k < a.nk && ok; ++k) {
#pragma unroll
      for (int u = 0; u <= H; ++u) {
        ok = warp_wait(smem_u32(&bars->empty[slot]), turn, s_abort, 1);
        if (!ok) break;
        if (elect_one()) {
          const uint32_t fb = smem_u32(&bars->full[slot]);
          if (rank == 0) mbar_expect_tx(fb, 2 * kUnitBytes);
          tma_load_2d_pair(smem_u32(base + slot * kUnitBytes), u == 0 ? &map_w : &map_t, k * kPK,
                           u == 0 ? w0 : (int)t0 + (u - 1) * 128, map_to_cta(fb, 0));
        }
        __syncwarp();
        if (++slot == kUnits) { slot = 0; turn ^= 1; }
      }
    }
  } else if (warp == 1 && rank == 0) {
    constexpr uint32_t idesc = make_idesc(256, kBN, 0, 0);
    constexpr uint32_t hi_sw = desc_hi(1024, 2);
    const uint32_t base16 = ((smem_u32(base) >> 4) & 0x3FFFu) | (1u << 16);
    bool ok = true;
    int slot = 0;
    uint32_t turn = 0;
    int left = (H + 1) * a.nk;             // units still to come, the current one included
    for (int k = 0; k < a.nk && ok; ++k) {
      uint32_t lb = 0, bar_w = 0;
#pragma unroll
      for (int u = 0; u <= H; ++u) {
        ok = warp_wait(smem_u32(&bars->full[slot]), turn, s_abort, 2);
        if (!ok) break;
        const uint32_t lo = base16 + (uint32_t)slot * (kUnitBytes >> 4);
        // what the unit's last product arrives on: its ring barrier, or in the ring's last turn, which nobody
        // refills, the epilogue's (whose warps do not hold the ring back: a phase of `empty` could pass them by)
        const int i = kUnits - left;
        const uint32_t bar = smem_u32(i >= 0 && i < kCsUnits ? &bars->last[i] : &bars->empty[slot]);
        if (u == 0) {
          lb = lo;
          bar_w = bar;
        } else {
          tc_fence_after();
          if (elect_one()) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)            // +32 bytes along d per step
              tc_mma_pair(tmem_base + (u - 1) * kBN, lo + 2 * ks, hi_sw, lb + 2 * ks, hi_sw, idesc, (k | ks) != 0);
            tc_commit_pair(bar);                                         // frees the unit in both blocks
            if (u == H) tc_commit_pair(bar_w);
          }
          __syncwarp();
        }
        if (++slot == kUnits) { slot = 0; turn ^= 1; }
        --left;
      }
    }
    if (ok && elect_one()) tc_commit_pair(smem_u32(&bars->done));
    __syncwarp();
  } else if (warp >= 2) {
    // ---- epilogue: warps 2-5 the first accumulator (H = 1: its first 128 columns), 6-9 the second
    //      (its second 128 columns)
    const int quarter = warp & 3, hf = (warp - 2) >> 2;
    const int tok = H == 2 ? hf * 128 : 0, part0 = H == 2 ? 0 : hf, parts = H;      // tokens and columns of this warp
    const long long t = t0 + tok + quarter * 32 + lane;
    int p = 0;
    const long long row = t < a.T ? token_row(a, t, &p) : -1;
    if (row < 0) p = 0;
    const int w8 = warp - 2, first = (H + 1) * a.nk - kUnits;     // the units of the ring's last turn
    unsigned char* s_cs = base + (first + w8) % kUnits * kUnitBytes;
    unsigned char* s_out = base + (first + 8 + (w8 >> 1)) % kUnits * kUnitBytes + (w8 & 1) * (kUnitBytes / 2);
    // (16-byte reads of the table: a caller's own table may start on any 8 bytes)
    const bool staged = a.half <= kCsHalf && (a.half & 1) == 0 && ((uintptr_t)a.cs & 15) == 0;
    bool ok = true;
    if (n0 + part0 * 128 < a.rope_w && staged) {
      // the 32 tokens' table rows, a whole row per request: a look-up by every token on its own would
      // touch 32 rows per request (33 k clocks for a tile of rope columns)
      // (a wait that parks: eight warps that spin here for the whole main loop cost 2048 tokens 28.8 -> 30.8 us)
      ok = __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->last[w8]), 0, s_abort, 4));
      if (ok) {
#pragma unroll 16
        for (int k = 0; k < 32; ++k) {
          const int pk = __shfl_sync(0xffffffffu, p, k);
          if (2 * lane < a.half) {
            const float4 w = __ldg((const float4*)(a.cs + (long long)pk * a.half) + lane);
            float2* dst = (float2*)(s_cs + k * (kCsHalf * 8));
            dst[(2 * lane) ^ k] = make_float2(w.x, w.y);
            dst[(2 * lane + 1) ^ k] = make_float2(w.z, w.w);
          }
        }
        __syncwarp();
      }
    }
    ok = ok && __all_sync(0xffffffffu, mbar_wait(smem_u32(&bars->done), 0, s_abort, 3));
    tc_fence_after();
    if (ok) {
      const float2* cs_row = (const float2*)(s_cs + lane * (kCsHalf * 8));
      for (int part = part0; part < part0 + parts; ++part) {        // 128 columns: all rope or all latent
        const int g0 = n0 + part * 128;
        const bool rope = g0 < a.rope_w;
        bf16* const out = rope ? a.rope + g0 : a.latent + (g0 - a.rope_w);
        const long long pitch = rope ? a.rope_w : a.d_c;
#pragma unroll 2
        for (int cc = 0; cc < 4; ++cc) {
          float v[32];
          tc_ld32(tmem_base + ((uint32_t)(quarter * 32) << 16) + (uint32_t)(tok * 2 + part * 128 + cc * 32), v);
          float2 w[16];
          if (rope) {
            const int4* id4 = (const int4*)(s_idx + part * 64 + cc * 16);
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const int4 id = id4[k];
              if (staged) {
                w[4 * k] = cs_row[id.x ^ lane]; w[4 * k + 1] = cs_row[id.y ^ lane];
                w[4 * k + 2] = cs_row[id.z ^ lane]; w[4 * k + 3] = cs_row[id.w ^ lane];
              } else {
                const float2* src = a.cs + (long long)p * a.half;
                w[4 * k] = __ldg(src + id.x); w[4 * k + 1] = __ldg(src + id.y);
                w[4 * k + 2] = __ldg(src + id.z); w[4 * k + 3] = __ldg(src + id.w);
              }
            }
          }
          tc_wait_ld();
          if (rope) {
#pragma unroll
            for (int k = 0; k < 16; ++k) {
              const float x0 = v[2 * k], x1 = v[2 * k + 1];
              v[2 * k] = __fsub_rn(__fmul_rn(x0, w[k].x), __fmul_rn(x1, w[k].y));
              v[2 * k + 1] = __fadd_rn(__fmul_rn(x0, w[k].y), __fmul_rn(x1, w[k].x));
            }
          }
#pragma unroll
          for (int q = 0; q < 4; ++q) {
            uint32_t packed[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) {
              const bf162 y = __floats2bfloat162_rn(v[8 * q + 2 * k], v[8 * q + 2 * k + 1]);
              packed[k] = *(const uint32_t*)&y;
            }
            *(uint4*)(s_out + lane * 256 + (((cc * 4 + q) ^ (lane & 15)) << 4)) = make_uint4(packed[0], packed[1], packed[2], packed[3]);
          }
        }
        __syncwarp();
        // 256 bytes of two tokens' cache rows per request
#pragma unroll 8
        for (int k = 0; k < 16; ++k) {
          const int tk = 2 * k + (lane >> 4);
          const long long rk = __shfl_sync(0xffffffffu, row, tk);
          const uint4 y = *(const uint4*)(s_out + tk * 256 + (((lane ^ tk) & 15) << 4));
          if (rk >= 0) *(uint4*)(out + rk * pitch + (lane & 15) * 8) = y;
        }
        __syncwarp();
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (*s_abort) drain_after_abort();
  if (threadIdx.x == 0 && *s_abort) ekv_record(a.status, ELITEKV_ERR_TIMEOUT, (int)blockIdx.x | (*s_abort << 16), (int)blockIdx.y);
  cluster_sync_all();                      // the tensor core reads both blocks' shared memory until the end
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::2.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

}  // namespace

int ekv_launch_project_append(const elitekv_layer* L, const elitekv_cache* cache, const CacheView& cv,
                              const void* x, const int32_t* seq_id, const int32_t* pos, long long T,
                              cudaStream_t st) {
  const int rope_w = L->n_h * 2 * L->r;
  const int n_out = rope_w + L->d_c;
  if (L->d % kPK != 0 || rope_w % kPN != 0 || L->d_c % kPN != 0) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  if (T >= (1ll << 31)) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  // a grid's second dimension holds 65535 token tiles: more tokens than that in the smallest are several launches
  constexpr long long kMost = 65535ll * kPM;
  if (T > kMost) {
    for (long long t = 0; t < T; t += kMost) {
      const int rc = ekv_launch_project_append(L, cache, cv, (const bf16*)x + t * L->d, seq_id + t, pos + t,
                                               T - t < kMost ? T - t : kMost, st);
      if (rc != ELITEKV_OK) return rc;
    }
    return ELITEKV_OK;
  }
  ProjArgs a;
  a.seq_id = seq_id;
  a.pos = pos;
  a.T = T;
  a.rope = (bf16*)cache->rope;
  a.latent = (bf16*)cache->latent;
  a.cv = cv;
  a.idx = L->d_idx;
  a.cs = L->d_cs;
  a.rope_w = rope_w;
  a.d_c = L->d_c;
  a.half = L->d_h / 2;
  a.max_pos = L->max_pos;
  a.nk = L->d / kPK;
  a.status = L->d_status;
  // More than one token tile and an output width of whole 256-column tiles: the form whose blocks need
  // least time for the call.  All take whole waves over the chip; microseconds for 64 depth steps
  // measured on 7B shapes at 256 to 16384 tokens (one tile per block 28, 46, 67, 85 for 1 to 4 waves,
  // H = 1 33, 59, H = 2 50, 102, 152; other depths scale all three alike).
  const int smem_pair = kUnits * kUnitBytes + (int)sizeof(PairBarriers) + 16 + 128 * 4 + 1024;
  int form = 0;
  if (T > kPM && n_out % kBN == 0 && 2 * a.nk >= kUnits && smem_pair <= L->smem_optin) {
    const auto waves = [&](long long cols, long long rows, long long at_once) {
      return (n_out / cols * ((T + rows - 1) / rows) + at_once - 1) / at_once;
    };
    const long long t0 = 7 + 20 * waves(kPN, kPM, L->sm_count);
    const long long t1 = 4 + 29 * waves(kBN, 256, L->sm_count / 2);
    const long long t2 = 2 + 50 * waves(kBN, 512, L->sm_count / 2);
    form = t2 <= t1 && t2 <= t0 ? 2 : t1 <= t0 ? 1 : 0;
  }
  if (form != 0) {
    CUtensorMap b_x, b_w;
    int rcb = make_map(&b_x, x, (unsigned long long)T, (unsigned long long)L->d, 128);
    if (rcb == ELITEKV_OK) rcb = make_map(&b_w, L->d_WcatT, (unsigned long long)n_out, (unsigned long long)L->d, kBN / 2);
    if (rcb != ELITEKV_OK) return rcb;
    const auto kern = form == 2 ? project_append_pair_kernel<2> : project_append_pair_kernel<1>;
    EKV_CUDA_OK(ekv_allow_smem(kern, smem_pair));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(2 * (n_out / kBN)), (unsigned)((T + 256 * form - 1) / (256 * form)));
    cfg.blockDim = dim3(kBThreads);
    cfg.dynamicSmemBytes = (size_t)smem_pair;
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = 2;
    attr[0].val.clusterDim.y = 1;
    attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    EKV_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, b_x, b_w, a));
    EKV_CUDA_OK(cudaGetLastError());
    return ELITEKV_OK;
  }
  // Few tiles: clusters share a tile's depth, as many blocks (8, 4, 2) as let all clusters be resident at
  // once: 15, 33, 74 clusters of one block per SM (by the occupancy calculator; more take two waves).  us, cold,
  // with 8 / 4 / 2 / 1 blocks per tile, depth 4096: 8 tiles 16.4 / 18.4 / 20.5 / 32.8, 16 tiles 22.5 / 20.5 /
  // 22.5 / 32.8, 32 tiles 30.7 / 22.5 / 24.6 / 32.8, 64 tiles 53.2 / 34.8 / 28.7 / 36.9; 40 tiles of depth 5120
  // 38.9 / 30.8 / 29.4 / 40.9.
  const long long tiles = n_out / kPN * ((T + kPM - 1) / kPM);
  const int split = tiles <= 15 && a.nk >= 8 ? 8 : tiles <= 33 && a.nk >= 4 ? 4 : tiles <= 74 && a.nk >= 2 ? 2 : 1;
  const int smem = kPStages * kPStageBytes + (split > 1 ? kRecvBytes : 0) + (int)sizeof(ProjBarriers) + 64 + 1024;
  if (smem > L->smem_optin) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  CUtensorMap m_x, m_w;
  int rc = make_map(&m_x, x, (unsigned long long)T, (unsigned long long)L->d, kPM);
  if (rc == ELITEKV_OK) rc = make_map(&m_w, L->d_WcatT, (unsigned long long)n_out, (unsigned long long)L->d, kPN);
  if (rc != ELITEKV_OK) return rc;
  auto launch = [&](auto kern) -> int {
    EKV_CUDA_OK(ekv_allow_smem(kern, smem));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(n_out / kPN), (unsigned)((T + kPM - 1) / kPM), split);
    cfg.blockDim = dim3(kPThreads);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 1;
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = split;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    EKV_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, m_x, m_w, a));
    EKV_CUDA_OK(cudaGetLastError());
    return ELITEKV_OK;
  };
  return split == 8   ? launch(project_append_kernel<8>)
         : split == 4 ? launch(project_append_kernel<4>)
         : split == 2 ? launch(project_append_kernel<2>)
                      : launch(project_append_kernel<1>);
}
