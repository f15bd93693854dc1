// Cluster-resident split-K decode kernel for sm_100a (tcgen05 + TMEM + TMA + distributed shared
// memory).
//
// Bound: HBM.  Every cache byte has to enter an SM once, with enough bytes in flight all the time,
// and the serial chain of a tile (scores -> softmax -> value product) has to stay off that path.
// A token's latent row is too wide for one SM to hold tiles of it beside the absorbed queries of
// all heads and still prefetch, so a cluster of C blocks splits the LATENT axis: block c owns
// kw/C key columns and vw/C value columns (384 of them for all the LLaMA shapes: C = 2 at
// 87.5 %, 4 at 75 %, 5 for 13B, 8 at 50 %), the matching slice of the absorbed queries (resident
// for a whole plan item), a ring of 64-token tiles of its columns, and the matching rows of the
// output (TMEM).  A tile stays where TMA put it from the score product to the value product.
//
// The HEADS are split too, for the softmax: block c finishes heads [c HPC, (c+1) HPC), and reads
// the rope dims of those heads (128 columns of the rope plane for every supported shape).  Per tile
//   1. each block multiplies its columns: S_c [64 x n_h] = C[:, cols_c] . Q_abs[:, cols_c]^T
//      (score equation of Section 3.1 with B^k absorbed, Section 5);
//   2. reduce-scatter: four sender warps take S_c out of TMEM and st.async the columns of each
//      block's heads into that block's receive buffer (16 bytes per token and four heads);
//   3. the owner adds the C partial sums in rank order and the rope dot products (FP32 FMA, in
//      warps of their own that read the rope rows straight into registers), runs the online softmax of
//      its heads (Section 2.1; base 2, reference maximum moved only past a head room of 2^8), a warp
//      per four or eight heads and 64 tokens, so that no barrier lies on the way, and
//   4. all-gather: st.asyncs the bf16 probabilities into every block's P tile, in the layout the
//      value product wants, together with the factor by which older output has to be rescaled;
//   5. each block accumulates acc_c [vw/C x n_h] += C[:, cols_c]^T . P (the latent is key and
//      value source at once, Section 3.2), which frees the tile's ring slot.
// Steps 1-5 of a tile take longer than a tile takes to stream in, so two STREAMS of tiles (even and
// odd) are in flight, each with its own softmax warps, score columns, P tile, running maximum and
// output accumulator; the two accumulators are merged when an item ends.  All hand-over buffers
// are single: a block can only send tile i + 2 after its own score product of that tile, which is
// issued after its value product of tile i, which needed every peer's probabilities of tile i,
// which each peer sent after it had read the partial scores of tile i.
//
// Roles:
//   warps 0, 3   TMA producers of the latent tiles; warp 2 of the query slice of an item
//   warp 1   TMEM owner and MMA issuer: polls for whichever comes first, probabilities of the
//            oldest tile or data of the next one
//   warps 4-7    senders, tiles of both streams in turn
//   warps 8-11   rescale of an accumulator when a reference moved, merge and epilogue of an item
//   warps 12-15  rope dot products, tiles of both streams in turn
//   warps 16 on  softmax: stream x four (C = 2: eight) heads
// Every wait is bounded; on a timeout the block records ELITEKV_ERR_TIMEOUT, stops issuing work
// and leaves through the common exit (its peers then run into their own limit).
//
// Measured (CUDA events around the kernel, L2 flushed before each step; in brackets the kernel that the
// shape had before): 7B 75 % 16 x 4096 68 us, 3.9 TB/s (78 us, resident tiles on block pairs); ragged
// 64 x [1024, 32768] 840 us, 5.5 TB/s (881, two passes); 13B 32 x 16384 566 us, 4.7 TB/s on 130 of 148
// SMs (773); 50 % 32 x 8192 492 us, 4.4 TB/s on 120 SMs (529); 75 % 32 x 8192 212 us, 5.1 TB/s (237);
// 87.5 % 107 us, 5.0 TB/s (130); S-LRD 184 us, 5.8 TB/s (199).  DRAM traffic 1.01 of the cache bytes.
// Back to back the long ones run at the board's power limit (clock 1.75-1.9 GHz), so bytes moved
// twice and products computed for padding cost time even where they would fit beside the loads.
#include <map>
#include <mutex>
#include <tuple>

#include "tc_ptx.cuh"

namespace {

constexpr int kT = 64;                 // tokens per tile
constexpr int kUnit = 16384;           // 128 columns of a tile: [2 chunks][64 tokens][64 bf16]
constexpr int kMaxRing = 12;           // units in the ring
constexpr int kTileBars = 8;           // tiles whose loads can be under way at once (more than the ring holds)
constexpr float kNoRef = -3.402823466e38f;   // reference maximum of a stream that has seen no finite score: any finite one moves
                                       // it, and a tile of scores that are all -inf has zero probabilities (not NaN)
constexpr int kFinSlots = 3;           // items whose softmax statistics can be under way at once

struct ClArgs {
  const int32_t* items;
  const int4* worker_rec;   // a worker's items and the first of them (PlanArgs)
  const int32_t* page_table;
  float* part_acc;          // [items][n_h][vw]
  float* part_ml;           // [items][n_h][2]
  const bf16* q_rope;       // [B][n_h][2r]
  const bf16* rope_plane;   // [cache rows][n_h 2r]
  int32_t* status;
  long long max_ctx, num_pages;
  int page_shift, page_mask, max_pages_per_seq;
  int vw;                   // value columns of a token (all blocks)
  int ku, vu;               // 128-column units of this block: scores, values
  int vchunk0;              // first 64-column chunk of the values (keys start at 0)
  int joint;                // values are the same columns as keys
  int n_ring;               // units in the ring
  float scale_log2e;
};

struct __align__(8) ClBarriers {
  uint64_t empty[kMaxRing], key_full[kTileBars], val_full[kTileBars];   // val_full: separated latents
  uint64_t q_full, q_free, s_full[2], p_full[2], rope_full[2], rope_free[2], recv_full[2][4];
  uint64_t cmd_full, cmd_done, acc_full, fin_full[kFinSlots];
};

// C blocks per cluster; LPH 16-byte pieces hold a head's rope dims
template <int C_, int LPH_>
struct Cl {
  static constexpr int C = C_, LPH = LPH_;
  static constexpr int HPC = 16 / LPH;            // heads a block finishes
  static constexpr int NH = C * HPC;              // heads of the layer
  static constexpr int NP = (NH + 15) & ~15;      // value-product columns (M = 128 wants multiples of 16)
  static constexpr int QUADS = HPC / 4;           // groups of four heads
  static constexpr int QW = QUADS > 2 ? 2 : 1;    // ... per softmax warp
  static constexpr int SRC = QUADS * 256;         // floats per source: [quads][64 tokens][4 heads]
  static constexpr int ROPE_W = C * 128;          // n_h * 2r
  static constexpr int E = 8 / LPH;               // rope dot products per lane
  static constexpr int THREADS = 512 + 64 * (QUADS / QW);
};

struct ClSmem {
  int q, ring, rope, p, recv, corr, fin, fac, bars, total;
};
template <class K>
__host__ __device__ inline ClSmem cl_layout(int ku, int n_ring) {
  ClSmem s;
  int o = 0;
  s.ring = o;  o += n_ring * kUnit;
  s.q = o;     o += 2 * ku * K::NH * 128;
  // a P tile holds NH heads; the value product's columns past them read what follows (their results
  // are never used), which the buffers behind cover
  s.p = o;     o += 2 * (K::NH / 8) * 1024;
  s.recv = o;  o += 2 * K::C * K::SRC * 4;
  s.rope = o;  o += 2 * K::SRC * 4;
  s.corr = o;  o += 2 * K::NH * 4;
  s.fin = o;   o += kFinSlots * 2 * K::NH * 8;       // [item][stream][head] (m, l)
  s.fac = o;   o += 4 * 2 * K::NH * 4;               // [warp][stream][head] merge factors
  s.bars = o;  o += (int)sizeof(ClBarriers) + 64;    // + tmem base, abort, command
  s.total = o + 1024;
  return s;
}

// Warp-level wait that parks between probes.
__device__ __forceinline__ bool cl_wait(uint32_t bar, uint32_t parity, volatile int* abort_flag, int why) {
  for (unsigned i = 0; i < kWaitLimit; ++i) {
    if (__any_sync(0xffffffffu, mbar_try_wait(bar, parity))) return true;
    if ((i & 255) == 255 && __any_sync(0xffffffffu, *abort_flag != 0)) return false;
  }
  if (*abort_flag == 0) *abort_flag = why;
  return false;
}
__device__ __forceinline__ bool cl_test(uint32_t bar, uint32_t parity) {
  return __any_sync(0xffffffffu, mbar_test_wait(bar, parity));
}

// Position of a role in the worker's sequence of tiles.
struct ClCursor {
  int item, t, nt, seq, tok0, ntok;
};
__device__ __forceinline__ void cl_settle(const int32_t* items, int hi, ClCursor& c) {
  while (c.item < hi) {
    const int4 v = __ldcg((const int4*)items + c.item);
    c.seq = v.x;
    c.tok0 = v.y;
    c.ntok = v.z;
    c.nt = (v.z + kT - 1) / kT;
    if (c.t < c.nt) return;
    c.t -= c.nt;
    ++c.item;
  }
}
__device__ __forceinline__ void cl_advance(const int32_t* items, int hi, ClCursor& c, int by) {
  c.t += by;
  if (c.t < c.nt) return;
  c.t -= c.nt;
  ++c.item;
  cl_settle(items, hi, c);
}

__device__ __forceinline__ uint32_t pack_bf16(float lo, float hi) {
  const bf162 v = __floats2bfloat162_rn(lo, hi);
  return *(const uint32_t*)&v;
}
__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

template <int C, int LPH>
__global__ void __launch_bounds__(Cl<C, LPH>::THREADS, 1)
decode_cl_kernel(const __grid_constant__ CUtensorMap map_lat, const __grid_constant__ CUtensorMap map_q, const ClArgs a) {
  using K = Cl<C, LPH>;
  constexpr int NH = K::NH, NP = K::NP, HPC = K::HPC;
  extern __shared__ unsigned char smem_raw[];
  const uint32_t rank = cluster_ctarank();
  const int worker = blockIdx.x / C;
  const int NR = a.n_ring, ku = a.ku, vu = a.vu;
  const int nut = a.joint ? ku : ku + vu;          // units per tile
  const ClSmem L = cl_layout<K>(ku, NR);

  unsigned char* base = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  unsigned char* s_ring = base + L.ring;
  float* s_corr = (float*)(base + L.corr);
  ClBarriers* bars = (ClBarriers*)(base + L.bars);
  uint32_t* s_tmem = (uint32_t*)(bars + 1);
  volatile int* s_abort = (volatile int*)(s_tmem + 1);
  volatile int* s_cmd = s_abort + 1;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  if (threadIdx.x == 32) {
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&map_lat) : "memory");
    asm volatile("prefetch.tensormap [%0];" ::"l"((uint64_t)&map_q) : "memory");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < kMaxRing; ++i) {
      mbar_init(smem_u32(&bars->empty[i]), 1);
    }
    for (int i = 0; i < kTileBars; ++i) {          // an arrival (with its bytes) per unit
      mbar_init(smem_u32(&bars->key_full[i]), ku);
      mbar_init(smem_u32(&bars->val_full[i]), vu);
    }
    mbar_init(smem_u32(&bars->q_full), 1);
    mbar_init(smem_u32(&bars->q_free), 1);
    for (int s = 0; s < 2; ++s) {
      mbar_init(smem_u32(&bars->s_full[s]), 1);
      mbar_init(smem_u32(&bars->p_full[s]), 1);
      mbar_init(smem_u32(&bars->rope_full[s]), 4);
      mbar_init(smem_u32(&bars->rope_free[s]), K::QUADS / K::QW);
      for (int q = 0; q < 4; ++q) mbar_init(smem_u32(&bars->recv_full[s][q]), 1);
    }
    mbar_init(smem_u32(&bars->cmd_full), 1);
    mbar_init(smem_u32(&bars->cmd_done), 4);
    mbar_init(smem_u32(&bars->acc_full), 1);
    for (int i = 0; i < kFinSlots; ++i) mbar_init(smem_u32(&bars->fin_full[i]), 1);
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
  }
  // TMEM columns: two accumulators of vu blocks x NP, then the two score buffers
  uint32_t tmem_cols = 32;
  while ((int)tmem_cols < 2 * vu * NP + 2 * NH) tmem_cols <<= 1;
  if (warp == 1) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(s_tmem)), "r"(tmem_cols) : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  cluster_sync_all();                    // every peer's barriers exist before any remote store
  tc_fence_after();
  const uint32_t tmem_base = *s_tmem;
  const uint32_t tmem_s0 = tmem_base + 2 * vu * NP;
  // Everything above touched only this cluster's own state; the plan, the queries and the cache
  // come from kernels earlier in the stream.
  ekv_pdl_wait();
  ekv_pdl_trigger();
  // one trip to L2 (worker_first, then the item: 0.7 us more before the first load)
  const int4 rec = __ldcg(a.worker_rec + 2 * worker), rec_n = __ldcg(a.worker_rec + 2 * worker + 1);
  const int item_lo = rec.x, item_hi = rec.y;
  const ClCursor c0{item_lo, 0, (rec_n.x + kT - 1) / kT, rec.z, rec.w, rec_n.x};      // the worker's first tile

  // first cache row of a tile (tiles start on multiples of 64 tokens and pages hold a multiple
  // of 64 tokens, so a tile never straddles pages)
  auto tile_row = [&](const ClCursor& c, bool report) -> int {
    const int t_abs = c.tok0 + c.t * kT;
    if (a.page_table == nullptr) return (int)((long long)c.seq * a.max_ctx + t_abs);
    const int pi = t_abs >> a.page_shift;
    int page = pi < a.max_pages_per_seq ? a.page_table[(long long)c.seq * a.max_pages_per_seq + pi] : -1;
    if (page < 0 || page >= a.num_pages) {
      if (report) ekv_record(a.status, ELITEKV_ERR_BAD_PAGE, c.seq, page);
      page = 0;
    }
    return (int)(((long long)page << a.page_shift) + (t_abs & a.page_mask));
  };
  const uint64_t pol_drop = make_l2_policy_evict_first();

  // ================================================================ warps 0, 3: latent tiles
  // Ring units are dealt alternately.  A tile's cache row is a dependent trip to the page table (1000
  // clocks), so the rows of 32 tiles of an item are looked up at once, one per lane.
  if (warp == 0 || warp == 3) {
    const bool report = warp == 0 && rank == 0;
    unsigned slot = 0, par = 0, g = 0, n = warp == 3 ? 1 : 0;     // n even: this warp's unit
    int my_row = 0, first_row = -1;                        // rows of tiles [first_row, first_row + 32) of the item
    ClCursor c = c0;
    bool ok = true;
    while (ok && c.item < item_hi) {
      if (c.t == 0 || c.t == first_row + 32) {
        first_row = c.t;
        ClCursor m = c;
        m.t += lane;
        my_row = m.t < c.nt ? tile_row(m, report) : 0;
      }
      const int row = __shfl_sync(0xffffffffu, my_row, c.t - first_row);
      for (int u = 0; u < nut; ++u, ++n) {
        if ((n & 1) == 0) {
          ok = cl_wait(smem_u32(&bars->empty[slot]), par ^ 1, s_abort, 1);
          if (!ok) break;
          // key units first, then (separated latents) value units
          const int chunk = u < ku ? (int)rank * 2 * ku + 2 * u : a.vchunk0 + (int)rank * 2 * vu + 2 * (u - ku);
          if (elect_one()) {
            const uint32_t fb = smem_u32(u < ku ? &bars->key_full[g % kTileBars] : &bars->val_full[g % kTileBars]);
            mbar_expect_tx(fb, (uint32_t)kUnit);
            tma_load_3d_hint(smem_u32(s_ring) + slot * kUnit, &map_lat, 0, row, chunk, fb, pol_drop);
          }
          __syncwarp();
        }
        if (++slot == (unsigned)NR) { slot = 0; par ^= 1; }
      }
      ++g;
      cl_advance(a.items, item_hi, c, 1);
    }
  }
  // ================================================================ warp 2: this block's slice of the item's queries
  else if (warp == 2) {
    const uint64_t pol_keep = make_l2_policy_evict_last();
    for (int item = item_lo; item < item_hi; ++item) {
      const int seq = item == item_lo ? rec.z : __ldcg(a.items + 4 * item);
      // the previous item's last score product has read the old ones
      if (item > item_lo && !cl_wait(smem_u32(&bars->q_free), (unsigned)(item - item_lo - 1) & 1, s_abort, 12)) break;
      if (elect_one()) {
        const uint32_t qb = smem_u32(&bars->q_full);
        mbar_expect_tx(qb, (uint32_t)(2 * ku * NH * 128));
        tma_load_3d_hint(smem_u32(base + L.q), &map_q, 0, seq * NH, (int)rank * 2 * ku, qb, pol_keep);
      }
      __syncwarp();
    }
  }
  // ================================================================ warp 1: MMA issuer
  else if (warp == 1) {
    constexpr uint32_t idesc_s = make_idesc(64, NH, 0, 0);   // S = C . Q^T, K-major both
    constexpr uint32_t idesc_pv = make_idesc(128, NP, 1, 1);     // acc = C^T . P, MN-major both
    constexpr uint32_t hi_sw = desc_hi(1024, 2);                 // 128-byte swizzle, 1024 bytes between 8-row groups
    constexpr uint32_t hi_p = desc_hi(kT * 16, 0);               // P: no swizzle, 1024 bytes between 8-head groups
    constexpr uint32_t kQChunk16 = (NH * 128) >> 4;
    // 14-bit start-address fields: the shared-window address of a block of non-zero rank carries
    // the rank above the offset, which must not spill into the neighbouring descriptor fields
    auto lo16 = [&](const unsigned char* p) { return ((smem_u32(p) >> 4) & 0x3FFFu) | (1u << 16); };
    const uint32_t ring16 = (smem_u32(s_ring) >> 4) & 0x3FFFu, q16 = lo16(base + L.q);
    const uint32_t empty0 = smem_u32(&bars->empty[0]);
    ClCursor cs = c0, cp = c0;
    unsigned s_slot = 0;                             // ring position of the first unit of the next score product
    unsigned p_slot = a.joint ? 0 : ku;              // ... and of the next value product
    unsigned gs = 0, gp = 0;                         // tiles whose scores / values have been issued
    unsigned n_q = 0, n_cmd = 0;                     // items whose queries were taken, commands given
    bool epi_open = false;
    unsigned idle = 0;
    while (cp.item < item_hi) {
      bool moved = false;
      // ---- value product of the oldest tile, as soon as all blocks' probabilities are here (and, with
      //      separated latents, its value units: the score product has waited for the others)
      if (gp < gs && cl_test(smem_u32(&bars->p_full[gp & 1]), (gp >> 1) & 1) &&
          (a.joint || cl_test(smem_u32(&bars->val_full[gp % kTileBars]), (gp / kTileBars) & 1))) {
        const unsigned s = gp & 1;
        const bool first = cp.t < 2;                 // first tile of this stream in the item: overwrites
        bool mv = false;                             // a reference moved: rescale this stream's output first
#pragma unroll
        for (int h = 0; h < NH; h += 32)
          if (NH % 32 == 0 || h + lane < NH) mv |= s_corr[s * NH + h + lane] != 1.f;
        fence_proxy_async();                         // P arrived through ordinary (remote) stores
        tc_fence_after();
        const int nvalid = min(kT, cp.ntok - cp.t * kT);
        const bool last = cp.t == cp.nt - 1;
        const uint32_t lo_p = desc_lo(smem_u32(base + L.p) + s * (NH / 8) * 1024, 128);
        uint32_t d = tmem_base + s * vu * NP;
        if (first) {
          if (epi_open) {                            // the previous item's output still leaves TMEM
            if (!cl_wait(smem_u32(&bars->cmd_done), (n_cmd - 1) & 1, s_abort, 13)) break;
            tc_fence_after();
            epi_open = false;
          }
        } else if (__any_sync(0xffffffffu, mv)) {
          if (elect_one()) {
            *s_cmd = (int)s;
            mbar_arrive(smem_u32(&bars->cmd_full));
          }
          __syncwarp();
          if (!cl_wait(smem_u32(&bars->cmd_done), n_cmd & 1, s_abort, 14)) break;
          tc_fence_after();
          ++n_cmd;
        }
        if (nvalid == kT) {
          if (elect_one()) {
            unsigned sl = p_slot;
#pragma unroll 1
            for (int u = 0; u < vu; ++u, d += NP) {
              const uint32_t la = (ring16 + sl * (kUnit >> 4)) | (512u << 16);     // two 64-column atoms 8 KB apart
              tc_mma_w(d, la, hi_sw, lo_p, hi_p, idesc_pv, !first);
              tc_mma_w(d, la + 128, hi_sw, lo_p + 16, hi_p, idesc_pv, 1);          // +16 tokens: 2048 bytes in A, 256 in P
              tc_mma_w(d, la + 256, hi_sw, lo_p + 32, hi_p, idesc_pv, 1);
              tc_mma_w(d, la + 384, hi_sw, lo_p + 48, hi_p, idesc_pv, 1);
              tc_commit(empty0 + sl * 8);
              if (++sl == (unsigned)NR) sl = 0;
            }
            if (last) {
              tc_commit(smem_u32(&bars->acc_full));
              *s_cmd = 2;                            // item complete: merge and write it
              mbar_arrive(smem_u32(&bars->cmd_full));
            }
          }
        } else {
          // ragged end of a sequence: rows past its last token inside the last 16-token step become
          // exact zeros so that zero-probability rows cannot inject NaN/Inf bit patterns
          const int ksteps = (nvalid + 15) >> 4;
          unsigned sl = p_slot;
          for (int u = 0; u < vu; ++u) {
            unsigned char* unit = s_ring + sl * kUnit;
            for (int e = lane; e < (ksteps * 16 - nvalid) * 16; e += 32) {
              const int rrow = nvalid + (e >> 4), c16 = e & 15;
              *(uint4*)(unit + (c16 >> 3) * 8192 + rrow * 128 + (c16 & 7) * 16) = make_uint4(0, 0, 0, 0);
            }
            if (++sl == (unsigned)NR) sl = 0;
          }
          fence_proxy_async();
          __syncwarp();
          if (elect_one()) {
            sl = p_slot;
#pragma unroll 1
            for (int u = 0; u < vu; ++u, d += NP) {
              const uint32_t la = (ring16 + sl * (kUnit >> 4)) | (512u << 16);
              for (int k = 0; k < ksteps; ++k)
                tc_mma_w(d, la + 128 * k, hi_sw, lo_p + 16 * k, hi_p, idesc_pv, !first || k > 0);
              tc_commit(empty0 + sl * 8);
              if (++sl == (unsigned)NR) sl = 0;
            }
            if (last) {
              tc_commit(smem_u32(&bars->acc_full));
              *s_cmd = 2;
              mbar_arrive(smem_u32(&bars->cmd_full));
            }
          }
        }
        __syncwarp();
        if (last) {
          ++n_cmd;
          epi_open = true;
        }
        p_slot += nut;
        if (p_slot >= (unsigned)NR) p_slot -= NR;
        ++gp;
        cl_advance(a.items, item_hi, cp, 1);
        moved = true;
      }
      // ---- score product of the next tile (at most two tiles ahead of the value product: one per stream)
      if (cs.item < item_hi && gs < gp + 2 && cl_test(smem_u32(&bars->key_full[gs % kTileBars]), (gs / kTileBars) & 1) &&
          (cs.t != 0 || cl_test(smem_u32(&bars->q_full), n_q & 1))) {
        const unsigned s = gs & 1;
        const bool q_last = cs.t == cs.nt - 1;
        if (elect_one()) {
          // arm the stream's probabilities of this tile: bf16 [NH][64] + a factor per head
          mbar_expect_tx(smem_u32(&bars->p_full[s]), (uint32_t)(NH * kT * 2 + NH * 4));
          const uint32_t d = tmem_s0 + s * NH;
          uint32_t lb = q16;
          unsigned sl = s_slot;
#pragma unroll 1
          for (int u = 0; u < ku; ++u, lb += 2 * kQChunk16) {
            const uint32_t la = (ring16 + sl * (kUnit >> 4)) | (1u << 16);
#pragma unroll
            for (int ks = 0; ks < 8; ++ks)           // two 64-column chunks, +32 bytes along K per step
              tc_mma_w(d, la + (ks >> 2) * 512 + 2 * (ks & 3), hi_sw, lb + (ks >> 2) * kQChunk16 + 2 * (ks & 3), hi_sw,
                       idesc_s, (u + ks) != 0);
            if (!a.joint) tc_commit(empty0 + sl * 8);          // a key unit of separated latents is done
            if (++sl == (unsigned)NR) sl = 0;
          }
          tc_commit(smem_u32(&bars->s_full[s]));
          if (q_last) tc_commit(smem_u32(&bars->q_free));
        }
        __syncwarp();
        if (q_last) ++n_q;
        s_slot += nut;
        if (s_slot >= (unsigned)NR) s_slot -= NR;
        ++gs;
        cl_advance(a.items, item_hi, cs, 1);
        moved = true;
      }
      if (moved) {
        idle = 0;
      } else {
        ++idle;
        if ((idle & 1023) == 1023 && __any_sync(0xffffffffu, *s_abort != 0)) break;
        if (idle > kSpinLimit) {
          if (*s_abort == 0) *s_abort = 4;
          break;
        }
      }
    }
  }
  // ================================================================ warps 4-7: senders
  else if (warp >= 4 && warp < 8) {
    const int quarter = warp & 3;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const uint32_t b0 = smem_u32(base);
    uint32_t rb[C];                                  // shared-window base of every block of the cluster
#pragma unroll
    for (int p = 0; p < C; ++p) rb[p] = map_to_cta(b0, p);
    const uint32_t off_bar0 = (uint32_t)((unsigned char*)&bars->recv_full[0][0] - base);
    const int t = 16 * quarter + (lane & 15);        // token of this lane's score row (M = 64: 16 rows per warp)
    ClCursor c = c0;
    for (unsigned g = 0; c.item < item_hi; ++g, cl_advance(a.items, item_hi, c, 1)) {
      const unsigned s = g & 1;
      const uint32_t off_recv = (uint32_t)L.recv + (s * C + rank) * (K::SRC * 4) + t * 16;
      const uint32_t off_bar = off_bar0 + s * 32;
      if (!cl_wait(smem_u32(&bars->s_full[s]), (g >> 1) & 1, s_abort, 6)) break;
      tc_fence_after();
      const uint32_t tm = tmem_s0 + s * NH + lane_base;
#pragma unroll
      for (int col = 0; col < NH; col += 32) {       // 32 (or a last 8) columns at a time
        float v[32];
        if (col + 32 <= NH) tc_ld32(tm + col, v);
        else tc_ld8(tm + col, v);
        tc_wait_ld();
        if (lane < 16) {
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            if (col + 4 * j < NH) {
              const int h = col + 4 * j, p = h / HPC, quad = (h % HPC) / 4;
              st_async_f4(rb[p] + off_recv + quad * 1024, make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]),
                          rb[p] + off_bar + quad * 8);
            }
          }
        }
      }
      tc_fence_before();
    }
  }
  // ================================================================ warps 8-11: rescale, merge, epilogue
  else if (warp >= 8 && warp < 12) {
    const int quarter = warp & 3;
    const uint32_t lane_base = (uint32_t)(quarter * 32) << 16;
    const float2* s_fin = (const float2*)(base + L.fin);
    float* fac = (float*)(base + L.fac) + quarter * 2 * NH;
    ClCursor c = c0;
    unsigned n_cmd = 0, g0 = 0;                      // commands taken; tiles before the item
    while (c.item < item_hi) {
      if (!cl_wait(smem_u32(&bars->cmd_full), n_cmd & 1, s_abort, 15)) break;
      ++n_cmd;
      const int cmd = *s_cmd;
      if (cmd < 2) {                                 // rescale stream cmd's accumulator
        tc_fence_after();
        for (int u = 0; u < vu; ++u) {
#pragma unroll 1
          for (int col = 0; col < NH; col += 8) {
            float v[8];
            const uint32_t addr = tmem_base + (uint32_t)((cmd * vu + u) * NP + col) + lane_base;
            tc_ld8(addr, v);
            tc_wait_ld();
#pragma unroll
            for (int j = 0; j < 8; ++j) v[j] *= s_corr[cmd * NH + col + j];
            tc_st8(addr, v);
          }
        }
        tc_wait_st();
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive(smem_u32(&bars->cmd_done));
        continue;
      }
      const int k = c.item - item_lo;
      const int slot = k % kFinSlots;
      const bool both = c.nt > 1;
      const int only = (int)(g0 & 1);                // a one-tile item went through one stream
      if (threadIdx.x == 256) mbar_expect_tx(smem_u32(&bars->fin_full[slot]), (uint32_t)((both ? 2 : 1) * NH * 8));
      if (!cl_wait(smem_u32(&bars->fin_full[slot]), (unsigned)(k / kFinSlots) & 1, s_abort, 16)) break;
      // merge factors of the two streams (every warp its own copy), and the item's statistics
      for (int v = lane; v < NH; v += 32) {
        const float2 x0 = s_fin[(slot * 2 + 0) * NH + v], x1 = s_fin[(slot * 2 + 1) * NH + v];
        const float m0 = both || only == 0 ? x0.x : -INFINITY, m1 = both || only == 1 ? x1.x : -INFINITY;
        const float M = fmaxf(m0, m1);
        const float f0 = m0 == -INFINITY ? 0.f : exp2f(m0 - M), f1 = m1 == -INFINITY ? 0.f : exp2f(m1 - M);
        fac[v] = f0;
        fac[NH + v] = f1;
        if (rank == 0 && quarter == 0)
          __stcg((float2*)(a.part_ml + ((size_t)c.item * NH + v) * 2),      // (no finite score in the whole item: weightless)
                 make_float2(M > kNoRef ? M : -INFINITY, (f0 != 0.f ? x0.y * f0 : 0.f) + (f1 != 0.f ? x1.y * f1 : 0.f)));
      }
      __syncwarp();
      // a [128 columns x heads] block leaves TMEM with one thread per latent column: for a fixed
      // head the lanes of a warp hold 32 consecutive columns, 128-byte stores from registers
      // (The factors are read before the stores: behind one, each read of shared memory would wait for it.  From the
      // last value product to the last store 2.1 us, 2.9 with a factor read per store.)
      float* dst = a.part_acc + (size_t)c.item * NH * a.vw + (size_t)rank * vu * 128 + quarter * 32 + lane;
      if (!cl_wait(smem_u32(&bars->acc_full), (unsigned)k & 1, s_abort, 10)) break;
      tc_fence_after();
#pragma unroll 1
      for (int col = 0; col < NH; col += 8) {
        float f0[8], f1[8];
#pragma unroll
        for (int j = 0; j < 8; j += 4) {
          *(float4*)&f0[j] = *(const float4*)&fac[col + j];
          *(float4*)&f1[j] = *(const float4*)&fac[NH + col + j];
        }
#pragma unroll 1
        for (int u = 0; u < vu; ++u) {
          float v0[8], v1[8];
          const uint32_t at = tmem_base + (uint32_t)(u * NP + col) + lane_base;
          if (both || only == 0) tc_ld8(at, v0);
          if (both || only == 1) tc_ld8(at + vu * NP, v1);
          tc_wait_ld();
          float* out = dst + (size_t)col * a.vw + u * 128;
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            float y = 0.f;
            if (both || only == 0) y = v0[j] * f0[j];
            if (both || only == 1) y = fmaf(v1[j], f1[j], y);
            __stcg(out + (size_t)j * a.vw, y);
          }
        }
      }
      tc_fence_before();
      __syncwarp();                                  // the factors may be overwritten
      if (lane == 0) mbar_arrive(smem_u32(&bars->cmd_done));
      g0 += (unsigned)c.nt;
      cl_advance(a.items, item_hi, c, c.nt - c.t);
    }
  }
  // ================================================================ warps 12-15: rope dot products
  else if (warp >= 12 && warp < 16) {
    // A block's heads have 256 bytes of a rope row.  Lane of load i takes 16 of them of token
    // 16 quarter + 2 i + (lane >> 4): whole 256-byte pieces per half warp, straight into registers one
    // tile ahead, and drawn into L2 kAhead tiles ahead of that.
    constexpr int kAhead = 2;
    const int quarter = warp & 3, piece = lane & 15;
    const bf16* plane = a.rope_plane + rank * 128 + piece * 8;
    ClCursor c = c0, ld = c0, pf = c0;               // tiles computed, loaded, prefetched next
    int row_q[kAhead + 1] = {};                      // cache rows of the tiles between ld and pf
    int n_q = 0;
    uint4 raw[8];
    auto prefetch = [&] {
      if (pf.item >= item_hi) return;
      const int row = tile_row(pf, false), nvalid = min(kT, pf.ntok - pf.t * kT);
      // 16 rows of two 128-byte lines each: one line per lane
      const int t = 16 * quarter + (lane >> 1);
      if (t < nvalid)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.rope_plane + ((size_t)row + t) * K::ROPE_W + rank * 128 + (lane & 1) * 64));
#pragma unroll
      for (int i = 0; i <= kAhead; ++i)
        if (i == n_q) row_q[i] = row;
      ++n_q;
      cl_advance(a.items, item_hi, pf, 1);
    };
    auto load = [&] {
      if (ld.item >= item_hi) return;
      const int nvalid = min(kT, ld.ntok - ld.t * kT);
      const bf16* src = plane + (size_t)row_q[0] * K::ROPE_W;
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int t = 16 * quarter + 2 * i + (lane >> 4);
        raw[i] = make_uint4(0, 0, 0, 0);
        if (t < nvalid) raw[i] = ld_stream_v4(src + (size_t)t * K::ROPE_W);
      }
#pragma unroll
      for (int i = 0; i < kAhead; ++i) row_q[i] = row_q[i + 1];
      --n_q;
      cl_advance(a.items, item_hi, ld, 1);
    };
#pragma unroll
    for (int i = 0; i <= kAhead; ++i) prefetch();
    load();
    float qr[8];
    for (unsigned g = 0; c.item < item_hi; ++g, cl_advance(a.items, item_hi, c, 1)) {
      const unsigned s = g & 1;
      if (c.t == 0) {
        const uint32_t* src = (const uint32_t*)(a.q_rope + (size_t)c.seq * K::ROPE_W + rank * 128 + piece * 8);
#pragma unroll
        for (int k = 0; k < 4; ++k) {                // 4-byte aligned
          const uint32_t v = __ldcg(src + k);
          qr[2 * k] = bf_lo(v);
          qr[2 * k + 1] = bf_hi(v);
        }
      }
      float rp[K::E];
      {
        float d[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint32_t* w = (const uint32_t*)&raw[i];
          float acc = 0.f;
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            acc = fmaf(qr[2 * k], bf_lo(w[k]), acc);
            acc = fmaf(qr[2 * k + 1], bf_hi(w[k]), acc);
          }
          d[i] = acc;
        }
        // sum over the LPH lanes of a head, each lane ending with E tokens of its own
        if constexpr (LPH == 1) {
#pragma unroll
          for (int e = 0; e < 8; ++e) rp[e] = d[e];
        } else {
          const bool o0 = lane & 1, o1 = lane & 2;
          float d1[4];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            const float give = o0 ? d[2 * k] : d[2 * k + 1], keep = o0 ? d[2 * k + 1] : d[2 * k];
            d1[k] = keep + __shfl_xor_sync(0xffffffffu, give, 1);
          }
#pragma unroll
          for (int e = 0; e < K::E; ++e) {
            if constexpr (LPH == 2) {
              rp[e] = d1[e];
            } else {
              const float give = o1 ? d1[2 * e] : d1[2 * e + 1], keep = o1 ? d1[2 * e + 1] : d1[2 * e];
              rp[e] = keep + __shfl_xor_sync(0xffffffffu, give, 2);
            }
          }
        }
      }
      load();
      prefetch();
      // the stream's softmax warps have taken tile g - 2
      if (g >= 2 && !cl_wait(smem_u32(&bars->rope_free[s]), ((g >> 1) - 1) & 1, s_abort, 5)) break;
      const int hh = piece / LPH;
      float* dst = (float*)(base + L.rope) + s * K::SRC + (hh >> 2) * 256 +
                   (16 * quarter + 2 * (lane & (LPH - 1)) + (lane >> 4)) * 4 + (hh & 3);
#pragma unroll
      for (int e = 0; e < K::E; ++e) dst[8 * LPH * e] = rp[e];
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->rope_full[s]));
    }
  }
  // ================================================================ warps 16 on: softmax
  else if (warp >= 16) {
    constexpr int QW = K::QW, WPS = K::QUADS / QW;   // quads per warp, warps per stream
    const int s = (warp - 16) / WPS, q0 = (warp - 16) % WPS * QW;            // stream; first quad
    const int v0 = (int)rank * HPC + 4 * q0;                                 // first head
    const uint32_t b0 = smem_u32(base);
    uint32_t rb[C];
#pragma unroll
    for (int p = 0; p < C; ++p) rb[p] = map_to_cta(b0, p);
    const uint32_t off_p_bar = (uint32_t)((unsigned char*)&bars->p_full[s] - base);
    const float* recv = (const float*)(base + L.recv) + s * C * K::SRC + q0 * 256 + lane * 4;    // tokens lane, lane + 32
    const float* rope = (const float*)(base + L.rope) + s * K::SRC + q0 * 256 + lane * 4;
    const uint32_t off_p = (uint32_t)L.p + (uint32_t)(s * (NH / 8) * 1024 + (v0 >> 3) * 1024 + (lane >> 3) * 128 + (lane & 7) * 16 + (v0 & 7) * 2);
    const uint32_t off_corr = (uint32_t)L.corr + (uint32_t)(s * NH + v0) * 4u;
    float m_ref[4 * QW], l_sum[4 * QW];
    bool fresh = true;                               // the next tile is this stream's first of its item
    unsigned par = 0;
    ClCursor c = c0;
    if (s) cl_advance(a.items, item_hi, c, 1);
    while (c.item < item_hi) {
      if (lane < QW) mbar_expect_tx(smem_u32(&bars->recv_full[s][q0 + lane]), (uint32_t)(C * 1024));
      if (fresh) {
#pragma unroll
        for (int h = 0; h < 4 * QW; ++h) {
          m_ref[h] = kNoRef;
          l_sum[h] = 0.f;
        }
      }
      const int nv = c.ntok - c.t * kT;                // tokens of the tile
      ClCursor nx = c;
      cl_advance(a.items, item_hi, nx, 2);
      // ---- rope part, computed ahead
      if (!cl_wait(smem_u32(&bars->rope_full[s]), par, s_abort, 8)) break;
      float x[2][4 * QW];
#pragma unroll
      for (int e = 0; e < 2; ++e)
#pragma unroll
        for (int q = 0; q < QW; ++q) *(float4*)&x[e][4 * q] = *(const float4*)(rope + q * 256 + e * 128);
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&bars->rope_free[s]));
      // ---- full scores: sources in rank order
      bool ok = true;
#pragma unroll
      for (int q = 0; q < QW; ++q) ok = ok && cl_wait(smem_u32(&bars->recv_full[s][q0 + q]), par, s_abort, 9);
      if (!ok) break;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const bool live = lane + 32 * e < nv;
#pragma unroll
        for (int q = 0; q < QW; ++q) {
          float4 y = *(const float4*)(recv + q * 256 + e * 128);
#pragma unroll
          for (int p = 1; p < C; ++p) {
            const float4 z = *(const float4*)(recv + p * K::SRC + q * 256 + e * 128);
            y.x += z.x; y.y += z.y; y.z += z.z; y.w += z.w;
          }
          x[e][4 * q] = live ? (x[e][4 * q] + y.x) * a.scale_log2e : -INFINITY;
          x[e][4 * q + 1] = live ? (x[e][4 * q + 1] + y.y) * a.scale_log2e : -INFINITY;
          x[e][4 * q + 2] = live ? (x[e][4 * q + 2] + y.z) * a.scale_log2e : -INFINITY;
          x[e][4 * q + 3] = live ? (x[e][4 * q + 3] + y.w) * a.scale_log2e : -INFINITY;
        }
      }
      // ---- does a reference have to move?  (always on an item's first tile; rarely after it)
      bool over = false;
#pragma unroll
      for (int h = 0; h < 4 * QW; ++h) over |= fmaxf(x[0][h], x[1][h]) > m_ref[h] + 8.f;      // head-room of 2^8
      float corr[4 * QW];
#pragma unroll
      for (int h = 0; h < 4 * QW; ++h) corr[h] = 1.f;
      if (__any_sync(0xffffffffu, over)) {
#pragma unroll
        for (int h = 0; h < 4 * QW; ++h) {
          const float tm = ord2f(__reduce_max_sync(0xffffffffu, f2ord(fmaxf(x[0][h], x[1][h]))));
          if (tm > m_ref[h] + 8.f) {
            corr[h] = exp2f(m_ref[h] - tm);          // first tile of an item: 0, nothing to rescale yet
            m_ref[h] = tm;
            l_sum[h] *= corr[h];
            if (fresh) corr[h] = 1.f;
          }
        }
      }
      // ---- probabilities, rounded as the tensor core will see them, into every block's P tile
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        uint32_t w[2 * QW];
#pragma unroll
        for (int k = 0; k < 2 * QW; ++k) {
          w[k] = pack_bf16(exp2f(x[e][2 * k] - m_ref[2 * k]), exp2f(x[e][2 * k + 1] - m_ref[2 * k + 1]));
          l_sum[2 * k] += bf_lo(w[k]);
          l_sum[2 * k + 1] += bf_hi(w[k]);
        }
#pragma unroll
        for (int p = 0; p < C; ++p) {
          if constexpr (QW == 2) st_async_v4(rb[p] + off_p + e * 512, w[0], w[1], w[2], w[3], rb[p] + off_p_bar);
          else st_async_v2(rb[p] + off_p + e * 512, w[0], w[1], rb[p] + off_p_bar);
        }
      }
      if (lane < C) {        // the factors: lane p sends to block p
        uint32_t dst = rb[0];
#pragma unroll
        for (int p = 1; p < C; ++p) dst = lane == p ? rb[p] : dst;
#pragma unroll
        for (int q = 0; q < QW; ++q)
          st_async_f4(dst + off_corr + 16 * q, make_float4(corr[4 * q], corr[4 * q + 1], corr[4 * q + 2], corr[4 * q + 3]), dst + off_p_bar);
      }
      // ---- this stream's last tile of the item: its softmax statistics go to every block
      fresh = nx.item != c.item;
      if (fresh) {
        const int k = c.item - item_lo;
        const uint32_t off_fin = (uint32_t)L.fin + (uint32_t)(((k % kFinSlots) * 2 + s) * NH + v0) * 8u;
        const uint32_t off_bar = (uint32_t)((unsigned char*)&bars->fin_full[k % kFinSlots] - base);
#pragma unroll
        for (int h = 0; h < 4 * QW; h += 2) {
          const float l0 = warp_sum(l_sum[h]), l1 = warp_sum(l_sum[h + 1]);
          if (lane == 0)
#pragma unroll
            for (int p = 0; p < C; ++p)
              st_async_f4(rb[p] + off_fin + 8 * h, make_float4(m_ref[h], l0, m_ref[h + 1], l1), rb[p] + off_bar);
        }
      }
      c = nx;
      par ^= 1;
    }
  }

  // ============================================================== teardown
  __syncwarp();
  if (*s_abort) drain_after_abort();
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x == 0 && *s_abort) ekv_record(a.status, ELITEKV_ERR_TIMEOUT, worker | (*s_abort << 16), (int)rank);
  cluster_sync_all();                    // no block leaves while a peer may still write into it
  if (warp == 1) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem_base), "r"(tmem_cols) : "memory");
  }
}

// ---------------------------------------------------------------- host side
// 3-D view of a [rows][cols] bf16 matrix as [cols / 64][rows][64]: a box [box_chunks][box_rows][64]
// arrives as one 128-byte-swizzled operand tile per 64-column chunk.
int cl_make_map(CUtensorMap* m, const void* ptr, unsigned long long rows, unsigned long long cols, unsigned box_rows,
                unsigned box_chunks) {
  EncodeTiledFn fn = encode_fn();
  if (!fn) return ELITEKV_ERR_CUDA;
  cuuint64_t dims[3] = {64, rows, cols / 64};
  cuuint64_t strides[2] = {cols * sizeof(bf16), 64 * sizeof(bf16)};
  cuuint32_t box[3] = {64, box_rows, box_chunks};
  cuuint32_t estr[3] = {1, 1, 1};
  CUresult r = fn(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(ptr), dims, strides, box, estr,
                  CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                  CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  return r == CUDA_SUCCESS ? ELITEKV_OK : ELITEKV_ERR_CUDA;
}

// Blocks per cluster: the block's heads have 128 rope columns together.
int cl_c(const elitekv_layer* L) { return L->n_h * 2 * L->r / 128; }

// Calls f with the kernel and its traits for the layer's shape.
template <class F>
int cl_with(const elitekv_layer* L, F f) {
  switch (cl_c(L) * 10 + 2 * L->r / 8) {
    case 21: return f(decode_cl_kernel<2, 1>, Cl<2, 1>());
    case 42: return f(decode_cl_kernel<4, 2>, Cl<4, 2>());
    case 52: return f(decode_cl_kernel<5, 2>, Cl<5, 2>());
    case 84: return f(decode_cl_kernel<8, 4>, Cl<8, 4>());
    default: return -1;
  }
}

// ring units and shared memory of a shape; 0 when it does not fit
template <class K>
int cl_ring(const elitekv_layer* L, int* smem) {
  const int ku = L->kw / 128 / K::C, vu = L->vw / 128 / K::C;
  const int nut = L->voff == 0 ? ku : ku + vu;
  if (2 * vu * K::NP + 2 * K::NH > 512) return 0;
  int nr = (L->smem_optin - cl_layout<K>(ku, 0).total) / kUnit;
  if (nr > kMaxRing) nr = kMaxRing;
  if (nr < 2 * nut || nr / nut + 2 > kTileBars) return 0;       // a tile per stream; a barrier per tile under way
  *smem = cl_layout<K>(ku, nr).total;
  return nr;
}

template <class K>
cudaLaunchAttribute cl_cluster_attr() {
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = K::C;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  return at;
}

}  // namespace

// Shapes: n_h 2r = 128 C with C in {2, 4, 5, 8} (two, four, or eight heads per 64 rope columns), and
// key and value latents that split into whole 128-column units per block.
int ekv_cl_supported(const elitekv_layer* L, const elitekv_cache* cache) {
  if (L->r <= 0 || (L->n_h * 2 * L->r) % 128 != 0 || (2 * L->r) % 8 != 0) return 0;
  const int C = cl_c(L);
  if (C < 2 || C > 8 || L->n_h % C != 0 || 2 * L->r / 8 * (L->n_h / C) != 16) return 0;
  if (L->kw % (128 * C) != 0 || L->vw % (128 * C) != 0) return 0;
  int smem = 0;
  if (cl_with(L, [&](auto, auto k) { return cl_ring<decltype(k)>(L, &smem); }) <= 0) return 0;
  if (cache && cache->page_table && (cache->page_size % kT != 0)) return 0;
  return 1;
}

// Clusters the device holds at once.  A property of kernel, ring size and device that takes the
// runtime milliseconds to work out, so each combination is asked once per process.
int ekv_cl_max_clusters(const elitekv_layer* L) {
  static std::mutex mutex;
  static std::map<std::tuple<int, int, int>, int> known;      // (device, blocks per cluster, shared memory)
  const int n = cl_with(L, [&](auto kern, auto k) -> int {
    using K = decltype(k);
    int smem = 0, n_cl = 0;
    if (cl_ring<K>(L, &smem) <= 0) return 0;
    std::lock_guard<std::mutex> lock(mutex);
    const auto key = std::make_tuple(L->device, K::C, smem);
    const auto it = known.find(key);
    if (it != known.end()) return it->second;
    if (ekv_allow_smem(kern, smem) != cudaSuccess) return 0;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(K::C);
    cfg.blockDim = dim3(K::THREADS);
    cfg.dynamicSmemBytes = smem;
    cudaLaunchAttribute attr[1] = {cl_cluster_attr<K>()};
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    if (cudaOccupancyMaxActiveClusters(&n_cl, kern, &cfg) != cudaSuccess) {
      cudaGetLastError();
      return 0;
    }
    known[key] = n_cl;
    return n_cl;
  });
  return n > 0 ? n : 0;
}

int ekv_cl_workers(const elitekv_layer* L) { return L->cl_clusters > 0 ? L->cl_clusters : 1; }
int ekv_cl_max_items(const elitekv_layer* L, int B) { return ekv_cl_workers(L) + B; }

int ekv_launch_decode_cl(const elitekv_layer* L, const elitekv_cache* cache, const CacheView& cv,
                         const void* q_rope, const void* q_abs, int B, const DecodeScratch& ws,
                         cudaStream_t st) {
  if (!ekv_cl_supported(L, cache) || ws.rows > 1) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  const unsigned long long rows =
      cv.page_table ? (unsigned long long)cv.num_pages << cv.page_shift : (unsigned long long)cv.max_ctx * cv.n_seqs;
  if (rows >= (1ull << 31)) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  return cl_with(L, [&](auto kern, auto k) -> int {
    using K = decltype(k);
    int smem = 0;
    ClArgs a;
    a.n_ring = cl_ring<K>(L, &smem);
    a.ku = L->kw / 128 / K::C;
    a.vu = L->vw / 128 / K::C;
    a.joint = L->voff == 0;
    a.vchunk0 = L->voff / 64;
    CUtensorMap m_lat, m_q;
    int rc = cl_make_map(&m_lat, cache->latent, rows, L->d_c, kT, 2);
    if (rc == ELITEKV_OK)
      rc = cl_make_map(&m_q, q_abs, (unsigned long long)B * L->n_h, L->kw, K::NH, 2 * a.ku);
    if (rc != ELITEKV_OK) return rc;
    a.items = ws.items;
    a.worker_rec = ws.worker_rec;
    a.page_table = cv.page_table;
    a.part_acc = ws.part_acc;
    a.part_ml = ws.part_ml;
    a.q_rope = (const bf16*)q_rope;
    a.rope_plane = (const bf16*)cache->rope;
    a.status = L->d_status;
    a.max_ctx = cv.max_ctx;
    a.num_pages = cv.num_pages;
    a.page_shift = cv.page_shift;
    a.page_mask = cv.page_mask;
    a.max_pages_per_seq = cv.max_pages_per_seq;
    a.vw = L->vw;
    a.scale_log2e = L->scale * 1.4426950408889634f;
    EKV_CUDA_OK(ekv_allow_smem(kern, smem));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(ws.n_workers * K::C));
    cfg.blockDim = dim3(K::THREADS);
    cfg.dynamicSmemBytes = (size_t)smem;
    cfg.stream = st;
    cudaLaunchAttribute attr[2] = {cl_cluster_attr<K>()};
    attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    // Clusters of an odd number of blocks only all fit when they are placed on an empty device: launched
    // while the kernel before drains, one of the 26 clusters of 13B waited for another to end (875 us
    // a step instead of 618).  The others start as dependents (7B B16 74.7 us a step, 76.7 without).
    cfg.numAttrs = K::C % 2 ? 1 : 2;
    EKV_CUDA_OK(cudaLaunchKernelEx(&cfg, kern, m_lat, m_q, a));
    EKV_CUDA_OK(cudaGetLastError());
    return ELITEKV_OK;
  });
}
