// RoPElite search scoring (Algorithm 1, Section 3.1), all heads of all layers side by side.
//
// For one head the search compares the attention scores s = q K^T (pre-softmax, Section 2.1) with
// RoPE on every chunk against the scores with RoPE on the elite chunks e plus one candidate j
// only, over every decoding step of a calibration sequence (query position m, key position
// n <= m, token t at position t), and picks the candidate with the smallest L1 distance.
//
// Chunk i contributes to the score of the pair (m, n)
//     rotated:  a_i cos(phi) - b_i sin(phi),   plain:  a_i,
//     a_i = q_{m,2i} k_{n,2i} + q_{m,2i+1} k_{n,2i+1},  b_i = q_{m,2i+1} k_{n,2i} - q_{m,2i} k_{n,2i+1},
//     phi = (m - n) theta_i                                                   (Eq. 1a / 1b)
// so with D_i = a_i (cos(phi) - 1) - b_i sin(phi) the difference between the fully rotated score
// and the trial score is  R - D_j,  R = sum of D_i over the chunks not in e.  One pass over the
// pairs therefore yields the distances of ALL candidates of a round:  dist[j] = sum |R - D_j|.
// With both vectors rotated by HALF their angle, q' = q e^{i m theta/2}, k' = k e^{i n theta/2},
//     D_i = -2 sin((m - n) theta_i / 2) (q'_y k'_x - q'_x k'_y),
// three FP32 operations instead of six, and just as exact at small angles (the sine is a factor,
// nothing cancels).  The common sign is dropped: D_i = s_i t_i, s = 2 sin(.), t = q'_y k'_x - q'_x k'_y.
//
// Bound: FP32 pipe, issue and shared-memory reads (the contraction is 2 deep).  Two rows at a time in packed
// operations (all but the add with |.|).
//   Resident form: a thread owns 16 (8, 4) query rows x 4 keys, sums R over the free chunks (multiply, two FMA) and goes over
//     them once more for |R - D_j| (the same, and the add): 7 operations per pair and chunk, 15 16-byte shared-memory
//     reads a chunk and pass for 64 pairs.  All chunks' operands of a 128 x 128 tile lie in shared memory, staged once
//     for both passes.
//   Staged form: R is kept between rounds (four bytes a pair in the workspace) and loses the chunk that was chosen, so that a
//     round takes 4 operations per pair and chunk; it is summed afresh in the first round and where its norm has
//     fallen so far that the rounding errors of what was taken out would show (ropelite_select_kernel).  A thread owns 8 x 8
//     pairs: 12 reads a chunk, a byte of which takes as long for a broadcast as for 32 different words.  Rows and
//     keys are rotated once per search and come by the copy engine, three copies per chunk, four chunks a stage (six small
//     copies per chunk kept warps waiting: 9.4 ms instead of 8.4); three blocks of four warps share an SM and
//     drift apart, so that one's start and waits lie under the others' operations.  A pass that sums R stages every chunk
//     twice, and there is the rotation: one round is the resident form's, several are this one's.
// 32 heads x 2048 tokens x d_h 128: one round 1.53 ms resident, 1.76 staged; eight 11.8 and 8.34 (9.1 with kept R on 16 x 4 tiles
// of one block per SM).  A later round takes 0.95 ms, 0.49 of 148 SMs x 128 lanes x 1.965 GHz for the causal pairs' operations.
// Short calibrations cannot fill the device with such tiles: there a thread owns 4 x 4 pairs, and up to 128
// tokens a form with the 64 D_i of one pair in registers is the faster one (rl_carve).
//
// distance kernels: grid (items, heads); an item is 128, 64 or 32 query rows x up to `span` key tiles of 128.  The slice of
// the sine table that a tile's relative positions need comes with its keys; the table is
// zero at negative relative positions, which is the causal mask.  Item results go to a
// [head][item][chunk] array; the select kernel adds them in a fixed order (the result does not
// depend on scheduling), masks the chunks already chosen and takes the first minimum.
//
// The kernels of a search are a chain of programmatic dependent launches: one is resident while the one before it
// still writes.  What a kernel reads of its predecessors (tables, rotated rows, item results, masks, states) comes
// behind ekv_pdl_wait, by the copy engine or with plain loads, from L2 where other blocks write the same line: never
// ld.global.nc, which a compiler may make of a `const __restrict__` pointer and move in front of the wait.
// Distance blocks that are placed while blocks of another kernel hold some of the SMs come to lie two on an SM beside
// an empty one, half as fast in a call of one block an SM (16 heads x 150 tokens x d_h 128, one round, 53 us; now 45).  So the
// kernels in front of them trigger at their end, the select kernel a launch latency before it, unless there are SMs
// for the blocks of both (rl_apart).
#include "tc_ptx.cuh"

namespace {

constexpr int kRlKeys = 128;      // keys per stage
constexpr int kRlAcc = 8;         // lanes of a warp that keep running distances
constexpr int kRlPad = 256;       // zeros in front of the sine table: negative relative positions

// TR query rows and TK keys per thread: in blocks of 4 warps with 8 keys, of 8 with 4
template <int TR_, int TK_>
struct Rl {
  static constexpr int TR = TR_, TK = TK_, NW = TK == 8 ? 4 : 8, THREADS = 32 * NW;
  static constexpr int LANES = kRlKeys / TK;             // lanes that share a thread tile's rows
  static constexpr int WROWS = TR * (32 / LANES);        // query rows per warp
  static constexpr int ROWS = NW * WROWS;                // ... per block
  static constexpr int SPAN = kRlKeys + ROWS;            // sine table entries of a stage (relative positions)
  static_assert(ROWS <= kRlKeys && kRlKeys % ROWS == 0 && SPAN <= kRlPad, "a stage's slice lies inside the table");
};
// the staged form's
template <int TR_, int TK_>
struct RlRing : Rl<TR_, TK_> {
  static constexpr int VALUES = TR_ * TK_ / 4;           // 16-byte pieces of a thread's sums R
  // chunks per stage, stages, and steps between a stage's load and its use (the other warps may be behind the
  // first one, which loads, by the stages that are left)
  static constexpr int PART = TK_ == 8 ? 4 : 8, STAGES = TK_ == 8 ? 6 : 5, AHEAD = TK_ == 8 ? 3 : 4;
};
typedef RlRing<8, 8> RlLarge;
typedef RlRing<4, 4> RlFew;

// What a search keeps of a head from one round to the next, beside its sums R.
struct __align__(16) RlState {
  float norm;       // largest distance of the round that last summed R afresh
  int last;         // chunk chosen in the round before
  int fresh;        // the next round sums R afresh
  int failed;       // a wait ran out: no more results for this head
};

// entries of a chunk's sine table: entry x holds 2 sin((x - kRlPad) theta / 2), zero up to kRlPad
__host__ __device__ inline int rl_sin_len(int n) { return (n + 127) / 128 * 128 + kRlPad; }

// (cos, sin)(pos theta_i / 2) laid out [pos][chunk], and the sine table [chunk][...];
// double precision, rounded once
__global__ void ropelite_table_kernel(float2* __restrict__ cs, float* __restrict__ sn, int n, int half, int d_h,
                                      double base, unsigned long long* __restrict__ masks, RlState* __restrict__ state, int heads, int early) {
  ekv_pdl_wait();
  if (early) ekv_pdl_trigger();
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int len = rl_sin_len(n);
  for (long long h = e; h < heads; h += (long long)gridDim.x * blockDim.x) {
    if (masks) masks[h] = 0;                 // a search begins with no chunk chosen
    if (state) state[h] = RlState{0.f, 0, 1, 0};
  }
  if (e >= (long long)len * half) return;
  const int i = (int)(e % half), x = (int)(e / half);
  const int pos = x - kRlPad;
  float s2 = 0.f;
  if (pos > 0) {
    const double theta = pow(base, -2.0 * (double)i / (double)d_h);
    double s, c;
    sincos(0.5 * (double)pos * theta, &s, &c);
    s2 = (float)(2.0 * s);
    if (pos < n) cs[(size_t)pos * half + i] = make_float2((float)c, (float)s);
  } else if (pos == 0) {
    cs[i] = make_float2(1.f, 0.f);
  }
  sn[(size_t)i * len + x] = s2;
}

// four chunks (16 bytes) of a query or key row, rotated by half their angle
__device__ __forceinline__ void rl_rotate4(const bf16* row, const float2* cs, float2* out) {
  const uint4 raw = *(const uint4*)row;
  const uint32_t w[4] = {raw.x, raw.y, raw.z, raw.w};
  const float4 c01 = *(const float4*)cs, c23 = *((const float4*)cs + 1);      // (a sector: the second half from L1)
  const float2 c[4] = {{c01.x, c01.y}, {c01.z, c01.w}, {c23.x, c23.y}, {c23.z, c23.w}};
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float x = __uint_as_float(w[u] << 16), y = __uint_as_float(w[u] & 0xffff0000u);
    out[u] = make_float2(x * c[u].x - y * c[u].y, x * c[u].y + y * c[u].x);
  }
}

// Rows of Q and K rotated by half their angle, zeros past the last token, laid out as the distance kernel
// copies them, per head Q [row tile][chunk][x, y][tile rows], K [tile of 128 keys][chunk][x, y][keys]; the first four of every
// eight keys of a tile come before the others where a thread takes eight.  Every row tile, key tile and round reads them.
// Grid (rows / 64, heads, Q or K), 256 threads.
__global__ void ropelite_rotate_kernel(const bf16* __restrict__ Q, const bf16* __restrict__ K, const float2* cs,
                                       float* __restrict__ rot, int n, int n_pad, int half, int q_rows, int split) {
  ekv_pdl_wait();
  const int row = blockIdx.x * 64 + threadIdx.x % 64, head = blockIdx.y, k = blockIdx.z;
  const bf16* src = (k ? K : Q) + ((size_t)head * n + row) * 2 * half;
  const int tile = k ? kRlKeys : q_rows, in = row % tile;
  float* x = rot + ((size_t)head * 2 + k) * 2 * half * n_pad + (size_t)(row - in) * 2 * half +
             (k && split ? (in >> 2 & 1) * 64 + (in >> 3) * 4 + (in & 3) : in);
  for (int i = threadIdx.x / 64 * 4; i < half; i += 16) {
    float2 v[4] = {};
    if (row < n) rl_rotate4(src + 2 * i, cs + (size_t)row * half + i, v);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      x[(size_t)(i + u) * 2 * tile] = v[u].x;
      x[(size_t)(i + u) * 2 * tile + tile] = v[u].y;
    }
  }
}

// one chunk of a stage
template <class F>
struct __align__(16) RlChunk {
  float kx[kRlKeys], ky[kRlKeys], qx[F::ROWS], qy[F::ROWS], sn[F::SPAN];
};
template <int HALF, class F>
struct RlSmem {
  RlChunk<F> ring[F::STAGES][F::PART];
  float acc[HALF][F::NW * kRlAcc];     // running distances
  uint64_t full[F::STAGES], empty[F::STAGES];
  int list[HALF];                      // chunks in the order in which a tile needs them
  int n_hi;                            // end of the block's keys; 0: a wait ran out
};

// Two rows (r, r + 1) at a time: packed fp32 operations, each element rounded as by itself
typedef unsigned long long rl2;
__device__ __forceinline__ rl2 rl_pack(float lo, float hi) {
  rl2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(lo), "f"(hi));
  return d;
}
__device__ __forceinline__ float2 rl_unpack(rl2 a) {
  float2 d;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(d.x), "=f"(d.y) : "l"(a));
  return d;
}
__device__ __forceinline__ rl2 rl_mul(rl2 a, rl2 b) {
  rl2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ rl2 rl_fma(rl2 a, rl2 b, rl2 c) {
  rl2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}

// where a chunk's operands lie: chunk i of planes, or one of a stage
template <class Planes>
struct RlOfPlanes {
  const Planes& p;
  const int i;
  __device__ __forceinline__ const float* kx(int at) const { return &p.kx[i][at]; }
  __device__ __forceinline__ const float* ky(int at) const { return &p.ky[i][at]; }
  __device__ __forceinline__ const float* qx(int at) const { return &p.qx[i][at]; }
  __device__ __forceinline__ const float* qy(int at) const { return &p.qy[i][at]; }
  __device__ __forceinline__ const float* sn(int at) const { return &p.sn[i][at]; }
};
template <class F>
struct RlOfStage {
  const RlChunk<F>& p;
  __device__ __forceinline__ const float* kx(int at) const { return &p.kx[at]; }
  __device__ __forceinline__ const float* ky(int at) const { return &p.ky[at]; }
  __device__ __forceinline__ const float* qx(int at) const { return &p.qx[at]; }
  __device__ __forceinline__ const float* qy(int at) const { return &p.qy[at]; }
  __device__ __forceinline__ const float* sn(int at) const { return &p.sn[at]; }
};

// operands of a thread's pairs for one chunk; kNeg: t with its sign turned
template <class F>
struct RlOps {
  rl2 a[F::TK], b[F::TK];            // keys: t = q_y a + q_x b
  rl2 qx[F::TR / 2], qy[F::TR / 2];
  rl2 s[(F::TR + F::TK) / 2][2];     // [v][0]: table entries 2 v, 2 v + 1; [v][1]: 2 v + 1, 2 v + 2
};
// rg: the thread's group of TR rows in the block; lk: its group of TK keys
template <class F, bool kNeg, class At>
__device__ __forceinline__ void rl_load(RlOps<F>& o, const At& ch, int rg, int lk) {
  constexpr int TR = F::TR, TK = F::TK;
#pragma unroll
  for (int h = 0; h < TK / 4; ++h) {       // (the keys' first fours come before their second ones: lanes read consecutive 16 bytes)
    const float4 kx = *(const float4*)ch.kx(kRlKeys / 2 * h + 4 * lk), ky = *(const float4*)ch.ky(kRlKeys / 2 * h + 4 * lk);
    const float x[4] = {kx.x, kx.y, kx.z, kx.w}, y[4] = {ky.x, ky.y, ky.z, ky.w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const float a = kNeg ? -x[j] : x[j], b = kNeg ? y[j] : -y[j];
      o.a[4 * h + j] = rl_pack(a, a);
      o.b[4 * h + j] = rl_pack(b, b);
    }
  }
  // entry u of the stage's slice: relative position (m0 - n0) - 128 + u; this thread's pairs need
  // u = TR rg + r - (TK lk + j) + 128, from TR rg - TK lk + 128 - TK on
  const float4* sp = (const float4*)ch.sn(TR * rg - TK * lk + kRlKeys - TK);
  float e[TR + TK];
#pragma unroll
  for (int u = 0; u < (TR + TK) / 4; ++u) *(float4*)&e[4 * u] = sp[u];
#pragma unroll
  for (int v = 0; v < (TR + TK) / 2; ++v) {
    o.s[v][0] = rl_pack(e[2 * v], e[2 * v + 1]);
    if (2 * v + 2 < TR + TK) o.s[v][1] = rl_pack(e[2 * v + 1], e[2 * v + 2]);
  }
  const ulonglong2* qx = (const ulonglong2*)ch.qx(TR * rg);
  const ulonglong2* qy = (const ulonglong2*)ch.qy(TR * rg);
#pragma unroll
  for (int u = 0; u < TR / 4; ++u) {
    const ulonglong2 vx = qx[u], vy = qy[u];
    o.qx[2 * u] = vx.x; o.qx[2 * u + 1] = vx.y;
    o.qy[2 * u] = vy.x; o.qy[2 * u + 1] = vy.y;
  }
}
// table pair of rows 2 r, 2 r + 1 and key j: entries 2 r - j + TK and the next
template <class F>
__device__ __forceinline__ rl2 rl_sin(const RlOps<F>& o, int r, int j) { return o.s[(2 * r - j + F::TK) / 2][(2 * r - j + F::TK) & 1]; }

// R += D of a chunk (kNeg: R -= D)
template <class F, bool kNeg, class At>
__device__ __forceinline__ void rl_add(rl2 (&R)[F::TR / 2][F::TK], const At& ch, int rg, int lk) {
  RlOps<F> o;
  rl_load<F, kNeg>(o, ch, rg, lk);
#pragma unroll
  for (int r = 0; r < F::TR / 2; ++r)
#pragma unroll
    for (int j = 0; j < F::TK; ++j) {
      const rl2 t = rl_fma(o.qx[r], o.b[j], rl_mul(o.qy[r], o.a[j]));
      R[r][j] = rl_fma(rl_sin(o, r, j), t, R[r][j]);
    }
}
// the thread's share of the distance of a chunk: sum of |R - D| over its pairs
template <class F, class At>
__device__ __forceinline__ float rl_distance(const rl2 (&R)[F::TR / 2][F::TK], const At& ch, int rg, int lk) {
  constexpr int TK = F::TK;
  RlOps<F> o;
  rl_load<F, true>(o, ch, rg, lk);
  float v[TK] = {};
#pragma unroll
  for (int r = 0; r < F::TR / 2; ++r)
#pragma unroll
    for (int j = 0; j < TK; ++j) {
      const rl2 t = rl_fma(o.qx[r], o.b[j], rl_mul(o.qy[r], o.a[j]));
      const float2 x = rl_unpack(rl_fma(rl_sin(o, r, j), t, R[r][j]));
      v[j] += fabsf(x.x);
      v[j] += fabsf(x.y);
    }
  float d = (v[0] + v[1]) + (v[2] + v[3]);
  if constexpr (TK == 8) d += (v[4] + v[5]) + (v[6] + v[7]);
  return d;
}
// Wait that parks between probes.  One that runs out sets the block's last key to 0, so that its warps leave with their next
// tile, and the lane loads no more stages.  Lanes that differ meet again at the end of the step.  (The same with a vote
// per wait, a flag that the loops test or a budget of probes for all waits of a thread: 1 to 3 % of a search.)
__device__ __forceinline__ bool rl_wait(uint32_t bar, uint32_t parity, volatile int* n_hi, unsigned limit) {
  unsigned tries = 0;
  while (!mbar_try_wait(bar, parity))
    if (++tries > limit) { *n_hi = 0; return false; }
  return true;
}
__device__ __forceinline__ void rl_bulk(void* dst, const void* src, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(smem_u32(dst)),
               "l"((uint64_t)src), "r"(bytes), "r"(bar)
               : "memory");
}

// Tiles of 128 keys in a head's row tiles below mt (a row tile ends at the diagonal).
template <class F>
__host__ __device__ inline long long rl_tiles_below(int mt) {
  constexpr int q = kRlKeys / F::ROWS;
  const long long a = mt / q, b = mt % q;
  return q * (a * (a + 1) / 2) + b * (a + 1);
}

// item -> (row tile, group of `span` key tiles), long rows first
template <int ROWS>
__device__ __forceinline__ void rl_item(int n, int span, int item, int* mt, int* kg) {
  *mt = (n + ROWS - 1) / ROWS - 1;
  *kg = item;
  for (;; --*mt) {
    const int groups = ((*mt + 1) * ROWS + kRlKeys * span - 1) / (kRlKeys * span);
    if (*kg < groups) return;
    *kg -= groups;
  }
}

// R summed in every round, with the operands of all chunks of a key tile resident in shared memory: staged once for
// both passes, rotated by the block itself, so that nothing is kept in the workspace.
template <int HALF, class F>
struct RlResident {
  float kx[HALF][kRlKeys], ky[HALF][kRlKeys], sn[HALF][F::SPAN], qx[HALF][F::ROWS], qy[HALF][F::ROWS];
  float acc[HALF][F::NW * kRlAcc];     // running distances
  int list[HALF];                      // chunks not chosen yet
};
template <int HALF, class F>
__global__ void __launch_bounds__(F::THREADS)
ropelite_distance_resident_kernel(const bf16* __restrict__ Q, const bf16* __restrict__ K, int n, const float2* cs, const float* sn,
                                  const unsigned long long* masks, int span, float* __restrict__ partial /* [heads][items][HALF] */) {
  constexpr int d_h = 2 * HALF, NW = F::NW, THREADS = F::THREADS, ROWS = F::ROWS, SPAN = F::SPAN;
  static_assert(F::TK == 4, "a warp's lanes cover the keys");
  extern __shared__ __align__(128) unsigned char smem_rl[];
  RlResident<HALF, F>& sm = *(RlResident<HALF, F>*)smem_rl;
  const int head = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int mt, kg;
  rl_item<ROWS>(n, span, blockIdx.x, &mt, &kg);
  ekv_pdl_wait();
  ekv_pdl_trigger();
  const int m0 = mt * ROWS;
  const int n_lo = kg * span * kRlKeys, n_hi = min(n_lo + span * kRlKeys, m0 + ROWS);
  const unsigned long long mask = masks ? __ldcg(masks + head) : 0ull;
  const int n_free = HALF - __popcll(HALF == 64 ? mask : mask & ((1ull << (HALF & 63)) - 1));
  float* out = partial + ((size_t)head * gridDim.x + blockIdx.x) * HALF;
  if (n_free <= 1) {                 // a single free chunk: R = D_j for every pair
    for (int j = threadIdx.x; j < HALF; j += THREADS) out[j] = 0.f;
    return;
  }
  if (threadIdx.x < HALF && !((mask >> threadIdx.x) & 1ull))
    sm.list[threadIdx.x - __popcll(mask & ((1ull << threadIdx.x) - 1))] = threadIdx.x;
  const bf16* Qh = Q + (size_t)head * n * d_h;
  const bf16* Kh = K + (size_t)head * n * d_h;
  // (consecutive threads take consecutive rows: the transposed stores hit different banks)
  for (int e = threadIdx.x; e < ROWS * (HALF / 4); e += THREADS) {
    const int rr = e % ROWS, g4 = e / ROWS;
    float2 v[4] = {};
    if (m0 + rr < n) rl_rotate4(Qh + (size_t)(m0 + rr) * d_h + g4 * 8, cs + (size_t)(m0 + rr) * HALF + g4 * 4, v);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      sm.qx[g4 * 4 + u][rr] = v[u].x;
      sm.qy[g4 * 4 + u][rr] = v[u].y;
    }
  }
  for (int e = threadIdx.x; e < HALF * NW * kRlAcc; e += THREADS) (&sm.acc[0][0])[e] = 0.f;
  const int sn_len = rl_sin_len(n);

  for (int n0 = n_lo; n0 < n_hi; n0 += kRlKeys) {
    __syncthreads();
    // entry u holds relative position (m0 - n0) - 128 + u
    const int x0 = m0 - n0 - kRlKeys + kRlPad;
    for (int e = threadIdx.x; e < HALF * (SPAN / 4); e += THREADS) {
      const int i = e / (SPAN / 4), u = (e % (SPAN / 4)) * 4;
      cp_async16(&sm.sn[i][u], sn + (size_t)i * sn_len + x0 + u);
    }
    cp_async_commit();
#pragma unroll
    for (int e = threadIdx.x; e < kRlKeys * (HALF / 4); e += THREADS) {
      const int nn = e % kRlKeys, g4 = e / kRlKeys;         // 4 chunks = 8 elements = 16 bytes
      float2 v[4] = {};
      if (n0 + nn < n) rl_rotate4(Kh + (size_t)(n0 + nn) * d_h + g4 * 8, cs + (size_t)(n0 + nn) * HALF + g4 * 4, v);
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        sm.kx[g4 * 4 + u][nn] = v[u].x;
        sm.ky[g4 * 4 + u][nn] = v[u].y;
      }
    }
    cp_async_wait<0>();
    __syncthreads();
    // every pair of this warp lies above the diagonal, or its rows past the last token
    if (n0 > m0 + F::TR * warp + F::TR - 1 || m0 + F::TR * warp >= n) continue;
    rl2 R[F::TR / 2][F::TK];
#pragma unroll
    for (int r = 0; r < F::TR / 2; ++r)
#pragma unroll
      for (int j = 0; j < F::TK; ++j) R[r][j] = 0ull;
#pragma unroll 8
    for (int c = 0; c < n_free; ++c) rl_add<F, false>(R, RlOfPlanes<RlResident<HALF, F>>{sm, sm.list[c]}, warp, lane);
#pragma unroll 8
    for (int c = 0; c < n_free; ++c) {
      const int i = sm.list[c];
      float d = rl_distance<F>(R, RlOfPlanes<RlResident<HALF, F>>{sm, i}, warp, lane);
      d += __shfl_xor_sync(0xffffffffu, d, 16);
      d += __shfl_xor_sync(0xffffffffu, d, 8);
      if (lane < kRlAcc) sm.acc[i][warp * kRlAcc + lane] += d;
    }
  }
  // block result: threads in a fixed order
  __syncthreads();
  for (int j = warp; j < HALF; j += NW) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < NW * kRlAcc; w += 32) v += sm.acc[j][w + lane];
    v = warp_sum(v);
    if (lane == 0) out[j] = v;
  }
}

// kSilent (self-test): stages are awaited that nobody fills, every wait with a short limit
template <int HALF, class F, bool kSilent = false>
__global__ void __launch_bounds__(F::THREADS, F::TR == 8 ? 3 : 2)
ropelite_distance_kernel(const float* rot /* [heads]: Q, K (ropelite_rotate_kernel) */, int n, int n_pad,
                         const float* sn, const unsigned long long* masks, int span,
                         float* __restrict__ partial /* [heads][items][HALF] */,
                         ulonglong2* kept /* [heads][tiles][VALUES][THREADS], null: R is not kept */,
                         RlState* state, int first_round, int last_round) {
  constexpr int TR = F::TR, TK = F::TK, NW = F::NW, THREADS = F::THREADS, ROWS = F::ROWS;
  extern __shared__ __align__(128) unsigned char smem_rl[];
  RlSmem<HALF, F>& sm = *(RlSmem<HALF, F>*)smem_rl;
  const int head = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int mt, kg;
  rl_item<ROWS>(n, span, blockIdx.x, &mt, &kg);
  ekv_pdl_wait();
  ekv_pdl_trigger();
  const int m0 = mt * ROWS;
  const int n_lo = kg * span * kRlKeys, n_hi = min(n_lo + span * kRlKeys, m0 + ROWS);
  const unsigned long long mask = masks ? __ldcg(masks + head) : 0ull;
  const int4 kept_state = __ldcg((const int4*)&state[head]);      // RlState
  // one trip to L2 for both, and meanwhile:
  if (threadIdx.x == 0) {
    for (int i = 0; i < F::STAGES; ++i) {
      mbar_init(smem_u32(&sm.full[i]), 1);
      mbar_init(smem_u32(&sm.empty[i]), NW);
    }
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    fence_proxy_async();
  }
  for (int e = threadIdx.x; e < HALF * NW * kRlAcc; e += THREADS) (&sm.acc[0][0])[e] = 0.f;
  const int n_free = HALF - __popcll(HALF == 64 ? mask : mask & ((1ull << (HALF & 63)) - 1));
  float* out = partial + ((size_t)head * gridDim.x + blockIdx.x) * HALF;
  if (n_free <= 1 || kept_state.w) {      // a single free chunk: R = D_j for every pair; or no result any more
    for (int j = threadIdx.x; j < HALF; j += THREADS) out[j] = kept_state.w ? NAN : 0.f;
    return;
  }
  const bool fresh = kept == nullptr || first_round || kept_state.z;
  // one that R has to lose, then the free ones
  const int n_old = fresh ? 0 : 1, n_list = n_old + n_free, parts = (n_list + F::PART - 1) / F::PART;
  if (threadIdx.x < HALF && !((mask >> threadIdx.x) & 1ull))
    sm.list[n_old + threadIdx.x - __popcll(mask & ((1ull << threadIdx.x) - 1))] = threadIdx.x;
  if (threadIdx.x == 0) {
    if (!fresh) sm.list[0] = kept_state.y;
    sm.n_hi = n_hi;
  }
  if (kept)
    kept += (head * rl_tiles_below<F>((n + ROWS - 1) / ROWS) + rl_tiles_below<F>(mt)) * (F::VALUES * THREADS) + threadIdx.x;
  const float* rot_h = rot + (size_t)head * 4 * HALF * n_pad;
  const int sn_len = rl_sin_len(n);
  __syncthreads();

  // Steps of the block: for each key tile the parts of its list, twice where R is summed afresh.  The first
  // warp loads them.
  const int tile_steps = fresh ? 2 * parts : parts;
  constexpr unsigned kLimit = kSilent ? 1024 : kWaitLimit;
  int load_n0 = n_lo, load_step = 0, load_slot = 0;
  uint32_t load_parity = 1;
  volatile int* const last_key = &sm.n_hi;
  auto load = [&] {
    if (load_n0 < n_hi) {
      if (!rl_wait(smem_u32(&sm.empty[load_slot]), load_parity, last_key, kLimit)) { load_n0 = n_hi; return; }
      const int c0 = load_step % parts * F::PART, cn = min(F::PART, n_list - c0);
      const uint32_t bar = smem_u32(&sm.full[load_slot]);
      if (lane == 0) mbar_expect_tx(bar, (uint32_t)(cn * sizeof(RlChunk<F>)));      // (the phase waits for it, whatever lands before)
      for (int e = kSilent ? 3 * cn : lane; e < 3 * cn; e += 32) {
        const int c = e / 3, what = e - 3 * c;
        const int i = sm.list[c0 + c];
        RlChunk<F>& ch = sm.ring[load_slot][c];
        const float* k = rot_h + (size_t)2 * HALF * (n_pad + load_n0) + (size_t)i * 2 * kRlKeys;
        if (what == 0) rl_bulk(ch.kx, k, 2 * sizeof(ch.kx), bar);
        else if (what == 1) rl_bulk(ch.qx, rot_h + (size_t)2 * HALF * m0 + (size_t)i * 2 * ROWS, 2 * sizeof(ch.qx), bar);
        else rl_bulk(ch.sn, sn + (size_t)i * sn_len + m0 - load_n0 - kRlKeys + kRlPad, sizeof(ch.sn), bar);
      }
      if (++load_step == tile_steps) { load_step = 0; load_n0 += kRlKeys; }
    }
    if (++load_slot == F::STAGES) { load_slot = 0; load_parity ^= 1; }
  };
  if (warp == 0)
    for (int i = 0; i < F::AHEAD; ++i) load();

  const int rg = warp * (32 / F::LANES) + lane / F::LANES, lk = lane % F::LANES;
  int slot = 0;
  uint32_t parity = 0;
  for (int n0 = n_lo; n0 < __shfl_sync(0xffffffffu, *last_key, 0); n0 += kRlKeys) {
    // pairs of this warp that are not all above the diagonal, nor its rows past the last token
    const bool live = n0 < m0 + F::WROWS * (warp + 1) && m0 + F::WROWS * warp < n;
    rl2 R[TR / 2][TK];
    ulonglong2* const keep_at = kept + (size_t)(n0 / kRlKeys) * (F::VALUES * THREADS);
    if (fresh) {
#pragma unroll
      for (int r = 0; r < TR / 2; ++r)
#pragma unroll
        for (int j = 0; j < TK; ++j) R[r][j] = 0ull;
    } else {
      if (live) {
#pragma unroll
        for (int u = 0; u < F::VALUES; ++u) {
          const ulonglong2 v = __ldcs(keep_at + u * THREADS);
          R[u / (TK / 2)][u % (TK / 2) * 2] = v.x;
          R[u / (TK / 2)][u % (TK / 2) * 2 + 1] = v.y;
        }
      }
      if (n0 + kRlKeys < *last_key && (threadIdx.x & 7) == 0) {      // the next tile's come into L2 meanwhile
#pragma unroll
        for (int u = 0; u < F::VALUES; ++u)
          asm volatile("prefetch.global.L2 [%0];" ::"l"(keep_at + (F::VALUES + u) * THREADS));
      }
    }
#pragma unroll 1
    for (int step = 0; step < tile_steps; ++step) {
      if (warp == 0) load();
      if (!rl_wait(smem_u32(&sm.full[slot]), parity, last_key, kLimit)) load_n0 = n_hi;
      if (live) {
        const bool sum = fresh && step < parts;
        int c = 0;
        const int part = sum || !fresh ? step : step - parts, cn = min(F::PART, n_list - part * F::PART);
        const RlChunk<F>* ring = sm.ring[slot];
        if (sum) {
#pragma unroll 4
          for (; c < cn; ++c) rl_add<F, false>(R, RlOfStage<F>{ring[c]}, rg, lk);
        } else {
          if (part == 0) {
            if (!fresh) {                        // R loses the chunk chosen in the round before
              rl_add<F, true>(R, RlOfStage<F>{ring[0]}, rg, lk);
              c = 1;
            }
            if (kept && !last_round) {
#pragma unroll
              for (int u = 0; u < F::VALUES; ++u) __stcs(keep_at + u * THREADS, make_ulonglong2(R[u / (TK / 2)][u % (TK / 2) * 2], R[u / (TK / 2)][u % (TK / 2) * 2 + 1]));
            }
          }
#pragma unroll 4
          for (; c < cn; ++c) {
            float d = rl_distance<F>(R, RlOfStage<F>{ring[c]}, rg, lk);
            d += __shfl_xor_sync(0xffffffffu, d, 16);
            d += __shfl_xor_sync(0xffffffffu, d, 8);
            if (lane < kRlAcc) sm.acc[part * F::PART + c][warp * kRlAcc + lane] += d;
          }
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(smem_u32(&sm.empty[slot]));
      if (++slot == F::STAGES) { slot = 0; parity ^= 1; }
    }
  }
  __syncthreads();
  if (sm.n_hi == 0) {
    // the stages loaded and not yet used (fewer than there are) have time to land
    if (warp == 0)
      while (slot != load_slot) {
        for (unsigned i = 0; i < 1024 && !mbar_try_wait(smem_u32(&sm.full[slot]), parity); ++i) {}
        if (++slot == F::STAGES) { slot = 0; parity ^= 1; }
      }
    drain_after_abort();
    if (threadIdx.x == 0) state[head].failed = 1;
  }
  // block result: threads in a fixed order
  const float bad = sm.n_hi == 0 ? NAN : 0.f;
  for (int c = n_old + warp; c < n_list; c += NW) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < NW * kRlAcc; w += 32) v += sm.acc[c][w + lane];
    v = warp_sum(v);
    if (lane == 0) out[sm.list[c]] = v + bad;
  }
}

// Small calls (rl_form): a block is 16 query rows and all their keys, 64 at a time; a thread takes one pair
// at a time and holds its D_i in registers.  9 loads and operations per pair and chunk instead of 7 packed
// ones, but no pair is computed that the causal rule leaves out, and a block's chain is short.
constexpr int kRsRows = 16, kRsKeys = 64, kRsWarps = 4;
template <int HALF>
struct RsSmem {
  float2 k[HALF][kRsKeys], q[kRsRows][HALF];
  float sn[HALF][kRsKeys + kRsRows];
  float red[kRsWarps][HALF];
};
template <int HALF>
__global__ void __launch_bounds__(32 * kRsWarps)
ropelite_distance_small_kernel(const bf16* __restrict__ Q, const bf16* __restrict__ K, int n,
                               const float2* cs, const float* sn, const unsigned long long* masks,
                               float* __restrict__ partial /* [heads][row tiles][HALF] */) {
  constexpr int d_h = 2 * HALF, THREADS = 32 * kRsWarps;
  extern __shared__ __align__(128) unsigned char smem_rl[];
  RsSmem<HALF>& sm = *(RsSmem<HALF>*)smem_rl;
  const int head = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  ekv_pdl_wait();
  ekv_pdl_trigger();
  const int m0 = blockIdx.x * kRsRows, m_last = min(m0 + kRsRows, n) - 1;
  const unsigned long long mask = masks ? __ldcg(masks + head) : 0ull;
  const bf16* Qh = Q + (size_t)head * n * d_h;
  const bf16* Kh = K + (size_t)head * n * d_h;
  for (int e = threadIdx.x; e < kRsRows * (HALF / 4); e += THREADS) {
    const int rr = e / (HALF / 4), g4 = e % (HALF / 4);
    float2 v[4] = {};
    if (m0 + rr < n) rl_rotate4(Qh + (size_t)(m0 + rr) * d_h + g4 * 8, cs + (size_t)(m0 + rr) * HALF + g4 * 4, v);
#pragma unroll
    for (int u = 0; u < 4; ++u) sm.q[rr][g4 * 4 + u] = v[u];
  }
  float acc[HALF];
#pragma unroll
  for (int j = 0; j < HALF; ++j) acc[j] = 0.f;
  const int sn_len = rl_sin_len(n);
  for (int n0 = 0; n0 <= m_last; n0 += kRsKeys) {
    __syncthreads();
    const int x0 = m0 - n0 - kRsKeys + kRlPad;              // entry u: relative position (m0 - n0) - 64 + u
    for (int e = threadIdx.x; e < HALF * ((kRsKeys + kRsRows) / 4); e += THREADS) {
      const int i = e / ((kRsKeys + kRsRows) / 4), u = e % ((kRsKeys + kRsRows) / 4) * 4;
      cp_async16(&sm.sn[i][u], sn + (size_t)i * sn_len + x0 + u);
    }
    cp_async_commit();
    for (int e = threadIdx.x; e < kRsKeys * (HALF / 4); e += THREADS) {
      const int nn = e % kRsKeys, g4 = e / kRsKeys;
      if (n0 + nn > m_last) continue;
      float2 v[4];
      rl_rotate4(Kh + (size_t)(n0 + nn) * d_h + g4 * 8, cs + (size_t)(n0 + nn) * HALF + g4 * 4, v);
#pragma unroll
      for (int u = 0; u < 4; ++u) sm.k[g4 * 4 + u][nn] = v[u];
    }
    cp_async_wait<0>();
    __syncthreads();
#pragma unroll 1
    for (int e = 0; e < kRsRows / kRsWarps * (kRsKeys / 32); ++e) {
      const int rr = warp + e / (kRsKeys / 32) * kRsWarps, nn = lane + e % (kRsKeys / 32) * 32;
      if (n0 + nn > m0 + rr || m0 + rr >= n) continue;      // causal pairs only
      const int u = rr - nn + kRsKeys;
      float d[HALF], R = 0.f;
#pragma unroll
      for (int i = 0; i < HALF; ++i) {
        const float2 q = sm.q[rr][i], k = sm.k[i][nn];
        d[i] = __fmul_rn(sm.sn[i][u], fmaf(q.y, k.x, -(q.x * k.y)));      // rounded: the last free chunk's R - D_j is 0
        if (!((mask >> i) & 1ull)) R = __fadd_rn(R, d[i]);
      }
#pragma unroll
      for (int j = 0; j < HALF; ++j) acc[j] += fabsf(R - d[j]);
    }
  }
#pragma unroll
  for (int j = 0; j < HALF; ++j) {
    const float v = warp_sum(acc[j]);
    if (lane == 0) sm.red[warp][j] = v;
  }
  __syncthreads();
  if (threadIdx.x < HALF) {
    float v = 0.f;
#pragma unroll
    for (int w = 0; w < kRsWarps; ++w) v += sm.red[w][threadIdx.x];
    partial[((size_t)head * gridDim.x + blockIdx.x) * HALF + threadIdx.x] = v;
  }
}

// One block per head: adds the items' results in a fixed order, writes the round's distances
// (+inf for chunks already chosen) and, when `elite_idx` is given, appends the first minimum to
// the head's list and to its mask.
constexpr int kRlSelect = 8;      // threads per chunk
__global__ void ropelite_select_kernel(const float* partial, int n_items, int half, unsigned long long* masks, float* __restrict__ dist_out,
                                       int32_t* __restrict__ elite_idx, int r, int round,
                                       RlState* state /* null: forms without waits */, int keep, int early) {
  __shared__ float s_d[kRlSelect][64];
  ekv_pdl_wait();
  if (early) ekv_pdl_trigger();
  const int head = blockIdx.x, j = threadIdx.x & 63, part = threadIdx.x >> 6;
  const unsigned long long mask = masks ? __ldcg(masks + head) : 0ull;
  float v = 0.f;
  if (j < half) {
    const float* src = partial + (size_t)head * n_items * half + j;
#pragma unroll 4
    for (int t = part; t < n_items; t += kRlSelect) v += __ldcg(src + (size_t)t * half);
  }
  s_d[part][j] = v;
  __syncthreads();
  ekv_pdl_trigger();
  if (threadIdx.x < 64) {
    v = INFINITY;
    if (j < half && !((mask >> j) & 1ull)) {
      v = 0.f;
#pragma unroll
      for (int p = 0; p < kRlSelect; ++p) v += s_d[p][j];
    }
    if (j < half && dist_out) dist_out[(size_t)head * half + j] = v;
    s_d[0][j] = v;
  }
  __syncthreads();
  if (threadIdx.x == 0 && elite_idx && state && __ldcg(&state[head].failed)) {
    elite_idx[(size_t)head * r + round] = -1;
  } else if (threadIdx.x == 0 && elite_idx) {
    int best = 0;
    for (int c = 1; c < half; ++c)
      if (s_d[0][c] < s_d[0][best]) best = c;
    elite_idx[(size_t)head * r + round] = best;
    masks[head] = mask | (1ull << best);
    if (keep) {
      // The winner's distance is the L1 norm of the next round's R.  Taking chunks out of a kept R adds
      // rounding errors of the size of the R that was summed; below a quarter of it, or where anything
      // is not finite, R is summed afresh, so that the errors stay of the size of those of a sum.
      float norm = __ldcg(&state[head].norm);
      if (round == 0 || __ldcg(&state[head].fresh)) {
        norm = 0.f;
        for (int c = 0; c < half; ++c)
          if (!((mask >> c) & 1ull)) norm = fmaxf(norm, s_d[0][c]);
      }
      state[head].norm = norm;
      state[head].last = best;
      state[head].fresh = !(4.f * s_d[0][best] >= norm && norm < INFINITY);
    }
  }
}

enum RlKind { kRlSmall, kRlResident, kRlStaged };
struct RlCarve {
  size_t off_cs, off_sin, off_partial, off_masks, off_state, off_rot, off_kept, total;
  RlKind kind;
  int tr, span, items;          // rows per thread, key tiles per item, items per head
  int group;                    // heads that go through their rounds together
  bool keep;                    // their sums R are kept between rounds
};
inline size_t rl_align(size_t x) { return (x + 255) & ~(size_t)255; }

// Key tiles per item: whole rows cut into at most 16 items, at least 4 tiles long (an item starts anew: its queries,
// its barriers, the first stage's latency); single tiles where that would leave most of the
// device without work (fewer blocks than four for each of 148 SMs).
constexpr int kRlSms = 148;
long long rl_count(int n, int rows, int span) {
  long long k = 0;
  for (int m = rows; m < n + rows; m += rows) k += (m + kRlKeys * span - 1) / (kRlKeys * span);
  return k;
}
inline int rl_pad_n(int n) { return (n + kRlKeys - 1) / kRlKeys * kRlKeys; }
template <class F>
size_t rl_kept_bytes_of(int n) {
  return (size_t)rl_tiles_below<F>((n + F::ROWS - 1) / F::ROWS) * F::VALUES * F::THREADS * sizeof(ulonglong2);
}
size_t rl_kept_bytes(int tr, int n) {
  return tr == 8 ? rl_kept_bytes_of<RlLarge>(n) : rl_kept_bytes_of<RlFew>(n);
}
// Scratch of a head in the staged form: its rotated rows (2 MB at 2048 tokens of d_h 128) and its sums R, four bytes for
// each pair of its tiles (9 MB; 137 MB at 8192 tokens).  Heads are independent, so a call whose heads need more than
// kRlScratch takes them through its rounds in groups.  A head of over 22000 tokens needs more by itself:
// its R is summed in every round.
constexpr size_t kRlScratch = (size_t)1 << 30;
RlCarve rl_layout(int heads, int n, int half, RlKind kind, int tr, bool keep) {
  RlCarve c;
  c.kind = kind;
  c.tr = tr;
  c.span = 1;
  if (kind == kRlSmall) {
    c.items = (n + kRsRows - 1) / kRsRows;
  } else {
    const int tiles = (n + kRlKeys - 1) / kRlKeys, span = tiles > 64 ? (tiles + 15) / 16 : 4;
    if (heads * rl_count(n, 8 * tr, span) >= 4 * kRlSms) c.span = span;
    c.items = (int)rl_count(n, 8 * tr, c.span);
  }
  const size_t rot = kind == kRlStaged ? sizeof(float) * 4 * (size_t)half * rl_pad_n(n) : 0;
  const size_t kept = kind == kRlStaged ? rl_kept_bytes(tr, n) : 0;
  c.keep = keep && kind == kRlStaged && rot + kept <= kRlScratch;
  const size_t per_head = rot + (c.keep ? kept : 0);
  c.group = heads;
  if (per_head * heads > kRlScratch) c.group = per_head < kRlScratch ? (int)(kRlScratch / per_head) : 1;
  size_t o = 0;
  c.off_cs = o;      o = rl_align(o + sizeof(float2) * (size_t)half * n);
  c.off_sin = o;     o = rl_align(o + sizeof(float) * (size_t)half * rl_sin_len(n));
  c.off_partial = o; o = rl_align(o + sizeof(float) * (size_t)c.group * c.items * half);
  c.off_masks = o;   o = rl_align(o + sizeof(unsigned long long) * (size_t)heads);
  c.off_state = o;   o = kind == kRlStaged ? rl_align(o + sizeof(RlState) * (size_t)heads) : o;
  c.off_rot = o;     o = rl_align(o + (size_t)c.group * rot);
  c.off_kept = o;    o = rl_align(o + (c.keep ? (size_t)c.group * kept : 0));
  c.total = o;
  return c;
}

// Which form, for a device of 148 SMs: the one whose blocks should take least time in all.  The tables hold
// microseconds: a call (tables, rotation), what a round costs beside its tiles, then a round of which every SM has one,
// two or three blocks of one key tile each and every further wave of `fit` blocks an SM, for a round that sums R and for
// one that keeps it.  A round's tiles cost in proportion to its free chunks.  Over 1 to 64 heads of 129 to 2048
// tokens and 1 to 8 rounds (1320 calls) the choice takes 1.002 of the best form's time in the mean, 1.12 at worst.
// Us at d_h 128 (resident 16, 8, 4 rows / staged 8, 4 rows): one round 8 x 150 60, 40, 31 / 67, 45; 32 x 1000 433, 549,
// 736 / 627, 742; 32 x 2048 1538, 1842, 2649 / 1760, 2520; three rounds 8 x 150 176, 114, 87 / 144, 95; 32 x 1000 1286,
// 1629, 2186 / 1315, 1578; 32 x 2048 4574, 5475, 7899 / 3708, 5404.  Forms of 4 rows are for calls of few blocks: from
// three an SM on another one is faster.
struct RlForm {
  RlKind kind;
  int tr, fit;                    // rows per thread, blocks per SM
  float call, round;
  float first[3], first_wave;
  float later[3], later_wave;     // staged, R kept
  float several;                  // share of a wave's time where items have several tiles
};
constexpr int kRlForms = 5;
constexpr float kRlNever = 1e12f;
const RlForm kRlForms128[kRlForms] = {
    {kRlResident, 16, 1, 2.f, 5.f, {53.7f}, 53.7f, {}, 0.f, 0.91f},
    {kRlResident, 8, 1, 2.f, 4.5f, {33.5f}, 33.5f, {}, 0.f, 0.92f},
    {kRlResident, 4, 2, 2.f, 4.f, {24.7f, 48.9f}, kRlNever, {}, 0.f, 1.f},
    {kRlStaged, 8, 3, 11.f, 5.f, {54.f, 69.f, 85.f}, 86.f, {33.5f, 42.5f, 53.f}, 49.f, 1.f},
    {kRlStaged, 4, 2, 9.f, 5.f, {32.f, 42.f}, kRlNever, {20.3f, 25.5f}, kRlNever, 1.f}};
const RlForm kRlForms64[kRlForms] = {
    {kRlResident, 16, 2, 2.f, 4.f, {28.4f, 56.5f}, 56.5f, {}, 0.f, 0.87f},
    {kRlResident, 8, 2, 2.f, 8.f, {13.8f, 27.5f}, 27.5f, {}, 0.f, 0.96f},
    {kRlResident, 4, 2, 2.f, 8.5f, {8.6f, 16.8f}, kRlNever, {}, 0.f, 1.f},
    {kRlStaged, 8, 3, 9.f, 5.f, {24.5f, 34.f, 44.5f}, 43.f, {17.3f, 22.8f, 28.8f}, 26.f, 1.f},
    {kRlStaged, 4, 2, 6.f, 5.f, {14.5f, 20.f}, kRlNever, {9.9f, 12.5f}, kRlNever, 1.f}};

double rl_time(const RlForm& f, const RlCarve& c, int heads, int n, int half, int rounds) {
  const long long blocks = heads * rl_count(n, 8 * f.tr, 1);
  const auto tiles = [&](const float* per, float wave) -> double {
    const long long per_sm = (blocks + kRlSms - 1) / kRlSms - 1;
    // (items of several tiles end apart: 0.4 tiles' time for each that one can have)
    if (c.span > 1 && wave < kRlNever) return ((double)blocks / (kRlSms * f.fit) + 0.4 * c.span) * wave * f.several;
    return per[per_sm % f.fit] + per_sm / f.fit * (double)wave;
  };
  const double first = tiles(f.first, f.first_wave), later = c.keep ? tiles(f.later, f.later_wave) : first;
  double t = f.call;
  for (int k = 0; k < rounds; ++k) t += f.round + (k ? later : first) * (half + (k && c.keep) - k) / half;
  return t;
}

// The layout of a call of `rounds` rounds that brings `room` bytes; the least one where that is too little for any.
RlCarve rl_carve(int heads, int n, int half, int rounds, size_t room) {
  // Up to 64 tokens the small form is the fastest one while a few of its blocks share an SM, up to 128 tokens while each
  // has its own: a search of few tokens is a chain of small launches, its time that of one block.
  const long long small = (long long)heads * ((n + kRsRows - 1) / kRsRows);
  if (n <= 2 * kRsKeys && small <= (n > kRsKeys ? 1 : half == 64 ? 2 : 4) * kRlSms) return rl_layout(heads, n, half, kRlSmall, 1, false);
  const RlForm* forms = half == 64 ? kRlForms128 : kRlForms64;
  RlCarve best;
  best.total = SIZE_MAX;
  double least = INFINITY;
  for (int i = 0; i < kRlForms; ++i) {
    const RlCarve c = rl_layout(heads, n, half, forms[i].kind, forms[i].tr, rounds > 1);
    const double t = c.total <= room ? rl_time(forms[i], c, heads, n, half, rounds) : INFINITY;
    if (t < least || (least == INFINITY && c.total < best.total)) {
      least = t;
      best = c;
    }
  }
  return best;
}

int rl_check(int heads, int n, int d_h) {
  if (heads <= 0 || n <= 0) return ELITEKV_ERR_INVALID_ARG;
  if (d_h != 64 && d_h != 128) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  if ((long long)n > (1 << 20) || heads > 65535) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  return ELITEKV_OK;
}

// One round of the group's heads.  Q, K (the small form's), masks and state are the group's first.
struct RlRound {
  const bf16 *Q, *K;
  const unsigned long long* masks;
  RlState* state;
  bool keep;                    // R is kept for the next round
  int first, last;              // round of the search
  bool silent;                  // self-test (ropelite_distance_kernel)
};
template <int HALF>
int rl_launch_half(const RlRound& d, int heads, int n, const RlCarve& c, unsigned char* base, cudaStream_t st) {
  const float2* cs = (const float2*)(base + c.off_cs);
  const float* sn = (const float*)(base + c.off_sin);
  float* partial = (float*)(base + c.off_partial);
  const dim3 grid((unsigned)c.items, (unsigned)heads);
  if (c.kind == kRlSmall) {
    const auto kern = ropelite_distance_small_kernel<HALF>;
    EKV_CUDA_OK(ekv_allow_smem(kern, sizeof(RsSmem<HALF>)));
    EKV_CUDA_OK(ekv_launch_pdl(kern, grid, dim3(32 * kRsWarps), sizeof(RsSmem<HALF>), st, d.Q, d.K, n, cs, sn, d.masks, partial));
  } else if (c.kind == kRlResident) {
    const auto launch = [&](auto form) -> int {
      using F = decltype(form);
      const auto kern = ropelite_distance_resident_kernel<HALF, F>;
      EKV_CUDA_OK(ekv_allow_smem(kern, sizeof(RlResident<HALF, F>)));
      EKV_CUDA_OK(ekv_launch_pdl(kern, grid, dim3(F::THREADS), sizeof(RlResident<HALF, F>), st, d.Q, d.K, n, cs, sn, d.masks, c.span,
                                 partial));
      return ELITEKV_OK;
    };
    const int rc = c.tr == 16 ? launch(Rl<16, 4>()) : c.tr == 8 ? launch(Rl<8, 4>()) : launch(Rl<4, 4>());
    if (rc != ELITEKV_OK) return rc;
  } else {
    const auto launch = [&](auto form) -> int {
      using F = decltype(form);
      const auto kern = HALF == 32 && F::TR == 4 && d.silent ? ropelite_distance_kernel<HALF, F, HALF == 32 && F::TR == 4>
                                                             : ropelite_distance_kernel<HALF, F>;
      EKV_CUDA_OK(ekv_allow_smem(kern, sizeof(RlSmem<HALF, F>)));
      EKV_CUDA_OK(ekv_launch_pdl(kern, grid, dim3(F::THREADS), sizeof(RlSmem<HALF, F>), st, (const float*)(base + c.off_rot), n,
                                 rl_pad_n(n), sn, d.masks, c.span, partial,
                                 d.keep ? (ulonglong2*)(base + c.off_kept) : nullptr, d.state, d.first, d.last));
      return ELITEKV_OK;
    };
    const int rc = c.tr == 8 ? launch(RlLarge()) : launch(RlFew());
    if (rc != ELITEKV_OK) return rc;
  }
  EKV_CUDA_OK(cudaGetLastError());
  return ELITEKV_OK;
}
int rl_launch_distance(const RlRound& d, int heads, int n, int d_h, const RlCarve& c, unsigned char* base, cudaStream_t st) {
  return d_h == 128 ? rl_launch_half<64>(d, heads, n, c, base, st) : rl_launch_half<32>(d, heads, n, c, base, st);
}
int rl_launch_rotate(const bf16* Q, const bf16* K, int heads, int n, int d_h, const RlCarve& c, unsigned char* base, cudaStream_t st) {
  if (c.kind != kRlStaged) return ELITEKV_OK;
  EKV_CUDA_OK(ekv_launch_pdl(ropelite_rotate_kernel, dim3((unsigned)rl_pad_n(n) / 64, (unsigned)heads, 2), dim3(256), 0, st, Q, K,
                             (const float2*)(base + c.off_cs), (float*)(base + c.off_rot), n, rl_pad_n(n), d_h / 2,
                             c.tr == 8 ? RlLarge::ROWS : RlFew::ROWS, (int)(c.tr == 8)));
  EKV_CUDA_OK(cudaGetLastError());
  return ELITEKV_OK;
}

// one block per SM, whatever the other kernel's blocks hold
int rl_apart(long long blocks) { return blocks <= kRlSms; }
RlState* rl_state(const RlCarve& c, unsigned char* base) { return c.kind == kRlStaged ? (RlState*)(base + c.off_state) : nullptr; }
int rl_launch_table(const RlCarve& c, unsigned char* base_ptr, int n, int d_h, float base, unsigned long long* masks, int heads,
                    cudaStream_t st) {
  const long long total = (long long)rl_sin_len(n) * (d_h / 2);
  EKV_CUDA_OK(ekv_launch_pdl(ropelite_table_kernel, dim3((unsigned)((total + 255) / 256)), dim3(256), 0, st,
                             (float2*)(base_ptr + c.off_cs), (float*)(base_ptr + c.off_sin), n, d_h / 2, d_h, (double)base, masks,
                             rl_state(c, base_ptr), heads,
                             c.kind != kRlStaged && rl_apart((total + 255) / 256 + (long long)c.items * heads)));
  EKV_CUDA_OK(cudaGetLastError());
  return ELITEKV_OK;
}

}  // namespace

extern "C" int elitekv_ropelite_workspace_size(int32_t n_heads, int32_t n, int32_t d_h, size_t* bytes) {
  if (!bytes) return ELITEKV_ERR_INVALID_ARG;
  const int rc = rl_check(n_heads, n, d_h);
  if (rc != ELITEKV_OK) return rc;
  // what any of its forms can use
  *bytes = rl_carve(n_heads, n, d_h / 2, 1, SIZE_MAX).total;
  if (rl_carve(n_heads, n, d_h / 2, 1, SIZE_MAX).kind != kRlSmall)
    for (int i = 0; i < kRlForms; ++i) {
      const size_t total = rl_layout(n_heads, n, d_h / 2, kRlForms128[i].kind, kRlForms128[i].tr, true).total;
      if (total > *bytes) *bytes = total;
    }
  return ELITEKV_OK;
}

extern "C" int elitekv_ropelite_workspace_size_rounds(int32_t n_heads, int32_t n, int32_t d_h, int32_t rounds, size_t* bytes) {
  if (!bytes) return ELITEKV_ERR_INVALID_ARG;
  const int rc = rl_check(n_heads, n, d_h);
  if (rc != ELITEKV_OK) return rc;
  if (rounds < 0 || rounds > d_h / 2) return ELITEKV_ERR_INVALID_ARG;
  *bytes = rl_carve(n_heads, n, d_h / 2, rounds, rounds > 0 ? SIZE_MAX : 0).total;
  return ELITEKV_OK;
}

extern "C" int elitekv_ropelite_distances(const void* Q, const void* K, int32_t n_heads, int32_t n, int32_t d_h,
                                          float rope_base, const uint64_t* elite_mask, void* workspace,
                                          size_t workspace_bytes, float* dist, elitekv_stream_t stream) {
  if (!Q || !K || !workspace || !dist) return ELITEKV_ERR_INVALID_ARG;
  if (((uintptr_t)Q & 15) || ((uintptr_t)K & 15)) return ELITEKV_ERR_INVALID_ARG;
  int rc = rl_check(n_heads, n, d_h);
  if (rc != ELITEKV_OK) return rc;
  const int half = d_h / 2;
  const RlCarve c = rl_carve(n_heads, n, half, 1, workspace_bytes);
  if (((uintptr_t)workspace & 255) || workspace_bytes < c.total) return ELITEKV_ERR_WORKSPACE_TOO_SMALL;
  unsigned char* base = (unsigned char*)workspace;
  float* partial = (float*)(base + c.off_partial);
  cudaStream_t st = (cudaStream_t)stream;
  rc = rl_launch_table(c, base, n, d_h, rope_base, nullptr, n_heads, st);
  if (rc != ELITEKV_OK) return rc;
  unsigned long long* masks = (unsigned long long*)elite_mask;
  RlState* state = rl_state(c, base);
  for (int h0 = 0; h0 < n_heads; h0 += c.group) {
    const int heads = n_heads - h0 < c.group ? n_heads - h0 : c.group;
    const size_t at = (size_t)h0 * n * d_h;
    const RlRound d{(const bf16*)Q + at, (const bf16*)K + at, masks ? masks + h0 : nullptr, state ? state + h0 : nullptr, false, 1, 1, false};
    rc = rl_launch_rotate(d.Q, d.K, heads, n, d_h, c, base, st);
    if (rc == ELITEKV_OK) rc = rl_launch_distance(d, heads, n, d_h, c, base, st);
    if (rc != ELITEKV_OK) return rc;
    EKV_CUDA_OK(ekv_launch_pdl(ropelite_select_kernel, dim3(heads), dim3(64 * kRlSelect), 0, st, partial, c.items, half,
                               masks ? masks + h0 : nullptr, dist + (size_t)h0 * half, nullptr, 0, 0, nullptr, 0, 0));
    EKV_CUDA_OK(cudaGetLastError());
  }
  return ELITEKV_OK;
}

namespace {

int rl_search(const RlCarve& c, const void* Q, const void* K, int n_heads, int n, int d_h, float rope_base, int r, void* workspace,
              size_t workspace_bytes, int32_t* elite_idx, float* dist_trace, cudaStream_t st, bool silent) {
  const int half = d_h / 2;
  if (((uintptr_t)workspace & 255) || workspace_bytes < c.total) return ELITEKV_ERR_WORKSPACE_TOO_SMALL;
  unsigned char* base = (unsigned char*)workspace;
  float* partial = (float*)(base + c.off_partial);
  unsigned long long* masks = (unsigned long long*)(base + c.off_masks);
  RlState* state = rl_state(c, base);
  const bool keep = c.keep && r > 1;
  int rc = rl_launch_table(c, base, n, d_h, rope_base, masks, n_heads, st);
  if (rc != ELITEKV_OK) return rc;
  for (int h0 = 0; h0 < n_heads; h0 += c.group) {
    const int heads = n_heads - h0 < c.group ? n_heads - h0 : c.group;
    const size_t at = (size_t)h0 * n * d_h;
    rc = r > 0 ? rl_launch_rotate((const bf16*)Q + at, (const bf16*)K + at, heads, n, d_h, c, base, st) : ELITEKV_OK;
    if (rc != ELITEKV_OK) return rc;
    for (int round = 0; round < r; ++round) {
      rc = rl_launch_distance(RlRound{(const bf16*)Q + at, (const bf16*)K + at, masks + h0, state ? state + h0 : nullptr, keep, round == 0, round == r - 1, silent},
                              heads, n, d_h, c, base, st);
      if (rc != ELITEKV_OK) return rc;
      EKV_CUDA_OK(ekv_launch_pdl(ropelite_select_kernel, dim3(heads), dim3(64 * kRlSelect), 0, st, partial, c.items, half, masks + h0,
                                 dist_trace ? dist_trace + ((size_t)round * n_heads + h0) * half : nullptr,
                                 elite_idx + (size_t)h0 * r, r, round, state ? state + h0 : nullptr, (int)keep, rl_apart((long long)(c.items + 1) * heads)));
      EKV_CUDA_OK(cudaGetLastError());
    }
  }
  return ELITEKV_OK;
}

}  // namespace

extern "C" int elitekv_ropelite_search(const void* Q, const void* K, int32_t n_heads, int32_t n, int32_t d_h,
                                       float rope_base, int32_t r, void* workspace, size_t workspace_bytes,
                                       int32_t* elite_idx, float* dist_trace, elitekv_stream_t stream) {
  if (!Q || !K || !workspace || !elite_idx) return ELITEKV_ERR_INVALID_ARG;
  if (((uintptr_t)Q & 15) || ((uintptr_t)K & 15)) return ELITEKV_ERR_INVALID_ARG;
  const int rc = rl_check(n_heads, n, d_h);
  if (rc != ELITEKV_OK) return rc;
  if (r < 0 || r > d_h / 2) return ELITEKV_ERR_INVALID_ARG;
  return rl_search(rl_carve(n_heads, n, d_h / 2, r, workspace_bytes), Q, K, n_heads, n, d_h, rope_base, r, workspace, workspace_bytes, elite_idx,
                   dist_trace, (cudaStream_t)stream, false);
}

// The distance kernel with stages that nobody fills, on two heads of 130 tokens and d_h 64, two rounds.
extern "C" int elitekv_selftest_search_timeout(const void* Q, const void* K, void* workspace, size_t workspace_bytes,
                                               int32_t* elite_idx, float* dist_trace, elitekv_stream_t stream) {
  if (!Q || !K || !workspace || !elite_idx || !dist_trace || ((uintptr_t)Q & 15) || ((uintptr_t)K & 15)) return ELITEKV_ERR_INVALID_ARG;
  return rl_search(rl_layout(2, 130, 32, kRlStaged, 4, true), Q, K, 2, 130, 64, 10000.f, 2, workspace, workspace_bytes, elite_idx, dist_trace, (cudaStream_t)stream, true);
}
