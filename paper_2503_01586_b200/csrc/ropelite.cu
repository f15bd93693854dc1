// RoPElite search scoring (Algorithm 1, Section 3.1), all heads of all layers in one launch.
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
// Bound: FP32 pipe and issue (the contraction is 2 deep).  A thread owns 16 query rows x 4 keys, sums R
// over the free chunks (t: multiply, FMA; R: FMA), then goes over the chunks once more for |R - D_j|
// (FMA, add with |.|): 7 operations per pair and chunk, D_i is never stored, and the 64 pairs of a
// thread share their operands, 15 16-byte shared-memory loads per chunk and pass.  Two rows at a time
// with packed operations (all but the add with |.|): 43 % fewer instructions at the same number of
// fp32 operations; pairs of neighbouring table entries are formed in registers.  32 heads x 2048 tokens
// x d_h 128: 1.48 ms a round (1.58 with scalar operations, 1.53 with the chunk loops unrolled twice
// and not eight times; 0.54 of 148 SMs x 128 lanes x 1.965 GHz).  The form that holds the 64 D_i of one
// pair in registers took 3.04 ms: 9 operations and three loads per pair and chunk, shared-memory bound.
// Short calibrations cannot fill the device with 128 x 128 tiles: there a thread owns 8 or 4 rows, and up
// to 128 tokens the register form is the faster one (rl_form; one head of 64 tokens, four rounds: 235 us on
// one such tile, 72 us).
//
// distance kernel: grid (items, heads), 256 threads; an item is 128 (64, 32) query rows x up to `span` key
// tiles of 128.  Per key tile the rotated keys (x plane, y plane, [chunk][key]) and the slice of
// the sine table that the tile's relative positions need are staged in shared memory; the table is
// zero at negative relative positions, which is the causal mask.  Item results go to a
// [head][item][chunk] array; the select kernel adds them in a fixed order (the result does not
// depend on scheduling), masks the chunks already chosen and takes the first minimum.
#include <initializer_list>

#include "common.cuh"

namespace {

constexpr int kRlKeys = 128;      // keys per stage
constexpr int kRlTK = 4;          // ... per thread
constexpr int kRlAcc = 8;         // lanes of a warp that keep running distances
constexpr int kRlPad = 256;       // zeros in front of the sine table: negative relative positions
static_assert(kRlKeys == 32 * kRlTK, "thread tiles cover the block's keys");

// blocks of 8 warps with TR query rows per warp (and thread): 16, or 8 or 4 where that fills the device better
template <int TR_>
struct Rl {
  static constexpr int TR = TR_, NW = 8, THREADS = 32 * NW;
  static constexpr int ROWS = NW * TR;                   // query rows per block
  static constexpr int SPAN = kRlKeys + ROWS;            // sine table entries of a stage (relative positions)
  static_assert(ROWS <= 128 && SPAN <= kRlPad, "a stage's slice lies inside the table");
};

// entries of a chunk's sine table: entry x holds 2 sin((x - kRlPad) theta / 2), zero up to kRlPad
__host__ __device__ inline int rl_sin_len(int n) { return (n + 127) / 128 * 128 + kRlPad; }

// (cos, sin)(pos theta_i / 2) laid out [pos][chunk], and the sine table [chunk][...];
// double precision, rounded once
__global__ void ropelite_table_kernel(float2* __restrict__ cs, float* __restrict__ sn, int n, int half, int d_h,
                                      double base) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  const int len = rl_sin_len(n);
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
  const float4 c01 = __ldg((const float4*)cs), c23 = __ldg((const float4*)cs + 1);
  const float2 c[4] = {{c01.x, c01.y}, {c01.z, c01.w}, {c23.x, c23.y}, {c23.z, c23.w}};
#pragma unroll
  for (int u = 0; u < 4; ++u) {
    const float x = __uint_as_float(w[u] << 16), y = __uint_as_float(w[u] & 0xffff0000u);
    out[u] = make_float2(x * c[u].x - y * c[u].y, x * c[u].y + y * c[u].x);
  }
}

template <int HALF, class F>
struct RlSmem {
  float kx[HALF][kRlKeys], ky[HALF][kRlKeys];
  float sn[HALF][F::SPAN];
  float qx[HALF][F::ROWS], qy[HALF][F::ROWS];
  float acc[HALF][F::NW * kRlAcc];     // running distances
  int list[HALF];                    // chunks not chosen yet
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

// operands of a thread's 4 TR pairs for one chunk; kNeg: t with its sign turned
template <int TR>
struct RlOps {
  rl2 a[kRlTK], b[kRlTK];            // keys: t = q_y a + q_x b
  rl2 qx[TR / 2], qy[TR / 2];
  rl2 s[(TR + kRlTK) / 2][2];        // [v][0]: table entries 2 v, 2 v + 1; [v][1]: 2 v + 1, 2 v + 2
};
template <int HALF, class F, bool kNeg>
__device__ __forceinline__ void rl_load(RlOps<F::TR>& o, const RlSmem<HALF, F>& sm, int i, int warp, int lane) {
  constexpr int TR = F::TR;
  const float4 kx = *(const float4*)&sm.kx[i][lane * kRlTK], ky = *(const float4*)&sm.ky[i][lane * kRlTK];
  const float x[kRlTK] = {kx.x, kx.y, kx.z, kx.w}, y[kRlTK] = {ky.x, ky.y, ky.z, ky.w};
#pragma unroll
  for (int j = 0; j < kRlTK; ++j) {
    const float a = kNeg ? -x[j] : x[j], b = kNeg ? y[j] : -y[j];
    o.a[j] = rl_pack(a, a);
    o.b[j] = rl_pack(b, b);
  }
  // entry u of the stage's slice: relative position (m0 - n0) - 128 + u; this thread's pairs need
  // u = TR warp + r - (4 lane + j) + 128, from TR warp - 4 lane + 124 on
  const float4* sp = (const float4*)&sm.sn[i][TR * warp - kRlTK * lane + kRlKeys - kRlTK];
  float e[TR + kRlTK];
#pragma unroll
  for (int u = 0; u < (TR + kRlTK) / 4; ++u) *(float4*)&e[4 * u] = sp[u];
#pragma unroll
  for (int v = 0; v < (TR + kRlTK) / 2; ++v) {
    o.s[v][0] = rl_pack(e[2 * v], e[2 * v + 1]);
    if (2 * v + 2 < TR + kRlTK) o.s[v][1] = rl_pack(e[2 * v + 1], e[2 * v + 2]);
  }
  const ulonglong2* qx = (const ulonglong2*)&sm.qx[i][TR * warp];
  const ulonglong2* qy = (const ulonglong2*)&sm.qy[i][TR * warp];
#pragma unroll
  for (int u = 0; u < TR / 4; ++u) {
    const ulonglong2 vx = qx[u], vy = qy[u];
    o.qx[2 * u] = vx.x; o.qx[2 * u + 1] = vx.y;
    o.qy[2 * u] = vy.x; o.qy[2 * u + 1] = vy.y;
  }
}
// table pair of rows 2 r, 2 r + 1 and key j: entries 2 r - j + 4 and the next
template <int TR>
__device__ __forceinline__ rl2 rl_sin(const RlOps<TR>& o, int r, int j) { return o.s[(2 * r - j + kRlTK) / 2][(2 * r - j + kRlTK) & 1]; }

// What a search keeps of a head from one round to the next, beside its sums R.
struct RlState {
  float norm;       // largest distance of the round that last summed R afresh
  int last;         // chunk chosen in the round before
  int fresh;        // the next round sums R afresh
};

// Tiles of 128 keys in a head's row tiles below mt (a row tile ends at the diagonal).
template <class F>
__host__ __device__ inline long long rl_tiles_below(int mt) {
  constexpr int q = kRlKeys / F::ROWS;
  const long long a = mt / q, b = mt % q;
  return q * (a * (a + 1) / 2) + b * (a + 1);
}

template <int HALF, class F>
__global__ void __launch_bounds__(F::THREADS)
ropelite_distance_kernel(const bf16* __restrict__ Q, const bf16* __restrict__ K, int n,
                         const float2* __restrict__ cs, const float* __restrict__ sn,
                         const unsigned long long* __restrict__ masks, int span,
                         float* __restrict__ partial /* [heads][items][HALF] */,
                         ulonglong2* __restrict__ kept /* [heads][tiles][TR][THREADS], null: R is not kept */,
                         const RlState* __restrict__ state, int first_round, int last_round) {
  constexpr int d_h = 2 * HALF, TR = F::TR, NW = F::NW, THREADS = F::THREADS, ROWS = F::ROWS, SPAN = F::SPAN;
  extern __shared__ __align__(16) unsigned char smem_rl[];
  RlSmem<HALF, F>& sm = *(RlSmem<HALF, F>*)smem_rl;
  const int head = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // item -> (row tile, group of key tiles), long rows first
  int mt = (n + ROWS - 1) / ROWS - 1, kg = blockIdx.x;
  for (;; --mt) {
    const int groups = ((mt + 1) * ROWS + kRlKeys * span - 1) / (kRlKeys * span);
    if (kg < groups) break;
    kg -= groups;
  }
  const int m0 = mt * ROWS;
  const int n_lo = kg * span * kRlKeys, n_hi = min(n_lo + span * kRlKeys, m0 + ROWS);
  const unsigned long long mask = masks ? masks[head] : 0ull;
  const int n_free = HALF - __popcll(HALF == 64 ? mask : mask & ((1ull << (HALF & 63)) - 1));
  float* out = partial + ((size_t)head * gridDim.x + blockIdx.x) * HALF;
  if (n_free <= 1) {                 // a single free chunk: R = D_j for every pair
    for (int j = threadIdx.x; j < HALF; j += THREADS) out[j] = 0.f;
    return;
  }
  if (threadIdx.x < HALF && !((mask >> threadIdx.x) & 1ull))
    sm.list[threadIdx.x - __popcll(mask & ((1ull << threadIdx.x) - 1))] = threadIdx.x;
  const bool fresh = kept == nullptr || first_round || state[head].fresh;
  const int chosen = fresh ? 0 : state[head].last;
  if (kept)
    kept += (head * rl_tiles_below<F>((n + ROWS - 1) / ROWS) + rl_tiles_below<F>(mt)) * (TR * THREADS) + threadIdx.x;
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
    // pairs of this warp that are not all above the diagonal, nor its rows past the last token
    const bool live = n0 <= m0 + TR * warp + TR - 1 && m0 + TR * warp < n;
    rl2 R[TR / 2][kRlTK];
    ulonglong2* const keep_at = kept + (size_t)(n0 / kRlKeys) * (TR * THREADS);
    if (!fresh && live) {                        // lands while the tile is staged
#pragma unroll
      for (int u = 0; u < TR; ++u) {
        const ulonglong2 v = __ldcs(keep_at + u * THREADS);
        R[u / 2][u % 2 * 2] = v.x;
        R[u / 2][u % 2 * 2 + 1] = v.y;
      }
    }
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
    if (!live) continue;
    if (fresh) {
#pragma unroll
      for (int r = 0; r < TR / 2; ++r)
#pragma unroll
        for (int j = 0; j < kRlTK; ++j) R[r][j] = 0ull;
#pragma unroll 8
      for (int c = 0; c < n_free; ++c) {
        RlOps<TR> o;
        rl_load<HALF, F, false>(o, sm, sm.list[c], warp, lane);
#pragma unroll
        for (int r = 0; r < TR / 2; ++r)
#pragma unroll
          for (int j = 0; j < kRlTK; ++j) {
            const rl2 t = rl_fma(o.qx[r], o.b[j], rl_mul(o.qy[r], o.a[j]));
            R[r][j] = rl_fma(rl_sin(o, r, j), t, R[r][j]);
          }
      }
    } else {                                     // R loses the chunk chosen in the round before
      RlOps<TR> o;
      rl_load<HALF, F, true>(o, sm, chosen, warp, lane);
#pragma unroll
      for (int r = 0; r < TR / 2; ++r)
#pragma unroll
        for (int j = 0; j < kRlTK; ++j) {
          const rl2 t = rl_fma(o.qx[r], o.b[j], rl_mul(o.qy[r], o.a[j]));
          R[r][j] = rl_fma(rl_sin(o, r, j), t, R[r][j]);
        }
    }
    if (kept && !last_round) {
#pragma unroll
      for (int u = 0; u < TR; ++u) __stcs(keep_at + u * THREADS, make_ulonglong2(R[u / 2][u % 2 * 2], R[u / 2][u % 2 * 2 + 1]));
    }
#pragma unroll 8
    for (int c = 0; c < n_free; ++c) {
      RlOps<TR> o;
      const int i = sm.list[c];
      rl_load<HALF, F, true>(o, sm, i, warp, lane);
      float v[kRlTK] = {};
#pragma unroll
      for (int r = 0; r < TR / 2; ++r)
#pragma unroll
        for (int j = 0; j < kRlTK; ++j) {
          const rl2 t = rl_fma(o.qx[r], o.b[j], rl_mul(o.qy[r], o.a[j]));
          const float2 x = rl_unpack(rl_fma(rl_sin(o, r, j), t, R[r][j]));
          v[j] += fabsf(x.x);
          v[j] += fabsf(x.y);
        }
      float d = (v[0] + v[1]) + (v[2] + v[3]);
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
                               const float2* __restrict__ cs, const float* __restrict__ sn,
                               const unsigned long long* __restrict__ masks,
                               float* __restrict__ partial /* [heads][row tiles][HALF] */) {
  constexpr int d_h = 2 * HALF, THREADS = 32 * kRsWarps;
  extern __shared__ __align__(16) unsigned char smem_rl[];
  RsSmem<HALF>& sm = *(RsSmem<HALF>*)smem_rl;
  const int head = blockIdx.y, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * kRsRows, m_last = min(m0 + kRsRows, n) - 1;
  const unsigned long long mask = masks ? masks[head] : 0ull;
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
__global__ void ropelite_select_kernel(const float* __restrict__ partial, int n_items, int half,
                                       unsigned long long* __restrict__ masks, float* __restrict__ dist_out,
                                       int32_t* __restrict__ elite_idx, int r, int round,
                                       RlState* __restrict__ state) {
  __shared__ float s_d[kRlSelect][64];
  const int head = blockIdx.x, j = threadIdx.x & 63, part = threadIdx.x >> 6;
  const unsigned long long mask = masks ? masks[head] : 0ull;
  float v = 0.f;
  if (j < half) {
    const float* src = partial + (size_t)head * n_items * half + j;
#pragma unroll 4
    for (int t = part; t < n_items; t += kRlSelect) v += src[(size_t)t * half];
  }
  s_d[part][j] = v;
  __syncthreads();
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
  if (threadIdx.x == 0 && elite_idx) {
    int best = 0;
    for (int c = 1; c < half; ++c)
      if (s_d[0][c] < s_d[0][best]) best = c;
    elite_idx[(size_t)head * r + round] = best;
    masks[head] = mask | (1ull << best);
    if (state) {
      // The winner's distance is the L1 norm of the next round's R.  Taking chunks out of a kept R adds
      // rounding errors of the size of the R that was summed; below a quarter of it, or where anything
      // is not finite, R is summed afresh, so that the errors stay of the size of those of a sum.
      float norm = state[head].norm;
      if (round == 0 || state[head].fresh) {
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

struct RlCarve {
  size_t off_cs, off_sin, off_partial, off_masks, off_state, total;
  size_t off_kept, total_kept;  // the sums R of kept_heads heads behind the rest
  int tr, span, items;          // rows per thread (1: the small form), key tiles per item, items per head
  int kept_heads;               // heads that a search takes through its rounds together (0: R is not kept)
};
inline size_t rl_align(size_t x) { return (x + 255) & ~(size_t)255; }

// Key tiles per item: whole rows cut into at most 16 items, at least 4 tiles long (the rotated
// queries of an item are prepared anew); single tiles where that would leave most of the
// device without work (fewer blocks than four for each of 148 SMs).
long long rl_count(int n, int rows, int span) {
  long long k = 0;
  for (int m = rows; m < n + rows; m += rows) k += (m + kRlKeys * span - 1) / (kRlKeys * span);
  return k;
}
// Which form, for a device of 148 SMs.  A search of few tokens is a chain of small launches: its time is
// that of one block.  Up to 64 tokens the small form is the faster one while a few of its blocks share an
// SM, up to 128 tokens while each has its own.  Four rounds, d_h 128, us (small / 4 / 8 / 16 rows per
// thread): 4 heads x 64 tokens 72 / 129 / 163 / 173, 4 x 128 105 / 133 / 171 / 246, 32 x 128 - / 132 / 172 / 250,
// 32 x 300 - / 427 / 308 / 391, 16 x 512 - / 522 / 440 / 460, 16 x 1024 - / 1606 / 1111 / 894.  Beyond it the
// form whose blocks take least time in all, in whole rounds over the device: a key tile of a block takes
// 24, 33 and 52 us at d_h 128, and in the same proportions at d_h 64.
void rl_form(int heads, int n, int half, RlCarve* c) {
  constexpr int kSms = 148;
  const long long small = (long long)heads * ((n + kRsRows - 1) / kRsRows);
  c->span = 1;
  if (n <= 2 * kRsKeys && small <= (n > kRsKeys ? 1 : half == 64 ? 2 : 4) * kSms) {
    c->tr = 1;
    c->items = (n + kRsRows - 1) / kRsRows;
    return;
  }
  long long best = 0;
  for (const int tr : {16, 8, 4}) {
    const int cost = tr == 16 ? 52 : tr == 8 ? 33 : 24;
    const long long t = (heads * rl_count(n, 8 * tr, 1) + kSms - 1) / kSms * cost;
    if (tr == 16 || t < best) {
      best = t;
      c->tr = tr;
    }
  }
  const int tiles = (n + kRlKeys - 1) / kRlKeys, span = tiles > 64 ? (tiles + 15) / 16 : 4;
  if (heads * rl_count(n, 8 * c->tr, span) >= 4 * kSms) c->span = span;
  c->items = (int)rl_count(n, 8 * c->tr, c->span);
}
// The sums R of a head, four bytes for each pair of its tiles (9 MB at 2048 tokens, 137 MB at 8192).  Heads are
// independent, so a search whose heads need more than kRlKeptMost takes them through its rounds in groups;
// one head of over 22000 tokens alone needs more, and its R is summed in every round.
constexpr size_t kRlKeptMost = (size_t)1 << 30;
template <class F>
size_t rl_kept_bytes_of(int n) {
  return (size_t)rl_tiles_below<F>((n + F::ROWS - 1) / F::ROWS) * F::TR * F::THREADS * sizeof(ulonglong2);
}
size_t rl_kept_bytes(int tr, int n) {
  return tr == 16 ? rl_kept_bytes_of<Rl<16>>(n) : tr == 8 ? rl_kept_bytes_of<Rl<8>>(n) : rl_kept_bytes_of<Rl<4>>(n);
}
RlCarve rl_carve(int heads, int n, int half) {
  RlCarve c;
  rl_form(heads, n, half, &c);
  size_t o = 0;
  c.off_cs = o;      o = rl_align(o + sizeof(float2) * (size_t)half * n);
  c.off_sin = o;     o = rl_align(o + sizeof(float) * (size_t)half * rl_sin_len(n));
  c.off_partial = o; o = rl_align(o + sizeof(float) * (size_t)heads * c.items * half);
  c.off_masks = o;   o = rl_align(o + sizeof(unsigned long long) * (size_t)heads);
  c.off_state = o;   o = rl_align(o + sizeof(RlState) * (size_t)heads);
  c.total = o;
  c.off_kept = o;
  const size_t per_head = rl_kept_bytes(c.tr, n);
  c.kept_heads = c.tr == 1 || per_head > kRlKeptMost ? 0 : (int)(kRlKeptMost / per_head < (size_t)heads ? kRlKeptMost / per_head : (size_t)heads);
  c.total_kept = o + (size_t)c.kept_heads * per_head;
  return c;
}

int rl_check(int heads, int n, int d_h) {
  if (heads <= 0 || n <= 0) return ELITEKV_ERR_INVALID_ARG;
  if (d_h != 64 && d_h != 128) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  if ((long long)n > (1 << 20) || heads > 65535) return ELITEKV_ERR_UNSUPPORTED_SHAPE;
  return ELITEKV_OK;
}

struct RlKeep {
  ulonglong2* kept;             // null: R is summed in every round
  const RlState* state;
  int first_round, last_round;
};
template <int HALF>
int rl_launch_half(const void* Q, const void* K, int heads, int n, const RlCarve& c, unsigned char* base,
                   const unsigned long long* masks, const RlKeep& k, cudaStream_t st) {
  const float2* cs = (const float2*)(base + c.off_cs);
  const float* sn = (const float*)(base + c.off_sin);
  float* partial = (float*)(base + c.off_partial);
  const dim3 grid((unsigned)c.items, (unsigned)heads);
  if (c.tr == 1) {
    const auto kern = ropelite_distance_small_kernel<HALF>;
    EKV_CUDA_OK(ekv_allow_smem(kern, sizeof(RsSmem<HALF>)));
    kern<<<grid, 32 * kRsWarps, sizeof(RsSmem<HALF>), st>>>((const bf16*)Q, (const bf16*)K, n, cs, sn, masks, partial);
  } else {
    const auto launch = [&](auto form) -> int {
      using F = decltype(form);
      const auto kern = ropelite_distance_kernel<HALF, F>;
      EKV_CUDA_OK(ekv_allow_smem(kern, sizeof(RlSmem<HALF, F>)));
      kern<<<grid, F::THREADS, sizeof(RlSmem<HALF, F>), st>>>((const bf16*)Q, (const bf16*)K, n, cs, sn, masks, c.span, partial,
                                                              k.kept, k.state, k.first_round, k.last_round);
      return ELITEKV_OK;
    };
    const int rc = c.tr == 16 ? launch(Rl<16>()) : c.tr == 8 ? launch(Rl<8>()) : launch(Rl<4>());
    if (rc != ELITEKV_OK) return rc;
  }
  EKV_CUDA_OK(cudaGetLastError());
  return ELITEKV_OK;
}
int rl_launch_distance(const void* Q, const void* K, int heads, int n, int d_h, const RlCarve& c, unsigned char* base,
                       const unsigned long long* masks, const RlKeep& k, cudaStream_t st) {
  return d_h == 128 ? rl_launch_half<64>(Q, K, heads, n, c, base, masks, k, st)
                    : rl_launch_half<32>(Q, K, heads, n, c, base, masks, k, st);
}

int rl_launch_table(const RlCarve& c, unsigned char* base_ptr, int n, int d_h, float base, cudaStream_t st) {
  const long long total = (long long)rl_sin_len(n) * (d_h / 2);
  ropelite_table_kernel<<<(unsigned)((total + 255) / 256), 256, 0, st>>>(
      (float2*)(base_ptr + c.off_cs), (float*)(base_ptr + c.off_sin), n, d_h / 2, d_h, (double)base);
  EKV_CUDA_OK(cudaGetLastError());
  return ELITEKV_OK;
}

}  // namespace

extern "C" int elitekv_ropelite_workspace_size(int32_t n_heads, int32_t n, int32_t d_h, size_t* bytes) {
  if (!bytes) return ELITEKV_ERR_INVALID_ARG;
  const int rc = rl_check(n_heads, n, d_h);
  if (rc != ELITEKV_OK) return rc;
  *bytes = rl_carve(n_heads, n, d_h / 2).total_kept;
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
  const RlCarve c = rl_carve(n_heads, n, half);
  if (((uintptr_t)workspace & 255) || workspace_bytes < c.total) return ELITEKV_ERR_WORKSPACE_TOO_SMALL;
  unsigned char* base = (unsigned char*)workspace;
  float* partial = (float*)(base + c.off_partial);
  cudaStream_t st = (cudaStream_t)stream;
  rc = rl_launch_table(c, base, n, d_h, rope_base, st);
  if (rc != ELITEKV_OK) return rc;
  rc = rl_launch_distance(Q, K, n_heads, n, d_h, c, base, (const unsigned long long*)elite_mask, RlKeep{nullptr, nullptr, 1, 1}, st);
  if (rc != ELITEKV_OK) return rc;
  ropelite_select_kernel<<<n_heads, 64 * kRlSelect, 0, st>>>(partial, c.items, half,
                                                 (unsigned long long*)elite_mask, dist, nullptr, 0, 0, nullptr);
  EKV_CUDA_OK(cudaGetLastError());
  return ELITEKV_OK;
}

extern "C" int elitekv_ropelite_search(const void* Q, const void* K, int32_t n_heads, int32_t n, int32_t d_h,
                                       float rope_base, int32_t r, void* workspace, size_t workspace_bytes,
                                       int32_t* elite_idx, float* dist_trace, elitekv_stream_t stream) {
  if (!Q || !K || !workspace || !elite_idx) return ELITEKV_ERR_INVALID_ARG;
  if (((uintptr_t)Q & 15) || ((uintptr_t)K & 15)) return ELITEKV_ERR_INVALID_ARG;
  int rc = rl_check(n_heads, n, d_h);
  if (rc != ELITEKV_OK) return rc;
  const int half = d_h / 2;
  if (r < 0 || r > half) return ELITEKV_ERR_INVALID_ARG;
  const RlCarve c = rl_carve(n_heads, n, half);
  if (((uintptr_t)workspace & 255) || workspace_bytes < c.total) return ELITEKV_ERR_WORKSPACE_TOO_SMALL;
  unsigned char* base = (unsigned char*)workspace;
  float* partial = (float*)(base + c.off_partial);
  unsigned long long* masks = (unsigned long long*)(base + c.off_masks);
  RlState* state = (RlState*)(base + c.off_state);
  cudaStream_t st = (cudaStream_t)stream;
  rc = rl_launch_table(c, base, n, d_h, rope_base, st);
  if (rc != ELITEKV_OK) return rc;
  EKV_CUDA_OK(cudaMemsetAsync(masks, 0, sizeof(unsigned long long) * (size_t)n_heads, st));
  // a smaller workspace than the one asked for serves the form that keeps nothing
  const bool keep = c.kept_heads > 0 && r > 1 && workspace_bytes >= c.total_kept;
  const int group = keep ? c.kept_heads : n_heads;
  for (int h0 = 0; h0 < n_heads; h0 += group) {
    const int heads = n_heads - h0 < group ? n_heads - h0 : group;
    const bf16 *Qg = (const bf16*)Q + (size_t)h0 * n * d_h, *Kg = (const bf16*)K + (size_t)h0 * n * d_h;
    for (int round = 0; round < r; ++round) {
      rc = rl_launch_distance(Qg, Kg, heads, n, d_h, c, base, masks + h0,
                              RlKeep{keep ? (ulonglong2*)(base + c.off_kept) : nullptr, state + h0, round == 0, round == r - 1}, st);
      if (rc != ELITEKV_OK) return rc;
      ropelite_select_kernel<<<heads, 64 * kRlSelect, 0, st>>>(partial, c.items, half, masks + h0,
                                                     dist_trace ? dist_trace + ((size_t)round * n_heads + h0) * half : nullptr,
                                                     elite_idx + (size_t)h0 * r, r, round, keep ? state + h0 : nullptr);
      EKV_CUDA_OK(cudaGetLastError());
    }
  }
  return ELITEKV_OK;
}
