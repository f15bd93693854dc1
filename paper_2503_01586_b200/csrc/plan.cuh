// Work plans (plan.cu has the description), one block of kPlanThreads threads: shared by the
// stand-alone kernel and by the kernel that prepares a whole decode step.
#pragma once

#include "common.cuh"

constexpr int kPlanThreads = 256;
constexpr int kPlanStage = 4096;       // items whose worker ids are staged in shared memory

// T: what tiles are summed in.  Lengths of up to 2^31 - 1 tokens in tiles of one pass 2^31 with two sequences;
// what a device's memory holds is far below it (plan_narrow), and 64-bit sums there cost a step of one
// sequence 0.6 us of 39.
template <class T>
struct __align__(16) PlanShared {        // the block's shared memory
  long long total;
  T warp_tot[kPlanThreads / 32], g0[kPlanThreads], tiles[kPlanThreads];
  int first[kPlanThreads], len[kPlanThreads];
  short w0[kPlanThreads], wk[kPlanStage];    // wk: worker of each item (n_workers < 32768)
};

// The threads that make a plan.  A step's plan is run once, by one block, with instructions that are not in the caches:
// most of its time.  So the last warp makes the same trip at once and without effect, with made-up lengths, one turn
// of each loop, while the others still wait for the kernel before (or, where there is none, beside them).
constexpr int kPlanWorkers = kPlanThreads - 32;
struct PlanTeam {
  int threads;      // of which thread t is one
  bool dry;         // the last warp, by itself
  __device__ __forceinline__ void sync() const {
    if (dry) __syncwarp();
    else asm volatile("bar.sync 1, %0;" ::"r"(threads) : "memory");
  }
};

// exclusive scan over the team (warp shuffles + one shared array of warp totals)
template <class V, class T>
__device__ __forceinline__ V block_exclusive_scan(const PlanTeam& team, V v, T* warp_tot, V* total) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  V incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const V x = __shfl_up_sync(0xffffffffu, incl, o);
    if (lane >= o) incl += x;
  }
  if (lane == 31 && !team.dry) warp_tot[warp] = incl;
  team.sync();
  V before = 0, all = 0;
#pragma unroll
  for (int w = 0; w < kPlanThreads / 32; ++w) {
    const V t = w < team.threads / 32 ? (V)warp_tot[w] : 0;
    if (w < warp) before += t;
    all += t;
  }
  if (team.dry) {      // (its own warp's, so that the trip goes on as with lengths)
    before = 0;
    all = __shfl_sync(0xffffffffu, incl, 31);
  }
  team.sync();
  *total = all;
  return before + incl - v;
}

// Length of sequence b as the kernels may use it: a length beyond what the cache can hold per
// sequence (or a negative one) is recorded as BAD_POSITION and clamped, so that no kernel
// downstream walks into another sequence's rows.  Only `report` threads record.
__device__ __forceinline__ int checked_len(const int32_t* seq_lens, int b, long long max_len, int32_t* status,
                                           bool report) {
  int n = seq_lens[b];
  if (n < 0 || n > max_len) {
    if (report && status) ekv_record(status, ELITEKV_ERR_BAD_POSITION, b, n);
    n = n < 0 ? 0 : (int)max_len;
  }
  return n;
}

struct PlanArgs {
  const int32_t* seq_lens;
  int B, tile, n_workers;      // n_workers 0: the even plan
  int max_items;
  int32_t* items;
  int32_t* seq_first;
  int32_t* worker_first;
  int32_t* zero_ints;          // cleared beside the plan (the combine's arrival counters)
  int n_zero;
  long long max_len;           // tokens one sequence can hold: longer (or negative) lengths are recorded and clamped
  int32_t* status;
  int overhead;
  int4* worker_rec;            // balanced plans, optional: [n_workers][2], what worker_first and items say of a worker's
                               // first item in one place: first item, end of the items, sequence, first token | token count
};
// B lengths of up to max_len tokens make less than 2^31 tiles, and the tile that holds the last token ends below 2^31
inline bool plan_narrow(int B, int tile, long long max_len, int overhead) {
  return max_len + tile <= 0x7fffffffLL && (max_len / tile + 1 + overhead) * B <= 0x7fffffffLL;
}
inline bool plan_narrow(const PlanArgs& a) { return plan_narrow(a.B, a.tile, a.max_len, a.overhead); }

// 32-bit division where the operands allow it (a 64-bit one is a subroutine of over 100 instructions)
__device__ __forceinline__ long long plan_div(long long x, long long y) {
  return ((unsigned long long)(x | y) >> 32) == 0 ? (long long)((unsigned)x / (unsigned)y) : x / y;
}
template <class T>
__device__ __forceinline__ T plan_tiles(int n, int tile) {
  return sizeof(T) == 8 ? (T)plan_div((long long)n + tile - 1, tile) : ((T)n + tile - 1) / tile;
}

// One copy of the division for all its uses: see plan_quick
static __device__ __noinline__ unsigned plan_udiv(unsigned x, unsigned y) { return x / y; }

// Balanced plan of up to 32 sequences, a lane per sequence: every warp has the whole batch in its registers, so there
// is no barrier and no shared memory.  A form with the uses of a search and of an item unrolled and inlined one by one
// took 10 us cold, 2 us when it ran a second time at once.  So there is one copy of each here, items and workers are chunks
// of one loop: 2.8 us behind the wait for one sequence, 3.0 for 16.  (The even plan has hundreds of items, for which
// a warp per 32 is the slower way: the smallest model's step 15.9 us, 14.6 with plan_small.)
// False, with nothing but the counters and reports written, where a product does not fit 32 bits.
// The arithmetic is that of plan_balanced below.
__device__ __forceinline__ bool plan_quick_ok(const PlanArgs& a) { return a.n_workers > 0 && a.B <= 32; }
__device__ __forceinline__ bool plan_quick(const PlanArgs& a, bool dry) {
  constexpr unsigned kAll = 0xffffffffu;
  const int t = threadIdx.x, lane = t & 31, B = a.B;
  const unsigned overhead = a.overhead;
  int n = 0;
  if (dry) n = lane < B ? a.tile : 0;
  else if (lane < B) n = checked_len(a.seq_lens, lane, a.max_len, a.status, t < 32);
  if (!dry)
    for (int i = t; i < a.n_zero; i += kPlanWorkers) a.zero_ints[i] = 0;
  const unsigned tiles = n > 0 ? plan_udiv((unsigned)n + a.tile - 1, (unsigned)a.tile) + overhead : 0;
  // inclusive sums
  unsigned g1 = 0, pieces = 0, w0 = 0, f1 = 0, total = 1, nw = 1;
#pragma unroll 1
  for (int pass = 0; pass < 2; ++pass) {
    unsigned v = pass ? pieces : tiles;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const unsigned x = __shfl_up_sync(kAll, v, o);
      if (lane >= o) v += x;
    }
    if (pass) {
      f1 = v;
      break;
    }
    g1 = v;
    total = max(__shfl_sync(kAll, v, 31), 1u);
    if (total >= plan_udiv(kAll, (unsigned)a.n_workers)) return false;
    nw = min(total, (unsigned)a.n_workers);
    w0 = plan_udiv((g1 - tiles + overhead + 1) * nw - 1, total);
    const unsigned last = plan_udiv(g1 * nw - 1, total);
    if (tiles > 0) pieces = last - w0 + 1;
  }
  const unsigned g0 = g1 - tiles, first = f1 - pieces;
  const int n_items = (int)__shfl_sync(kAll, f1, 31);
  if (!dry && t <= B) a.seq_first[t] = t < B ? (int)first : n_items;
  // chunks of 32 items, then of 31 workers (and the one behind them, whose first item ends the last one's)
  const int item_chunks = (a.max_items + 31) / 32, chunks = item_chunks + (a.n_workers + 31) / 31;
#pragma unroll 1
  for (int c = dry ? 0 : t >> 5; c < chunks; c += dry ? chunks : kPlanWorkers / 32) {
    const bool wk = c >= item_chunks;
    const unsigned i = wk ? (c - item_chunks) * 31 + lane : c * 32 + lane;
    // the sequence of item i, or of the first position of worker i's range: the last one whose first item (first
    // position) is not past it; an empty sequence has that of the one behind it
    const unsigned key = wk ? g0 : first, x = wk ? plan_udiv(min(i, nw) * total, nw) : i;
    int s = 0;
#pragma unroll 1
    for (int o = 16; o > 0; o >>= 1) {
      const unsigned k = __shfl_sync(kAll, key, s + o);      // (s + o <= 31)
      if (s + o < B && k <= x) s += o;
    }
    const unsigned g = __shfl_sync(kAll, g0, s), tl = __shfl_sync(kAll, tiles, s), sw = __shfl_sync(kAll, w0, s);
    const unsigned len = (unsigned)__shfl_sync(kAll, n, s), f = __shfl_sync(kAll, first, s);
    const unsigned j = wk ? (i > sw ? i - sw : 0) : i - f, w = sw + j, base = g + overhead;
    const unsigned ta = max(base, plan_udiv(w * total, nw)) - base, tb = min(g + tl, plan_udiv((w + 1) * total, nw)) - base;
    const int tok0 = (int)(ta * a.tile), ntok = (int)min(tb * a.tile, len) - tok0;
    const int lo = i < nw ? (int)(f + j) : n_items, hi = __shfl_down_sync(kAll, lo, 1);
    if (dry) continue;
    if (!wk) {
      if (i < (unsigned)a.max_items) *(int4*)(a.items + 4 * i) = (int)i < n_items ? make_int4(s, tok0, ntok, (int)w) : make_int4(-1, 0, 0, 0);
    } else if (lane < 31 && (int)i <= a.n_workers) {
      a.worker_first[i] = lo;
      if (a.worker_rec && (int)i < a.n_workers) {
        a.worker_rec[2 * i] = make_int4(lo, hi, s, tok0);
        a.worker_rec[2 * i + 1] = make_int4(ntok, 0, 0, 0);
      }
    }
  }
  return true;
}

// Batches of at most a sequence per thread: both plans in one trip for the lengths, two scans and one
// pass with a thread per ITEM.  (A thread per sequence that writes the sequence's items one after the
// other, two 64-bit divisions each, took twice as long as the query preparation beside it; this form, cold and without
// the warming trip, 4.0 us for one sequence in 33 items and 5.0 for 16.)  The arithmetic is
// that of plan_even and plan_balanced below.
__device__ __forceinline__ bool plan_small_ok(const PlanArgs& a) {
  return a.B <= kPlanThreads && a.n_workers + a.B <= kPlanStage;
}
template <class T>
__device__ __forceinline__ void plan_small(const PlanArgs& a, PlanShared<T>& sh, const PlanTeam team) {
  const bool dry = team.dry;      // nothing is written, shared memory neither: what a dry trip reads there is anybody's
  T *const warp_tot = sh.warp_tot, *const s_g0 = sh.g0, *const s_tiles = sh.tiles;
  int *const s_first = sh.first, *const s_len = sh.len;
  short *const s_w0 = sh.w0, *const s_wk = sh.wk;
  const int t = dry ? threadIdx.x % 32 : threadIdx.x, B = a.B;
  const bool balanced = a.n_workers > 0;
  const int overhead = balanced ? a.overhead : 0;      // empty tiles in front of every sequence
  int n = 0;
  if (dry) n = t < B ? a.tile : 0;
  else if (t < B) n = checked_len(a.seq_lens, t, a.max_len, a.status, true);
  if (!dry)
    for (int i = t; i < a.n_zero; i += team.threads) a.zero_ints[i] = 0;
  const T tiles = n > 0 ? (T)plan_div((long long)n + a.tile - 1, a.tile) + overhead : 0;
  T sum;
  const T g0 = block_exclusive_scan(team, tiles, warp_tot, &sum);
  const long long total = sum > 0 ? sum : 1;
  const long long nw = balanced ? (total < a.n_workers ? total : a.n_workers) : 1;
  auto bound = [&](long long w) -> long long { return plan_div(w * total, nw); };
  auto owner = [&](long long g) -> int { return (int)plan_div((g + 1) * nw - 1, total); };
  int pieces = 0, w0 = 0;
  if (tiles > 0) {
    if (balanced) {
      w0 = owner(g0 + overhead);
      pieces = owner((long long)g0 + tiles - 1) - w0 + 1;
    } else {
      const long long budget = a.max_items - B > 0 ? a.max_items - B : 1;
      const long long target = plan_div(total + budget - 1, budget);
      pieces = (int)plan_div(tiles + target - 1, target);
    }
  }
  int n_items;
  const int first = block_exclusive_scan(team, pieces, warp_tot, &n_items);
  if (t < B && !dry) {
    a.seq_first[t] = first;
    s_first[t] = first; s_g0[t] = g0; s_len[t] = n; s_tiles[t] = tiles; s_w0[t] = (short)w0;
  }
  if (t == 0 && !dry) a.seq_first[B] = n_items;
  team.sync();
  for (int it = t; it < a.max_items; it += dry ? a.max_items : team.threads) {
    int4 item = make_int4(-1, 0, 0, 0);
    if (it < n_items) {
      int lo = 0, hi = B;                    // the last sequence whose first item is not past this one
      while (hi - lo > 1) {
        const int mid = (lo + hi) >> 1;
        if (s_first[mid] <= it) lo = mid; else hi = mid;
      }
      const int j = it - s_first[lo], len = s_len[lo];
      const T tl = s_tiles[lo];
      int ta, tb, w = 0;                     // tiles of the sequence
      if (balanced) {
        const long long base = (long long)s_g0[lo] + overhead;
        w = s_w0[lo] + j;
        ta = (int)(max(base, bound(w)) - base);
        tb = (int)(min((long long)s_g0[lo] + tl, bound(w + 1)) - base);
        if (!dry) s_wk[it] = (short)w;
      } else {
        const int np = (lo + 1 < B ? s_first[lo + 1] : n_items) - s_first[lo];
        ta = (int)plan_div((long long)tl * j, np);
        tb = (int)plan_div((long long)tl * (j + 1), np);
      }
      const int tok0 = ta * a.tile;
      item = make_int4(lo, tok0, (int)min((T)tb * a.tile, (T)len) - tok0, w);
    }
    if (!dry) *(int4*)(a.items + 4 * it) = item;
  }
  if (!balanced) return;
  team.sync();
  const int held = dry ? 1 : min(n_items, a.max_items);
  for (int w = t; w <= a.n_workers; w += dry ? a.n_workers + 1 : team.threads) {
    int lo = 0, hi = held;                   // first item whose worker is >= w
    while (lo < hi) {
      const int mid = (lo + hi) >> 1;
      if (s_wk[mid] < w) lo = mid + 1; else hi = mid;
    }
    if (dry) continue;
    a.worker_first[w] = lo;
    if (a.worker_rec && w < a.n_workers) {
      const bool any = lo < held && s_wk[lo] == w;
      int end = lo;                          // (a worker has few items)
      while (end < held && s_wk[end] == w) ++end;
      const int4 x = any ? *(const int4*)(a.items + 4 * lo) : make_int4(0, 0, 0, 0);
      a.worker_rec[2 * w] = make_int4(lo, end, x.x, x.y);
      a.worker_rec[2 * w + 1] = make_int4(x.z, 0, 0, 0);
    }
  }
}

template <class T>
__device__ __forceinline__ void plan_even(const PlanArgs& a, PlanShared<T>& sh) {
  const int B = a.B, tile = a.tile, max_items = a.max_items, n_zero = a.n_zero;
  int32_t* __restrict__ items = a.items;
  int32_t* __restrict__ seq_first = a.seq_first;
  int32_t* __restrict__ zero_ints = a.zero_ints;
  T* const warp_tot = sh.warp_tot;
  long long& s_total = sh.total;
  const int t = threadIdx.x;
  for (int i = t; i < n_zero; i += blockDim.x) zero_ints[i] = 0;
  if (t == 0) s_total = 0;
  __syncthreads();
  long long local = 0;
  for (int b = t; b < B; b += blockDim.x) {
    int n = checked_len(a.seq_lens, b, a.max_len, a.status, true);
    local += n > 0 ? plan_tiles<T>(n, tile) : 0;
  }
  if (local) atomicAdd((unsigned long long*)&s_total, (unsigned long long)local);
  __syncthreads();
  const long long total = s_total;
  const long long budget = max_items - B > 0 ? max_items - B : 1;
  long long target = (total + budget - 1) / budget;
  if (target < 1) target = 1;

  int carry = 0;
  for (int b0 = 0; b0 < B; b0 += blockDim.x) {
    const int b = b0 + t;
    int n = 0, tiles = 0, pieces = 0;
    if (b < B) {
      n = checked_len(a.seq_lens, b, a.max_len, a.status, false);
      tiles = n > 0 ? (int)plan_tiles<T>(n, tile) : 0;
      pieces = (int)((tiles + target - 1) / target);
    }
    int chunk_total;
    const int first = carry + block_exclusive_scan(PlanTeam{kPlanThreads, false}, pieces, warp_tot, &chunk_total);
    if (b < B) {
      seq_first[b] = first;
      for (int j = 0; j < pieces; ++j) {
        const int ta = (int)((long long)tiles * j / pieces);
        const int tb = (int)((long long)tiles * (j + 1) / pieces);
        const int tok0 = ta * tile;
        const int tok1 = (int)min((T)tb * tile, (T)n);
        const int it = first + j;
        if (it < max_items) *(int4*)(items + 4 * it) = make_int4(b, tok0, tok1 - tok0, 0);
      }
    }
    carry += chunk_total;
  }
  if (t == 0) seq_first[B] = carry;
  for (int it = carry + t; it < max_items; it += blockDim.x) *(int4*)(items + 4 * it) = make_int4(-1, 0, 0, 0);
}

// Balanced plan for kernels whose blocks walk several items: worker w of `n_workers` owns the
// global tile range [w*total/n, (w+1)*total/n), n = min(n_workers, total) (integer division: the
// ranges differ by at most one tile and none is empty); an item is the
// intersection of one worker's range with one sequence.  Items come out in global order, so they
// are grouped by sequence (seq_first) and by worker (worker_first).  items[i] = (sequence, first
// token, token count, worker).
// Starting an item costs a worker about as much as `overhead` tiles (new queries, a partial
// result to write out), and a worker whose range contains the start of a sequence has one item
// more than the others.  The tile list therefore carries `overhead` empty tiles in front of every
// sequence: they take room in a worker's quota and hold no tokens.
template <class T>
__device__ __forceinline__ void plan_balanced(const PlanArgs& a, PlanShared<T>& sh) {
  const int B = a.B, tile = a.tile, n_workers = a.n_workers, max_items = a.max_items, overhead = a.overhead, n_zero = a.n_zero;
  int32_t* __restrict__ items = a.items;
  int32_t* __restrict__ seq_first = a.seq_first;
  int32_t* __restrict__ worker_first = a.worker_first;
  int32_t* __restrict__ zero_ints = a.zero_ints;
  T* const warp_tot = sh.warp_tot;
  long long& s_total = sh.total;
  short* const s_wk = sh.wk;
  const int t = threadIdx.x;
  for (int i = t; i < n_zero; i += blockDim.x) zero_ints[i] = 0;
  if (t == 0) s_total = 0;
  __syncthreads();
  long long local = 0;
  for (int b = t; b < B; b += blockDim.x) {
    int n = checked_len(a.seq_lens, b, a.max_len, a.status, true);
    local += n > 0 ? plan_tiles<T>(n, tile) + overhead : 0;
  }
  if (local) atomicAdd((unsigned long long*)&s_total, (unsigned long long)local);
  __syncthreads();
  const long long total = s_total > 0 ? s_total : 1;
  // first position of worker w's range, and the worker that owns position g
  // (with fewer positions than workers only the first `total` workers get a range, of one each)
  const long long nw = total < n_workers ? total : n_workers;
  auto bound = [&](long long w) -> long long { return w * total / nw; };
  auto owner = [&](long long g) -> int { return (int)(((g + 1) * nw - 1) / total); };
  T carry_tiles = 0;
  int carry_items = 0;
  {
    for (int b0 = 0; b0 < B; b0 += blockDim.x) {
      const int b = b0 + t;
      int n = 0;
      T tiles = 0;
      if (b < B) {
        n = checked_len(a.seq_lens, b, a.max_len, a.status, false);
        tiles = n > 0 ? plan_tiles<T>(n, tile) + overhead : 0;     // with the empty tiles in front
      }
      T chunk_tiles;
      const T g0 = carry_tiles + block_exclusive_scan(PlanTeam{kPlanThreads, false}, tiles, warp_tot, &chunk_tiles);
      int pieces = 0, w0 = 0;
      if (tiles > 0) {
        w0 = owner(g0 + overhead);                                // workers that hold real tiles
        const int w1 = owner(g0 + tiles - 1);
        pieces = w1 - w0 + 1;
      }
      int chunk_items;
      const int first = carry_items + block_exclusive_scan(PlanTeam{kPlanThreads, false}, pieces, warp_tot, &chunk_items);
      if (b < B) {
        seq_first[b] = first;
        for (int j = 0; j < pieces; ++j) {
          const long long ga = max((long long)g0 + overhead, bound(w0 + j));
          const long long gb = min((long long)g0 + tiles, bound(w0 + j + 1));
          const int tok0 = (int)(ga - g0 - overhead) * tile;
          const int tok1 = (int)min((T)(gb - g0 - overhead) * tile, (T)n);
          const int it = first + j;
          if (it < max_items) *(int4*)(items + 4 * it) = make_int4(b, tok0, tok1 - tok0, w0 + j);
          if (it < kPlanStage) s_wk[it] = (short)(w0 + j);
        }
      }
      carry_tiles += chunk_tiles;
      carry_items += chunk_items;
    }
  }
  if (t == 0) seq_first[B] = carry_items;
  for (int it = carry_items + t; it < max_items; it += blockDim.x) *(int4*)(items + 4 * it) = make_int4(-1, 0, 0, 0);
  // worker_first[w] = number of items of workers below w (items are ordered by worker; a worker
  // without items gets an empty range).  The worker ids of up to kPlanStage items are kept in
  // shared memory while they are written, so that this is a binary search per worker instead of
  // a second trip to global memory.
  __syncthreads();
  const int n_items = min(carry_items, max_items);
  if (n_items <= kPlanStage) {
    for (int w = t; w <= n_workers; w += blockDim.x) {
      int lo = 0, hi = n_items;              // first item whose worker is >= w
      while (lo < hi) {
        const int mid = (lo + hi) >> 1;
        if (s_wk[mid] < w) lo = mid + 1; else hi = mid;
      }
      worker_first[w] = lo;
    }
  } else {
    for (int w = t; w <= n_workers; w += blockDim.x) worker_first[w] = n_items;
    __syncthreads();
    for (int it = t; it < n_items; it += blockDim.x) {
      const int wk = items[4 * it + 3];
      if (it == 0 || items[4 * (it - 1) + 3] != wk) worker_first[wk] = it;
    }
    __syncthreads();
    if (t == 0)       // unset entries still hold the item count; an entry may not exceed its successor
      for (int w = n_workers - 1; w >= 0; --w)
        if (worker_first[w] > worker_first[w + 1]) worker_first[w] = worker_first[w + 1];
  }
}

template <class T>
__device__ __forceinline__ void plan_large(const PlanArgs& a, PlanShared<T>& sh) {
  if (a.n_workers > 0) plan_balanced(a, sh);
  else plan_even(a, sh);
  if (a.worker_rec) {
    __syncthreads();
    for (int w = threadIdx.x; w < a.n_workers; w += kPlanThreads) {
      const int lo = a.worker_first[w], hi = a.worker_first[w + 1];
      const int4 x = lo < hi ? *(const int4*)(a.items + 4 * lo) : make_int4(0, 0, 0, 0);
      a.worker_rec[2 * w] = make_int4(lo, hi, x.x, x.y);
      a.worker_rec[2 * w + 1] = make_int4(x.z, 0, 0, 0);
    }
  }
}
// A whole plan, with the wait for the kernels before in front of the first trip to memory.  (Where every thread has a
// sequence there is no warp to spare for the dry trip.  A dry trip of the whole block in front of the wait is as
// good behind a running kernel, and 1.5 to 2 us more where there is none: an isolated step of the smallest model 21.7 us,
// 20.3 so; 12 x 900 39.8 and 37.9.  With one 87.5 % 16 x 1500 takes 32.3 us a step back to back, 33.2 so.)
// kAlone: the kernel is nothing but a plan, and triggers behind the wait.  In front of it, attention blocks came to wait on
// SMs that blocks of the query preparation were yet to leave (87.5 % from hidden states, 32 x 8192: 127.2 us, 120.5 now).
template <bool kAlone, class T>
__device__ __forceinline__ void plan_behind_wait(const PlanArgs& a, PlanShared<T>& sh) {
  const bool spare = plan_small_ok(a) && a.B <= kPlanWorkers, dry = spare && threadIdx.x >= kPlanWorkers;
  if (!dry) {
    ekv_pdl_wait();
    if (kAlone) ekv_pdl_trigger();
  }
  if (sizeof(T) == 4 && plan_quick_ok(a) && spare) {
    const bool done = plan_quick(a, dry);
    if (done || dry) return;
  }
  if (plan_small_ok(a)) {
    plan_small(a, sh, PlanTeam{dry ? 32 : spare ? kPlanWorkers : kPlanThreads, dry});
    return;
  }
  plan_large(a, sh);
}
