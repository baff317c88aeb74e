// Batched group-by and join: thousands of uneven instances in two persistent
// launches instead of several launches (and host round trips) per instance.
//
// Most of the paper's kernel time at small scale factors sits in launches
// too small to fill the GPU (Sec. 5.3).  Here every instance is cut into
// tiles of blockDim x ITEMS rows; each CTA of a persistent grid (sized to the
// resident capacity) takes the next work item (a group-by's tiles by 32, a
// join's probe tiles by up to 8) from one atomic work counter, finds its
// instance in the items' prefix sums, split 32 ways a round by a warp, and
// processes it.  Launch A: join builds and group-by aggregation (independent).  Launch
// B: join probes (after every build) and group-by compaction (after every
// aggregation).  The caller zeroes the counters and tables before A, so one
// batch is one memset plus two launches, which a CUDA graph replays.
//
// Tables follow the single-instance kernels: open addressing on stored keys
// key ^ 2^63 (0 = empty, INT64_MIN on a side path), zero-identity aggregate
// words, bounded probing with an overflow flag per instance, from the key's
// home sector of four slots.  A thread probes alone (W = 1: one sector a load)
// or W = 2, 4 or 8 threads together, each reading one slot of a W-slot window.
// Group-by instances whose groups fit pre-aggregate each work item in a
// shared-memory table (smtab.cuh) and merge it into the global table.
#include <cooperative_groups.h>

#include <type_traits>

#include "batch.cuh"
#include "smtab.cuh"

namespace cg = cooperative_groups;

namespace rel {

namespace {

constexpr int BATCH_SMEM_PROBES = 32;

// Instance of a work item (start[i] <= item < start[i + 1]), found by a whole
// warp: every round splits the range 32 ways, so 4096 instances take three
// dependent loads instead of twelve.
__device__ __forceinline__ int find_instance(const long long* start, int n, long long item) {
  const int lane = threadIdx.x & 31;
  int lo = 0, len = n;  // start[lo] <= item < start[lo + len]
  while (len > 1) {
    const int step = (len + 31) >> 5;
    const int at = lo + lane * step;
    const bool le = lane * step < len && __ldg(start + at) <= item;
    const int k = 31 - __clz(__ballot_sync(0xffffffffu, le));  // lane 0 always votes
    lo += k * step;
    len = len - k * step < step ? len - k * step : step;
  }
  return lo;
}

// The next work item of a launch (warp 0): total items, the first `split` of
// which belong to `first`, the rest to `second`; *inst < 0 when none is left.
__device__ __forceinline__ void next_item(unsigned long long* ctr, long long total, long long split,
                                          const long long* first, int n_first,
                                          const long long* second, int n_second,
                                          long long* item, int* inst) {
  unsigned long long t = 0;
  if ((threadIdx.x & 31) == 0) t = atomicAdd(ctr, 1ull);
  const long long x = (long long)__shfl_sync(0xffffffffu, t, 0);
  const int i = x >= total  ? -1
                : x < split ? find_instance(first, n_first, x)
                            : find_instance(second, n_second, x - split);
  if ((threadIdx.x & 31) == 0) {
    *item = x;
    *inst = i;
  }
}

__device__ __forceinline__ uint64_t encode_word(int op, int64_t v) {
  return op == REL_COUNT ? 1ull
         : op == REL_MIN ? (uint64_t)v ^ MIN_FLIP
         : op == REL_MAX ? (uint64_t)v ^ MAX_FLIP
                         : (uint64_t)v;
}

__device__ __forceinline__ void red_global(unsigned long long* w, int op, uint64_t x) {
  if (op == REL_MIN || op == REL_MAX)
    redg_max(w, x);
  else
    redg_add(w, x);
}

// The encoded words of one row (or of a pre-aggregated slot) for aggregate a.
struct Words {
  uint64_t w[BATCH_MAX_AGGS];
};

__device__ __forceinline__ Words row_words(const BatchGb& g, int64_t v) {
  Words x;
#pragma unroll
  for (int a = 0; a < BATCH_MAX_AGGS; ++a) x.w[a] = a < g.n_aggs ? encode_word(g.ops[a], v) : 0;
  return x;
}

__device__ __forceinline__ void red_words(const BatchGb& g, unsigned long long* t, const Words& x) {
#pragma unroll
  for (int a = 0; a < BATCH_MAX_AGGS; ++a)
    if (a < g.n_aggs) red_global(t + a, g.ops[a], x.w[a]);
}

__device__ __forceinline__ void side_update(const BatchGb& g, BatchStatus* st, const Words& x) {
  atomicAdd(&st->n_side, 1ull);
  red_words(g, st->side_aggs, x);
}

// Global tables are walked from the first slot of the key's home sector (four
// keys, 32 bytes): one 256-bit load shows four slots for the price of one, so
// at half load 96 of 100 rows end at their first load.
__device__ __forceinline__ uint64_t home_slot(const BatchGb& g, uint64_t ek) {
  return home_sector(ek, g.log2_slots);
}
// Slot of ek at or after slot s (the first of a sector), claiming the first
// empty one; ~0 when the table overflowed.  Out of line: the rare path.
__device__ __noinline__ uint64_t global_claim(const BatchGb& g, BatchStatus* st, uint64_t ek,
                                              uint64_t s) {
  const uint64_t mask = (1ull << g.log2_slots) - 1;
  for (uint32_t i = 0; i < g.max_probe; i += 4) {
    uint64_t k[4];
    ld_sector(g.tkeys + s, k);
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (k[q] == 0) {
        k[q] = atomicCAS((unsigned long long*)(g.tkeys + s + q), 0ull, (unsigned long long)ek);
        if (k[q] == 0) k[q] = ek;
      }
      if (k[q] == ek) return s + q;
    }
    s = (s + 4) & mask;
    if ((i & 31) == 28 && ld_relaxed_u32(&st->overflow)) return ~0ull;  // already overflowed
  }
  atomicOr(&st->overflow, 1u);
  return ~0ull;
}

__device__ __forceinline__ void global_update(const BatchGb& g, BatchStatus* st, uint64_t ek,
                                              const Words& x) {
  const uint64_t s = global_claim(g, st, ek, home_slot(g, ek));
  if (s != ~0ull) red_words(g, g.taggs + s * (uint64_t)g.n_aggs, x);
}

// A row outside the fast paths, out of line: INT64_MIN to the side
// accumulator, any other key to the global table.
__device__ __noinline__ void rare_row(const BatchGb& g, BatchStatus* st, uint64_t ek, uint64_t v) {
  const Words x = row_words(g, (int64_t)v);
  if (ek == 0)
    side_update(g, st, x);
  else
    global_update(g, st, ek, x);
}

// W threads probe together: each reads one slot of a W-slot window; a key
// found anywhere in the window is updated, else the lowest empty slot is
// claimed.  Slots are never freed, so every inserter of a key meets the same
// first window with room and finds the key there.  (ek, v, valid) is the
// calling thread's row; the group serves its W rows one after another.
template <int W>
__device__ __noinline__ void global_update_coop(const BatchGb& g, BatchStatus* st, uint64_t ek,
                                                int64_t v, bool valid) {
  const auto tile = cg::tiled_partition<W>(cg::this_thread_block());
  const uint64_t mask = (1ull << g.log2_slots) - 1;
  const int rank = (int)tile.thread_rank();
  for (int r = 0; r < W; ++r) {
    const uint64_t k = tile.shfl(ek, r);
    const int64_t vr = tile.shfl(v, r);
    if (!tile.shfl((int)valid, r)) continue;
    const Words x = row_words(g, vr);
    if (k == 0) {
      if (rank == 0) side_update(g, st, x);
      continue;
    }
    const uint64_t base = home_slot(g, k);
    bool done = false;
    for (uint32_t i = 0; i < g.max_probe && !done; i += W) {
      if ((i & 31) == 32 - W && tile.any(ld_relaxed_u32(&st->overflow) != 0)) {
        done = true;  // already overflowed: the result is discarded
        break;
      }
      const uint64_t s = (base + i + rank) & mask;
      const uint64_t cur = ld_relaxed(g.tkeys + s);
      const unsigned hit = tile.ballot(cur == k);
      if (hit) {
        if (rank == __ffs(hit) - 1) red_words(g, g.taggs + s * (uint64_t)g.n_aggs, x);
        done = true;
        break;
      }
      unsigned emp = tile.ballot(cur == 0);
      while (emp) {
        const int leader = __ffs(emp) - 1;
        unsigned long long res = 0;
        if (rank == leader) {
          res = atomicCAS((unsigned long long*)(g.tkeys + s), 0ull, (unsigned long long)k);
          if (res == 0 || res == k) red_words(g, g.taggs + s * (uint64_t)g.n_aggs, x);
        }
        res = tile.shfl(res, leader);
        if (res == 0 || res == k) {
          done = true;
          break;
        }
        emp &= ~(1u << leader);
      }
    }
    if (!done && rank == 0) atomicOr(&st->overflow, 1u);
  }
}

// Rows base + j / 2 * 2 * B + 2 * tid + {0, 1} (j < U) below end; ek = 0 where
// there is none.  vec: both columns allow two rows per load.
template <class KT, int U>
__device__ __forceinline__ uint32_t load_rows(const BatchGb& g, bool vec, long long base,
                                              long long end, uint64_t (&ek)[U], uint64_t (&v)[U]) {
  const KT* keys = (const KT*)g.keys;
  const int B = blockDim.x;
  if (vec && base + (long long)B * U <= end) {
#pragma unroll
    for (int j = 0; j < U; j += 2) {
      const long long r = base + (long long)j * B + 2 * threadIdx.x;
      if constexpr (sizeof(KT) == 8) {
        const longlong2 k = __ldcs((const longlong2*)(keys + r));
        ek[j] = (uint64_t)k.x ^ KEY_FLIP;
        ek[j + 1] = (uint64_t)k.y ^ KEY_FLIP;
      } else {
        const int2 k = __ldcs((const int2*)(keys + r));
        ek[j] = (uint64_t)(int64_t)k.x ^ KEY_FLIP;
        ek[j + 1] = (uint64_t)(int64_t)k.y ^ KEY_FLIP;
      }
      const longlong2 x = __ldcs((const longlong2*)(g.vals + r));
      v[j] = (uint64_t)x.x;
      v[j + 1] = (uint64_t)x.y;
    }
    return (1u << U) - 1;
  }
  uint32_t ok = 0;
#pragma unroll
  for (int j = 0; j < U; ++j) {
    const long long r = base + (long long)(j / 2) * 2 * B + 2 * threadIdx.x + (j & 1);
    const bool in = r < end;
    ek[j] = in ? (uint64_t)(int64_t)__ldcs(keys + r) ^ KEY_FLIP : 0;
    v[j] = in && g.vals ? (uint64_t)__ldcs((const long long*)g.vals + r) : 0;
    ok |= (in ? 1u : 0u) << j;
  }
  return ok;
}

// Rows into the CTA's shared-memory table (smtab.cuh), cleared before and
// merged into the instance's global table after: one update per distinct key
// of the work item.
template <class KT, int NA>
__device__ __noinline__ void shared_rows(const BatchGb& g, BatchStatus* st, long long r0,
                                            long long r1, uint8_t* sm) {
  constexpr int U = NA == 4 ? 2 : 4;  // rows per thread in flight (registers)
  SmTab<NA> t;
  t.bind(sm, (uint32_t)g.smem_slots);
  t.clear();
  const bool vec = g.vals && (uintptr_t)g.keys % (2 * sizeof(KT)) == 0 && (uintptr_t)g.vals % 16 == 0;
  const long long step = (long long)blockDim.x * U;
  uint64_t ek[U], v[U];
  uint32_t ok = load_rows<KT, U>(g, vec, r0, r1, ek, v);
  __syncthreads();
  for (; r0 < r1; r0 += step) {
    uint64_t nek[U], nv[U];
    const uint32_t nok = load_rows<KT, U>(g, vec, r0 + step, r1, nek, nv);
    uint32_t rare = 0, slot[U];
#pragma unroll
    for (int j = 0; j < U; ++j) rare |= (ek[j] == 0 ? 1u : 0u) << j;
    rare &= ok;
    rare |= t.find(ek, BATCH_SMEM_PROBES, slot);
    if (rare) {
#pragma unroll
      for (int j = 0; j < U; ++j)
        if (rare >> j & 1) rare_row(g, st, ek[j], v[j]);
    }
    __syncwarp();
    t.add(slot, v);
#pragma unroll
    for (int j = 0; j < U; ++j) {
      ek[j] = nek[j];
      v[j] = nv[j];
    }
    ok = nok;
  }
  __syncthreads();
  for (uint32_t s = threadIdx.x; s < (uint32_t)g.smem_slots; s += blockDim.x) {
    const uint64_t k = t.key_of(s);
    if (k == 0) continue;
    uint64_t w[NA];
    t.words(s, w);
    Words x;
#pragma unroll
    for (int a = 0; a < BATCH_MAX_AGGS; ++a) {
      x.w[a] = 0;
      if (a < g.n_aggs) {
        const int op = g.ops[a];
        x.w[a] = op == REL_SUM ? w[0] : w[1];
        if constexpr (NA == 4) x.w[a] = op == REL_MIN ? w[2] : op == REL_MAX ? w[3] : x.w[a];
      }
    }
    global_update(g, st, k, x);
  }
  __syncthreads();
}

// Rows straight into the instance's global table (W = 1): two home sectors in
// flight per thread, then both rows' reductions.  The few rows that leave
// their home sector are finished in a loop of their own, inline: a call there
// would store its caller's registers to local memory for every warp (7 rows in
// 10 have such a lane), which writes through to L2 beside the reductions.
template <class KT>
__device__ __noinline__ void global_rows(const BatchGb& g, BatchStatus* st, long long r0,
                                         long long r1) {
  constexpr int U = 2;
  const bool vec = g.vals && (uintptr_t)g.keys % (2 * sizeof(KT)) == 0 && (uintptr_t)g.vals % 16 == 0;
  const long long step = (long long)blockDim.x * U;
  uint64_t* const tk = g.tkeys;
  unsigned long long* const ta = g.taggs;
  const uint64_t mask = (1ull << g.log2_slots) - 1;
  for (; r0 < r1; r0 += step) {
    uint64_t ek[U], v[U], s[U];
    const uint32_t ok = load_rows<KT, U>(g, vec, r0, r1, ek, v);
    uint32_t miss = 0, put = ok;
    {
      uint64_t k[U][4];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        s[j] = home_slot(g, ek[j]);
        ld_sector(tk + s[j], k[j]);
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const uint64_t e = ek[j];
        const uint32_t at = in_sector(k[j], e);
        if (at == 4) {
          miss |= 1u << j;
          if (k[j][3] != 0) s[j] = (s[j] + 4) & mask;  // the home sector is full
        } else {
          s[j] += at;
        }
        if (e == 0) {  // no row, or INT64_MIN
          if (ok >> j & 1) rare_row(g, st, 0, v[j]);
          put &= ~(1u << j);
        }
      }
    }
    miss &= put;
    for (uint32_t i = 0; miss; i += 4) {
      const bool second = !(miss & 1);
      const uint64_t e = second ? ek[1] : ek[0];
      uint64_t w = second ? s[1] : s[0], k[4];
      ld_sector(tk + w, k);
      uint32_t at = in_sector(k, e);
      if (at == 4 && k[3] == 0) at = claim_in_sector(tk + w, k, e);  // room as loaded
      bool done = at != 4;
      w = done ? w + at : (w + 4) & mask;
      if (!done && ((i & 31) == 28 && ld_relaxed_u32(&st->overflow))) {  // already overflowed
        done = true;
        put &= ~(miss & (0u - miss));
      } else if (!done && i >= 2 * g.max_probe) {
        atomicOr(&st->overflow, 1u);
        done = true;
        put &= ~(miss & (0u - miss));
      }
      if (second) s[1] = w; else s[0] = w;
      if (done) miss &= miss - 1;
    }
    __syncwarp();
#pragma unroll
    for (int j = 0; j < U; ++j)
      if (put >> j & 1) red_words(g, ta + s[j] * (uint64_t)g.n_aggs, row_words(g, (int64_t)v[j]));
  }
}

// Work item t of a group-by: g.span consecutive tiles of B x ITEMS rows.
template <int ITEMS, int W>
__device__ __forceinline__ void gb_tile(const BatchGb& g, BatchStatus* st, long long t,
                                        uint8_t* sm) {
  const int B = blockDim.x;
  const long long rows = (long long)B * ITEMS * g.span;
  const long long r0 = t * rows, r1 = r0 + rows < g.n_rows ? r0 + rows : g.n_rows;
  const bool k32 = g.key_type == REL_I32;
  if (g.smem_slots) {
    bool minmax = false;
    for (int a = 0; a < g.n_aggs; ++a) minmax |= g.ops[a] == REL_MIN || g.ops[a] == REL_MAX;
    if (minmax)
      k32 ? shared_rows<int, 4>(g, st, r0, r1, sm) : shared_rows<long long, 4>(g, st, r0, r1, sm);
    else
      k32 ? shared_rows<int, 2>(g, st, r0, r1, sm) : shared_rows<long long, 2>(g, st, r0, r1, sm);
  } else if (W == 1) {
    k32 ? global_rows<int>(g, st, r0, r1) : global_rows<long long>(g, st, r0, r1);
  } else {
    for (long long r = r0; r < r1; r += B) {
      const long long i = r + threadIdx.x;
      const bool in = i < r1;
      int64_t k = 0, v = 0;
      if (in) {
        k = k32 ? (int64_t)__ldcs((const int*)g.keys + i) : (int64_t)__ldcs((const long long*)g.keys + i);
        if (g.vals) v = (int64_t)__ldcs((const long long*)g.vals + i);
      }
      global_update_coop<W>(g, st, (uint64_t)k ^ KEY_FLIP, v, in);
    }
  }
}

// Build rows into their partition's table: every build row claims the first
// empty slot from its home sector on.  The table is at most half full, so the
// home sector's first slot is tried without a look, BUILD_U rows at a time.
template <int ITEMS>
__device__ __forceinline__ void build_tile(const BatchJoin& J, BatchStatus* st, long long t) {
  constexpr int BUILD_U = 4;
  const int B = blockDim.x;
  const uint64_t mask = (1ull << J.log2_slots) - 1;
  for (int j0 = 0; j0 < ITEMS; j0 += BUILD_U) {
    const long long r0 = t * (long long)B * ITEMS + (long long)j0 * B + threadIdx.x;
    uint64_t ek[BUILD_U], s[BUILD_U];
    JoinVal v[BUILD_U];
    unsigned long long got[BUILD_U];
#pragma unroll
    for (int j = 0; j < BUILD_U; ++j) {
      const long long r = r0 + (long long)j * B;
      const bool in = r < J.n_build;
      ek[j] = in ? (uint64_t)__ldcs((const long long*)J.bkeys + r) ^ KEY_FLIP : 0;
      v[j] = JoinVal{in ? __ldcs((const long long*)J.bpay + r) : 0, (int32_t)r, 0};
      if (in && ek[j] == 0) J.side[atomicAdd(&st->n_side, 1ull)] = v[j];
    }
#pragma unroll
    for (int j = 0; j < BUILD_U; ++j) {
      s[j] = home_sector(ek[j], J.log2_slots);
      got[j] = 1;
      if (ek[j] != 0)
        got[j] = atomicCAS((unsigned long long*)(J.tkeys + s[j]), 0ull, (unsigned long long)ek[j]);
    }
#pragma unroll
    for (int j = 0; j < BUILD_U; ++j) {
      if (ek[j] == 0) continue;
      for (uint32_t i = 0; got[j] != 0 && i < J.max_probe; ++i) {
        s[j] = (s[j] + 1) & mask;
        got[j] = ld_relaxed(J.tkeys + s[j]);
        if (got[j] == 0)
          got[j] = atomicCAS((unsigned long long*)(J.tkeys + s[j]), 0ull, (unsigned long long)ek[j]);
      }
      if (got[j] == 0)
        J.tvals[s[j]] = v[j];
      else
        atomicOr(&st->overflow, 1u);
    }
  }
}

// Persistent launch A: join builds, then group-by tiles, from one counter.
template <int ITEMS, int W>
__global__ void __launch_bounds__(512, 2) batch_a(const __grid_constant__ BatchArgs a) {
  extern __shared__ __align__(16) uint8_t bsm[];
  __shared__ long long s_item;
  __shared__ int s_inst;
  __shared__ union {
    BatchGb g;
    BatchJoin j;
  } s_desc;
  const long long n_build = a.n_j ? a.jb_tiles[a.n_j] : 0;
  const long long total = n_build + (a.n_g ? a.gb_tiles[a.n_g] : 0);
  for (;;) {
    // warp 0 takes the next item and finds its instance; the CTA copies that
    // instance's descriptor into shared memory
    if (threadIdx.x < 32)
      next_item(a.ctr, total, n_build, a.jb_tiles, a.n_j, a.gb_tiles, a.n_g, &s_item, &s_inst);
    __syncthreads();
    const long long item = s_item;
    const int i = s_inst;
    if (i < 0) break;
    const bool is_build = item < n_build;
    {
      const uint4* src = is_build ? (const uint4*)(a.jn + i) : (const uint4*)(a.gb + i);
      const int words = (is_build ? sizeof(BatchJoin) : sizeof(BatchGb)) / sizeof(uint4);
      if ((int)threadIdx.x < words) ((uint4*)&s_desc)[threadIdx.x] = src[threadIdx.x];
    }
    __syncthreads();
    if (is_build) {
      build_tile<ITEMS>(s_desc.j, a.jst + i, item - a.jb_tiles[i]);
    } else {
      gb_tile<ITEMS, W>(s_desc.g, a.gst + i, item - n_build - a.gb_tiles[i], bsm);
    }
    __syncthreads();
  }
}

__device__ __forceinline__ int64_t decode_word(int op, uint64_t w) {
  return op == REL_MIN ? (int64_t)(w ^ MIN_FLIP) : op == REL_MAX ? (int64_t)(w ^ MAX_FLIP) : (int64_t)w;
}

// Compaction of a tile of slots: a thread's ITEMS keys are read together and a
// warp takes one output claim for all of them.
template <int ITEMS>
__device__ __forceinline__ void compact_tile(const BatchGb& g, BatchStatus* st, long long t) {
  const int B = blockDim.x;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const long long slots = 1ll << g.log2_slots;
  const long long s0 = t * (long long)B * ITEMS + threadIdx.x;
  uint64_t k[ITEMS];
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) {
    const long long s = s0 + (long long)j * B;
    k[j] = s < slots ? g.tkeys[s] : 0;
  }
  uint32_t total = 0;
#pragma unroll
  for (int j = 0; j < ITEMS; ++j) total += __popc(__ballot_sync(0xffffffffu, k[j] != 0));
  if (total) {
    unsigned long long wb = 0;
    if (lane == 0) wb = atomicAdd(&st->n_out, (unsigned long long)total);
    wb = __shfl_sync(0xffffffffu, wb, 0);
#pragma unroll
    for (int j = 0; j < ITEMS; ++j) {
      const unsigned m = __ballot_sync(0xffffffffu, k[j] != 0);
      const unsigned long long pos = wb + __popc(m & lt);
      if (k[j] != 0 && pos < (unsigned long long)g.out_capacity) {
        g.out_keys[pos] = (int64_t)(k[j] ^ KEY_FLIP);
        const unsigned long long* w = g.taggs + (uint64_t)(s0 + (long long)j * B) * g.n_aggs;
#pragma unroll
        for (int a = 0; a < BATCH_MAX_AGGS; ++a)
          if (a < g.n_aggs) g.out_aggs[a][pos] = decode_word(g.ops[a], w[a]);
      }
      wb += __popc(m);
    }
  }
  if (t == 0 && threadIdx.x == 0 && st->n_side > 0) {
    const unsigned long long pos = atomicAdd(&st->n_out, 1ull);
    if (pos < (unsigned long long)g.out_capacity) {
      g.out_keys[pos] = INT64_MIN;
#pragma unroll
      for (int a = 0; a < BATCH_MAX_AGGS; ++a)
        if (a < g.n_aggs) g.out_aggs[a][pos] = decode_word(g.ops[a], st->side_aggs[a]);
    }
  }
}

// Matches of key e in the sector at slot s: bit q for slot s + q.  *last: an
// empty slot ends the key's sequence (slots fill in order).
__device__ __forceinline__ uint32_t match_sector(const uint64_t* tk, uint64_t s, uint64_t e,
                                                 bool* last) {
  uint64_t k[4];
  asm volatile("ld.global.nc.v4.u64 {%0, %1, %2, %3}, [%4];"
               : "=l"(k[0]), "=l"(k[1]), "=l"(k[2]), "=l"(k[3])
               : "l"(tk + s));
  *last = k[3] == 0;
  return (k[0] == e ? 1u : 0u) | (k[1] == e ? 2u : 0u) | (k[2] == e ? 4u : 0u) | (k[3] == e ? 8u : 0u);
}

// Probe rows [r0, r1): PROBE_U rows per thread have their home sectors and
// first matches in flight together, and a warp's first matches take one output
// claim; a row's further matches (build keys that repeat), sequences that go on
// past the home sector and INT64_MIN rows are finished in a slower loop.
__device__ __forceinline__ void probe_rows(const BatchJoin& J, BatchStatus* st, long long r0,
                                           long long r1) {
  constexpr int PROBE_U = 4;
  const int B = blockDim.x;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const uint64_t mask = (1ull << J.log2_slots) - 1;
  const unsigned long long n_side = st->n_side, cap = (unsigned long long)J.capacity;
  for (; r0 < r1; r0 += (long long)B * PROBE_U) {
    uint64_t ek[PROBE_U], s[PROBE_U];
    uint32_t m[PROBE_U], more = 0, side = 0;
#pragma unroll
    for (int j = 0; j < PROBE_U; ++j) {
      const long long r = r0 + (long long)j * B + threadIdx.x;
      ek[j] = r < r1 ? (uint64_t)__ldcs((const long long*)J.pkeys + r) ^ KEY_FLIP : 0;
      side |= (r < r1 && ek[j] == 0 ? 1u : 0u) << j;
    }
#pragma unroll
    for (int j = 0; j < PROBE_U; ++j) {
      s[j] = home_sector(ek[j], J.log2_slots);
      m[j] = 0;
      bool last = true;
      if (ek[j] != 0) m[j] = match_sector(J.tkeys, s[j], ek[j], &last);
      more |= (last ? 0u : 1u) << j;
    }
    JoinVal v[PROBE_U];
    uint32_t total = 0;
#pragma unroll
    for (int j = 0; j < PROBE_U; ++j) {
      const unsigned h = __ballot_sync(0xffffffffu, m[j] != 0);
      total += __popc(h);
      if (m[j]) v[j] = J.tvals[s[j] + __ffs(m[j]) - 1];
    }
    if (total) {
      unsigned long long wb = 0;
      if (lane == 0) wb = atomicAdd(&st->n_out, (unsigned long long)total);
      wb = __shfl_sync(0xffffffffu, wb, 0);
#pragma unroll
      for (int j = 0; j < PROBE_U; ++j) {
        const unsigned h = __ballot_sync(0xffffffffu, m[j] != 0);
        if (m[j]) {
          const unsigned long long pos = wb + __popc(h & lt);
          if (pos < cap) {
            __stcs(J.o_pi + pos, (int32_t)(r0 + (long long)j * B + threadIdx.x));
            __stcs(J.o_bi + pos, v[j].bidx);
            __stcs((long long*)J.o_pay + pos, (long long)v[j].payload);
          }
          m[j] &= m[j] - 1;
        }
        wb += __popc(h);
      }
    }
#pragma unroll
    for (int j = 0; j < PROBE_U; ++j) {
      const bool sd = side >> j & 1;
      bool go = sd || m[j] != 0 || (more >> j & 1);
      uint64_t w = sd ? 0 : s[j];
      uint32_t mm = m[j], steps = 0;
      bool last = !(more >> j & 1);
      while (__any_sync(0xffffffffu, go)) {
        bool hit = false;
        JoinVal x{0, 0, 0};
        if (go) {
          if (sd) {
            if (w < n_side) {
              x = J.side[w++];
              hit = true;
            }
          } else {
            while (mm == 0 && !last && steps < J.max_probe) {
              w = (w + 4) & mask;
              steps += 4;
              mm = match_sector(J.tkeys, w, ek[j], &last);
            }
            if (mm) {
              x = J.tvals[w + __ffs(mm) - 1];
              mm &= mm - 1;
              hit = true;
            }
          }
          go = hit;
        }
        const unsigned h = __ballot_sync(0xffffffffu, hit);
        if (!h) continue;
        unsigned long long wb = 0;
        if (lane == 0) wb = atomicAdd(&st->n_out, (unsigned long long)__popc(h));
        wb = __shfl_sync(0xffffffffu, wb, 0);
        if (hit) {
          const unsigned long long pos = wb + __popc(h & lt);
          if (pos < cap) {
            J.o_pi[pos] = (int32_t)(r0 + (long long)j * B + threadIdx.x);
            J.o_bi[pos] = x.bidx;
            J.o_pay[pos] = x.payload;
          }
        }
      }
    }
  }
}

// Probe work item t of a join: J.span tiles.
template <int ITEMS>
__device__ __forceinline__ void probe_tile(const BatchJoin& J, BatchStatus* st, long long t) {
  const long long rows = (long long)blockDim.x * ITEMS * J.span;
  const long long r0 = t * rows;
  probe_rows(J, st, r0, r0 + rows < J.n_probe ? r0 + rows : J.n_probe);
}

// Persistent launch B: join probes, then group-by compaction.  Three CTAs per
// SM: both halves wait on L2 round trips (512 group-bys and 64 joins, 512 x 4:
// 812 -> 712 us against two CTAs, in spite of 56 bytes of spills).
template <int ITEMS>
__global__ void __launch_bounds__(512, 3) batch_b(const __grid_constant__ BatchArgs a) {
  __shared__ long long s_item;
  __shared__ int s_inst;
  __shared__ union {
    BatchGb g;
    BatchJoin j;
  } s_desc;
  const long long n_probe = a.n_j ? a.jp_tiles[a.n_j] : 0;
  const long long total = n_probe + (a.n_g ? a.gc_tiles[a.n_g] : 0);
  for (;;) {
    if (threadIdx.x < 32)
      next_item(a.ctr + 1, total, n_probe, a.jp_tiles, a.n_j, a.gc_tiles, a.n_g, &s_item, &s_inst);
    __syncthreads();
    const long long item = s_item;
    const int i = s_inst;
    if (i < 0) break;
    const bool is_probe = item < n_probe;
    {
      const uint4* src = is_probe ? (const uint4*)(a.jn + i) : (const uint4*)(a.gb + i);
      const int words = (is_probe ? sizeof(BatchJoin) : sizeof(BatchGb)) / sizeof(uint4);
      if ((int)threadIdx.x < words) ((uint4*)&s_desc)[threadIdx.x] = src[threadIdx.x];
    }
    __syncthreads();
    if (is_probe)
      probe_tile<ITEMS>(s_desc.j, a.jst + i, item - a.jp_tiles[i]);
    else
      compact_tile<ITEMS>(s_desc.g, a.gst + i, item - n_probe - a.gc_tiles[i]);
    __syncthreads();
  }
}

template <int ITEMS, int W>
rel_status launch_pair(const BatchArgs& a, int block, int smem, int grid_a, int grid_b,
                       cudaStream_t st) {
  relhost::launch_begin(relhost::K_BATCH_A, st);
  batch_a<ITEMS, W><<<grid_a, block, smem, st>>>(a);
  relhost::launch_end(relhost::K_BATCH_A, st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return relhost::cuda_fail(e, "launch(batch A)");
  relhost::launch_begin(relhost::K_BATCH_B, st);
  batch_b<ITEMS><<<grid_b, block, 0, st>>>(a);
  relhost::launch_end(relhost::K_BATCH_B, st);
  e = cudaGetLastError();
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "launch(batch B)");
}

template <int ITEMS, int W>
rel_status occ_pair(int block, int smem, int* pa, int* pb) {
  cudaError_t e = relhost::allow_smem(batch_a<ITEMS, W>);
  if (e != cudaSuccess) return relhost::cuda_fail(e, "cudaFuncSetAttribute(batch)");
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(pa, batch_a<ITEMS, W>, block, smem);
  if (e == cudaSuccess)
    e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(pb, batch_b<ITEMS>, block, 0);
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "occupancy(batch)");
}

template <int ITEMS, class F>
rel_status with_width(int width, F&& f) {
  switch (width) {
    case 1: return f(std::integral_constant<int, ITEMS>{}, std::integral_constant<int, 1>{});
    case 2: return f(std::integral_constant<int, ITEMS>{}, std::integral_constant<int, 2>{});
    case 4: return f(std::integral_constant<int, ITEMS>{}, std::integral_constant<int, 4>{});
    case 8: return f(std::integral_constant<int, ITEMS>{}, std::integral_constant<int, 8>{});
  }
  relhost::set_error("batch: probe width must be 1, 2, 4 or 8");
  return REL_E_INVALID;
}

template <class F>
rel_status with_config(int items, int width, F&& f) {
  switch (items) {
    case 4: return with_width<4>(width, f);
    case 8: return with_width<8>(width, f);
    case 16: return with_width<16>(width, f);
  }
  relhost::set_error("batch: items per thread must be 4, 8 or 16");
  return REL_E_INVALID;
}

}  // namespace

rel_status batch_launch(const BatchArgs& a, int block, int items, int width, int smem_bytes,
                        int grid_a, int grid_b, cudaStream_t st) {
  return with_config(items, width, [&](auto I, auto W) {
    return launch_pair<decltype(I)::value, decltype(W)::value>(a, block, smem_bytes, grid_a,
                                                               grid_b, st);
  });
}

size_t batch_smem_bytes(const BatchGb& g) {
  if (!g.smem_slots) return 0;
  bool minmax = false;
  for (int a = 0; a < g.n_aggs; ++a) minmax |= g.ops[a] == REL_MIN || g.ops[a] == REL_MAX;
  return minmax ? SmTab<4>::bytes((uint32_t)g.smem_slots) : SmTab<2>::bytes((uint32_t)g.smem_slots);
}

rel_status batch_occupancy(int block, int items, int width, int smem_bytes, int* per_sm_a,
                           int* per_sm_b) {
  return with_config(items, width, [&](auto I, auto W) {
    return occ_pair<decltype(I)::value, decltype(W)::value>(block, smem_bytes, per_sm_a, per_sm_b);
  });
}

}  // namespace rel
