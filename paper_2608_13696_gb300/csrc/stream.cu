// Streaming group-by for key/value rows: one int32 or int64 key column, one
// int64 value column, aggregates (sum, count[, min, max]) -- the shapes KV4 /
// KV2 of the fused kernel, without its staging ring.
//
// The paper's group-by kernels are issue-bound (Sec. 5, 7): instructions per
// DRAM sector, not bandwidth, limit them.  The kernels here keep the per-row
// path short.  Rows come straight from HBM in 16-byte vector loads (two rows per
// load and column, several rows per thread in flight, evict-first), with no
// shared-memory staging or barrier on the path.  By what the plan has:
//  * gb_smem_k: a CTA-shared table (smtab.cuh), the global one behind it;
//  * gb_pin_k: pinned hot keys (from the sample sketch) that are all the keys
//    there are, or all the sample had: a one-probe perfect-hash test, then
//    thread-private words in shared memory (one column per thread: no atomics,
//    no bank conflicts);
//  * gb_stream_k: pinned keys and others, whose rows issue their first slot read
//    of the global table before any is resolved, then claim or accumulate with
//    CAS / RED atomics, bounded probing;
//  * gb_glob_k: the global table alone;
//  * gb_ppass_stream_k and gb_part_l2_k: the partitioned plans' passes.
// At the end a CTA folds its own words into the global table, which the
// compaction kernel turns into the output.
#include "groupby.cuh"
#include "smtab.cuh"

namespace rel {

namespace {

constexpr int ST_BLOCK = 128;
constexpr int ST_U = 8;          // rows per thread per chunk (a multiple of 2)
// pinned keys with thread-private accumulators: 32 KB of them per CTA
template <int NA>
constexpr int pin_max() {
  return NA == 4 ? 8 : 16;
}
constexpr int ST_PIN_LIMIT = 16;

template <int NA>
__device__ __forceinline__ void words_of(uint64_t v, uint64_t (&w)[NA]) {
  w[0] = v;
  w[1] = 1;
  if constexpr (NA == 4) {
    w[2] = v ^ MIN_FLIP;
    w[3] = v ^ MAX_FLIP;
  }
}

// word a keeps an unsigned max (MIN / MAX) rather than a sum
template <int NA>
__device__ __forceinline__ constexpr bool umax_word(int a) {
  return NA == 4 && a >= 2;
}

template <int NA>
__device__ __forceinline__ void red_global(unsigned long long* t, const uint64_t (&w)[NA]) {
#pragma unroll
  for (int a = 0; a < NA; ++a) {
    if (umax_word<NA>(a))
      redg_max(t + a, w[a]);
    else
      redg_add(t + a, w[a]);
  }
}

// Claim-or-accumulate from a first slot whose content k is already loaded.
template <int NA>
__device__ __forceinline__ void global_resolve(const GbParams& p, uint64_t ek, uint64_t s,
                                               uint64_t k, const uint64_t (&w)[NA]) {
  const uint64_t mask = (1ull << p.log2_slots) - 1;
  for (uint32_t i = 0; i < p.max_probe; ++i) {
    if (k == 0) {
      k = atomicCAS((unsigned long long*)(p.tkeys + s), 0ull, (unsigned long long)ek);
      if (k == 0) k = ek;
    }
    if (k == ek) {
      red_global<NA>(p.taggs + s * (uint64_t)NA, w);
      return;
    }
    s = (s + 1) & mask;
    if ((i & 31) == 31 && ld_relaxed_u32(&p.hdr->overflow)) return;  // already overflowed
    k = __ldcg((const unsigned long long*)(p.tkeys + s));
  }
  atomicOr(&p.hdr->overflow, 1u);
}

template <int NA>
__device__ __forceinline__ void global_update(const GbParams& p, uint64_t ek,
                                              const uint64_t (&w)[NA]) {
  const uint64_t s = slot_of(ek, p.log2_slots);
  global_resolve<NA>(p, ek, s, __ldcg((const unsigned long long*)(p.tkeys + s)), w);
}

template <class KT>
struct KeyPair;
template <>
struct KeyPair<int64_t> {
  using V = longlong2;
  __device__ __forceinline__ static void split(const V& v, int64_t& a, int64_t& b) {
    a = v.x;
    b = v.y;
  }
};
template <>
struct KeyPair<int32_t> {
  using V = int2;
  __device__ __forceinline__ static void split(const V& v, int64_t& a, int64_t& b) {
    a = v.x;
    b = v.y;
  }
};

template <class KT, int NA>
__global__ void __launch_bounds__(ST_BLOCK, 6) gb_stream_k(const __grid_constant__ GbParams p) {
  extern __shared__ __align__(16) uint8_t sm[];
  // [pinned keys by slot: 32 x 8 B][dense id by slot: 32 B][key by dense id:
  //  16 x 8 B][CTA sums: 16 x 4 x 8 B][thread-private words: PM x NA x
  //  ST_BLOCK x 8 B]
  constexpr int PM = pin_max<NA>();
  uint64_t* pk = (uint64_t*)sm;
  uint8_t* dense = sm + 256;
  uint64_t* pkd = (uint64_t*)(sm + 288);
  unsigned long long* csum = (unsigned long long*)(sm + 416);
  uint64_t* acc = (uint64_t*)(sm + 416 + 8 * ST_PIN_LIMIT * 4);
  const int tid = threadIdx.x;
  const uint32_t tmask = p.tiny_slots - 1;

  {
    if (tid < 32) {
      const uint64_t k = tid < (int)p.tiny_slots ? p.tiny_init[tid] : 0;
      pk[tid] = k;
      const unsigned occ = __ballot_sync(0xffffffffu, k != 0);
      const int d = __popc(occ & ((1u << tid) - 1u));
      dense[tid] = (uint8_t)d;
      if (k != 0 && d < PM) pkd[d] = k;
    }
    for (int i = tid; i < PM * NA * ST_BLOCK; i += ST_BLOCK) acc[i] = 0;
    for (int i = tid; i < PM * NA; i += ST_BLOCK) csum[i] = 0;
  }
  __syncthreads();

  const KT* keys = (const KT*)p.col[p.key_col[0]];
  const int64_t* vals = (const int64_t*)p.col[p.r_a];
  const int64_t n = p.n_rows;
  constexpr int64_t CHUNK = (int64_t)ST_BLOCK * ST_U;
  const bool vec = ((uintptr_t)keys % (2 * sizeof(KT)) == 0) && ((uintptr_t)vals % 16 == 0);

  for (int64_t base = (int64_t)blockIdx.x * CHUNK; base < n; base += (int64_t)gridDim.x * CHUNK) {
    uint64_t ek[ST_U];
    uint64_t val[ST_U];
    bool ok[ST_U];
    // rows base + j * 2 * ST_BLOCK + 2 * tid + {0, 1}: 32 lanes cover a
    // contiguous 2 x 32-row stretch of every column per load
    if (vec && base + CHUNK <= n) {
#pragma unroll
      for (int j = 0; j < ST_U / 2; ++j) {
        const int64_t r = base + (int64_t)j * 2 * ST_BLOCK + 2 * tid;
        const typename KeyPair<KT>::V kv = __ldcs((const typename KeyPair<KT>::V*)(keys + r));
        const longlong2 vv = __ldcs((const longlong2*)(vals + r));
        int64_t k0, k1;
        KeyPair<KT>::split(kv, k0, k1);
        ek[2 * j] = (uint64_t)k0 ^ KEY_FLIP;
        ek[2 * j + 1] = (uint64_t)k1 ^ KEY_FLIP;
        val[2 * j] = (uint64_t)vv.x;
        val[2 * j + 1] = (uint64_t)vv.y;
        ok[2 * j] = ok[2 * j + 1] = true;
      }
    } else {
#pragma unroll
      for (int j = 0; j < ST_U; ++j) {
        const int64_t r = base + (int64_t)(j / 2) * 2 * ST_BLOCK + 2 * tid + (j & 1);
        ok[j] = r < n;
        ek[j] = ok[j] ? ((uint64_t)(int64_t)keys[r] ^ KEY_FLIP) : 0;
        val[j] = ok[j] ? (uint64_t)vals[r] : 0;
      }
    }
    bool need[ST_U];
#pragma unroll
    for (int j = 0; j < ST_U; ++j) {
      need[j] = false;
      if (!ok[j]) continue;
      uint64_t w[NA];
      words_of<NA>(val[j], w);
      {
        const uint32_t s = small_slot_of(ek[j], tmask, p.tiny_mult);
        if (pk[s] == ek[j] && ek[j] != 0) {
          uint64_t* t = acc + (size_t)dense[s] * NA * ST_BLOCK + tid;
#pragma unroll
          for (int a = 0; a < NA; ++a) {
            const uint64_t o = t[a * ST_BLOCK];
            t[a * ST_BLOCK] = umax_word<NA>(a) ? (o > w[a] ? o : w[a]) : o + w[a];
          }
          continue;
        }
      }
      if (ek[j] == 0) {  // INT64_MIN: the side accumulator
        atomicAdd(&p.hdr->n_side, 1ull);
        red_global<NA>(p.hdr->side_aggs, w);
        continue;
      }
      need[j] = true;
    }
    // global table: first slot reads of every remaining row, then resolve
    uint64_t gs[ST_U], gk[ST_U];
#pragma unroll
    for (int j = 0; j < ST_U; ++j) {
      if (!need[j]) continue;
      gs[j] = slot_of(ek[j], p.log2_slots);
      gk[j] = __ldcg((const unsigned long long*)(p.tkeys + gs[j]));
    }
#pragma unroll
    for (int j = 0; j < ST_U; ++j) {
      if (!need[j]) continue;
      uint64_t w[NA];
      words_of<NA>(val[j], w);
      global_resolve<NA>(p, ek[j], gs[j], gk[j], w);
    }
  }

  // fold the thread-private words into the global table
  {
    const int lane = tid & 31;
    for (int d = 0; d < PM; ++d) {
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        uint64_t x = acc[((size_t)d * NA + a) * ST_BLOCK + tid];
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          const uint64_t y = __shfl_xor_sync(0xffffffffu, x, o);
          x = umax_word<NA>(a) ? (x > y ? x : y) : x + y;
        }
        if (lane == 0 && x) {
          if (umax_word<NA>(a))
            atomicMax(csum + d * NA + a, (unsigned long long)x);
          else
            sadd64(csum + d * NA + a, x);
        }
      }
    }
  }
  __syncthreads();
  if (tid < PM && csum[tid * NA + 1] != 0) {  // word 1 counts rows
    uint64_t w[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) w[a] = csum[tid * NA + a];
    global_update<NA>(p, pkd[tid], w);
  }
}

// A row outside the fast path, out of line: INT64_MIN to the side accumulator,
// any other key to the global table.
template <int NA>
__device__ __noinline__ void rare_row(const GbParams& p, uint64_t ek, uint64_t val) {
  uint64_t w[NA];
  words_of<NA>(val, w);
  if (ek == 0) {
    atomicAdd(&p.hdr->n_side, 1ull);
    red_global<NA>(p.hdr->side_aggs, w);
  } else {
    global_update<NA>(p, ek, w);
  }
}

// A CTA's table into the global one (after a barrier behind the adds).
template <int NA>
__device__ __forceinline__ void merge_table(const GbParams& p, const SmTab<NA>& t) {
  for (uint32_t s = threadIdx.x; s < t.slots; s += blockDim.x) {
    const uint64_t k = t.key_of(s);
    if (k == 0) continue;
    uint64_t w[NA];
    t.words(s, w);
    global_update<NA>(p, k, w);
  }
}

// Rows into one shared-memory table per CTA (a plan with CTA-shared slots),
// merged into the global table at the end; rows the table has no room for go
// to the global table one by one.  Pinned and thread-private slots of the plan
// are not used (but see PIN_TABLE_SLOTS): on a hot key the table's adds
// serialise over a warp's lanes (15 ns a warp at worst), less than a second
// lookup costs every row.
constexpr int SG_U = 4;            // rows per thread per chunk
// largest table: the rest of the SM's 256 KB is L1, through which the rows come
// (1e8 rows, 3000 groups:
// 220 KB 1.45 ms, 168 KB 1.20)
constexpr uint32_t SG_MAX_BYTES = 168 * 1024;

template <class KT, int NA>
__global__ void __launch_bounds__(1024, 1) gb_smem_k(const __grid_constant__ GbParams p) {
  extern __shared__ __align__(16) uint8_t sm[];
  SmTab<NA> t;
  t.bind(sm, p.smem_slots);
  t.clear();
  const int tid = threadIdx.x, B = blockDim.x;
  const KT* keys = (const KT*)p.col[p.key_col[0]];
  const int64_t* vals = (const int64_t*)p.col[p.r_a];
  const int64_t n = p.n_rows;
  const int64_t CHUNK = (int64_t)B * SG_U, step = (int64_t)gridDim.x * CHUNK;
  const bool vec = ((uintptr_t)keys % (2 * sizeof(KT)) == 0) && ((uintptr_t)vals % 16 == 0);
  // rows base + j * 2 * B + 2 * tid + {0, 1}; the next chunk's loads go out
  // before this chunk is worked on
  auto load = [&](int64_t base, uint64_t(&ek)[SG_U], uint64_t(&val)[SG_U]) -> uint32_t {
    uint32_t ok = 0;
    if (vec && base + CHUNK <= n) {
#pragma unroll
      for (int j = 0; j < SG_U / 2; ++j) {
        const int64_t r = base + (int64_t)j * 2 * B + 2 * tid;
        int64_t k0, k1;
        KeyPair<KT>::split(__ldcs((const typename KeyPair<KT>::V*)(keys + r)), k0, k1);
        const longlong2 vv = __ldcs((const longlong2*)(vals + r));
        ek[2 * j] = (uint64_t)k0 ^ KEY_FLIP;
        ek[2 * j + 1] = (uint64_t)k1 ^ KEY_FLIP;
        val[2 * j] = (uint64_t)vv.x;
        val[2 * j + 1] = (uint64_t)vv.y;
      }
      return (1u << SG_U) - 1;
    }
#pragma unroll
    for (int j = 0; j < SG_U; ++j) {
      const int64_t r = base + (int64_t)(j / 2) * 2 * B + 2 * tid + (j & 1);
      const bool in = r < n;
      ek[j] = in ? (uint64_t)(int64_t)keys[r] ^ KEY_FLIP : 0;
      val[j] = in ? (uint64_t)vals[r] : 0;
      ok |= (in ? 1u : 0u) << j;
    }
    return ok;
  };
  uint64_t ek[SG_U], val[SG_U];
  uint32_t ok = 0;
  int64_t base = (int64_t)blockIdx.x * CHUNK;
  if (base < n) ok = load(base, ek, val);
  __syncthreads();
  // Warps that begin with 64 rows of one key -- the only one, or runs of rows
  // -- look for the like in every chunk (3e7 rows of one key, sum and count:
  // 146 -> 104 us; four aggregates, runs of 2500 keys 311 -> 220; 3e7 rows
  // without runs, 100 keys: 149, 151).
  bool same = false;
  if (base < n) {
    const uint64_t k = __shfl_sync(0xffffffffu, ek[0], 0);
    same = __all_sync(0xffffffffu, ek[0] == k && ek[1] == k && ok != 0);
  }
  for (; base < n; base += step) {
    uint64_t nek[SG_U], nval[SG_U];
    uint32_t nok = 0;
    if (base + step < n) nok = load(base + step, nek, nval);
    uint32_t rare = 0, slot[SG_U];  // INT64_MIN rows, and those without a slot
#pragma unroll
    for (int j = 0; j < SG_U; ++j) rare |= (ek[j] == 0 ? 1u : 0u) << j;
    rare &= ok;
    rare |= t.find(ek, (int)p.shared_probes, slot);
    if (rare) {
#pragma unroll
      for (int j = 0; j < SG_U; ++j)
        if (rare >> j & 1) rare_row<NA>(p, ek[j], val[j]);
    }
    __syncwarp();
    if (same)
      t.template add_same<SG_U, 2>(slot, val);
    else
      t.add(slot, val);
#pragma unroll
    for (int j = 0; j < SG_U; ++j) {
      ek[j] = nek[j];
      val[j] = nval[j];
    }
    ok = nok;
  }
  __syncthreads();
  merge_table<NA>(p, t);
}

// Every row straight into the global table: a plan without per-CTA slots.
// Bound by L2: per row one sector of four keys, and for MIN and MAX the pair
// read first and raised only when the row improves it, beside the reductions
// of sum and count (four reductions a row: 50 G rows/s at best; a 16-byte load
// and two: 74).  1e8 rows, 20000 groups: 3.22 ms with one-slot probes
// and four reductions, 2.11 ms.
template <class KT, int NA>
__global__ void __launch_bounds__(512, 2) gb_glob_k(const __grid_constant__ GbParams p) {
  constexpr int U = 2;
  const KT* keys = (const KT*)p.col[p.key_col[0]];
  const int64_t* vals = (const int64_t*)p.col[p.r_a];
  const int64_t n = p.n_rows, CHUNK = (int64_t)blockDim.x * U;
  const bool vec = ((uintptr_t)keys % (2 * sizeof(KT)) == 0) && ((uintptr_t)vals % 16 == 0);
  const uint64_t mask = (1ull << p.log2_slots) - 1;
  for (int64_t base = (int64_t)blockIdx.x * CHUNK; base < n; base += (int64_t)gridDim.x * CHUNK) {
    uint64_t ek[U] = {0, 0}, v[U] = {0, 0}, s[U];
    uint32_t put = 0;  // rows to add
    const int64_t r = base + U * threadIdx.x;
    if (vec && r + 1 < n) {
      int64_t k0, k1;
      KeyPair<KT>::split(__ldcs((const typename KeyPair<KT>::V*)(keys + r)), k0, k1);
      const longlong2 vv = __ldcs((const longlong2*)(vals + r));
      ek[0] = (uint64_t)k0 ^ KEY_FLIP;
      ek[1] = (uint64_t)k1 ^ KEY_FLIP;
      v[0] = (uint64_t)vv.x;
      v[1] = (uint64_t)vv.y;
      put = 3;
    } else {
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if (r + j >= n) continue;
        ek[j] = (uint64_t)(int64_t)keys[r + j] ^ KEY_FLIP;
        v[j] = (uint64_t)vals[r + j];
        put |= 1u << j;
      }
    }
    uint32_t miss = 0;
    {
      uint64_t k[U][4];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        s[j] = home_sector(ek[j], p.log2_slots);
        ld_sector(p.tkeys + s[j], k[j]);
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if (!(put >> j & 1)) continue;
        if (ek[j] == 0) {  // INT64_MIN
          rare_row<NA>(p, 0, v[j]);
          put &= ~(1u << j);
          continue;
        }
        const uint32_t at = in_sector(k[j], ek[j]);
        if (at != 4) {
          s[j] += at;
        } else {
          miss |= 1u << j;
          if (k[j][3] != 0) s[j] = (s[j] + 4) & mask;  // the home sector is full
        }
      }
    }
    // the few rows that leave their home sector, or open a group
    for (uint32_t i = 0; miss; i += 4) {
      const bool second = !(miss & 1);
      const uint64_t e = second ? ek[1] : ek[0];
      uint64_t w = second ? s[1] : s[0], k[4];
      ld_sector(p.tkeys + w, k);
      uint32_t at = in_sector(k, e);
      if (at == 4 && k[3] == 0) at = claim_in_sector(p.tkeys + w, k, e);  // room as loaded
      bool done = at != 4;
      w = done ? w + at : (w + 4) & mask;
      if (!done) {
        const bool over = i >= 2 * p.max_probe;
        if (over) atomicOr(&p.hdr->overflow, 1u);
        if (over || ((i & 31) == 28 && ld_relaxed_u32(&p.hdr->overflow))) {  // already overflowed
          done = true;
          put &= ~(miss & (0u - miss));
        }
      }
      if (second) s[1] = w; else s[0] = w;
      if (done) miss &= miss - 1;
    }
    __syncwarp();
    if constexpr (NA == 4) {
      uint64_t mn[U], mx[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        mn[j] = mx[j] = ~0ull;
        if (put >> j & 1)
          asm volatile("ld.relaxed.gpu.global.v2.u64 {%0, %1}, [%2];"
                       : "=l"(mn[j]), "=l"(mx[j])
                       : "l"(p.taggs + s[j] * 4 + 2)
                       : "memory");
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if ((v[j] ^ MIN_FLIP) > mn[j]) redg_max(p.taggs + s[j] * 4 + 2, v[j] ^ MIN_FLIP);
        if ((v[j] ^ MAX_FLIP) > mx[j]) redg_max(p.taggs + s[j] * 4 + 3, v[j] ^ MAX_FLIP);
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j) {
      if (!(put >> j & 1)) continue;
      redg_add(p.taggs + s[j] * NA, v[j]);
      redg_add(p.taggs + s[j] * NA + 1, 1);
    }
  }
}

// Rows of a plan whose groups are all pinned (a handful of keys): thread-private
// words only, updated without atomics, and HBM the bound.  Against gb_stream_k,
// which also carries rows that are not pinned at full speed: words of 28 bytes
// a key instead of 32 with MIN and MAX read as one and written only when
// raised, columns by hash slot instead of a second lookup, one wide CTA per SM.
// 2e8 rows of four keys: 0.742 -> 0.515 ms (6.2 TB/s, 92 % of the copy rate).
constexpr int PK_U = 4;             // rows per thread per chunk
constexpr int PK_MAX_BLOCK = 768;

template <int NA>
__host__ __device__ constexpr uint32_t pk_key_bytes() {  // per key and thread: sum, count, (min, max)
  return NA == 4 ? 28 : 12;
}
constexpr uint32_t PK_HEAD = 8 * TINY_MAX_SLOTS + 8 * TINY_MAX_SLOTS * 4;  // keys, reduced words

// TAB: a shared table takes the rows of other keys, for plans that expect more
// groups than a sketch found keys; without one they go to the global table row
// by row.
template <class KT, int NA, bool TAB>
__global__ void __launch_bounds__(PK_MAX_BLOCK, 1) gb_pin_k(const __grid_constant__ GbParams p) {
  extern __shared__ __align__(16) uint8_t sm[];
  uint64_t* pk = (uint64_t*)sm;  // pinned key of each slot (0: none)
  uint64_t* red = pk + TINY_MAX_SLOTS;
  const uint32_t S = p.tiny_slots, B = blockDim.x, tid = threadIdx.x, tmask = S - 1;
  // [min, max pairs][sums][counts], each [slot][thread]
  const uint32_t mm = smem_u32(sm) + PK_HEAD, sum = mm + (NA == 4 ? 16 * S * B : 0), cnt = sum + 8 * S * B;
  SmTab<NA> t;
  if (TAB) {
    t.bind(sm + PK_HEAD + (size_t)pk_key_bytes<NA>() * S * B, p.smem_slots);
    t.clear();
  }
  if (tid < TINY_MAX_SLOTS) pk[tid] = tid < S ? p.tiny_init[tid] : 0;
  for (uint32_t s = 0; s < S; ++s) {
    if (NA == 4) {
      sts64(mm + 16 * (s * B + tid), 0);
      sts64(mm + 16 * (s * B + tid) + 8, 0);
    }
    sts64(sum + 8 * (s * B + tid), 0);
    sts32(cnt + 4 * (s * B + tid), 0);
  }
  __syncthreads();
  const KT* keys = (const KT*)p.col[p.key_col[0]];
  const int64_t* vals = (const int64_t*)p.col[p.r_a];
  const int64_t n = p.n_rows, CHUNK = (int64_t)B * PK_U, step = (int64_t)gridDim.x * CHUNK;
  const bool vec = ((uintptr_t)keys % (2 * sizeof(KT)) == 0) && ((uintptr_t)vals % 16 == 0);
  auto load = [&](int64_t base, uint64_t(&ek)[PK_U], uint64_t(&val)[PK_U]) -> uint32_t {
    uint32_t ok = 0;
    if (vec && base + CHUNK <= n) {
#pragma unroll
      for (int j = 0; j < PK_U; j += 2) {
        const int64_t r = base + (int64_t)j * B + 2 * tid;
        int64_t k0, k1;
        KeyPair<KT>::split(__ldcs((const typename KeyPair<KT>::V*)(keys + r)), k0, k1);
        const longlong2 vv = __ldcs((const longlong2*)(vals + r));
        ek[j] = (uint64_t)k0 ^ KEY_FLIP;
        ek[j + 1] = (uint64_t)k1 ^ KEY_FLIP;
        val[j] = (uint64_t)vv.x;
        val[j + 1] = (uint64_t)vv.y;
      }
      return (1u << PK_U) - 1;
    }
#pragma unroll
    for (int j = 0; j < PK_U; ++j) {
      const int64_t r = base + (int64_t)(j / 2) * 2 * B + 2 * tid + (j & 1);
      const bool in = r < n;
      ek[j] = in ? (uint64_t)(int64_t)keys[r] ^ KEY_FLIP : 0;
      val[j] = in ? (uint64_t)vals[r] : 0;
      ok |= (in ? 1u : 0u) << j;
    }
    return ok;
  };
  uint64_t ek[PK_U], val[PK_U];
  int64_t base = (int64_t)blockIdx.x * CHUNK;
  uint32_t ok = base < n ? load(base, ek, val) : 0;
  for (; base < n; base += step) {
    uint64_t nek[PK_U], nval[PK_U];
    const uint32_t nok = base + step < n ? load(base + step, nek, nval) : 0;
    uint32_t s[PK_U];
    bool hit[PK_U];
#pragma unroll
    for (int j = 0; j < PK_U; ++j) {
      s[j] = small_slot_of(ek[j], tmask, p.tiny_mult);
      hit[j] = pk[s[j]] == ek[j] && ek[j] != 0;
    }
#pragma unroll
    for (int j = 0; j < PK_U; ++j) {
      if (hit[j]) {
        const uint32_t at = s[j] * B + tid;
        const uint64_t o = lds64(sum + 8 * at);
        const uint32_t c = lds32(cnt + 4 * at);
        if constexpr (NA == 4) {
          uint64_t mn, mx;
          lds128(mm + 16 * at, mn, mx);
          const uint64_t a = val[j] ^ MIN_FLIP, b = val[j] ^ MAX_FLIP;
          if (a > mn) sts64(mm + 16 * at, a);
          if (b > mx) sts64(mm + 16 * at + 8, b);
        }
        sts64(sum + 8 * at, o + val[j]);
        sts32(cnt + 4 * at, c + 1);
      } else if (!TAB && (ok >> j & 1)) {
        rare_row<NA>(p, ek[j], val[j]);
      }
    }
    if constexpr (TAB) {
      bool other = false;
#pragma unroll
      for (int j = 0; j < PK_U; ++j) other |= !hit[j] && (ok >> j & 1);
      if (__any_sync(0xffffffffu, other)) {
        uint64_t e[PK_U];
        uint32_t slot[PK_U], rare = 0;
#pragma unroll
        for (int j = 0; j < PK_U; ++j) {
          e[j] = hit[j] ? 0 : ek[j];
          rare |= (!hit[j] && ek[j] == 0 ? 1u : 0u) << j;  // INT64_MIN
        }
        rare &= ok;
        rare |= t.find(e, (int)p.shared_probes, slot);
        if (rare) {
#pragma unroll
          for (int j = 0; j < PK_U; ++j)
            if (rare >> j & 1) rare_row<NA>(p, ek[j], val[j]);
        }
        __syncwarp();
        t.add(slot, val);
      }
    }
#pragma unroll
    for (int j = 0; j < PK_U; ++j) {
      ek[j] = nek[j];
      val[j] = nval[j];
    }
    ok = nok;
  }
  __syncthreads();
  // one warp per (slot, word): the threads' words folded, then the groups
  const uint32_t warp = tid >> 5, lane = tid & 31;
  for (uint32_t q = warp; q < S * NA; q += B / 32) {
    const uint32_t g = q / NA, a = q % NA;
    uint64_t v = 0;
    for (uint32_t i = lane; i < B; i += 32) {
      const uint32_t at = g * B + i;
      const uint64_t y = a == 0 ? lds64(sum + 8 * at) : a == 1 ? (uint64_t)lds32(cnt + 4 * at)
                                                              : lds64(mm + 16 * at + 8 * (a - 2));
      v = umax_word<NA>(a) ? (v > y ? v : y) : v + y;
    }
#pragma unroll
    for (int o = 16; o; o >>= 1) {
      const uint64_t y = __shfl_xor_sync(0xffffffffu, v, o);
      v = umax_word<NA>(a) ? (v > y ? v : y) : v + y;
    }
    if (lane == 0) red[q] = v;
  }
  __syncthreads();
  if (tid < S && red[tid * NA + 1] != 0) {
    uint64_t w[NA];
#pragma unroll
    for (int a = 0; a < NA; ++a) w[a] = red[tid * NA + a];
    global_update<NA>(p, pk[tid], w);
  }
  if (TAB) merge_table<NA>(p, t);
}

// Partitioned variant, passes 1 and 2, streaming: a CTA counts its rows per
// partition (pass 1); after the scan, pass 2 writes each row as a (key,
// value) record.  Pinned hot keys never become records: pass 2 aggregates
// them in thread-private words and folds them into the spill table.  INT64_MIN
// rows go to the side accumulator in pass 2.
//
// Writing every record to its own partition costs one L2 write transaction
// per 16-byte record (measured: ~3.5 ms for 1.4e8 records, at any partition
// count from 256 to 16384).  So pass 2 sorts each chunk of SP_TILE records
// by level-1 bin (at most 2^PART_L1_BITS bins of consecutive partitions) in
// shared memory, claims each bin's run with one atomic on the bin's cursor
// and writes the runs contiguously; a second pass (gb_part_l2_k) does the
// same for the partitions inside each bin.  Record order inside a partition
// is arbitrary, which the aggregation does not see.
// Two 256-thread CTAs per SM: while one waits at a barrier of its sort, the
// other streams.  The pinned keys' words are laid out as in gb_pin_k (three
// loads and two stores a row, min and max stored only when they change) and
// for the keys there are: 2e8 Zipf(1.1) rows, 8 pinned keys taking a third of
// them, pass 2 with four words 1843 -> 1520 us (four 64-bit words each before,
// 64 KB per CTA whatever the keys), with two words 1417; 2e8 uniform rows,
// none pinned, 1364.  Reads and writes alone are 0.8 ms.
constexpr int SP_BLOCK = 256;
constexpr int SP_MIN_BLOCKS = 2;
constexpr int SP_TILE = SP_BLOCK * ST_U;  // rows of one chunk, records sorted at once
constexpr int SP_BINS = 1 << PART_L1_BITS;
constexpr int SP_BAD = 15;  // wsum[SP_BAD] != 0: a claim overran its bin
static_assert(SP_BLOCK >= SP_BINS, "one thread per level-1 bin");
// shared memory of pass 2 after the pinned words: bin counts, local and
// global bases, bin ends, warp sums, then the tile's records and their bins
constexpr size_t SP_SORT_SMEM = 4 * 4 * SP_BINS + 64 + 16 * SP_TILE + SP_TILE;
constexpr uint32_t SP_HEAD = 416 + 8 * ST_PIN_LIMIT * 4;

template <class KT, int NA, bool PIN, bool SCATTER>
__global__ void __launch_bounds__(SP_BLOCK, SP_MIN_BLOCKS) gb_ppass_stream_k(const __grid_constant__ GbParams p) {
  extern __shared__ __align__(16) uint8_t sm[];
  constexpr int PM = pin_max<NA>();
  uint64_t* pk = (uint64_t*)sm;
  uint8_t* dense = sm + 256;
  uint64_t* pkd = (uint64_t*)(sm + 288);
  unsigned long long* csum = (unsigned long long*)(sm + 416);
  // thread-private words of the pinned keys there are, each [key][thread]:
  // min and max side by side, sums, 32-bit counts
  uint32_t n_hot = 0;
  if (PIN && SCATTER)
    for (uint32_t i = 0; i < p.tiny_slots; ++i) n_hot += p.tiny_init[i] != 0;
  const uint32_t mm = smem_u32(sm) + SP_HEAD, sum = mm + (NA == 4 ? 16 : 0) * SP_BLOCK * n_hot,
                 cnt = sum + 8 * SP_BLOCK * n_hot;
  uint8_t* const rest = sm + SP_HEAD + (size_t)pk_key_bytes<NA>() * SP_BLOCK * n_hot;
  unsigned int* ctr = (unsigned int*)rest;  // pass 1: [P] counts
  // pass 2
  unsigned int* cnt1 = (unsigned int*)rest;
  unsigned int* lb = cnt1 + SP_BINS;
  unsigned int* gb1 = lb + SP_BINS;
  unsigned int* end1 = gb1 + SP_BINS;
  unsigned int* wsum = end1 + SP_BINS;
  PartRec* recbuf = (PartRec*)(wsum + 16);
  uint8_t* slot_bin = (uint8_t*)(recbuf + SP_TILE);
  const int tid = threadIdx.x;
  const uint32_t P = 1u << p.part_bits;
  const uint32_t shift1 = p.part_bits > PART_L1_BITS ? p.part_bits - PART_L1_BITS : 0;
  const uint32_t B1 = P >> shift1;  // level-1 bins
  PartRec* const out1 = shift1 ? p.recs1 : p.recs;
  const uint32_t tmask = p.tiny_slots - 1;
  if (PIN) {
    if (tid < 32) {
      const uint64_t k = tid < (int)p.tiny_slots ? p.tiny_init[tid] : 0;
      pk[tid] = k;
      const unsigned occ = __ballot_sync(0xffffffffu, k != 0);
      const int d = __popc(occ & ((1u << tid) - 1u));
      dense[tid] = (uint8_t)d;
      if (k != 0 && d < PM) pkd[d] = k;
    }
    if (SCATTER) {
      for (uint32_t i = 4 * tid; i < pk_key_bytes<NA>() * SP_BLOCK * n_hot; i += 4 * SP_BLOCK) sts32(mm + i, 0);
      for (int i = tid; i < PM * NA; i += SP_BLOCK) csum[i] = 0;
    }
  }
  if (!SCATTER) {
    for (uint32_t i = tid; i < P; i += SP_BLOCK) ctr[i] = 0;
  } else {
    if (tid < (int)B1) {
      cnt1[tid] = 0;
      end1[tid] = (unsigned int)p.part_start[(tid + 1) << shift1];
    }
    if (tid == 0) wsum[SP_BAD] = 0;
  }
  const int lane = tid & 31, warp = tid >> 5;
  __syncthreads();

  const KT* keys = (const KT*)p.col[p.key_col[0]];
  const int64_t* vals = (const int64_t*)p.col[p.r_a];
  const int64_t n = p.n_rows;
  constexpr int64_t CHUNK = (int64_t)SP_BLOCK * ST_U;
  const bool vec = ((uintptr_t)keys % (2 * sizeof(KT)) == 0) && ((uintptr_t)vals % 16 == 0);
  // rows base + j * 2 * SP_BLOCK + 2 * tid + {0, 1}; the next chunk's loads
  // go out before this chunk is worked on (the pass is bound by load latency)
  auto load = [&](int64_t base, uint64_t(&ek)[ST_U], uint64_t(&val)[ST_U], uint32_t& ok) {
    if (vec && base + CHUNK <= n) {
#pragma unroll
      for (int j = 0; j < ST_U / 2; ++j) {
        const int64_t r = base + (int64_t)j * 2 * SP_BLOCK + 2 * tid;
        int64_t k0, k1;
        KeyPair<KT>::split(__ldcs((const typename KeyPair<KT>::V*)(keys + r)), k0, k1);
        ek[2 * j] = (uint64_t)k0 ^ KEY_FLIP;
        ek[2 * j + 1] = (uint64_t)k1 ^ KEY_FLIP;
        if (SCATTER) {
          const longlong2 vv = __ldcs((const longlong2*)(vals + r));
          val[2 * j] = (uint64_t)vv.x;
          val[2 * j + 1] = (uint64_t)vv.y;
        }
      }
      ok = (1u << ST_U) - 1;
      return;
    }
    ok = 0;
#pragma unroll
    for (int j = 0; j < ST_U; ++j) {
      const int64_t r = base + (int64_t)(j / 2) * 2 * SP_BLOCK + 2 * tid + (j & 1);
      const bool in = r < n;
      ek[j] = in ? ((uint64_t)(int64_t)keys[r] ^ KEY_FLIP) : 0;
      if (SCATTER) val[j] = in ? (uint64_t)vals[r] : 0;
      ok |= (in ? 1u : 0u) << j;
    }
  };
  const int64_t step = (int64_t)gridDim.x * CHUNK;
  uint64_t ek[ST_U], val[ST_U];
  uint32_t okm = 0;
  if ((int64_t)blockIdx.x * CHUNK < n) load((int64_t)blockIdx.x * CHUNK, ek, val, okm);
  for (int64_t base = (int64_t)blockIdx.x * CHUNK; base < n; base += step) {
    uint64_t nek[ST_U], nval[ST_U];
    uint32_t nok = 0;
    if (base + step < n) load(base + step, nek, nval, nok);
    // The chunk's rows go through the steps below together, each step's
    // shared-memory lookups and atomics for all ST_U rows in flight at once
    // (one chain per row would leave the SM waiting on their latency).
    // pinned key? (thread-private accumulation)
    uint32_t pinm = 0;
    if (PIN) {
      uint32_t sl[ST_U];
      uint64_t pv[ST_U];
#pragma unroll
      for (int j = 0; j < ST_U; ++j) {
        sl[j] = small_slot_of(ek[j], tmask, p.tiny_mult);
        pv[j] = pk[sl[j]];
      }
#pragma unroll
      for (int j = 0; j < ST_U; ++j)
        pinm |= ((okm >> j & 1) && pv[j] == ek[j] && ek[j] != 0 ? 1u : 0u) << j;
      if (SCATTER && pinm) {
        uint32_t dd[ST_U];
#pragma unroll
        for (int j = 0; j < ST_U; ++j) dd[j] = dense[sl[j]];
#pragma unroll
        for (int j = 0; j < ST_U; ++j) {
          if (!(pinm >> j & 1)) continue;
          const uint32_t at = dd[j] * SP_BLOCK + tid;
          const uint64_t o = lds64(sum + 8 * at);
          const uint32_t c = lds32(cnt + 4 * at);
          if constexpr (NA == 4) {
            uint64_t mn, mx;
            lds128(mm + 16 * at, mn, mx);
            const uint64_t lo = val[j] ^ MIN_FLIP, hi = val[j] ^ MAX_FLIP;
            if (lo > mn) sts64(mm + 16 * at, lo);
            if (hi > mx) sts64(mm + 16 * at + 8, hi);
          }
          sts64(sum + 8 * at, o + val[j]);
          sts32(cnt + 4 * at, c + 1);
        }
      }
    }
    // INT64_MIN rows (stored key 0): the side accumulator
    uint32_t sidem = 0;
#pragma unroll
    for (int j = 0; j < ST_U; ++j) sidem |= ((okm >> j & 1) && ek[j] == 0 ? 1u : 0u) << j;
    sidem &= ~pinm;
    if (SCATTER && sidem) {
#pragma unroll
      for (int j = 0; j < ST_U; ++j) {
        if (!(sidem >> j & 1)) continue;
        uint64_t w[NA];
        words_of<NA>(val[j], w);
        atomicAdd(&p.hdr->n_side, 1ull);
        red_global<NA>(p.hdr->side_aggs, w);
      }
    }
    // every other row is a record of its partition
    const uint32_t recm = okm & ~pinm & ~sidem;
    uint32_t part[ST_U];
#pragma unroll
    for (int j = 0; j < ST_U; ++j) part[j] = part_of(ek[j], p.part_bits);
    if (!SCATTER) {
#pragma unroll
      for (int j = 0; j < ST_U; ++j)
        if (recm >> j & 1) atomicAdd(&ctr[part[j]], 1u);
    } else {
      // sort the chunk's records by level-1 bin: ranks within the bins ...
      uint32_t rank[ST_U];
#pragma unroll
      for (int j = 0; j < ST_U; ++j)
        if (recm >> j & 1) rank[j] = atomicAdd(&cnt1[part[j] >> shift1], 1u);
      __syncthreads();
      // ... the bins' local bases (exclusive scan over threads 0..B1-1), one
      // global claim per non-empty bin, and the counts cleared for the next
      // chunk (every thread has read its count by the barrier before) ...
      const uint32_t c = tid < (int)B1 ? cnt1[tid] : 0u;
      uint32_t incl = c;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      if (lane == 31 && warp < SP_BINS / 32) wsum[warp] = incl;
      __syncthreads();
      uint32_t nrec = 0, before = 0;
#pragma unroll
      for (int w = 0; w < SP_BINS / 32; ++w) {
        before += w < warp ? wsum[w] : 0u;
        nrec += wsum[w];
      }
      if (tid < (int)B1) {
        lb[tid] = before + incl - c;
        // output position of local slot i of this bin: i + delta (mod 2^32);
        // a claim past the bin's end (the passes disagreed) voids the call and
        // stops this CTA's writes
        if (c) {
          const uint32_t g = atomicAdd(p.cursor1 + tid, c);
          if (g + c > end1[tid]) {
            atomicOr(&p.hdr->timeout, 2u);
            wsum[SP_BAD] = 1;
          }
          gb1[tid] = g - (before + incl - c);
        }
        cnt1[tid] = 0;
      }
      __syncthreads();
      // ... the records into place in shared memory ...
#pragma unroll
      for (int j = 0; j < ST_U; ++j) {
        if (!(recm >> j & 1)) continue;
        const uint32_t b = part[j] >> shift1;
        const uint32_t sl = lb[b] + rank[j];
        PartRec r;
        r.ek = ek[j];
        r.val = (long long)val[j];
        recbuf[sl] = r;
        slot_bin[sl] = (uint8_t)b;
      }
      __syncthreads();
      // ... and out: consecutive threads write consecutive records of a run.
      // No barrier after: the next chunk touches only the cleared counts
      // before its first barrier, which every thread reaches after this.
      if (!wsum[SP_BAD])  // uniform: never past a bin
        for (uint32_t i = tid; i < nrec; i += SP_BLOCK) out1[i + gb1[slot_bin[i]]] = recbuf[i];
    }
#pragma unroll
    for (int j = 0; j < ST_U; ++j) {
      ek[j] = nek[j];
      if (SCATTER) val[j] = nval[j];
    }
    okm = nok;
  }
  __syncthreads();
  if (!SCATTER) {
    for (uint32_t i = tid; i < P; i += SP_BLOCK) p.hist[(size_t)i * p.fixed_grid + blockIdx.x] = ctr[i];
    return;
  }
  if (PIN) {
    for (uint32_t d = 0; d < n_hot; ++d) {
#pragma unroll
      for (int a = 0; a < NA; ++a) {
        const uint32_t at = d * SP_BLOCK + tid;
        uint64_t x = a == 0 ? lds64(sum + 8 * at) : a == 1 ? (uint64_t)lds32(cnt + 4 * at)
                                                           : lds64(mm + 16 * at + 8 * (a - 2));
#pragma unroll
        for (int o = 16; o; o >>= 1) {
          const uint64_t y = __shfl_xor_sync(0xffffffffu, x, o);
          x = umax_word<NA>(a) ? (x > y ? x : y) : x + y;
        }
        if (lane == 0 && x) {
          if (umax_word<NA>(a))
            atomicMax(csum + d * NA + a, (unsigned long long)x);
          else
            sadd64(csum + d * NA + a, x);
        }
      }
    }
    __syncthreads();
    if (tid < PM && csum[tid * NA + 1] != 0) {
      uint64_t w[NA];
#pragma unroll
      for (int a = 0; a < NA; ++a) w[a] = csum[tid * NA + a];
      global_update<NA>(p, pkd[tid], w);
    }
  }
}

size_t ppass_smem(const GbParams& p, int na, bool pin, bool scatter) {
  size_t b = SP_HEAD;
  if (pin && scatter)
    for (uint32_t i = 0; i < p.tiny_slots; ++i)
      if (p.tiny_init[i] != 0) b += (size_t)(na == 4 ? pk_key_bytes<4>() : pk_key_bytes<2>()) * SP_BLOCK;
  return b + (scatter ? SP_SORT_SMEM : 4ull << p.part_bits);
}

// CTAs of a pass that fit on the SMs at once (at most cap), or 0.
template <class KT, int NA, bool PIN, bool SCATTER>
uint32_t ppass_grid(const GbParams& p, uint32_t cap) {
  auto kern = gb_ppass_stream_k<KT, NA, PIN, SCATTER>;
  const size_t smem = ppass_smem(p, NA, PIN, SCATTER);
  if (relhost::allow_smem(kern) != cudaSuccess)
    return 0;
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, SP_BLOCK, smem) != cudaSuccess)
    return 0;
  const uint32_t g = (uint32_t)relhost::device_sms() * (uint32_t)(occ > 0 ? occ : 0);
  return g < cap ? g : cap;
}

// The histogram pass runs p.fixed_grid CTAs (its counts are laid out per
// CTA); the scatter pass, whose positions come from the bins' cursors, runs
// as many CTAs as fit.
template <class KT, int NA, bool PIN, bool SCATTER>
rel_status launch_ppass(const GbParams& p, cudaStream_t st) {
  auto kern = gb_ppass_stream_k<KT, NA, PIN, SCATTER>;
  const size_t smem = ppass_smem(p, NA, PIN, SCATTER);
  cudaError_t e = relhost::allow_smem(kern);
  if (e != cudaSuccess) return relhost::cuda_fail(e, "cudaFuncSetAttribute(partition pass)");
  const uint32_t grid = SCATTER ? ppass_grid<KT, NA, PIN, SCATTER>(p, 1u << 16) : p.fixed_grid;
  if (grid < 1) return relhost::set_error("group-by: partition pass does not fit"), REL_E_UNSUPPORTED;
  const int id = SCATTER ? relhost::K_GB_PSCATTER : relhost::K_GB_PHIST;
  relhost::launch_begin(id, st);
  kern<<<grid, SP_BLOCK, smem, st>>>(p);
  relhost::launch_end(id, st);
  e = cudaGetLastError();
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "launch(partition pass)");
}

template <class KT, int NA>
rel_status ppass_dispatch(const GbParams& p, bool scatter, cudaStream_t st) {
  const bool pin = p.tiny_frozen && p.tiny_slots;
  if (pin)
    return scatter ? launch_ppass<KT, NA, true, true>(p, st) : launch_ppass<KT, NA, true, false>(p, st);
  return scatter ? launch_ppass<KT, NA, false, true>(p, st) : launch_ppass<KT, NA, false, false>(p, st);
}

size_t stream_smem(int na) {
  return 416 + 8 * ST_PIN_LIMIT * 4 + (size_t)8 * (na == 4 ? pin_max<4>() : pin_max<2>()) * na * ST_BLOCK;
}

// One wave of resident CTAs, at most one per chunk.
template <class K>
rel_status launch_rows(K kern, int block, size_t smem, int64_t chunk, const GbParams& p,
                       cudaStream_t st) {
  cudaError_t e = relhost::allow_smem(kern);
  if (e != cudaSuccess) return relhost::cuda_fail(e, "cudaFuncSetAttribute(stream)");
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, block, smem);
  if (e != cudaSuccess) return relhost::cuda_fail(e, "occupancy(stream)");
  if (occ < 1) return relhost::set_error("group-by: stream kernel does not fit"), REL_E_UNSUPPORTED;
  const int64_t chunks = (p.n_rows + chunk - 1) / chunk;
  int64_t grid = (int64_t)relhost::device_sms() * occ;
  if (grid > chunks) grid = chunks;
  if (grid < 1) grid = 1;
  relhost::launch_begin(relhost::K_GB_STREAM, st);
  kern<<<(int)grid, block, smem, st>>>(p);
  relhost::launch_end(relhost::K_GB_STREAM, st);
  e = cudaGetLastError();
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "launch(stream)");
}

// Pinned keys that gb_stream_k keeps in thread-private words.
bool pins_fit(const GbParams& p, int na, int n_hot) {
  return p.tiny_frozen && p.tiny_slots <= 32 && n_hot <= (na == 4 ? pin_max<4>() : pin_max<2>());
}

template <class KT, int NA, bool TAB>
rel_status launch_pin(const GbParams& p, cudaStream_t st) {
  int block = p.n_rows > (int64_t)relhost::device_sms() * 4096 ? PK_MAX_BLOCK : 128;
  const size_t per = p.tiny_slots * pk_key_bytes<NA>(), head = PK_HEAD + (TAB ? SmTab<NA>::bytes(p.smem_slots) : 0);
  while (block > 128 && head + per * block > 184 * 1024) block -= 128;  // (L1)
  return launch_rows(gb_pin_k<KT, NA, TAB>, block, head + per * block, (int64_t)block * PK_U, p, st);
}

// The largest table beside pinned keys that were all the keys of the sample
// (a plan for at most half as many groups, though the sample has a few keys):
// nearly every row is pinned, and three or four frequent keys meet on their
// slots in gb_smem_k (1.45e8 rows of three Zipf(1.5) keys, four aggregates: 652
// us there, 402 here; 3e7 rows of ten keys in runs, two aggregates: 140, 80).
constexpr uint32_t PIN_TABLE_SLOTS = 1024;

template <class KT, int NA>
rel_status dispatch_layers(const GbParams& p, cudaStream_t st) {
  int n_hot = 0;
  for (uint32_t i = 0; i < p.tiny_slots && p.tiny_frozen; ++i) n_hot += p.tiny_init[i] != 0;
  if (p.all_pinned && p.smem_slots && p.smem_slots <= PIN_TABLE_SLOTS && pins_fit(p, NA, n_hot)) {
    GbParams q = p;
    if (q.smem_slots < 256) q.smem_slots = 256;
    return launch_pin<KT, NA, true>(q, st);
  }
  if (p.smem_slots || (p.tiny_slots && !pins_fit(p, NA, n_hot))) {
    // 1024 resident threads per SM whatever the table's size; small inputs in
    // small CTAs, so that more SMs take part
    const int64_t small = (int64_t)relhost::device_sms() * 2048;
    GbParams q = p;
    // A plan's table is half full (with first-come or too many pinned
    // thread-private slots instead: its few groups in 256 slots).  Where the
    // rows pay for clearing and merging it, up to four times the slots keep
    // more keys in their home bucket (1e8 rows, 400 groups: 1024 slots 0.64
    // ms, 4096 slots 0.50 ms), as long as two CTAs fit; a plan at the largest
    // table gets what one CTA per SM can hold.
    if (q.smem_slots < 256) q.smem_slots = 256;
    if (p.n_rows > 8 * small)
      while (q.smem_slots < 4 * p.smem_slots && SmTab<NA>::bytes(2 * q.smem_slots) <= SG_MAX_BYTES / 2)
        q.smem_slots *= 2;
    if (p.smem_slots == SHARED_MAX_SLOTS) q.smem_slots = SmTab<NA>::fit(SG_MAX_BYTES);
    const size_t smem = SmTab<NA>::bytes(q.smem_slots);
    const int block = smem > 110 * 1024 ? 1024 : smem > 54 * 1024 || p.n_rows > small ? 512 : 256;
    return launch_rows(gb_smem_k<KT, NA>, block, smem, (int64_t)block * SG_U, q, st);
  }
  const bool pin = p.tiny_frozen && p.tiny_slots;
  if (pin && p.all_pinned) return launch_pin<KT, NA, false>(p, st);
  if (pin) return launch_rows(gb_stream_k<KT, NA>, ST_BLOCK, stream_smem(NA), ST_BLOCK * ST_U, p, st);
  const int block = p.n_rows > (int64_t)relhost::device_sms() * 2048 ? 512 : 128;
  return launch_rows(gb_glob_k<KT, NA>, block, 0, (int64_t)block * 2, p, st);
}

}  // namespace

bool gb_stream_shape(int shape) {
  return shape == SHAPE_KV4_64 || shape == SHAPE_KV4_32 || shape == SHAPE_KV2_64 ||
         shape == SHAPE_KV2_32;
}

// Level 2 of the streaming scatter: every tile of PART_TILE level-1 records
// (tiles never straddle a bin) is sorted by partition inside its bin in
// shared memory; each partition's run is claimed with one atomic on the
// partition's cursor and written contiguously.  Persistent grid; tile t
// belongs to the last bin b with l2_tiles[b] <= t.  Bound by its shared memory
// (ranks by atomics, the records' scattered stores) and by the barriers between:
// four CTAs of 256 threads and 2048 records per SM rather than two of 512 and
// 4096, 942 -> 872 us for the 1.4e8 records of 2e8 Zipf(1.1) rows and 1246 ->
// 1144 for 2e8 uniform ones (reads and writes alone: 0.66 and 0.94 ms).
constexpr int L2_BLOCK = 256;
constexpr int L2_U = PART_TILE / L2_BLOCK;
constexpr int L2_MAX_SUB = 1 << (PART_MAX_BITS - PART_L1_BITS);
constexpr size_t L2_SMEM = 16 * PART_TILE + PART_TILE;

__global__ void __launch_bounds__(L2_BLOCK, 4) gb_part_l2_k(const __grid_constant__ GbParams p) {
  extern __shared__ __align__(16) uint8_t sm[];
  PartRec* recbuf = (PartRec*)sm;
  uint8_t* slot_bin = sm + 16 * PART_TILE;
  __shared__ unsigned int tp[SP_BINS + 1];
  __shared__ unsigned int cnt[L2_MAX_SUB], lb[L2_MAX_SUB], gb[L2_MAX_SUB];
  __shared__ int bad;  // a claim overran its partition: this CTA writes no more
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const uint32_t shift1 = p.part_bits - PART_L1_BITS;  // > 0: launched only then
  const uint32_t B1 = 1u << PART_L1_BITS;
  const uint32_t B2 = 1u << shift1;
  for (uint32_t i = tid; i <= B1; i += L2_BLOCK) tp[i] = p.l2_tiles[i];
  if (tid < (int)B2) cnt[tid] = 0;
  if (tid == 0) bad = 0;
  __syncthreads();
  const uint32_t T = tp[B1];
  for (uint32_t t = blockIdx.x; t < T; t += gridDim.x) {
    uint32_t lo = 0, hi = B1;  // tp[lo] <= t < tp[hi]
    while (hi - lo > 1) {
      const uint32_t mid = (lo + hi) >> 1;
      if (tp[mid] <= t) lo = mid; else hi = mid;
    }
    const uint32_t first = lo << shift1;  // first partition of the bin
    const unsigned long long s1 = p.part_start[first];
    const unsigned long long e1 = p.part_start[first + B2];
    const unsigned long long t0 = s1 + (unsigned long long)(t - tp[lo]) * PART_TILE;
    const unsigned long long t1 = t0 + PART_TILE < e1 ? t0 + PART_TILE : e1;
    PartRec r[L2_U];
    uint32_t sr[L2_U];  // partition within the bin | rank within it << 8
#pragma unroll
    for (int u = 0; u < L2_U; ++u) {
      const unsigned long long i = t0 + (unsigned long long)u * L2_BLOCK + tid;
      sr[u] = 0;
      if (i < t1) {
        const longlong2 v = __ldcs((const longlong2*)(p.recs1 + i));
        r[u].ek = (unsigned long long)v.x;
        r[u].val = v.y;
        sr[u] = part_of((uint64_t)v.x, p.part_bits) & (B2 - 1);
      }
    }
#pragma unroll
    for (int u = 0; u < L2_U; ++u)
      if (t0 + (unsigned long long)u * L2_BLOCK + tid < t1) sr[u] |= atomicAdd(&cnt[sr[u]], 1u) << 8;
    __syncthreads();
    // warp 0: local bases, one claim per non-empty partition, partition ends,
    // counts cleared for the next tile
    if (warp == 0) {
      constexpr int PER = L2_MAX_SUB / 32;
      uint32_t cb[PER], sum = 0;
#pragma unroll
      for (int k = 0; k < PER; ++k) {
        const uint32_t bn = lane * PER + k;
        cb[k] = bn < B2 ? cnt[bn] : 0u;
        sum += cb[k];
      }
      uint32_t incl = sum;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
      }
      uint32_t run = incl - sum;
#pragma unroll
      for (int k = 0; k < PER; ++k) {
        const uint32_t bn = lane * PER + k;
        if (bn < B2) {
          lb[bn] = run;
          if (cb[k]) {  // position of local slot i: i + delta (see the level-1 pass)
            const uint32_t g = atomicAdd(p.cursor + first + bn, cb[k]);
            if (g + cb[k] > (uint32_t)p.part_start[first + bn + 1]) {
              atomicOr(&p.hdr->timeout, 2u);
              bad = 1;
            }
            gb[bn] = g - run;
          }
          cnt[bn] = 0;
        }
        run += cb[k];
      }
    }
    __syncthreads();
#pragma unroll
    for (int u = 0; u < L2_U; ++u) {
      if (t0 + (unsigned long long)u * L2_BLOCK + tid >= t1) continue;
      const uint32_t sub = sr[u] & 0xFFu;
      const uint32_t sl = lb[sub] + (sr[u] >> 8);
      recbuf[sl] = r[u];
      slot_bin[sl] = (uint8_t)sub;
    }
    __syncthreads();
    // no barrier after the writes: the next tile touches only the cleared
    // counts before its first barrier
    const uint32_t nrec = (uint32_t)(t1 - t0);
    if (!bad)  // uniform: never past a partition
      for (uint32_t i = tid; i < nrec; i += L2_BLOCK) p.recs[i + gb[slot_bin[i]]] = recbuf[i];
  }
}

rel_status gb_launch_part_l2(const GbParams& p, cudaStream_t st) {
  if (p.part_bits <= PART_L1_BITS || p.part_bits > PART_MAX_BITS || !p.recs1)
    return relhost::set_error("group-by: level-2 scatter needs more than 2^%d partitions", PART_L1_BITS),
           REL_E_INVALID;
  cudaError_t e = cudaFuncSetAttribute(gb_part_l2_k, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       (int)L2_SMEM);
  if (e != cudaSuccess) return relhost::cuda_fail(e, "cudaFuncSetAttribute(level-2 scatter)");
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, gb_part_l2_k, L2_BLOCK, L2_SMEM);
  if (e != cudaSuccess || occ < 1) return relhost::cuda_fail(e, "occupancy(level-2 scatter)");
  const int grid = relhost::device_sms() * occ;
  relhost::launch_begin(relhost::K_GB_PL2, st);
  gb_part_l2_k<<<grid, L2_BLOCK, L2_SMEM, st>>>(p);
  relhost::launch_end(relhost::K_GB_PL2, st);
  e = cudaGetLastError();
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "launch(level-2 scatter)");
}

uint32_t gb_ppass_stream_grid(const GbParams& p, int shape, uint32_t cap) {
  const bool pin = p.tiny_frozen && p.tiny_slots;
  switch (shape) {
    case SHAPE_KV4_64:
      return pin ? ppass_grid<int64_t, 4, true, false>(p, cap) : ppass_grid<int64_t, 4, false, false>(p, cap);
    case SHAPE_KV4_32:
      return pin ? ppass_grid<int32_t, 4, true, false>(p, cap) : ppass_grid<int32_t, 4, false, false>(p, cap);
    case SHAPE_KV2_64:
      return pin ? ppass_grid<int64_t, 2, true, false>(p, cap) : ppass_grid<int64_t, 2, false, false>(p, cap);
    case SHAPE_KV2_32:
      return pin ? ppass_grid<int32_t, 2, true, false>(p, cap) : ppass_grid<int32_t, 2, false, false>(p, cap);
    default: return 0;
  }
}

bool gb_ppass_stream_eligible(const GbParams& p, int shape, int n_hot) {
  if (!gb_stream_shape(shape) || p.fixed_grid < 1) return false;
  const int na = (shape == SHAPE_KV4_64 || shape == SHAPE_KV4_32) ? 4 : 2;
  const int pmax = na == 4 ? pin_max<4>() : pin_max<2>();
  if (p.tiny_slots && !(p.tiny_frozen && p.tiny_slots <= 32 && n_hot <= pmax)) return false;
  return ppass_smem(p, na, p.tiny_slots != 0, true) * SP_MIN_BLOCKS <= 227 * 1024 &&
         ppass_smem(p, na, p.tiny_slots != 0, false) * SP_MIN_BLOCKS <= 227 * 1024;
}

rel_status gb_launch_ppass_stream(const GbParams& p, int shape, bool scatter, cudaStream_t st) {
  switch (shape) {
    case SHAPE_KV4_64: return ppass_dispatch<int64_t, 4>(p, scatter, st);
    case SHAPE_KV4_32: return ppass_dispatch<int32_t, 4>(p, scatter, st);
    case SHAPE_KV2_64: return ppass_dispatch<int64_t, 2>(p, scatter, st);
    case SHAPE_KV2_32: return ppass_dispatch<int32_t, 2>(p, scatter, st);
  }
  relhost::set_error("group-by: partition pass needs a key/value shape");
  return REL_E_INVALID;
}

rel_status gb_launch_stream(const GbParams& p, int shape, cudaStream_t st) {
  if (p.n_rows == 0) return REL_OK;
  switch (shape) {
    case SHAPE_KV4_64: return dispatch_layers<int64_t, 4>(p, st);
    case SHAPE_KV4_32: return dispatch_layers<int32_t, 4>(p, st);
    case SHAPE_KV2_64: return dispatch_layers<int64_t, 2>(p, st);
    case SHAPE_KV2_32: return dispatch_layers<int32_t, 2>(p, st);
  }
  relhost::set_error("group-by: stream kernel needs a key/value shape");
  return REL_E_INVALID;
}

}  // namespace rel
