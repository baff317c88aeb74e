// Group-by and exact distinct count for any descriptor: the filter, the packed
// key and the product-form aggregates are read from the launch parameters.
//
// The staged kernel (gb_main) keeps a row's words in an array indexed at run
// time and its tables slot by slot, and leaves rows its 2048-slot table cannot
// hold to one-at-a-time global updates (1e7 rows, 3500 groups, four
// aggregates: 4.2 ms).  Here nothing of a row is kept in an indexed array:
//  * a thread takes four consecutive rows; each column is loaded where it is
//    used, four values at a time (one 4- to 32-byte load), so a second use
//    comes from L1 and no staging or barrier sits on the path;
//  * filter and key first; then the four rows' slots are found together, in
//    the CTA's shared-memory table (the search of smtab.cuh) or, for what has
//    no place there, in the global table (home sectors of four keys);
//  * then one aggregate after the other: load, multiply, update the four rows'
//    word.  Shared words are separate arrays per aggregate, sums as in
//    smtab.cuh (two biased 32-bit halves), counts one 32-bit array.
// Instruction issue bounds it (60 % of the slots, 10.5 warp instructions a row;
// 1e7 rows, 3500 groups, four aggregates: 0.15 ms).
#include <algorithm>

#include "gen.cuh"
#include "smtab.cuh"

namespace rel {

namespace {

constexpr int GEN_U = 4;  // consecutive rows per thread
// What a table may take: the rest of the SM's 256 KB is L1, through which the
// columns stream.
constexpr uint32_t GEN_MAX_SMEM = 168 * 1024;

// Shared words of one aggregate: SUM 8 bytes (two arrays of 4), MIN / MAX 8,
// COUNT none of its own.
__host__ __device__ inline uint32_t word_bytes(int op) { return op == REL_COUNT ? 0 : 8; }

__host__ inline size_t gen_smem(const GbParams& p, uint32_t slots) {
  size_t per = 4;  // row counts
  for (int a = 0; a < p.n_aggs; ++a) per += word_bytes(p.aop[a]);
  return (size_t)slots * 8 + (size_t)(slots + 32) * per;
}

// Four values of one column as loaded: 4, 16 or 32 bytes.  Loading and
// unpacking are apart so that several columns' loads are in flight before the
// first value is used.
struct Raw4 {
  longlong2 a, b;
};

// From row r on (rows beyond n: 0); full: aligned, all four rows there.
__device__ __forceinline__ Raw4 load_raw(const GbParams& p, int c, int64_t r, bool full) {
  const uint8_t* q = p.col[c];
  const int t = p.ctype[c];
  Raw4 x;
  x.a = x.b = make_longlong2(0, 0);
  if (full) {
    if (t == REL_I64) {
      x.a = __ldg((const longlong2*)(q + 8 * r));
      x.b = __ldg((const longlong2*)(q + 8 * r) + 1);
    } else if (t == REL_I32) {
      x.a = __ldg((const longlong2*)(q + 4 * r));
    } else {
      x.a.x = (long long)__ldg((const unsigned int*)(q + r));
    }
    return x;
  }
  if (t == REL_I64) {
    const long long* v = (const long long*)q + r;
    if (r < p.n_rows) x.a.x = __ldg(v);
    if (r + 1 < p.n_rows) x.a.y = __ldg(v + 1);
    if (r + 2 < p.n_rows) x.b.x = __ldg(v + 2);
    if (r + 3 < p.n_rows) x.b.y = __ldg(v + 3);
  } else {
    uint64_t w[2] = {0, 0};
#pragma unroll
    for (int j = 0; j < GEN_U; ++j) {
      if (r + j >= p.n_rows) continue;
      if (t == REL_I32)
        w[j / 2] |= (uint64_t)(uint32_t)__ldg((const int*)q + r + j) << (32 * (j & 1));
      else
        w[0] |= (uint64_t)__ldg(q + r + j) << (8 * j);
    }
    x.a = make_longlong2((long long)w[0], (long long)w[1]);
  }
  return x;
}

__device__ __forceinline__ void unpack(const GbParams& p, int c, const Raw4& x, int64_t (&v)[GEN_U]) {
  const int t = p.ctype[c];
  if (t == REL_I64) {
    v[0] = x.a.x; v[1] = x.a.y; v[2] = x.b.x; v[3] = x.b.y;
  } else if (t == REL_I32) {
    v[0] = (int32_t)x.a.x; v[1] = x.a.x >> 32; v[2] = (int32_t)x.a.y; v[3] = x.a.y >> 32;
  } else {
#pragma unroll
    for (int j = 0; j < GEN_U; ++j) v[j] = ((uint32_t)x.a.x >> (8 * j)) & 255;
  }
}

__device__ __forceinline__ void load4(const GbParams& p, int c, int64_t r, bool full,
                                      int64_t (&v)[GEN_U]) {
  unpack(p, c, load_raw(p, c, r, full), v);
}

// Clears the bits of keep whose row fails range filter i.  Columns of at most
// 32 bits are compared in 32 bits.
__device__ __forceinline__ uint32_t filter4(const GbParams& p, int i, const Raw4& x, uint32_t keep) {
  const int64_t lo = p.pred_lo[i], hi = p.pred_hi[i];
  const int c = p.pred_col[i], t = p.ctype[c];
  if (t == REL_I64) {
    int64_t v[GEN_U];
    unpack(p, c, x, v);
#pragma unroll
    for (int j = 0; j < GEN_U; ++j)
      if (v[j] < lo || v[j] > hi) keep &= ~(1u << j);
    return keep;
  }
  if (lo > INT32_MAX || hi < INT32_MIN) return 0;
  const int l = lo < INT32_MIN ? INT32_MIN : (int)lo, h = hi > INT32_MAX ? INT32_MAX : (int)hi;
  int v[GEN_U];
  if (t == REL_I32) {
    v[0] = (int)x.a.x; v[1] = (int)(x.a.x >> 32); v[2] = (int)x.a.y; v[3] = (int)(x.a.y >> 32);
  } else {
#pragma unroll
    for (int j = 0; j < GEN_U; ++j) v[j] = ((uint32_t)x.a.x >> (8 * j)) & 255;
  }
#pragma unroll
  for (int j = 0; j < GEN_U; ++j)
    if (v[j] < l || v[j] > h) keep &= ~(1u << j);
  return keep;
}

// Inputs of aggregate a for four rows.
__device__ __forceinline__ void agg4(const GbParams& p, int a, int64_t r, bool full,
                                     uint64_t (&x)[GEN_U]) {
  int64_t v[GEN_U];
  load4(p, p.abase[a], r, full, v);
#pragma unroll
  for (int j = 0; j < GEN_U; ++j) x[j] = (uint64_t)v[j];
  for (int f = 0; f < p.anf[a]; ++f) {
    const uint64_t c = (uint64_t)p.ac[a][f], s = (uint64_t)p.as[a][f];
    load4(p, p.afcol[a][f], r, full, v);
#pragma unroll
    for (int j = 0; j < GEN_U; ++j) x[j] *= c + s * (uint64_t)v[j];
  }
}

// Global slot of key e, walking from its home sector and claiming the first
// empty slot; *claimed when this call put it there.  ~0 when the table
// overflowed.
__device__ __forceinline__ uint64_t global_slot(const GbParams& p, uint64_t e, bool* claimed) {
  const uint64_t mask = (1ull << p.log2_slots) - 1;
  uint64_t s = home_sector(e, p.log2_slots);
  *claimed = false;
  for (uint32_t i = 0; i < p.max_probe; i += 4) {
    uint64_t k[4];
    ld_sector(p.tkeys + s, k);
    uint32_t at = in_sector(k, e);
    if (at == 4 && k[3] == 0) {  // room as loaded
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if (at != 4 || k[q] != 0) continue;
        const uint64_t old =
            atomicCAS((unsigned long long*)(p.tkeys + s + q), 0ull, (unsigned long long)e);
        *claimed = old == 0;
        if (old == 0 || old == e) at = q;
      }
    }
    if (at != 4) return s + at;
    s = (s + 4) & mask;
    if ((i & 31) == 28 && ld_relaxed_u32(&p.hdr->overflow)) return ~0ull;  // already overflowed
  }
  atomicOr(&p.hdr->overflow, 1u);
  return ~0ull;
}

// Global slots of the rows of mask m, found two at a time; rows of an
// overflowed table come back as ~0.  Returns the number claimed.
__device__ __forceinline__ uint32_t global_slots(const GbParams& p, const uint64_t (&ek)[GEN_U],
                                                 uint32_t m, uint64_t (&gs)[GEN_U]) {
  uint32_t n = 0, miss = 0;
#pragma unroll
  for (int h = 0; h < GEN_U; h += 2) {
    uint64_t k[2][4];
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      gs[h + q] = home_sector(ek[h + q], p.log2_slots);
      if (m >> (h + q) & 1) ld_sector(p.tkeys + gs[h + q], k[q]);
    }
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      if (!(m >> (h + q) & 1)) continue;
      const uint32_t at = in_sector(k[q], ek[h + q]);
      if (at == 4) miss |= 1u << (h + q);
      else gs[h + q] += at;
    }
  }
  while (miss) {
    const uint32_t bit = miss & (0u - miss);
    uint64_t e = ek[0];
#pragma unroll
    for (int j = 1; j < GEN_U; ++j)
      if (bit == 1u << j) e = ek[j];
    bool c;
    const uint64_t s = global_slot(p, e, &c);
    n += c;
#pragma unroll
    for (int j = 0; j < GEN_U; ++j)
      if (bit == 1u << j) gs[j] = s;
    miss ^= bit;
  }
  __syncwarp();
  return n;
}

// A row whose key is INT64_MIN: the side accumulator.
__device__ __noinline__ void side_row(const GbParams& p, int64_t r) {
  atomicAdd(&p.hdr->n_side, 1ull);
  for (int a = 0; a < p.n_aggs; ++a) {
    const int op = p.aop[a];
    uint64_t x[GEN_U];
    if (op == REL_COUNT) {
      redg_add(p.hdr->side_aggs + a, 1);
      continue;
    }
    agg4(p, a, r, false, x);
    if (op == REL_SUM) redg_add(p.hdr->side_aggs + a, x[0]);
    else redg_max(p.hdr->side_aggs + a, x[0] ^ (op == REL_MIN ? MIN_FLIP : MAX_FLIP));
  }
}

// SM: a shared-memory table of p.smem_slots slots in front of the global one;
// SET: count distinct keys instead of aggregating.
template <bool SM, bool SET>
__global__ void __launch_bounds__(1024, 1) gb_gen_k(const __grid_constant__ GbParams p) {
  extern __shared__ __align__(16) uint8_t sm[];
  // [keys][row counts][words of aggregate 0][...]
  KeyTab t;
  const uint32_t n = p.smem_slots, stride = n + KeyTab::SPARE;
  uint32_t cnt = 0, words = 0;
  if (SM) {
    t.bind(smem_u32(sm), n);
    cnt = t.key + 8 * n;
    words = cnt + 4 * stride;
    uint32_t bytes = 8 * n;
    if (!SET) {
      bytes += 4 * stride;
      for (int a = 0; a < p.n_aggs; ++a) bytes += stride * word_bytes(p.aop[a]);
    }
    for (uint32_t i = 8 * threadIdx.x; i < bytes; i += 8 * blockDim.x) sts64(t.key + i, 0);
    __syncthreads();
  }
  unsigned long long claims = 0;
  // Whether to look for warps whose rows are all of one group (their words are
  // combined first): those that begin with such a chunk do
  bool same = true;
  bool aligned = true;
  for (int c = 0; c < p.n_cols; ++c) aligned &= (uintptr_t)p.col[c] % 16 == 0;
  const int64_t CHUNK = (int64_t)blockDim.x * GEN_U;
  for (int64_t base = (int64_t)blockIdx.x * CHUNK; base < p.n_rows; base += (int64_t)gridDim.x * CHUNK) {
    const int64_t r = base + GEN_U * threadIdx.x;
    const bool full = aligned && base + CHUNK <= p.n_rows;
    uint32_t keep = (1u << GEN_U) - 1;
    if (!full) {
#pragma unroll
      for (int j = 0; j < GEN_U; ++j)
        if (r + j >= p.n_rows) keep &= ~(1u << j);
    }
    int64_t v[GEN_U];
    uint64_t ek[GEN_U];
    // the first two key columns and the first filter column are in flight
    // together
    const Raw4 k0 = load_raw(p, p.key_col[0], r, full);
    Raw4 k1 = k0, f0 = k0;
    if (p.n_keys > 1) k1 = load_raw(p, p.key_col[1], r, full);
    if (p.n_preds > 0) f0 = load_raw(p, p.pred_col[0], r, full);
    unpack(p, p.key_col[0], k0, v);
#pragma unroll
    for (int j = 0; j < GEN_U; ++j)
      ek[j] = p.n_keys == 1 ? (uint64_t)v[j] : ((uint64_t)v[j] & p.key_mask[0]) << p.key_shift[0];
    for (int i = 1; i < p.n_keys; ++i) {
      if (i == 1) unpack(p, p.key_col[1], k1, v);
      else load4(p, p.key_col[i], r, full, v);
#pragma unroll
      for (int j = 0; j < GEN_U; ++j) ek[j] |= ((uint64_t)v[j] & p.key_mask[i]) << p.key_shift[i];
    }
    for (int i = 0; i < p.n_preds; ++i)
      keep = filter4(p, i, i == 0 ? f0 : load_raw(p, p.pred_col[i], r, full), keep);
    uint32_t side = 0;
#pragma unroll
    for (int j = 0; j < GEN_U; ++j) {
      ek[j] ^= KEY_FLIP;
      if (!(keep >> j & 1)) ek[j] = 0;
      else if (ek[j] == 0) side |= 1u << j;
    }
    keep &= ~side;
    if (side) {
      for (int j = 0; j < GEN_U; ++j) {
        if (!(side >> j & 1)) continue;
        if (SET) atomicAdd(&p.hdr->n_side, 1ull);
        else side_row(p, r + j);
      }
    }
    __syncwarp();
    uint32_t slot[GEN_U], left = keep;
    uint64_t gs[GEN_U] = {0, 0, 0, 0};
    if (SM) left = t.find(ek, (int)p.shared_probes, slot);
    if (!SM || __any_sync(0xffffffffu, left != 0)) {
      const uint32_t c = global_slots(p, ek, left, gs);
      if (SET) claims += c;
    }
    if (SET) continue;
    bool one = false;  // every row of the warp has the slot of its first
    if (SM) {
      if (same) {
        one = warp_same(slot[0]) && __all_sync(0xffffffffu, slot[1] == slot[0] && slot[2] == slot[0] &&
                                                                slot[3] == slot[0]);
        same = one || base != (int64_t)blockIdx.x * CHUNK;
      }
      if (one) {
        if ((threadIdx.x & 31) == 0) reds_add(cnt + 4 * slot[0], 32 * GEN_U);
      } else {
#pragma unroll
        for (int j = 0; j < GEN_U; ++j) reds_add(cnt + 4 * slot[j], 1);
      }
    }
#pragma unroll
    for (int j = 0; j < GEN_U; ++j)
      if (gs[j] == ~0ull) left &= ~(1u << j);  // the table overflowed
    uint32_t wa = words;  // the aggregate's shared words
    for (int a = 0; a < p.n_aggs; ++a) {
      const int op = p.aop[a];
      unsigned long long* g = p.taggs + a;
      if (op == REL_COUNT) {
        if (left) {
#pragma unroll
          for (int j = 0; j < GEN_U; ++j)
            if (left >> j & 1) redg_add(g + gs[j] * (uint64_t)p.n_aggs, 1);
        }
        continue;
      }
      uint64_t x[GEN_U];
      agg4(p, a, r, full, x);
      if (op == REL_SUM) {
        if (SM && one) {
          const uint64_t sum = warp_sum(x[0] + x[1] + x[2] + x[3]) + 32 * GEN_U * SUM_BIAS;
          if ((threadIdx.x & 31) == 0) {
            const uint32_t old = atoms_add(wa + 4 * slot[0], (uint32_t)sum);
            reds_add_nz(wa + 4 * (stride + slot[0]), high_with_carry(old, sum));
          }
        } else if (SM) {
          uint32_t old[GEN_U];
#pragma unroll
          for (int j = 0; j < GEN_U; ++j) old[j] = atoms_add(wa + 4 * slot[j], (uint32_t)(x[j] + SUM_BIAS));
#pragma unroll
          for (int j = 0; j < GEN_U; ++j)
            reds_add_nz(wa + 4 * (stride + slot[j]), high_with_carry(old[j], x[j] + SUM_BIAS));
        }
        if (left) {
#pragma unroll
          for (int j = 0; j < GEN_U; ++j)
            if (left >> j & 1) redg_add(g + gs[j] * (uint64_t)p.n_aggs, x[j]);
        }
      } else {
        const uint64_t flip = op == REL_MIN ? MIN_FLIP : MAX_FLIP;
        if (SM && one) {
          const uint64_t a = (x[0] ^ flip) > (x[1] ^ flip) ? x[0] ^ flip : x[1] ^ flip;
          const uint64_t b = (x[2] ^ flip) > (x[3] ^ flip) ? x[2] ^ flip : x[3] ^ flip;
          const uint64_t top = warp_max(a > b ? a : b);
          if ((threadIdx.x & 31) == 0) reds_raise64(wa + 8 * slot[0], top, lds64(wa + 8 * slot[0]));
        } else if (SM) {
#pragma unroll
          for (int j = 0; j < GEN_U; ++j)
            reds_raise64(wa + 8 * slot[j], x[j] ^ flip, lds64(wa + 8 * slot[j]));
        }
        if (left) {
#pragma unroll
          for (int j = 0; j < GEN_U; ++j)
            if (left >> j & 1) redg_max(g + gs[j] * (uint64_t)p.n_aggs, x[j] ^ flip);
        }
      }
      wa += stride * word_bytes(op);
    }
  }
  if (SM) {  // the CTA's groups (keys) into the global table (set)
    __syncthreads();
    for (uint32_t s = threadIdx.x; s < n; s += blockDim.x) {
      const uint64_t k = t.key_of(s);
      if (k == 0) continue;
      bool c;
      const uint64_t gs = global_slot(p, k, &c);
      claims += c;
      if (SET || gs == ~0ull) continue;
      const uint32_t rows = lds32(cnt + 4 * s);
      uint32_t wa = words;
      for (int a = 0; a < p.n_aggs; ++a) {
        const int op = p.aop[a];
        unsigned long long* g = p.taggs + gs * (uint64_t)p.n_aggs + a;
        if (op == REL_COUNT)
          redg_add(g, rows);
        else if (op == REL_SUM)
          redg_add(g, ((uint64_t)lds32(wa + 4 * (stride + s)) << 32 | lds32(wa + 4 * s)) -
                          (uint64_t)rows * SUM_BIAS);
        else
          redg_max(g, lds64(wa + 8 * s));
        wa += stride * word_bytes(op);
      }
    }
  }
  if (SET) {
#pragma unroll
    for (int o = 16; o; o >>= 1) claims += __shfl_xor_sync(0xffffffffu, claims, o);
    if ((threadIdx.x & 31) == 0 && claims) atomicAdd(&p.hdr->aux, claims);
    wait_for_earlier_kernels();
  }
}

// Distinct count of keys of at most 16 bits (one or two uint8 columns): a bit
// per possible key in shared memory, no hash and no search.  Bound by issue
// and HBM: 1e8 rows of (uint8, uint8) keys with an int32 filter 0.43 -> 0.22
// ms against the hashed count.
constexpr int BITS_WORDS = 65536 / 32;

__global__ void __launch_bounds__(512, 3) gb_gen_bits_k(const __grid_constant__ GbParams p) {
  __shared__ uint32_t seen[BITS_WORDS];
  for (int i = threadIdx.x; i < BITS_WORDS; i += blockDim.x) seen[i] = 0;
  __syncthreads();
  bool aligned = true;
  for (int c = 0; c < p.n_cols; ++c) aligned &= (uintptr_t)p.col[c] % 16 == 0;
  const int64_t CHUNK = (int64_t)blockDim.x * GEN_U;
  for (int64_t base = (int64_t)blockIdx.x * CHUNK; base < p.n_rows; base += (int64_t)gridDim.x * CHUNK) {
    const int64_t r = base + GEN_U * threadIdx.x;
    const bool full = aligned && base + CHUNK <= p.n_rows;
    uint32_t keep = (1u << GEN_U) - 1;
    if (!full) {
#pragma unroll
      for (int j = 0; j < GEN_U; ++j)
        if (r + j >= p.n_rows) keep &= ~(1u << j);
    }
    const Raw4 k0 = load_raw(p, p.key_col[0], r, full);
    Raw4 k1 = k0, f0 = k0;
    if (p.n_keys > 1) k1 = load_raw(p, p.key_col[1], r, full);
    if (p.n_preds > 0) f0 = load_raw(p, p.pred_col[0], r, full);
    for (int i = 0; i < p.n_preds; ++i)
      keep = filter4(p, i, i == 0 ? f0 : load_raw(p, p.pred_col[i], r, full), keep);
    // two 16-bit keys per word: (first column << 8) | second
    const uint32_t hi = p.n_keys > 1 ? (uint32_t)k0.a.x : 0u;
    const uint32_t lo = p.n_keys > 1 ? (uint32_t)k1.a.x : (uint32_t)k0.a.x;
    const uint32_t w[2] = {__byte_perm(lo, hi, 0x5140), __byte_perm(lo, hi, 0x7362)};
#pragma unroll
    for (int j = 0; j < GEN_U; ++j) {
      const uint32_t key = (w[j / 2] >> (16 * (j & 1))) & 0xFFFFu;
      const uint32_t bit = 1u << (key & 31);
      if ((keep >> j & 1) && !(*(volatile uint32_t*)(seen + (key >> 5)) & bit)) atomicOr(seen + (key >> 5), bit);
    }
  }
  __syncthreads();
  // this CTA's keys into the global bits; the first to set a bit counts its key
  unsigned long long claims = 0;
  for (int i = threadIdx.x; i < BITS_WORDS; i += blockDim.x)
    if (seen[i]) claims += __popc(seen[i] & ~atomicOr((uint32_t*)p.tkeys + i, seen[i]));
#pragma unroll
  for (int o = 16; o; o >>= 1) claims += __shfl_xor_sync(0xffffffffu, claims, o);
  if ((threadIdx.x & 31) == 0 && claims) atomicAdd(&p.hdr->aux, claims);
  wait_for_earlier_kernels();
}

template <class K>
rel_status launch_gen(K kern, int id, size_t smem, const GbParams& p, cudaStream_t st,
                      bool beside = false) {
  if (p.n_rows == 0) return REL_OK;
  cudaError_t e = relhost::allow_smem(kern);
  if (e != cudaSuccess) return relhost::cuda_fail(e, "cudaFuncSetAttribute(generic)");
  // 1024 resident threads per SM (64 registers each) whatever the table's
  // size; small inputs in small CTAs, so that more SMs take part
  const int block = smem > 110 * 1024 ? 1024 : p.n_rows > (int64_t)relhost::device_sms() * 2048 ? 512 : 256;
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, block, smem);
  if (e != cudaSuccess || occ < 1) return relhost::cuda_fail(e, "occupancy(generic)");
  const int64_t chunk = (int64_t)block * GEN_U, chunks = (p.n_rows + chunk - 1) / chunk;
  int64_t grid = (int64_t)(relhost::device_sms() - (beside ? 1 : 0)) * occ;
  if (grid > chunks) grid = chunks;
  relhost::launch_begin(id, st);
  e = relhost::launch(kern, (unsigned)grid, (unsigned)block, smem, st, beside, p);
  relhost::launch_end(id, st);
  if (e == cudaSuccess) e = cudaGetLastError();
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "launch(generic)");
}

}  // namespace

rel_status gb_launch_gen(const GbParams& p0, int64_t est, cudaStream_t st) {
  GbParams p = p0;
  if (!p.smem_slots && !p.tiny_slots)  // a plan without per-CTA layers
    return launch_gen(gb_gen_k<false, false>, relhost::K_GB_LAYERED, 0, p, st);
  // Slots for twice the groups, as many as fit one CTA per SM.  More groups
  // than that: a table for two CTAs per SM, searched only briefly, that
  // catches the frequent keys of a skewed input (and the few keys of one whose
  // plan knew no better than one group per row).
  size_t word = 12;
  for (int a = 0; a < p.n_aggs; ++a) word += word_bytes(p.aop[a]);
  const uint64_t fit1 = (GEN_MAX_SMEM - 32 * word) / word & ~15ull;
  const uint64_t fit2 = (GEN_MAX_SMEM / 2 - 32 * word) / word & ~15ull;
  const uint64_t want = est < 128 ? 256 : (2 * (uint64_t)est + 15) & ~15ull;
  const bool whole = 8 * fit1 >= 9 * (uint64_t)est;
  p.smem_slots = (uint32_t)(whole ? std::min(want, fit1) : fit2);
  p.shared_probes = whole ? 16 : 2;
  return launch_gen(gb_gen_k<true, false>, relhost::K_GB_LAYERED, gen_smem(p, p.smem_slots), p, st);
}

rel_status gb_launch_gen_set(const GbParams& p0, bool beside, cudaStream_t st) {
  GbParams p = p0;
  bool narrow = p.n_keys <= 2;  // and a set large enough for a bit per key
  for (int k = 0; k < p.n_keys; ++k) narrow &= p.ctype[p.key_col[k]] == REL_U8;
  if (narrow && (8ull << p.log2_slots) >= 4ull * BITS_WORDS)
    return launch_gen(gb_gen_bits_k, relhost::K_GB_KEYSET, 0, p, st, beside);
  // the keys the CTA has seen: few keys never reach the global set twice, and
  // a row of many keys is not searched for long
  p.smem_slots = 4096;
  p.shared_probes = 2;
  return launch_gen(gb_gen_k<true, true>, relhost::K_GB_KEYSET, 8 * (size_t)p.smem_slots, p, st, beside);
}

}  // namespace rel
