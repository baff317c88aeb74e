// Open-addressing aggregate table in shared memory, one per CTA: the layer
// the streaming group-by, the partition aggregation and the batched group-by
// share.  (sum, count[, min, max]) of one int64 value per key.
//
// Instruction issue and shared-memory wavefronts bound these kernels, not
// HBM, so the layout and the order of a row's work are chosen to spend few of
// either:
//  * one array per word.  A 32-byte slot puts a given word of every slot on
//    four of the 32 banks (16-byte slots: eight), so random slots conflict
//    eight deep and more; separate 4-byte arrays use all banks (an add costs
//    2.4 ns per warp and SM on random slots);
//  * a key's home is a bucket of two slots, read with one 16-byte load: at
//    half load 88 of 100 keys are there (97 at a quarter), where one-slot probing
//    makes some lane of nearly every warp walk four slots;
//  * a thread's rows are looked up together, then updated together by
//    straight-line code: the lanes of a warp that found their slots at
//    different probe depths have met again before the atomics, which are
//    issued once per row and not once per probe depth.  Rows that take no part
//    update a spare slot of their lane instead of branching around every
//    access;
//  * a sum is two 32-bit adds with a carry (a 64-bit shared add is a
//    compare-and-swap loop here); inputs are biased by SUM_BIAS, which the
//    reader takes off again (count x SUM_BIAS, exact mod 2^64), so that
//    values of either sign below 2^24 reach the high word only on a carry;
//  * MIN and MAX lie side by side, read with one 16-byte load and raised by
//    an atomic only when the row improves them.
// Counts are 32-bit: a table sees fewer than 2^32 rows.
#pragma once

#include "rel_internal.cuh"

namespace rel {

constexpr uint64_t SUM_BIAS = 1ull << 24;

__device__ __forceinline__ uint32_t lds32(uint32_t a) {
  uint32_t v;
  asm volatile("ld.volatile.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}
__device__ __forceinline__ void sts32(uint32_t a, uint32_t v) {
  asm volatile("st.volatile.shared.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
__device__ __forceinline__ void lds128(uint32_t a, uint64_t& x, uint64_t& y) {
  asm volatile("ld.volatile.shared.v2.u64 {%0, %1}, [%2];" : "=l"(x), "=l"(y) : "r"(a) : "memory");
}
__device__ __forceinline__ uint32_t atoms_add(uint32_t a, uint32_t v) {
  uint32_t o;
  asm volatile("atom.relaxed.cta.shared::cta.add.u32 %0, [%1], %2;"
               : "=r"(o)
               : "r"(a), "r"(v)
               : "memory");
  return o;
}
__device__ __forceinline__ void reds_add(uint32_t a, uint32_t v) {
  asm volatile("red.relaxed.cta.shared::cta.add.u32 [%0], %1;" ::"r"(a), "r"(v) : "memory");
}
// Predicated, without a branch: add v when it is not 0; raise to v when it is
// above cur; claim for k when cur is 0 (cur then holds what the slot held).
__device__ __forceinline__ void reds_add_nz(uint32_t a, uint32_t v) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.u32 p, %1, 0;\n\t"
      "@p red.relaxed.cta.shared::cta.add.u32 [%0], %1;\n\t}" ::"r"(a),
      "r"(v)
      : "memory");
}
__device__ __forceinline__ void reds_raise64(uint32_t a, uint64_t v, uint64_t cur) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.gt.u64 p, %1, %2;\n\t"
      "@p red.relaxed.cta.shared::cta.max.u64 [%0], %1;\n\t}" ::"r"(a),
      "l"(v), "l"(cur)
      : "memory");
}
__device__ __forceinline__ void atoms_claim(uint32_t a, uint64_t k, uint64_t& cur) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.eq.u64 p, %0, 0;\n\t"
      "@p atom.relaxed.cta.shared::cta.cas.b64 %0, [%1], 0, %2;\n\t}"
      : "+l"(cur)
      : "r"(a), "l"(k)
      : "memory");
}
// High word of x plus the carry of old + low word of x.
__device__ __forceinline__ uint32_t high_with_carry(uint32_t old, uint64_t x) {
  uint32_t h;
  asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %1, %2;\n\taddc.u32 %0, %3, 0;\n\t}"
      : "=r"(h)
      : "r"(old), "r"((uint32_t)x), "r"((uint32_t)(x >> 32)));
  return h;
}

// Over the 32 lanes of a warp, all of which take part: the sum mod 2^64 (16-bit
// halves of the low word cannot carry out of 32 bits), the largest.
__device__ __forceinline__ uint64_t warp_sum(uint64_t x) {
  const uint32_t a = __reduce_add_sync(0xffffffffu, (uint32_t)x & 0xFFFFu);
  const uint32_t b = __reduce_add_sync(0xffffffffu, (uint32_t)x >> 16);
  const uint32_t c = __reduce_add_sync(0xffffffffu, (uint32_t)(x >> 32));
  return (uint64_t)a + ((uint64_t)b << 16) + ((uint64_t)c << 32);
}
__device__ __forceinline__ uint64_t warp_max(uint64_t x) {
  const uint32_t h = (uint32_t)(x >> 32), top = __reduce_max_sync(0xffffffffu, h);
  return (uint64_t)top << 32 | __reduce_max_sync(0xffffffffu, h == top ? (uint32_t)x : 0u);
}
// Whether every lane holds the same.
__device__ __forceinline__ bool warp_same(uint32_t s) {
  return __all_sync(0xffffffffu, s == __shfl_sync(0xffffffffu, s, 0));
}

// The keys of a table: buckets of two slots.
struct KeyTab {
  static constexpr uint32_t SPARE = 32;  // slots past the table, one per lane, for idle rows
  uint32_t key;                          // shared address of the key array (16-byte aligned)
  uint32_t slots, idle;                  // an even number; this lane's spare slot

  __device__ __forceinline__ void bind(uint32_t addr, uint32_t n) {
    key = addr;
    slots = n;
    idle = n + (threadIdx.x & 31);
  }
  // First slot of the home bucket, from a multiplicative hash of the whole key
  // (a packed key's columns sit in different halves, so a folded 32-bit hash
  // would lay whole families of keys on the same few slots).
  __device__ __forceinline__ uint32_t home(uint64_t ek) const {
    return __umulhi((uint32_t)((ek * 0x9E3779B97F4A7C15ull) >> 32), slots >> 1) << 1;
  }
  __device__ __forceinline__ uint32_t next(uint32_t s) const {
    return s + 2 == slots ? 0 : s + 2;
  }
  __device__ __forceinline__ uint64_t key_of(uint32_t s) const { return lds64(key + 8 * s); }

  // Slots of U keys, inserting the new ones; a key of 0 takes no part and gets
  // the spare slot, as do rows that found no slot within `probes` further
  // buckets (returned as a mask).  Buckets fill in order and never empty, so
  // everyone who looks for a key walks the same slots and a claim is settled
  // by its compare-and-swap.  All lanes of the warp call this together: each
  // finishes the rows that did not end in their home bucket one by one, then
  // the warp is whole again.
  template <int U>
  __device__ __forceinline__ uint32_t find(const uint64_t (&ek)[U], int probes,
                                           uint32_t (&s)[U]) const {
    uint32_t miss = 0, left = 0;
    {
      uint64_t k0[U], k1[U];
#pragma unroll
      for (int j = 0; j < U; ++j) {
        s[j] = home(ek[j]);
        lds128(key + 8 * s[j], k0[j], k1[j]);
      }
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const bool e0 = k0[j] == ek[j], e1 = k1[j] == ek[j];
        if (!e0 && !e1) {
          miss |= 1u << j;
          if (k1[j] != 0) s[j] = next(s[j]);  // the bucket is full
        }
        if (!e0 && e1) s[j] |= 1;
        if (ek[j] == 0) {
          s[j] = idle;
          miss &= ~(1u << j);
        }
      }
    }
    while (miss) {
      const uint32_t bit = miss & (0u - miss);
      uint64_t k = ek[0], a, b;
      uint32_t w = s[0];
#pragma unroll
      for (int j = 1; j < U; ++j)
        if (bit == 1u << j) {
          k = ek[j];
          w = s[j];
        }
      lds128(key + 8 * w, a, b);
      if (a != k && b != k && b == 0) {  // room as loaded: claim it
        atoms_claim(key + 8 * w, k, a);
        if (a == 0) a = k;
        if (a != k) {
          atoms_claim(key + 8 * w + 8, k, b);
          if (b == 0) b = k;
        }
      }
      const bool done = a == k || b == k;
      w = a == k ? w : b == k ? w + 1 : next(w);
      if (done) {
        miss ^= bit;
      } else if (--probes <= 0) {
        left |= bit;
        miss ^= bit;
        probes = 1;
        w = idle;
      }
#pragma unroll
      for (int j = 0; j < U; ++j)
        if (bit == 1u << j) s[j] = w;
    }
    __syncwarp();
    return left;
  }
};

// NA = 4: sum, count, min, max; NA = 2: sum, count.
template <int NA>
struct SmTab : KeyTab {
  uint32_t mm, lo, hi, cnt;  // shared addresses of the word arrays

  __host__ __device__ static size_t bytes(uint32_t slots) {
    return (size_t)slots * 8 + (size_t)(slots + SPARE) * (12 + (NA == 4 ? 16 : 0));
  }
  // The most slots (a multiple of 16) a table of so many bytes holds.
  __host__ static uint32_t fit(size_t bytes) {
    const size_t word = 12 + (NA == 4 ? 16 : 0);
    return (uint32_t)((bytes - SPARE * word) / (8 + word)) & ~15u;
  }

  __device__ __forceinline__ void bind(void* base, uint32_t n) {  // n: a multiple of 16
    mm = smem_u32(base);
    KeyTab::bind(mm + (NA == 4 ? 16 * (n + SPARE) : 0), n);
    lo = key + 8 * n;
    hi = lo + 4 * (n + SPARE);
    cnt = hi + 4 * (n + SPARE);
  }
  // All threads of the CTA; a barrier must follow.
  __device__ __forceinline__ void clear() const {
    for (uint32_t a = mm + 16 * threadIdx.x; a < cnt + 4 * (slots + SPARE); a += 16 * blockDim.x)
      asm volatile("st.shared.v2.u64 [%0], {%1, %1};" ::"r"(a), "l"(0ull) : "memory");
  }

  // Add rows with values v to the groups of slots s.
  template <int U>
  __device__ __forceinline__ void add(const uint32_t (&s)[U], const uint64_t (&v)[U]) const {
    uint32_t old[U];
#pragma unroll
    for (int j = 0; j < U; ++j) old[j] = atoms_add(lo + 4 * s[j], (uint32_t)(v[j] + SUM_BIAS));
#pragma unroll
    for (int j = 0; j < U; ++j) reds_add(cnt + 4 * s[j], 1);
    if constexpr (NA == 4) {
      uint64_t mn[U], mx[U];
#pragma unroll
      for (int j = 0; j < U; ++j) lds128(mm + 16 * s[j], mn[j], mx[j]);
#pragma unroll
      for (int j = 0; j < U; ++j) {
        reds_raise64(mm + 16 * s[j], v[j] ^ MIN_FLIP, mn[j]);
        reds_raise64(mm + 16 * s[j] + 8, v[j] ^ MAX_FLIP, mx[j]);
      }
    }
#pragma unroll
    for (int j = 0; j < U; ++j) reds_add_nz(hi + 4 * s[j], high_with_carry(old[j], v[j] + SUM_BIAS));
  }

  // The same for a warp whose rows may all be of one slot: those are combined
  // first, as the adds of 32 lanes to one address take their turns (16 ns a warp
  // and SM).  G rows of a lane that lie together are looked at together.  (Warps
  // of two slots, as at the end of a run, cost as much in two parts as their adds
  // do.)  All lanes of the warp.
  template <int U, int G>
  __device__ __forceinline__ void add_same(const uint32_t (&s)[U], const uint64_t (&v)[U]) const {
#pragma unroll
    for (int j = 0; j < U; j += G) {
      uint32_t sg[G];
      uint64_t vg[G], sum = 0, mn = 0, mx = 0;
      bool own = true;
      const uint32_t first = __shfl_sync(0xffffffffu, s[j], 0);
#pragma unroll
      for (int q = 0; q < G; ++q) {
        sg[q] = s[j + q];
        vg[q] = v[j + q];
        own &= sg[q] == first;
        sum += vg[q];
        const uint64_t a = vg[q] ^ MIN_FLIP, b = vg[q] ^ MAX_FLIP;
        mn = mn > a ? mn : a;
        mx = mx > b ? mx : b;
      }
      // (rows without a slot are on a spare one, another in each lane)
      if (!__all_sync(0xffffffffu, own)) {
        add(sg, vg);
        continue;
      }
      sum = warp_sum(sum) + 32 * G * SUM_BIAS;
      if constexpr (NA == 4) {
        mn = warp_max(mn);
        mx = warp_max(mx);
      }
      if ((threadIdx.x & 31) == 0) {
        const uint32_t old = atoms_add(lo + 4 * first, (uint32_t)sum);
        reds_add(cnt + 4 * first, 32 * G);
        if constexpr (NA == 4) {
          uint64_t a, b;
          lds128(mm + 16 * first, a, b);
          reds_raise64(mm + 16 * first, mn, a);
          reds_raise64(mm + 16 * first + 8, mx, b);
        }
        reds_add_nz(hi + 4 * first, high_with_carry(old, sum));
      }
      __syncwarp();
    }
  }

  // The encoded words of a slot (after a barrier behind the adds).
  __device__ __forceinline__ void words(uint32_t s, uint64_t (&w)[NA]) const {
    const uint32_t c = lds32(cnt + 4 * s);
    w[0] = ((uint64_t)lds32(hi + 4 * s) << 32 | lds32(lo + 4 * s)) - (uint64_t)c * SUM_BIAS;
    w[1] = c;
    if constexpr (NA == 4) lds128(mm + 16 * s, w[2], w[3]);
  }
  __device__ __forceinline__ void clear_slot(uint32_t s) const {
    sts64(key + 8 * s, 0);
    sts32(lo + 4 * s, 0);
    sts32(hi + 4 * s, 0);
    sts32(cnt + 4 * s, 0);
    if constexpr (NA == 4) {
      sts64(mm + 16 * s, 0);
      sts64(mm + 16 * s + 8, 0);
    }
  }
};

}  // namespace rel
