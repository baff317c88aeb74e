// Hash equi-join kernels for sm_103a: build, count and probe.
//
// The paper's join runs three kernels over a hash table that is read
// randomly: insert (build), count (size the output) and retrieve (emit the
// matches), with the payload brought in by a separate gather (Sec. 7,
// Table 9), and finds count and retrieve bound by instruction issue and
// memory latency on GH200.  Here the table is an open-addressing array at
// load <= 1/2 of 16-byte slots (key, build row index) plus the table's own
// copy of the payload column -- 32 MB + 8 MB for a 10^6-row build side, small
// enough to stay in the GB300's L2 (whose random-access sweet spot is below
// ~64 MB) while the probe keys stream from HBM with evict-first loads and the
// outputs leave with streaming stores.  The payload gather is fused into the
// probe.  Slots come in pairs that fill one 32-byte sector: a key's sequence
// starts at its home pair and one 256-bit load shows both slots, so nine of
// ten unique keys (load 0.48) are decided by their first load; the others
// are finished in one loop per four rows, each lane on its own next row.
#include "join.cuh"

namespace rel {

namespace {

constexpr int J_BLOCK = 256;

// A pair of slots: keys a and b, build rows x and y.  Marked evict-last in L2
// so that the table outlives the streamed probe keys (evict-first) and the
// streamed outputs.
struct Pair {
  uint64_t a, b;
  int32_t x, y;
};
__device__ __forceinline__ Pair ld_pair(const JoinSlot* p, uint64_t pol) {
  unsigned long long k0, v0, k1, v1;
  asm volatile("ld.global.L2::cache_hint.v4.u64 {%0, %1, %2, %3}, [%4], %5;"
               : "=l"(k0), "=l"(v0), "=l"(k1), "=l"(v1)
               : "l"(p), "l"(pol));
  return Pair{k0, k1, (int32_t)(uint32_t)v0, (int32_t)(uint32_t)v1};
}
__device__ __forceinline__ uint64_t home_pair(uint64_t ek, int log2_slots) {
  return slot_of(ek, log2_slots) & ~1ull;
}

// Every build row claims the first empty slot from its home pair on, after a
// look at the pair: a claim that fails costs more than a look, above all in a
// table beyond L2 or with repeated keys (whole calls on 5e6 rows, each key three
// times: claims first 568 us, one slot a look 400, a pair 307; 10^6 different
// keys 71, 75, 68, the kernel 48 -> 45).  Bound by the latency of the claims.
__global__ void __launch_bounds__(J_BLOCK) join_build_k(const __grid_constant__ JoinParams p,
                                                        const int64_t* __restrict__ keys,
                                                        const int64_t* __restrict__ payload,
                                                        int64_t n) {
  const uint64_t mask = (1ull << p.log2_slots) - 1;
  bool dup = false;
  for (int64_t j = (int64_t)blockIdx.x * J_BLOCK + threadIdx.x; j < n;
       j += (int64_t)gridDim.x * J_BLOCK) {
    const uint64_t ek = (uint64_t)__ldcs((const long long*)keys + j) ^ KEY_FLIP;
    const long long pay = __ldcs((const long long*)payload + j);
    p.pay[j] = pay;  // the table's copy of the payload column
    if (ek == 0) {   // INT64_MIN: side list
      p.side[atomicAdd(&p.hdr->n_side, 1ull)] = JoinVal{pay, (int32_t)j, 0};
      continue;
    }
    // Two inserts of one key walk the same slots and claim them in order, so
    // the later one always meets the earlier one's: duplicates are always
    // noticed.
    uint64_t s = home_pair(ek, p.log2_slots);
    unsigned long long cur = 1;
    for (uint64_t i = 0; cur != 0 && i <= mask; i += 2) {
      uint64_t k[4];  // key, row, key, row
      ld_sector((const uint64_t*)(p.slots + s), k);
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        if (cur == 0) continue;
        cur = k[2 * q];
        if (cur == 0) cur = atomicCAS(&p.slots[s + q].ek, 0ull, (unsigned long long)ek);
        if (cur == 0) p.slots[s + q].bidx = (int32_t)j;
        dup |= cur == ek;
      }
      s = (s + 2) & mask;
    }
    if (cur != 0) atomicOr(&p.hdr->overflow, 1u);
  }
  if (dup) atomicOr(&p.hdr->dups, 1u);
}

constexpr int J_FLUSH = 256;             // matches of a warp that are written at once
constexpr int J_BUF = J_FLUSH + 32 * 4;  // ... and room for one more round
constexpr int J_CTAS = 4;

// Probe U rows per thread.
//  * Unique build keys (no duplicate seen while building): a row is done at its
//    first match, all of them in one round.
//  * Otherwise a row's sequence is walked to its first empty slot, all U rows a
//    pair further per round.
//  * Rows with key INT64_MIN walk the side list.
// A warp collects its matches (probe row, build row) in shared memory and, from
// J_FLUSH on, reserves the output with one atomic -- all warps take them from
// one address, which serves 1.6 G/s: one per 128 rows was 78 us of a 16e6-row
// probe -- gathers the payloads and writes all three columns densely.
// 16e6 rows into 10^6 keys, 90 % found: 241 -> 202 us, counting 156 -> 124;
// 400 009 rows into 60 013 keys three times each: 119 -> 41, counting 102 -> 24.
// Bound by instruction issue (half of the slots) and by the lookups that go on
// past the home pair, which hold up their warps.
template <bool EMIT, int U>
__global__ void __launch_bounds__(J_BLOCK, J_CTAS) join_probe_k(const __grid_constant__ JoinParams p,
                                                                const __grid_constant__ JoinOut o,
                                                                const int64_t* __restrict__ probe,
                                                                int64_t n) {
  __shared__ int2 bufs[EMIT ? J_BLOCK / 32 : 1][EMIT ? J_BUF : 1];
  int2* buf = bufs[EMIT ? threadIdx.x / 32 : 0];
  unsigned fill = 0;
  const int lane = threadIdx.x & 31;
  const unsigned lt = (1u << lane) - 1u;
  const uint64_t mask = (1ull << p.log2_slots) - 1;
  const bool unique = ld_relaxed_u32(&p.hdr->dups) == 0;
  const uint64_t n_side = p.hdr->n_side, cap = (uint64_t)o.capacity;
  const uint64_t pol = l2_evict_last_policy();
  const bool vec = (uintptr_t)probe % 16 == 0;
  unsigned long long counted = 0;
  constexpr int64_t TILE = (int64_t)J_BLOCK * U;
  // row of slot j
  auto row = [&](int64_t base, int j) -> int64_t {
    return U == 1 ? base + threadIdx.x : base + (j / 2) * 2 * J_BLOCK + 2 * threadIdx.x + (j & 1);
  };
  auto push = [&](bool h, int64_t r, int32_t b) {
    const unsigned v = __ballot_sync(0xffffffffu, h);
    if (h) buf[fill + __popc(v & lt)] = make_int2((int32_t)r, b);
    fill += __popc(v);
  };
  auto flush = [&]() {  // the warp converged; streaming stores keep the table in L2
    __syncwarp();
    unsigned long long wb = 0;
    if (lane == 0) wb = atomicAdd(&p.hdr->n_out, (unsigned long long)fill);
    wb = __shfl_sync(0xffffffffu, wb, 0);
    const unsigned room = wb >= cap ? 0 : cap - wb < fill ? (unsigned)(cap - wb) : fill;
    for (unsigned i = lane; i < room; i += 32 * 2) {
      int2 e[2];
      long long pay[2];
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (i + 32 * q < room) {
          e[q] = buf[i + 32 * q];
          pay[q] = __ldg(p.pay + e[q].y);
        }
#pragma unroll
      for (int q = 0; q < 2; ++q)
        if (i + 32 * q < room) {
          __stcs(o.probe_idx + wb + i + 32 * q, e[q].x);
          __stcs(o.build_idx + wb + i + 32 * q, e[q].y);
          __stcs((long long*)o.payload + wb + i + 32 * q, pay[q]);
        }
    }
    fill = 0;
    __syncwarp();
  };
  for (int64_t base = (int64_t)blockIdx.x * TILE; base < n; base += (int64_t)gridDim.x * TILE) {
    uint64_t ek[U], s[U];
    uint32_t side = 0;
    if (U > 1 && vec && base + TILE <= n) {
#pragma unroll
      for (int j = 0; j < U; j += 2) {
        const longlong2 kk = __ldcs((const longlong2*)(probe + row(base, j)));
        ek[j] = (uint64_t)kk.x ^ KEY_FLIP;
        ek[j + (U > 1)] = (uint64_t)kk.y ^ KEY_FLIP;
      }
#pragma unroll
      for (int j = 0; j < U; ++j) side |= (ek[j] == 0 ? 1u : 0u) << j;
    } else {
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const bool in = row(base, j) < n;
        ek[j] = in ? (uint64_t)__ldcs((const long long*)probe + row(base, j)) ^ KEY_FLIP : 0;
        side |= (in && ek[j] == 0 ? 1u : 0u) << j;
      }
    }
    uint32_t live = 0;
#pragma unroll
    for (int j = 0; j < U; ++j) {
      s[j] = home_pair(ek[j], p.log2_slots);
      live |= (ek[j] != 0 ? 1u : 0u) << j;
    }
    uint64_t walked = 0;
    do {
      Pair q[U];
      uint32_t m = 0;  // bit j: slot a of row j matches; bit 8 + j: slot b
#pragma unroll
      for (int j = 0; j < U; ++j)
        if (unique || (live >> j & 1)) q[j] = ld_pair(p.slots + s[j], pol);
#pragma unroll
      for (int j = 0; j < U; ++j) {
        if (!(live >> j & 1)) continue;
        m |= (q[j].a == ek[j] ? 1u : 0u) << j | (q[j].b == ek[j] ? 256u : 0u) << j;
        if (q[j].b == 0) live ^= 1u << j;  // an empty slot ends the sequence
        s[j] = (s[j] + 2) & mask;
      }
      if (unique) {
        live &= ~(m | m >> 8);
        // what the first pair did not decide: each lane on its own next row
        for (uint64_t i = 0; live && i <= U * mask; i += 2) {
          const uint32_t bit = live & (0u - live);
          uint64_t k = 0, w = 0;
#pragma unroll
          for (int j = 0; j < U; ++j)
            if (bit == 1u << j) {
              k = ek[j];
              w = s[j];
            }
          const Pair r = ld_pair(p.slots + w, pol);
          const bool e0 = r.a == k, e1 = r.b == k;
#pragma unroll
          for (int j = 0; j < U; ++j)
            if (bit == 1u << j) {
              s[j] = (w + 2) & mask;
              q[j].x = r.x;
              q[j].y = r.y;
            }
          m |= (e0 ? bit : 0u) | (e1 ? bit << 8 : 0u);
          if (e0 || e1 || r.b == 0) live ^= bit;
        }
        __syncwarp();
      }
      if (EMIT) {
#pragma unroll
        for (int j = 0; j < U; ++j) {
          const bool x = m >> j & 1, y = m >> (8 + j) & 1;
          push(x || (unique && y), row(base, j), x ? q[j].x : q[j].y);
          if (!unique) push(y, row(base, j), q[j].y);
        }
        if (fill >= J_FLUSH) flush();
      } else {
        counted += __popc(m);
      }
    } while (__any_sync(0xffffffffu, live != 0) && (walked += 2) <= mask);
    // INT64_MIN rows: every build row of the side list
    if (__any_sync(0xffffffffu, side != 0)) {
#pragma unroll
      for (int j = 0; j < U; ++j) {
        const unsigned m = __ballot_sync(0xffffffffu, side >> j & 1);
        if (!m) continue;
        if constexpr (!EMIT) {
          counted += side >> j & 1 ? n_side : 0;
        } else {
          for (uint64_t i = 0; i < n_side; ++i) {
            unsigned long long wb = 0;
            if (lane == 0) wb = atomicAdd(&p.hdr->n_out, (unsigned long long)__popc(m));
            wb = __shfl_sync(0xffffffffu, wb, 0) + __popc(m & lt);
            const JoinVal v = p.side[i];
            if ((side >> j & 1) && wb < cap) {
              o.probe_idx[wb] = (int32_t)row(base, j);
              o.build_idx[wb] = v.bidx;
              o.payload[wb] = v.payload;
            }
          }
        }
      }
    }
  }
  if (EMIT && fill) flush();
  if (!EMIT) {
#pragma unroll
    for (int off = 16; off; off >>= 1) counted += __shfl_xor_sync(0xffffffffu, counted, off);
    if (lane == 0 && counted) atomicAdd(&p.hdr->aux, counted);
  }
}

int grid_for(int64_t n, int per_sm_hint) {
  int64_t g = (n + J_BLOCK - 1) / J_BLOCK;
  const int64_t cap = (int64_t)relhost::device_sms() * per_sm_hint;
  if (g > cap) g = cap;
  return (int)(g < 1 ? 1 : g);
}

}  // namespace

rel_status join_launch_build(const JoinParams& p, const int64_t* keys, const int64_t* payload,
                             int64_t n, cudaStream_t st) {
  if (n == 0) return REL_OK;
  relhost::launch_begin(relhost::K_JOIN_BUILD, st);
  join_build_k<<<grid_for(n, 8), J_BLOCK, 0, st>>>(p, keys, payload, n);
  relhost::launch_end(relhost::K_JOIN_BUILD, st);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "launch(join build)");
}

rel_status join_launch_probe(const JoinParams& p, const JoinOut& o, const int64_t* probe,
                             int64_t n, bool emit, cudaStream_t st) {
  if (n == 0) return REL_OK;
  const int id = emit ? relhost::K_JOIN_PROBE : relhost::K_JOIN_COUNT;
  // one wave of resident CTAs, each walking the tiles: a second, partial
  // wave would leave most SMs idle at the end
  // rows per thread: 1 while the rows do not fill the chip, whose warps then
  // hold one lookup each (1e6 rows: 19 us against 24); above, 2 (4: spills or
  // two CTAs per SM, 220 - 290 us against 202 for 16e6 rows)
  const int u = n <= (int64_t)relhost::device_sms() * J_CTAS * J_BLOCK * 4 ? 1 : 2;
  auto kern = emit ? (u == 1 ? join_probe_k<true, 1> : join_probe_k<true, 2>)
                   : (u == 1 ? join_probe_k<false, 1> : join_probe_k<false, 2>);
  int occ = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, kern, J_BLOCK, 0) != cudaSuccess || occ < 1)
    occ = J_CTAS;
  const int64_t tile = (int64_t)J_BLOCK * u, tiles = (n + tile - 1) / tile;
  int64_t g = (int64_t)relhost::device_sms() * occ;
  if (g > tiles) g = tiles;
  relhost::launch_begin(id, st);
  kern<<<(int)g, J_BLOCK, 0, st>>>(p, o, probe, n);
  relhost::launch_end(id, st);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "launch(join probe)");
}

}  // namespace rel
