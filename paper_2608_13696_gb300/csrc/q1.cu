// The fused filter + product-form aggregation (ShapeQ1: keep lo <= date <= hi,
// key = two uint8 columns, sum(a), sum(b), sum(b * f0(d)), sum(b * f0(d) *
// f1(t)), count) with all groups pinned: a handful of groups over a fact table.
//
// HBM bounds it (38 bytes a row).  The staged kernel reached 59 % of the copy
// rate: its staging ring and 64-bit thread-private words left room for one
// 9-warp CTA per SM, too few to cover the words' read-add-write chains.  Here
// a thread loads four consecutive rows of every column straight to registers
// (11 loads in flight), and shared memory holds nothing but the words -- for
// each pinned group four 64-bit sums and a 32-bit count per thread, one column
// of words per thread, so no atomics and no bank conflicts -- which lets 24
// warps stay resident with eight groups.  Shared atomics instead of private
// words would meet on the few groups' slots (about 70 cycles a warp row
// against 20).  1e8 rows, 6 groups: 0.956 -> 0.537 ms (7.08 TB/s, the rate
// of a plain copy).
#include "groupby.cuh"

namespace rel {

namespace {

constexpr int Q1_U = 4;       // consecutive rows per thread
constexpr int Q1_MAX_HOT = 8;
constexpr int Q1_WORDS = 4;   // 64-bit sums; the count is a 32-bit word
// lookup[32] | keys[8] | reduced words[8][5], then the thread-private words
constexpr int Q1_HEAD = 4 * TINY_MAX_SLOTS + 8 * Q1_MAX_HOT + 8 * Q1_MAX_HOT * (Q1_WORDS + 1);

__host__ __device__ inline size_t q1_smem(int n_hot, int block) {
  return Q1_HEAD + (size_t)n_hot * block * (8 * Q1_WORDS + 4);
}

__device__ __forceinline__ void q1_global(const GbParams& p, uint64_t ek, const uint64_t (&w)[5]) {
  const uint64_t mask = (1ull << p.log2_slots) - 1;
  uint64_t s = slot_of(ek, p.log2_slots);
  for (uint32_t i = 0; i < p.max_probe; ++i) {
    uint64_t k = ld_relaxed(p.tkeys + s);
    if (k == 0) {
      k = atomicCAS((unsigned long long*)(p.tkeys + s), 0ull, (unsigned long long)ek);
      if (k == 0) k = ek;
    }
    if (k == ek) {
#pragma unroll
      for (int a = 0; a < 5; ++a) redg_add(p.taggs + s * 5 + a, w[a]);
      return;
    }
    s = (s + 1) & mask;
    if ((i & 31) == 31 && ld_relaxed_u32(&p.hdr->overflow)) return;  // already overflowed
  }
  atomicOr(&p.hdr->overflow, 1u);
}

// A kept row whose key the plan did not pin (the sample missed it).
__device__ __noinline__ void q1_rare(const GbParams& p, uint32_t key, uint64_t a, uint64_t b,
                                     uint64_t dp, uint64_t dt) {
  const uint64_t w[5] = {a, b, dp, dt, 1};
  q1_global(p, (uint64_t)key ^ KEY_FLIP, w);
}

__global__ void __launch_bounds__(1024, 1) gb_q1_k(const __grid_constant__ GbParams p, int n_hot) {
  extern __shared__ __align__(16) uint8_t sm[];
  uint32_t* look = (uint32_t*)sm;  // by hash slot: key | dense id << 16, or ~0
  uint64_t* hk = (uint64_t*)(sm + 4 * TINY_MAX_SLOTS);
  uint64_t* red = hk + Q1_MAX_HOT;
  const int B = blockDim.x, tid = threadIdx.x;
  uint64_t* acc = (uint64_t*)(sm + Q1_HEAD);               // [group][word][thread]
  uint32_t* cnt = (uint32_t*)(acc + (size_t)n_hot * Q1_WORDS * B);  // [group][thread]
  if (tid < TINY_MAX_SLOTS) {
    const uint64_t k = tid < (int)p.tiny_slots ? p.tiny_init[tid] : 0;
    const unsigned occ = __ballot_sync(0xffffffffu, k != 0);
    const int d = __popc(occ & ((1u << tid) - 1u));
    // a pinned key beyond 16 bits matches no row
    look[tid] = k != 0 && (k ^ KEY_FLIP) < 65536 ? (uint32_t)(k ^ KEY_FLIP) | (uint32_t)d << 16 : ~0u;
    if (k != 0) hk[d] = k;
  }
  for (int g = 0; g < n_hot; ++g) {
#pragma unroll
    for (int a = 0; a < Q1_WORDS; ++a) acc[(g * Q1_WORDS + a) * B + tid] = 0;
    cnt[g * B + tid] = 0;
  }
  __syncthreads();
  const int32_t* cd = (const int32_t*)p.col[p.r_pred];
  const uint8_t *c0 = p.col[p.r_k0], *c1 = p.col[p.r_k1];
  const int64_t *ca = (const int64_t*)p.col[p.r_a], *cb = (const int64_t*)p.col[p.r_b];
  const int64_t *cx = (const int64_t*)p.col[p.r_d], *ct = (const int64_t*)p.col[p.r_t];
  const int64_t lo = p.pred_lo[0], hi = p.pred_hi[0];
  const uint64_t k0 = (uint64_t)p.ac[2][0], s0 = (uint64_t)p.as[2][0];
  const uint64_t k1 = (uint64_t)p.ac[3][1], s1 = (uint64_t)p.as[3][1];
  const uint32_t tmask = p.tiny_slots - 1;
  const bool aligned = (((uintptr_t)cd | (uintptr_t)ca | (uintptr_t)cb | (uintptr_t)cx | (uintptr_t)ct) % 16 |
                        ((uintptr_t)c0 | (uintptr_t)c1) % 4) == 0;
  const int64_t CHUNK = (int64_t)B * Q1_U, n = p.n_rows;
  for (int64_t base = (int64_t)blockIdx.x * CHUNK; base < n; base += (int64_t)gridDim.x * CHUNK) {
    const int64_t r = base + Q1_U * tid;
    int32_t dt[Q1_U];
    uint32_t f0 = 0, f1 = 0, keep = 0;
    uint64_t a[Q1_U], b[Q1_U], x[Q1_U], t[Q1_U];
    if (aligned && base + CHUNK <= n) {
      const int4 d = __ldcs((const int4*)(cd + r));
      f0 = __ldcs((const unsigned int*)(c0 + r));
      f1 = __ldcs((const unsigned int*)(c1 + r));
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const longlong2 va = __ldcs((const longlong2*)(ca + r) + h), vb = __ldcs((const longlong2*)(cb + r) + h);
        const longlong2 vx = __ldcs((const longlong2*)(cx + r) + h), vt = __ldcs((const longlong2*)(ct + r) + h);
        a[2 * h] = va.x; a[2 * h + 1] = va.y;
        b[2 * h] = vb.x; b[2 * h + 1] = vb.y;
        x[2 * h] = vx.x; x[2 * h + 1] = vx.y;
        t[2 * h] = vt.x; t[2 * h + 1] = vt.y;
      }
      dt[0] = d.x; dt[1] = d.y; dt[2] = d.z; dt[3] = d.w;
      keep = (1u << Q1_U) - 1;
    } else {
#pragma unroll
      for (int j = 0; j < Q1_U; ++j) {
        const bool in = r + j < n;
        dt[j] = in ? cd[r + j] : 0;
        f0 |= (in ? (uint32_t)c0[r + j] : 0u) << (8 * j);
        f1 |= (in ? (uint32_t)c1[r + j] : 0u) << (8 * j);
        a[j] = in ? (uint64_t)ca[r + j] : 0;
        b[j] = in ? (uint64_t)cb[r + j] : 0;
        x[j] = in ? (uint64_t)cx[r + j] : 0;
        t[j] = in ? (uint64_t)ct[r + j] : 0;
        keep |= (in ? 1u : 0u) << j;
      }
    }
    // two 16-bit keys per word: (first column << 8) | second
    const uint32_t kw[2] = {__byte_perm(f1, f0, 0x5140), __byte_perm(f1, f0, 0x7362)};
    uint32_t key[Q1_U], l[Q1_U];
#pragma unroll
    for (int j = 0; j < Q1_U; ++j) {
      if ((int64_t)dt[j] < lo || (int64_t)dt[j] > hi) keep &= ~(1u << j);
      key[j] = (kw[j / 2] >> (16 * (j & 1))) & 0xFFFFu;
      l[j] = look[small_slot_of((uint64_t)key[j] ^ KEY_FLIP, tmask, p.tiny_mult)];
    }
#pragma unroll
    for (int j = 0; j < Q1_U; ++j) {
      if (!(keep >> j & 1)) continue;
      const uint64_t dp = b[j] * (k0 + s0 * x[j]), dq = dp * (k1 + s1 * t[j]);
      if ((l[j] & 0xFFFFu) != key[j] || l[j] == ~0u) {
        q1_rare(p, key[j], a[j], b[j], dp, dq);
        continue;
      }
      const uint32_t g = l[j] >> 16;
      uint64_t* w = acc + (size_t)g * Q1_WORDS * B + tid;
      uint32_t* c = cnt + g * B + tid;
      const uint64_t w0 = w[0], w1 = w[B], w2 = w[2 * B], w3 = w[3 * B];
      const uint32_t n0 = *c;
      w[0] = w0 + a[j];
      w[B] = w1 + b[j];
      w[2 * B] = w2 + dp;
      w[3 * B] = w3 + dq;
      *c = n0 + 1;
    }
  }
  __syncthreads();
  // one warp per (group, word): the threads' words summed, then the groups
  const int warp = tid >> 5, lane = tid & 31;
  for (int q = warp; q < n_hot * (Q1_WORDS + 1); q += B / 32) {
    const int g = q / (Q1_WORDS + 1), a = q % (Q1_WORDS + 1);
    uint64_t v = 0;
    for (int i = lane; i < B; i += 32)
      v += a < Q1_WORDS ? acc[(size_t)(g * Q1_WORDS + a) * B + i] : (uint64_t)cnt[g * B + i];
#pragma unroll
    for (int o = 16; o; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
    if (lane == 0) red[q] = v;
  }
  __syncthreads();
  if (tid < n_hot && red[tid * 5 + 4] != 0) {
    const uint64_t w[5] = {red[tid * 5], red[tid * 5 + 1], red[tid * 5 + 2], red[tid * 5 + 3],
                           red[tid * 5 + 4]};
    q1_global(p, hk[tid], w);
  }
}

}  // namespace

bool gb_q1_eligible(const GbParams& p, int n_hot) {
  // counts are 32 bits per thread, which sees its CTA's share of the rows: at
  // this limit no more than 2^40 / (SMs x 128), far below 2^32
  return p.tiny_frozen && p.tiny_slots <= TINY_MAX_SLOTS && n_hot >= 1 && n_hot <= Q1_MAX_HOT &&
         p.smem_slots == 0 && p.n_rows < (1ll << 40);
}

rel_status gb_launch_q1(const GbParams& p, int n_hot, cudaStream_t st) {
  if (p.n_rows == 0) return REL_OK;
  // one CTA per SM, whose words leave 70 KB of the SM's 256 to L1: the columns
  // stream through it (1e8 rows: 768 threads 0.537 ms; 1024, or 512 in two
  // CTAs, with 30 KB of L1 0.70); small inputs in small CTAs, so that more SMs take part
  int block = p.n_rows > (int64_t)relhost::device_sms() * 4096 ? 768 : 256;
  while (block > 128 && q1_smem(n_hot, block) > 184 * 1024) block -= 128;
  const size_t smem = q1_smem(n_hot, block);
  cudaError_t e = relhost::allow_smem(gb_q1_k);
  if (e != cudaSuccess) return relhost::cuda_fail(e, "cudaFuncSetAttribute(fused)");
  int occ = 0;
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, gb_q1_k, block, smem);
  if (e != cudaSuccess || occ < 1) return relhost::cuda_fail(e, "occupancy(fused)");
  const int64_t chunk = (int64_t)block * Q1_U, chunks = (p.n_rows + chunk - 1) / chunk;
  int64_t grid = (int64_t)relhost::device_sms() * occ;
  if (grid > chunks) grid = chunks;
  relhost::launch_begin(relhost::K_GB_LAYERED, st);
  gb_q1_k<<<(int)grid, block, smem, st>>>(p, n_hot);
  relhost::launch_end(relhost::K_GB_LAYERED, st);
  e = cudaGetLastError();
  return e == cudaSuccess ? REL_OK : relhost::cuda_fail(e, "launch(fused)");
}

}  // namespace rel
