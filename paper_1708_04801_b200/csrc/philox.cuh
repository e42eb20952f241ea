// Sample-index stream of the chains: Philox4x32-10 (Salmon, Moraes, Dror, Shaw, SC'11), written
// from the published definition, and the kernel that materialises each node's stream.
//
// Stands for Algorithm 1's "randomly shuffle the data on machine i; get the n-th example": the
// n-th example (1-based) of node j is row floor(u * m_j / 2^32) of its shard, u being output word
// (n-1)&3 of the block with counter ((n-1)>>2 low, (n-1)>>2 high, j, 0) and key (seed low, seed high).
#pragma once

#include "common.cuh"

namespace wpsgd {

// High 32 bits of a 32 x 32 -> 64 bit product, on the device and on the host.
__host__ __device__ __forceinline__ uint32_t mulhi32(uint32_t a, uint32_t b) {
#ifdef __CUDA_ARCH__
  return __umulhi(a, b);
#else
  return (uint32_t)(((unsigned long long)a * (unsigned long long)b) >> 32);
#endif
}

__host__ __device__ __forceinline__ uint4 philox4x32_10(uint4 c, uint32_t k0, uint32_t k1) {
#pragma unroll
  for (int i = 0; i < 10; ++i) {
    const uint32_t hi0 = mulhi32(0xD2511F53u, c.x), lo0 = 0xD2511F53u * c.x;
    const uint32_t hi1 = mulhi32(0xCD9E8D57u, c.z), lo1 = 0xCD9E8D57u * c.z;
    c = make_uint4(hi1 ^ c.y ^ k0, lo1, hi0 ^ c.w ^ k1, lo0);
    k0 += 0x9E3779B9u;
    k1 += 0xBB67AE85u;
  }
  return c;
}

// ---- shuffled order: one keyed permutation of the shard per node, cycled (Algorithm 1 read literally: "randomly
// shuffle the data on machine i", then "get the n-th example") -------------------------------------------------
// The n-th example is row pi((n-1) mod m). pi is a 4-round balanced Feistel network on 2w bits (2w = the even
// bit count >= 2 covering m-1) with cycle walking; round keys = the Philox block at counter (0, 0, node, 1);
// round function = a 32-bit multiply / xor-shift mixer masked to w bits.
__host__ __device__ __forceinline__ uint32_t mix_round(uint32_t x, uint32_t key) {
  uint32_t h = x ^ key;
  h *= 0x85EBCA6Bu;
  h ^= h >> 13;
  h *= 0xC2B2AE35u;
  h ^= h >> 16;
  return h;
}

__host__ __device__ __forceinline__ uint32_t shuffled_row(const uint4& keys, long long step0 /*0-based*/, uint32_t m) {
  if (m <= 1u) return 0u;
  int bits = 0;  // smallest bits with 2^bits >= m (m >= 2)
  while (bits < 32 && ((m - 1u) >> bits) != 0u) ++bits;
  if (bits < 2) bits = 2;
  if (bits & 1) ++bits;
  const int w = bits >> 1;
  const uint32_t mask = (w == 16) ? 0xFFFFu : ((1u << w) - 1u);
  const uint32_t kk[4] = {keys.x, keys.y, keys.z, keys.w};
  unsigned long long x = (unsigned long long)(step0 % (long long)m);
  // Every pass is a bijection of [0, 2^bits), so walking from a value below m returns below m; 2^bits < 4m, and
  // the expected number of passes is below 4. The loop bound only guards against a broken invariant.
  for (int guard = 0; guard < (1 << 20); ++guard) {
    uint32_t L = (uint32_t)(x >> w), R = (uint32_t)x & mask;
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const uint32_t t = (L ^ mix_round(R, kk[i])) & mask;
      L = R;
      R = t;
    }
    x = ((unsigned long long)L << w) | R;
    if (x < m) break;
  }
  return (uint32_t)(x < m ? x : 0ull);
}

// Row of step s + 1 of node j in a shard of m rows.
__host__ __device__ __forceinline__ uint32_t drawn_row(uint64_t seed, uint32_t j, long long s, uint32_t m) {
  const unsigned long long q = (unsigned long long)s >> 2;
  const uint4 o = philox4x32_10(make_uint4((uint32_t)q, (uint32_t)(q >> 32), j, 0u), (uint32_t)seed, (uint32_t)(seed >> 32));
  const int e = (int)(s & 3);
  return mulhi32(e == 0 ? o.x : (e == 1 ? o.y : (e == 2 ? o.z : o.w)), m);  // floor(u m / 2^32)
}

// Entries of steps b+1 .. b+steps of node j (shard of m rows) into out[0 .. steps), and the last one's row again into
// out[steps .. cnt). sampling 0: one counter value q (four consecutive steps) per (t0 + i * stride); sampling 1: one step
// per (t0 + i * stride).
__host__ __device__ __forceinline__ void emit_indices(int sampling, uint64_t seed, uint32_t j, long long b, long long steps, long long cnt, uint32_t m,
                                             uint32_t* __restrict__ out, long long t0, long long stride) {
  if (sampling == 1) {
    const uint4 keys = philox4x32_10(make_uint4(0u, 0u, j, 1u), (uint32_t)seed, (uint32_t)(seed >> 32));
    for (long long i = t0; i < cnt; i += stride) out[i] = shuffled_row(keys, b + (i < steps ? i : steps - 1), m);
    return;
  }
  const long long q_lo = b >> 2, q_hi = (b + steps - 1) >> 2;  // zero-based step s = n-1 lies in [b, b+steps)
  for (long long q = q_lo + t0; q <= q_hi; q += stride) {
    const uint4 o = philox4x32_10(make_uint4((uint32_t)q, (uint32_t)((unsigned long long)q >> 32), j, 0u),
                                  (uint32_t)seed, (uint32_t)(seed >> 32));
    const uint32_t w[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const long long s = (q << 2) + e;
      if (s >= b && s < b + steps) out[s - b] = mulhi32(w[e], m);  // floor(u m / 2^32)
    }
  }
  const long long t1 = stride - 1 - t0;  // the threads with the least to do above
  if (t1 < cnt - steps) {
    const uint32_t last = drawn_row(seed, j, b + steps - 1, m);
    for (long long i = steps + t1; i < cnt; i += stride) out[i] = last;
  }
}

// Per-node tables of a launch, one after the other in one buffer (built on the host, read by the kernels).
struct TableLayout {
  size_t shard_off, steps, first, idx_off, order, ids, total;
  __host__ __device__ explicit TableLayout(int k) {
    const size_t n = (size_t)k;
    shard_off = 0;                                     // [k+1] row offsets
    steps = shard_off + (n + 1) * sizeof(long long);   // [k] steps of this launch
    first = steps + n * sizeof(long long);             // [k] steps already run
    idx_off = first + n * sizeof(long long);           // [k+1] position of the node's stream: prefix sums of stream_entries
    order = idx_off + (n + 1) * sizeof(long long);     // [k+8] nodes, longest chain first, then -1
    ids = order + (n + 8) * sizeof(int);               // [k] node numbers that enter the counter
    total = (ids + n * sizeof(int) + 15) / 16 * 16;
  }
};
// The stream of a node is filled up to the next multiple of 64 steps with the row of its last step, so that kernels that take
// samples in groups always read valid rows, and only rows that the chain has visited: what fills a group up has the weight
// zero, but zero times a value that is not finite would reach the model.
__host__ __device__ __forceinline__ long long stream_entries(long long steps) { return (steps + 63) / 64 * 64; }

// Tables small enough travel as a kernel argument: no copy is enqueued for them.
template <int BYTES>
struct InlineTables {
  alignas(16) unsigned char b[BYTES];
};

// All nodes' streams for one launch of the chains. Node = blockIdx.y (+ gridDim.y per pass). BYTES > 0: the tables are the
// argument `t`, and block (0, 0) writes them to `tables` for the kernels that follow. What is written is read by chain kernels only, and
// those let the kernel after them start when their last block has ended (they do not call kernel_started): whoever read the
// old tables and streams is done when this kernel starts. So nothing has to be waited for first, and the streams are formed while
// the kernels before are still at work; the wait stands at the end (a kernel's completion implies that of all before it).
// `wait_first`: a stream kernel before this one was not followed by chains and may still be writing. 16 rounds of combine, set
// models, stream and short chains, squared loss: 32 x 512 fp32 369 -> 342 us; logistic, 100 x 200: 424 -> 388.
template <int BYTES>
__global__ void __launch_bounds__(256) index_stream_kernel(const __grid_constant__ InlineTables<(BYTES > 0 ? BYTES : 16)> t, int wait_first, int sampling,
                                                           uint64_t seed, int k, unsigned char* __restrict__ tables,
                                                           uint32_t* __restrict__ idx) {
  kernel_started();
  if (BYTES == 0 || wait_first) kernel_inputs_ready();
  const TableLayout L(k);
  const unsigned char* src = BYTES > 0 ? t.b : tables;
  if (BYTES > 0 && blockIdx.x == 0 && blockIdx.y == 0)
    for (size_t i = threadIdx.x; i < L.total / 16; i += blockDim.x) ((uint4*)tables)[i] = ((const uint4*)t.b)[i];
  const long long *off = (const long long*)(src + L.shard_off), *steps = (const long long*)(src + L.steps),
                  *first = (const long long*)(src + L.first), *idx_off = (const long long*)(src + L.idx_off);
  const int* ids = (const int*)(src + L.ids);
  for (int j = blockIdx.y; j < k; j += gridDim.y) {
    const long long cnt = stream_entries(steps[j]);
    if (cnt <= 0) continue;
    emit_indices(sampling, seed, (uint32_t)ids[j], first[j], steps[j], cnt, (uint32_t)(off[j + 1] - off[j]), idx + idx_off[j],
                 (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
  }
  kernel_inputs_ready();
}

// One node's stream, for callers that want to look at it.
__global__ void index_single_kernel(int sampling, uint64_t seed, int node, long long m, long long n_begin,
                                    long long count, uint32_t* __restrict__ out) {
  kernel_started();
  kernel_inputs_ready();
  if (count > 0)
    emit_indices(sampling, seed, (uint32_t)node, n_begin, count, count, (uint32_t)m, out,
                 (long long)blockIdx.x * blockDim.x + threadIdx.x, (long long)gridDim.x * blockDim.x);
}

}  // namespace wpsgd
