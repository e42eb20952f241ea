// Per-node SGD chains on dense rows, blocked form with B = 8 samples per block (algebra: chain_block.cuh) and the
// margins of a block taken from the model one block back.
//
// In the plain blocked form everything between two blocks is one dependent string: update of the model, margins
// p_b = X_b w_b of the next block (a dot product over all columns, summed over warps and over the cluster), recurrence,
// gamma back to the model. Here the margins are formed from the previous model,
//     q_b = X_b w_{b-1},   C_b = X_b X_{b-1}^T,   p_b = (1 - delta_{b-1}) q_b - C_b gamma_{b-1},
// (w_b = (1 - delta_{b-1}) w_{b-1} - X_{b-1}^T gamma_{b-1}, so this is X_b w_b in exact arithmetic). C_b is an 8 x 8
// block that does not depend on the model and is formed ahead together with the Gram block G_b = X_b X_b^T. What is left
// between two recurrences is an 8 x 8 matrix-vector product on registers of the recurrence warp; update, dot products and
// the exchange of their sums run beside the recurrence of the block before. A block period is then about half of
// (recurrence + update + dot products + exchange), or the longest of the roles below, instead of their sum.
//
// Roles of the warps of a CTA (one cluster of C CTAs per node, each CTA a column slice of whole 16-byte chunks):
//   recurrence   waits for the block's sums and its q sums, steps through the 8 samples, publishes gamma
//   sums of q    (C > 1; with one CTA the recurrence warp does it) adds up the model threads' shares of q_b, sends the eight sums to
//                every CTA of the cluster, and waits on behalf of the model warps for the rows that they read next
//   copy         one or two warps that request the rows of a block (one cp.async.bulk per row, never multicast) into a ring
//                of stages
//   constants    labels and step-size factors, four blocks at a time
//   feeder       waits on the mbarriers for the Gram sums and constants of the next block, for the recurrence (in clusters of more than
//                one CTA it also adds up the CTAs' sums)
//   gram         [X_b; X_{b-1}] X_b^T over the slice: one mma.m16n8k16 per 16 columns for bf16 rows (A = the 16 rows,
//                B = the first 8 of them again), 4 x 4 register tiles on the fp32 pipes for fp32 rows. Teams of one or
//                more warps take the blocks in turn
//   model        own the model in registers: update with gamma_b, then every thread's share of q_{b+2} into shared memory
//   realign      only when rows do not start on 16-byte boundaries or end inside a chunk: the copy warp then fetches the
//                16-byte granules that hold the row's slice, and these warps shift the bytes into the ring (bytes beyond
//                the row become zero)
// Recurrence, model, sum and feeder warps, whose hand-offs are on the dependent path, meet on named barriers (about 25 cycles
// one way); everything that runs ahead meets on mbarriers (waits with cluster scope only where another CTA completes them: the
// fence costs 70 cycles). Between CTAs of a cluster only sums travel: Gram sums (512 bytes) and q sums (32 bytes) of every CTA go
// to every CTA with st.async, and each CTA runs the recurrence redundantly.
//
// Code size. The loops of all roles run at the same time and share the instruction caches, and this is what the kernel reacts to most.
// With the hot code of all roles a tenth above what the SM's cache holds, everything ran 15 to 40 % slower (16 chains of 1024
// columns: 1050 cycles per block against 890 for the same source, 0.43 M against 0.02 M instruction requests beyond the SM).
// So: compiled for one or several CTAs and for realigned or aligned rows separately (1308 -> 1067), waits with as little inlined
// code as possible, 32-bit shared-memory addresses, loops kept rolled off the dependent path. And the warps of a role share
// schedulers by role (see launch_lag): the recurrence's scheduler has only short loops beside it (1058 -> 908).
//
// Buffers. Let g be the last block whose gamma a CTA has published. Its model warps hold rows up to block g + 3 in
// registers and have freed their stages, so it can have formed Gram sums up to block g + 3 + S (ring depth S) and q sums
// up to block g + 2. Publishing gamma_g took the q sums of block g from every CTA, which those sent after their own
// gamma_{g-2}: a peer may be two blocks behind. Tables read in the same CTA therefore have S + 4 entries, Gram sums from
// peers S + 6, q sums four; the shares of q inside a CTA two (the shares of block g + 2 follow gamma_g, which took q_g).
//
// What bounds a block, and what it measured (B200, 1965 MHz; cycles per block of 8 samples, 4 chains that have their SMs to
// themselves, squared and logistic loss alike): fp32, one CTA, 16 / 32 / 64 chunks of a row 735 / 805 / 1085; eight CTAs, 32 / 64 / 128
// chunks each 845 / 1160 / 1980, 256 chunks 3615; bf16, 32 / 64 / 128 / 256 chunks 885 / 1015 / 1330 / 2205; rows that do not start on 16 bytes,
// 32 / 64 / 128 chunks about 1000 / 1480 / 2920. With few chunks it is the string gamma -> update -> shares -> sum (430) -> cluster (280) -> steps
// over two blocks, and the instruction supply; from about 64 fp32 chunks per CTA on the Gram block (shared-memory reads, 8 wavefronts
// per chunk). Before the sums of q had a warp of their own and the code was cut: 16 / 32 (eight CTAs) / 64 bf16 chunks 815 / 1235 / 1350.
// Tried and taken back: rows by 16-byte copies of the threads instead of bulk copies (1900 against 1060 at d = 64); fp32 Gram
// products split into three units of 32 with a lane per chunk (1164 against 908 at d = 64), or as 4 x 8 tiles with different
// chunks in all lanes of a load (128 chunks: 2099 against 2022); partial sums to peers by plain stores that the reader polls
// (330 cycles one way, 260 with st.async and a barrier). Rings
// of more than 8 stages are taken where there is room and gain at most 1 % (12 chains of 999 columns, rows from DRAM: 1083 -> 1074);
// 5 stages cost 8 to 80 %.
//
// Leaving. Every wait on an mbarrier is bounded. One that runs out sets the status word and a flag in every CTA of the
// cluster; from then on a warp skips these waits and runs to the end of its loop, so that named barriers are still met by
// all their warps. Nobody exits before the cluster barrier at the end.
#pragma once

#include "chain_block.cuh"
#include "chain_mma16.cuh"

namespace wpsgd {

constexpr int LAG_B = 8;
constexpr int LAG_MAX_STAGES = 16;
constexpr int LAG_MAX_RAW_STAGES = 8;
constexpr int LAG_QBUF = 4;
constexpr int LAG_SUMS = 128;        // [8][8] G, then [8][8] C (a row per sample of the block)
constexpr int LAG_MAX_MODEL_WARPS = 8;           // (vectors of 8 bytes: at most half as many)
constexpr int LAG_MAX_MODEL_WARPS_REALIGNED = 4;
constexpr int LAG_GRAM_WARPS = 4;
// Shares of q that a model warp leaves for a sample: one per thread that owns a vector of 8 bytes, half as many for one of 16, a
// quarter for two. (Wide slices need the room for their rings: with half as many for two as well, 413 to 420 chunks and one CTA had
// three stages instead of four.)
__host__ __device__ constexpr int lag_q_shares(int vb, int nc) { return vb == 8 ? 32 : (nc == 1 ? 16 : 8); }
// Entries of a row of shares (64 or 128, absent ones zero), padded
__host__ __device__ constexpr int lag_q_row(int vb, int nc, bool realign) { return vb == 16 && (nc == 2 || realign) ? 68 : 132; }
static_assert(LAG_MAX_MODEL_WARPS / 2 * lag_q_shares(8, 1) <= 128 && LAG_MAX_MODEL_WARPS * lag_q_shares(16, 1) <= 128 &&
                  LAG_MAX_MODEL_WARPS_REALIGNED * lag_q_shares(16, 1) <= 64 && LAG_MAX_MODEL_WARPS * lag_q_shares(16, 2) <= 64,
              "a row holds the shares of all model warps");
constexpr int LAG_REALIGN_WARPS = 4;
constexpr int LAG_MAX_THREADS = 512;
constexpr int LAG_GROUP = 4;         // blocks whose constants are formed together
constexpr int LAG_GROUPS = 4;        // groups in flight
// The hinge step as one saturating FMA: clamp(2^40 (1 - t)) is 1 for t < 1 and 0 from 1 on, except that it lies between the
// two (both subgradients, so is what lies between) for 1 - t below 2^-40, far below the rounding of t.
constexpr float LAG_STEP = 1099511627776.0f;
constexpr int LAG_GAM = 20;          // -gamma_0..7 and -delta, every value twice, padded to 16 bytes

struct LagParams {
  BlockParams b;
  int chunks_per_cta;          // 16-byte chunks of a row owned by one CTA
  int gram_teams, gram_warps;  // teams, warps per team
  int model_warps;
  int raw_stages;              // blocks of fetched granules ahead of the realigning warps (0: rows need none)
  int realign_warps;           // realigning warps in all,
  int realign_rows;            // of which this many share a block
  int copy_warps;              // 1 or 2
  unsigned char role[LAG_MAX_THREADS / 32];  // what each warp does: numbered as in `place`
};

// Constants of a block
struct LagConst {
  float a[8];    // squared: beta_n = a_n r_n + b_n; hinge: beta_n = a_n clamp(2^40 + b_n r_n), b_n = -2^40 sc_n; logistic: a_n f(sc_n r_n)
  float b[8];
  float sc[8];
  float na_nv, ndl_nv, sc_max, pad[5];  // minus the product of the block's factors 1 - eta lambda, minus (1 - product), largest |sc_n|
};

struct LagSmem {
  size_t row_stride, raw_stride, ring, raw, red, part, tabs, q, qpart, cst, gam, tab, jet, full, empty, rfull, rempty, gbar, tbar, qbar, cfull, cempty, flag, total;
  __host__ __device__ LagSmem(int stages, size_t slice_bytes, int C, int gram_warps_all, int raw_stages, int q_row) {
    // odd multiples of 16 bytes: tile loads of 8 (or 4) rows at the same column never meet in a bank
    row_stride = slice_bytes + 16;
    if (row_stride % 32 == 0) row_stride += 16;
    raw_stride = slice_bytes + 32;
    ring = 0;
    raw = ring + (size_t)stages * LAG_B * row_stride;
    red = raw + (size_t)raw_stages * LAG_B * raw_stride;
    part = red + (C > 1 ? (size_t)(stages + 6) * C * LAG_SUMS * sizeof(float) : 0);  // [buffer][CTA][128]
    tabs = part + 2 * (size_t)gram_warps_all * LAG_SUMS * sizeof(float);             // [parity][gram warp][128]
    q = tabs + (size_t)(stages + 4) * LAG_SUMS * sizeof(float);
    qpart = q + (C > 1 ? LAG_QBUF * 64 * sizeof(float) : 0);                         // [LAG_QBUF][CTA / 4][sample][CTA % 4]
    cst = qpart + 2 * LAG_B * (size_t)q_row * sizeof(float);                              // [2][sample][model thread]
    gam = cst + LAG_GROUPS * LAG_GROUP * sizeof(LagConst);
    tab = gam + 2 * LAG_GAM * sizeof(float);                                       // powers of 1 - eta lambda
    jet = tab + 3 * 16 * sizeof(float);
    full = jet + 8 * 4 * sizeof(float);
    empty = full + LAG_MAX_STAGES * 8;
    rfull = empty + LAG_MAX_STAGES * 8;
    rempty = rfull + LAG_MAX_RAW_STAGES * 8;
    gbar = rempty + LAG_MAX_RAW_STAGES * 8;
    tbar = gbar + (LAG_MAX_STAGES + 6) * 8;
    qbar = tbar + (LAG_MAX_STAGES + 4) * 8;
    cfull = qbar + LAG_QBUF * 8;
    cempty = cfull + LAG_GROUPS * 8;
    flag = cempty + LAG_GROUPS * 8;  // and the address of the status word
    total = flag + 16;
  }
};

// Named barriers: 0 the CTA, then these
// (two of each where the arriving side can be a block ahead)
enum { LAG_BAR_GAMMA = 1, LAG_BAR_Q = 3, LAG_BAR_SUM = 5, LAG_BAR_TEAM = 7, LAG_BAR_START = 15 };

__device__ __forceinline__ void named_barrier(int id, int threads) {
  asm volatile("bar.sync %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void named_arrive(int id, int threads) {
  asm volatile("bar.arrive %0, %1;" ::"r"(id), "r"(threads) : "memory");
}
__device__ __forceinline__ void mbar_arrive(unsigned long long* bar) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(bar);
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(a) : "memory");
}
// try_wait with a suspend-time hint: the warp sleeps until the phase completes or about 20 microseconds have passed, so
// waiting roles take no issue slots from the ones that work
__device__ __forceinline__ bool mbar_sleep_wait(uint32_t a, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.acquire.cluster.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(a), "r"(parity), "r"(20000)
      : "memory");
  return ok != 0;
}

// the same for barriers that only this CTA's threads and copies complete: without the cost of a fence for the cluster
__device__ __forceinline__ bool mbar_sleep_wait_cta(uint32_t a, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(a), "r"(parity), "r"(20000)
      : "memory");
  return ok != 0;
}
// 4-byte store into the shared memory of a CTA of the cluster, counted on that CTA's barrier, where `yes`
__device__ __forceinline__ void st_async_f32_if(uint32_t addr, float v, uint32_t mbar, bool yes) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %3, 0;\n\t@p st.async.weak.shared::cluster.mbarrier::complete_tx::bytes.f32 [%0], %1, [%2];\n\t}" ::"r"(addr),
      "f"(v), "r"(mbar), "r"((int)yes)
      : "memory");
}
// one thread of a converged warp; the compiler knows that it is one
__device__ __forceinline__ bool elect_one() {
  uint32_t yes;
  asm volatile("{\n\t.reg .pred p;\n\telect.sync _|p, 0xffffffff;\n\tselp.u32 %0, 1, 0, p;\n\t}" : "=r"(yes));
  return yes != 0;
}

__device__ __forceinline__ float4 lds_f32x4(uint32_t a) {
  float4 v;
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void ldmatrix_x4(uint32_t (&r)[4], uint32_t a) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];" : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

// 16 or 8 bytes of a row as 32-bit words
template <int VB>
struct RowVec {
  uint32_t w[VB / 4];
  __device__ __forceinline__ void load(uint32_t a) {  // shared-window address
    if constexpr (VB == 16) asm volatile("ld.shared.v4.u32 {%0, %1, %2, %3}, [%4];" : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]) : "r"(a));
    else asm volatile("ld.shared.v2.u32 {%0, %1}, [%2];" : "=r"(w[0]), "=r"(w[1]) : "r"(a));
  }
};
// pair i of the vector's columns (bf16: one word holds a pair; fp32: words 2i and 2i + 1)
template <typename XT, int VB>
__device__ __forceinline__ float2 row_pair(const RowVec<VB>& v, int i) {
  if constexpr (sizeof(XT) == 2) return make_float2(__uint_as_float(v.w[i] << 16), __uint_as_float(v.w[i] & 0xffff0000u));
  else return make_float2(__uint_as_float(v.w[2 * i]), __uint_as_float(v.w[2 * i + 1]));
}

// A wait has run out: recorded in the status word and told to every CTA of the cluster. At `flag`: the flag itself, the status
// word's address 8 bytes on.
__device__ __noinline__ void lag_give_up(uint32_t flag, int where) {
  unsigned long long status;
  asm volatile("ld.shared.u64 %0, [%1+8];" : "=l"(status) : "r"(flag) : "memory");
  set_status((DevStatus*)status, DEV_TIMEOUT, where, (long long)blockIdx.x);
  for (uint32_t rr = 0; rr < cluster_nctarank(); ++rr) {
    uint32_t a;
    asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(flag), "r"(rr));
    st_shared_cluster(a, 1);
  }
}
// Bounded waits on mbarriers; a warp that has seen one run out (its own or the cluster's) waits no more. The code is inlined at
// every wait, so there is as little of it as possible.
struct LagWait {
  uint32_t flag;
  int polls;  // a poll lasts up to 20 microseconds
  bool dead;
  __device__ __forceinline__ LagWait(long long spin_limit, volatile int* g) : flag((uint32_t)__cvta_generic_to_shared((const void*)g)), dead(false) {
    polls = spin_limit < 64 ? 1 : (spin_limit > (1ll << 26) ? 1 << 20 : (int)(spin_limit >> 6));
  }
  template <bool CLUSTER>
  __device__ __forceinline__ void until(unsigned long long* bar, uint32_t parity, int where) {
    if (dead) return;
    const uint32_t a = (uint32_t)__cvta_generic_to_shared(bar);
    int left = polls;
    while (!(CLUSTER ? mbar_sleep_wait(a, parity) : mbar_sleep_wait_cta(a, parity))) {
      int told;
      asm volatile("ld.volatile.shared.s32 %0, [%1];" : "=r"(told) : "r"(flag) : "memory");
      if (told == 0 && --left >= 0) continue;
      if (told == 0) lag_give_up(flag, where);
      dead = true;
      break;
    }
  }
  // a barrier that other CTAs of the cluster complete, and one that only this CTA's threads and copies do
  __device__ __forceinline__ void cluster(unsigned long long* bar, uint32_t parity, int where) { until<true>(bar, parity, where); }
  __device__ __forceinline__ void operator()(unsigned long long* bar, uint32_t parity, int where) { until<false>(bar, parity, where); }
};

// Registers of the recurrence warp for one block and its eight steps, every lane the same except for the *_own values, which
// belong to sample lane & 7. r_n = p_n - sum_m beta_m G_mn is the bracket of the blocked form; the loss is taken at sc_n r_n.
template <int LOSS>
struct LagBlock {
  float G[BLK_PAIRS], ca[LAG_B], cb[LAG_B];
  float sc_own, ca_own, sc_max;
  // T: sums of the block, [8][8] Gram entries and [8][8] C^T
  __device__ __forceinline__ void load(const float* T, const LagConst& K, int n) {
#pragma unroll
    for (int n2 = 1; n2 < LAG_B; ++n2) {
      const float4 lo = *(const float4*)&T[n2 * 8];
      const float l4[4] = {lo.x, lo.y, lo.z, lo.w};
#pragma unroll
      for (int m = 0; m < 4; ++m)
        if (m < n2) G[n2 * (n2 - 1) / 2 + m] = l4[m];
      if (n2 > 4) {
        const float4 hi = *(const float4*)&T[n2 * 8 + 4];
        const float h4[4] = {hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int m = 4; m < 7; ++m)
          if (m < n2) G[n2 * (n2 - 1) / 2 + m] = h4[m - 4];
      }
    }
    if (LOSS == LOSS_LOGISTIC) {
      sc_own = K.sc[n];
      ca_own = K.a[n];
      sc_max = K.sc_max;
    } else {
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        const float4 v = ((const float4*)K.a)[i], u = ((const float4*)K.b)[i];
        ca[4 * i] = v.x; ca[4 * i + 1] = v.y; ca[4 * i + 2] = v.z; ca[4 * i + 3] = v.w;
        cb[4 * i] = u.x; cb[4 * i + 1] = u.y; cb[4 * i + 2] = u.z; cb[4 * i + 3] = u.w;
      }
    }
  }
  // sum_m ng_m C[n][m]: what the block before adds to the margin of sample n
  __device__ __forceinline__ float correction(const float* T, const float (&ng)[LAG_B], int n) const {
    const float4 lo = *(const float4*)&T[64 + n * 8], hi = *(const float4*)&T[64 + n * 8 + 4];
    const float row[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
    float acc0 = 0.0f, acc1 = 0.0f;
#pragma unroll
    for (int m = 0; m < LAG_B; m += 2) {
      acc0 = fmaf(ng[m], row[m], acc0);
      acc1 = fmaf(ng[m + 1], row[m + 1], acc1);
    }
    return acc0 + acc1;
  }
  // `margin`: for the hinge loss the smallest 2^40 |1 - t| of the samples, how near a decision came to its threshold
  __device__ __forceinline__ void steps(float r_own, const float* T, const LagConst& K, float4* jets, float (&beta)[LAG_B], float& margin) const {
    constexpr int B = LAG_B;
    const int lane = threadIdx.x & 31, n = lane & 7;
    if (LOSS == LOSS_LOGISTIC) {
      // the factor expanded around the block's margins as a cubic in r; beta's constant is in the coefficients
      float4 jet = logistic_jet(sc_own * r_own);
      const float c1 = ca_own * sc_own, c2 = c1 * sc_own;
      jet.x *= ca_own; jet.y *= c1; jet.z *= c2; jet.w *= c2 * sc_own;
      if (lane < B) jets[lane] = jet;
      __syncwarp();
      float dlt[B];
      float4 js[B];
#pragma unroll
      for (int m = 0; m < B; ++m) {
        js[m] = jets[m];
        dlt[m] = 0.0f;
      }
      float dmax = 0.0f;
#pragma unroll
      for (int m = 0; m < B; ++m) {
        if (m > 0) dmax = fmaxf(dmax, fabsf(dlt[m]));
        beta[m] = m == 0 ? js[0].x : logistic_factor_near(js[m], dlt[m]);
#pragma unroll
        for (int n2 = m + 1; n2 < B; ++n2) dlt[n2] = m == 0 ? -beta[0] * G[n2 * (n2 - 1) / 2] : fmaf(-beta[m], G[n2 * (n2 - 1) / 2 + m], dlt[n2]);
      }
      if (!(dmax * sc_max < LOGISTIC_DELTA_MAX)) {  // some step of the block moved a margin far: direct evaluation
        float rr = r_own;
#pragma unroll 1
        for (int m = 0; m < B; ++m) {
          const float bm = K.a[m] * logistic_factor(K.sc[m] * __shfl_sync(0xffffffffu, rr, m));
          if (n > m) rr = fmaf(-bm, T[n * 8 + m], rr);
#pragma unroll
          for (int e = 0; e < B; ++e)
            if (e == m) beta[e] = bm;
        }
      }
    } else {
      float r[B];
#pragma unroll
      for (int m = 0; m < B; ++m) r[m] = __shfl_sync(0xffffffffu, r_own, m);
#pragma unroll
      for (int m = 0; m < B; ++m) {
        if (LOSS == LOSS_HINGE) {
          const float far = fmaf(cb[m], r[m], LAG_STEP);
          beta[m] = ca[m] * __saturatef(far);  // 1 where sc r < 1, else 0
          margin = m == 0 ? fabsf(far) : fminf(margin, fabsf(far));
        } else beta[m] = fmaf(ca[m], r[m], cb[m]);
#pragma unroll
        for (int n2 = m + 1; n2 < B; ++n2) r[n2] = fmaf(-beta[m], G[n2 * (n2 - 1) / 2 + m], r[n2]);
      }
    }
  }
};
// -gamma_0..7 and -delta to the model warps, every value twice: the operand form of the packed FMA
__device__ __forceinline__ void lag_publish(float* dst, const float (&ng)[LAG_B], float ndl) {
  float4* gd = (float4*)dst;
  gd[0] = make_float4(ng[0], ng[0], ng[1], ng[1]);
  gd[1] = make_float4(ng[2], ng[2], ng[3], ng[3]);
  gd[2] = make_float4(ng[4], ng[4], ng[5], ng[5]);
  gd[3] = make_float4(ng[6], ng[6], ng[7], ng[7]);
  ((float2*)gd)[8] = make_float2(ndl, ndl);
}

// Sum of the model threads' shares of q for sample lane & 7, over this lane's quarter of them (lane >> 3): `n16` groups of 16
// entries, those from n16 on are zero
template <int QROW>
__device__ __forceinline__ float lag_sum_q(const float* qp, int n16) {
  const int lane = threadIdx.x & 31;
  const uint32_t src = (uint32_t)__cvta_generic_to_shared(qp) + (uint32_t)((lane & 7) * QROW + (lane >> 3) * 4) * 4u;
  const float4 a = lds_f32x4(src), b = lds_f32x4(src + 64u), c = lds_f32x4(src + 128u), d = lds_f32x4(src + 192u);
  float v = (((a.x + b.x) + (c.x + d.x)) + ((a.y + b.y) + (c.y + d.y))) + (((a.z + b.z) + (c.z + d.z)) + ((a.w + b.w) + (c.w + d.w)));
  if (n16 > 4) {
    const float4 e = lds_f32x4(src + 256u), f = lds_f32x4(src + 320u), g = lds_f32x4(src + 384u), h = lds_f32x4(src + 448u);
    v += (((e.x + f.x) + (g.x + h.x)) + ((e.y + f.y) + (g.y + h.y))) + (((e.z + f.z) + (g.z + h.z)) + ((e.w + f.w) + (g.w + h.w)));
  }
  return v;
}

// The recurrence warp's loop. What is published and kept for the next block is -gamma_m.
template <int LOSS, bool MULTI, int QROW>
__device__ __forceinline__ void lag_recurrence(int nb, int TB, int C, int NM, int n16, const float* tabs, const LagConst* cst, const float* q,
                                               const float* qpart, float* gam, float4* jets, unsigned long long* qbar,
                                               unsigned long long* cempty, LagWait& wait) {
  constexpr int B = LAG_B;
  const int lane = threadIdx.x & 31, n = lane & 7;
  const int bar_threads = 32 * (2 + NM), q_threads = MULTI ? 64 : bar_threads;
  float ng[B], ndl_prev = 0.0f;
#pragma unroll
  for (int m = 0; m < B; ++m) ng[m] = 0.0f;
  const float* T = tabs;
  const float* T_end = tabs + TB * LAG_SUMS;
  named_barrier(LAG_BAR_START, 64);  // sums and constants of block 0
#pragma unroll 1
  for (int b = 0; b < nb; ++b) {
    if (MULTI && lane == 0 && !wait.dead) mbar_arrive_expect_tx(&qbar[b & (LAG_QBUF - 1)], C * 32u);
    const LagConst& K = cst[b & (LAG_GROUP * LAG_GROUPS - 1)];
    LagBlock<LOSS> blk;
    blk.load(T, K, n);
    const float acc = blk.correction(T, ng, n);
    const float na_nv = K.na_nv, ndl_nv = K.ndl_nv;
    named_barrier(LAG_BAR_Q + (b & 1), q_threads);  // sums and constants of block b + 1 are there (one CTA: and the shares of q_b)
    float qv;
    if constexpr (!MULTI) {
      qv = lag_sum_q<QROW>(qpart + (b & 1) * (B * QROW), n16);
      qv += __shfl_xor_sync(0xffffffffu, qv, 8);
      qv += __shfl_xor_sync(0xffffffffu, qv, 16);
    } else {
      wait.cluster(&qbar[b & (LAG_QBUF - 1)], (uint32_t)(b / LAG_QBUF) & 1u, 4);
      const float* qs = q + (b & (LAG_QBUF - 1)) * 64 + n * 4;  // one sum per CTA (absent ones are zero)
      const float4 s4 = *(const float4*)qs, t4 = *(const float4*)(qs + 32);
      qv = ((s4.x + t4.x) + (s4.y + t4.y)) + ((s4.z + t4.z) + (s4.w + t4.w));
    }
    const float r_own = fmaf(ndl_prev, qv, qv) + acc;
    float beta[B], margin;
    blk.steps(r_own, T, K, jets, beta, margin);
#pragma unroll
    for (int m = 0; m < B; ++m) ng[m] = beta[m] * na_nv;
    if (lane == 0) lag_publish(gam + (b & 1) * LAG_GAM, ng, ndl_nv);
    named_arrive(LAG_BAR_GAMMA + (b & 1), bar_threads);
    ndl_prev = ndl_nv;
    if ((b & (LAG_GROUP - 1)) == LAG_GROUP - 1 && lane == 0 && !wait.dead) mbar_arrive(&cempty[(b / LAG_GROUP) & (LAG_GROUPS - 1)]);
    T += LAG_SUMS;
    if (T == T_end) T = tabs;
  }
}

// A_m (product of the factors before step m of its block of 8), eta_m / A_{m+1} and the block's end product for the
// decaying schedule, for the block and step of this lane (8 lanes per block; n0 = steps before the block, nv = its steps)
__device__ __forceinline__ void lag_decaying_factors(double eta0, double lam, long long n0, int nv, float& apw, float& cfac,
                                                     float& a_nv, float& dl_nv) {
  const int m = (int)(threadIdx.x & 7);
  // 1 / sqrt(n) and 1 / A from the fp32 special-function unit plus one Newton step in fp64 (relative error below 1e-12)
  const double nn = (double)(n0 + m + 1);
  double rs = (double)rsqrtf((float)nn);
  rs = rs * fma(-0.5 * nn, rs * rs, 1.5);
  const double eta = eta0 * rs;
  double ia = fma(-eta, lam, 1.0);
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    const double v = __shfl_up_sync(0xffffffffu, ia, o, 8);
    if (m >= o) ia *= v;
  }
  double ea = __shfl_up_sync(0xffffffffu, ia, 1, 8);
  if (m == 0) ea = 1.0;
  double rc = (double)__frcp_rn((float)ia);
  rc = rc * fma(-ia, rc, 2.0);
  const double a_end = __shfl_sync(0xffffffffu, ia, nv > 0 ? nv - 1 : 0, 8);
  apw = (float)ea;
  cfac = (float)(eta * rc);
  a_nv = nv > 0 ? (float)a_end : 1.0f;
  dl_nv = nv > 0 ? (float)(1.0 - a_end) : 0.0f;
}

// VB: bytes of a row that a model thread owns as one vector (fp32: 2 or 4 columns, bf16: 4 or 8), NC vectors per thread
// MULTI: a cluster of more than one CTA. REALIGN: rows pass through the realigning warps. Compiled for each, because what a kernel
// could do and does not fills the instruction cache all the same (see the note on code size).
template <typename XT, int VB, int NC, bool MULTI, bool REALIGN>
__global__ void __launch_bounds__(LAG_MAX_THREADS, 1) chain_lag_kernel(const LagParams lp) {
  constexpr int B = LAG_B;
  constexpr int V = 16 / (int)sizeof(XT);
  constexpr int VW = VB / (int)sizeof(XT);
  constexpr int QROW = lag_q_row(VB, NC, REALIGN);
  extern __shared__ __align__(16) unsigned char smem[];
  const BlockParams& bp = lp.b;
  const ChainParams& p = bp.c;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int S = bp.stages, TB = S + 4, GB = S + 6;
  const int NT = lp.gram_teams, NW = lp.gram_warps, NM = lp.model_warps;
  const uint32_t C = MULTI ? cluster_nctarank() : 1u, rank = MULTI ? cluster_ctarank() : 0u;
  const long long d = p.d;
  const long long c_first = (long long)rank * lp.chunks_per_cta * V;  // first column of the slice
  const long long c_left = d - c_first;
  const int ncols = (int)(c_left < 0 ? 0 : (c_left < (long long)lp.chunks_per_cta * V ? c_left : (long long)lp.chunks_per_cta * V));
  const int my_chunks = (ncols + V - 1) / V;
  const unsigned long long ld_bytes = (unsigned long long)p.ld * sizeof(XT);
  const LagSmem L(S, (size_t)lp.chunks_per_cta * 16, (int)C, NT * NW, REALIGN ? lp.raw_stages : 0, QROW);
  const uint32_t row_stride = (uint32_t)L.row_stride;
  unsigned char* ring = smem + L.ring;
  float* red = (float*)(smem + L.red);
  float* tabs = (float*)(smem + L.tabs);
  float* q = (float*)(smem + L.q);
  float* qpart = (float*)(smem + L.qpart);
  LagConst* cst = (LagConst*)(smem + L.cst);
  float* gam = (float*)(smem + L.gam);
  float* tab = (float*)(smem + L.tab);  // [0..8] a^k, [16..24] eta / a^{k+1}, [32..40] 1 - a^k
  unsigned long long* full = (unsigned long long*)(smem + L.full);
  unsigned long long* empty = (unsigned long long*)(smem + L.empty);
  unsigned long long* rfull = (unsigned long long*)(smem + L.rfull);
  unsigned long long* rempty = (unsigned long long*)(smem + L.rempty);
  unsigned long long* gbar = (unsigned long long*)(smem + L.gbar);
  unsigned long long* tbar = (unsigned long long*)(smem + L.tbar);
  unsigned long long* qbar = (unsigned long long*)(smem + L.qbar);
  unsigned long long* cfull = (unsigned long long*)(smem + L.cfull);
  unsigned long long* cempty = (unsigned long long*)(smem + L.cempty);
  volatile int* give_up = (volatile int*)(smem + L.flag);
  if (threadIdx.x <= B) {  // power tables in fp64, rounded once
    const double a = 1.0 - bp.eta_lambda;
    double pw = 1.0;
    for (int k = 0; k < (int)threadIdx.x; ++k) pw *= a;
    tab[threadIdx.x] = (float)pw;
    tab[16 + threadIdx.x] = (float)((double)p.eta0 / (pw * a));
    tab[32 + threadIdx.x] = (float)(1.0 - pw);
  }
  if (threadIdx.x == 32) {
    for (int s = 0; s < S; ++s) {
      mbar_init(&full[s], REALIGN ? lp.realign_rows : 2);  // (rows are requested in two groups of four)
      mbar_init(&empty[s], NM + 2 * NW);  // the block's own Gram team, the next block's, the model warps
    }
    for (int s = 0; REALIGN && s < lp.raw_stages; ++s) {
      mbar_init(&rfull[s], 2);
      mbar_init(&rempty[s], lp.realign_rows);
    }
    for (int s = 0; s < GB; ++s) mbar_init(&gbar[s], 1);
    for (int s = 0; s < TB; ++s) mbar_init(&tbar[s], 1);
    for (int s = 0; s < LAG_QBUF; ++s) mbar_init(&qbar[s], 1);
    for (int s = 0; s < LAG_GROUPS; ++s) {
      mbar_init(&cfull[s], 1);
      mbar_init(&cempty[s], 1);
    }
    *give_up = 0;
    *(DevStatus**)(smem + L.flag + 8) = p.status;
    mbar_fence_init();
  }
  {
    // ring and sums start at zero: row padding (half a tile of an odd chunk count, columns of idle threads) is read
    uint4* z = (uint4*)smem;
    const int n16 = (int)(L.tab / 16);
    for (int i = threadIdx.x; i < n16; i += blockDim.x) z[i] = make_uint4(0u, 0u, 0u, 0u);
  }
  fence_proxy_async_shared();
  kernel_inputs_ready();
  const int j = p.order[blockIdx.x / C];
  const long long n_run = p.n_steps[j];
  // (the stride taken from the argument once more: with one product for all, 32 fp32 chunks over a cluster took 3 % longer)
  const char* shard = (const char*)p.X + (unsigned long long)p.shard_off[j] * ((unsigned long long)p.ld * sizeof(XT)) + (size_t)c_first * sizeof(XT);
  const float* yshard = p.y + p.shard_off[j];
  const uint32_t* idx = p.idx + p.idx_off[j];  // padded to a multiple of 64 entries with the last step's row
  const int nb = (int)((n_run + B - 1) / B);  // the host sends chains of up to 2^33 steps here
  __syncthreads();
  if (MULTI) cluster_barrier();  // every CTA of the cluster runs and has set up its shared memory

  LagWait wait(bp.spin_limit, give_up);
  // recurrence, model warps, sums of q (more than one CTA), copy, constants, feeder, gram, realign
  const int place = lp.role[warp];
  const int first_part = 1 + NM;
  const int pl_copy = first_part + (MULTI ? 1 : 0), pl_const = pl_copy + lp.copy_warps, pl_feed = pl_const + 1, pl_gram = pl_feed + 1,
            pl_realign = pl_gram + NT * NW;
  const int n16 = (NM * lag_q_shares(VB, NC) + 15) / 16;  // groups of 16 shares of q

  if (place == 0) {
    // =========================== recurrence ==============================================================
    float4* jets = (float4*)(smem + L.jet);
    switch (p.loss) {
      case LOSS_HINGE: lag_recurrence<LOSS_HINGE, MULTI, QROW>(nb, TB, (int)C, NM, n16, tabs, cst, q, qpart, gam, jets, qbar, cempty, wait); break;
      case LOSS_LOGISTIC: lag_recurrence<LOSS_LOGISTIC, MULTI, QROW>(nb, TB, (int)C, NM, n16, tabs, cst, q, qpart, gam, jets, qbar, cempty, wait); break;
      default: lag_recurrence<LOSS_SQUARED, MULTI, QROW>(nb, TB, (int)C, NM, n16, tabs, cst, q, qpart, gam, jets, qbar, cempty, wait); break;
    }
  } else if (place < first_part) {
    // =========================== model ===================================================================
    const int mw = place - 1, mt = mw * 32 + lane, TM = NM * 32;
    const int bar_threads = 32 * (2 + NM);
    const uint32_t ring_a = (uint32_t)__cvta_generic_to_shared(ring), stage_bytes = B * row_stride;
    uint32_t off[NC];  // the thread's vectors in the first row of stage 0 (threads without columns: the row's zero padding)
    float2 w[NC][VW / 2];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      const int v0 = (i * TM + mt) * VW;
      off[i] = ring_a + (v0 < my_chunks * V ? (uint32_t)(i * TM + mt) * VB : (uint32_t)lp.chunks_per_cta * 16u);
      float w1[VW];
#pragma unroll
      for (int e = 0; e < VW; ++e) {
        w1[e] = 0.0f;
        if (v0 + e < ncols) {
          const long long c = c_first + v0 + e;
          if (p.resume) w1[e] = p.W[(size_t)j * d + c];
          else if (p.w0) w1[e] = p.w0[c];
        }
      }
#pragma unroll
      for (int e = 0; e < VW / 2; ++e) w[i][e] = make_float2(w1[2 * e], w1[2 * e + 1]);
    }
    // this thread's shares of q_blk (16-byte vectors: added up with those of the lane 16 away, half of the samples each; two of
    // them: then with those of the lane 8 away, a quarter each)
    auto put_q = [&](float (&v)[B], int blk) __attribute__((always_inline)) {
      float* qp = qpart + (blk & 1) * (B * QROW);
      if constexpr (VB == 16) {
        const bool hi = (lane & 16) != 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float send = hi ? v[i] : v[i + 4], keep = hi ? v[i + 4] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
        }
        if constexpr (NC == 2) {
          const bool hi8 = (lane & 8) != 0;
#pragma unroll
          for (int i = 0; i < 2; ++i) {
            const float send = hi8 ? v[i] : v[i + 2], keep = hi8 ? v[i + 2] : v[i];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
          }
          qp += (lane >> 3) * (2 * QROW) + mw * 8 + (lane & 7);
        } else {
          qp += (lane >> 4) * (4 * QROW) + mw * 16 + (lane & 15);
        }
#pragma unroll
        for (int i = 0; i < (NC == 2 ? 2 : 4); ++i) qp[i * QROW] = v[i];
      } else {
        qp += mt;
#pragma unroll
        for (int i = 0; i < B; ++i) qp[i * QROW] = v[i];
      }
      if (MULTI) named_arrive(LAG_BAR_SUM + (blk & 1), TM + 32);
      else named_arrive(LAG_BAR_Q + (blk & 1), bar_threads);
    };
    auto dot = [&](const RowVec<VB>& x, int i) __attribute__((always_inline)) -> float {
      float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int e = 0; e < VW / 2; ++e) s = __ffma2_rn(w[i][e], row_pair<XT, VB>(x, e), s);
      return s.x + s.y;
    };
    auto load_rows = [&](uint32_t stg, RowVec<VB> (&x)[NC][B]) __attribute__((always_inline)) {
#pragma unroll
      for (int i = 0; i < NC; ++i)
#pragma unroll
        for (int m = 0; m < B; ++m) x[i][m].load(off[i] + stg + (uint32_t)m * row_stride);
    };
    // the q rows are read ahead too where registers allow, else when they are needed
    constexpr bool AHEAD = NC == 1;
    RowVec<VB> xb[NC][B], xq[AHEAD ? 1 : NC][AHEAD ? B : 1];
    auto load_q = [&](uint32_t stg) __attribute__((always_inline)) {
      if constexpr (AHEAD) load_rows(stg, xq);
    };
    auto q_now = [&](uint32_t stg, float (&qa)[B]) __attribute__((always_inline)) {
#pragma unroll
      for (int m = 0; m < B; ++m) {
        if constexpr (AHEAD) {
          qa[m] = dot(xq[0][m], 0);
        } else {
          qa[m] = 0.0f;
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            xq[i][0].load(off[i] + stg + (uint32_t)m * row_stride);
            qa[m] += dot(xq[i][0], i);
          }
        }
      }
    };
    uint32_t sb = 0u, sq = 0u;  // offsets of the stages whose rows the update and q read next
    const uint32_t s_end = (uint32_t)S * stage_bytes;
    unsigned long long* free_b = empty;
    // blocks -2 and -1: no update, q_0 and q_1 from the initial model
    for (int blk = 0; blk < 3 && blk < nb; ++blk) wait(&full[blk], 0u, 1);
    if (nb > 0) {
      load_rows(0, xb);
      load_q(0);
    }
#pragma unroll 1
    for (int b = -2; b < nb; ++b) {
      if (b >= 0) {
        // w <- w + (-delta w - sum_m gamma_m x_m) once gamma_b is there (and the
        // rows of block b + 3); the small terms are added up before they meet w
        named_barrier(LAG_BAR_GAMMA + (b & 1), bar_threads);
        const float4* gd = (const float4*)(gam + (b & 1) * LAG_GAM);
        float2 gm[B];
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4 g4 = gd[i];
          gm[2 * i] = make_float2(g4.x, g4.y);
          gm[2 * i + 1] = make_float2(g4.z, g4.w);
        }
        const float2 ndl = ((const float2*)gd)[8];
#pragma unroll
        for (int i = 0; i < NC; ++i)
#pragma unroll
          for (int e = 0; e < VW / 2; ++e) {
            float2 s = __ffma2_rn(gm[0], row_pair<XT, VB>(xb[i][0], e), __fmul2_rn(ndl, w[i][e]));
            float2 t = __fmul2_rn(gm[4], row_pair<XT, VB>(xb[i][4], e));
#pragma unroll
            for (int m = 1; m < 4; ++m) {
              s = __ffma2_rn(gm[m], row_pair<XT, VB>(xb[i][m], e), s);
              t = __ffma2_rn(gm[m + 4], row_pair<XT, VB>(xb[i][m + 4], e), t);
            }
            w[i][e] = __fadd2_rn(w[i][e], __fadd2_rn(s, t));
          }
      }
      if (b + 2 < nb) {
        float qa[B];
        q_now(sq, qa);
        put_q(qa, b + 2);
      }
      if (b >= -1 && b + 1 < nb) {
        if (b >= 0) load_rows(sb, xb);
        __syncwarp();
        if (lane == 0 && !wait.dead) mbar_arrive(free_b);
        sb += stage_bytes;
        ++free_b;
        if (sb == s_end) { sb = 0u; free_b = empty; }
      }
      sq += stage_bytes;
      if (sq == s_end) sq = 0u;
      if (b + 3 < nb) load_q(sq);
    }
#pragma unroll
    for (int i = 0; i < NC; ++i)
#pragma unroll
      for (int e = 0; e < VW; ++e) {
        const int v0 = (i * TM + mt) * VW + e;
        if (v0 < ncols) p.W[(size_t)j * d + c_first + v0] = (e & 1) ? w[i][e / 2].y : w[i][e / 2].x;
      }
  } else if (MULTI && place < pl_copy) {
    // =========================== sums of q =================================================================
    // adds up the model threads' shares of q_b and sends the eight sums to every CTA: lane l sample l & 7, to the CTAs l >> 3
    // and (l >> 3) + 4
    const uint32_t d0 = (uint32_t)(lane >> 3) < C ? (uint32_t)(lane >> 3) : rank, d1 = (uint32_t)(lane >> 3) + 4u < C ? (uint32_t)(lane >> 3) + 4u : rank;
    float* q_own = q + (rank >> 2) * 32 + (lane & 7) * 4 + (rank & 3);
    const uint32_t q_dst0 = map_shared_rank(q_own, d0), q_dst1 = map_shared_rank(q_own, d1);
    const uint32_t q_bar0 = map_shared_rank(qbar, d0), q_bar1 = map_shared_rank(qbar, d1);
    // Then it waits, on behalf of the model warps, for the rows that they read after their next update: gamma of block b - 1 is let out
    // behind the rows of block b + 2.
    const int sum_threads = 32 * (NM + 1), bar_threads = 32 * (NM + 2);
    int sr = S == 3 ? 0 : 3;
    uint32_t rpar = S == 3 ? 1u : 0u;
#pragma unroll 1
    for (int b = 0; nb > 0; ++b) {
      if (b > 0) {
        if (b + 2 < nb) {
          wait(&full[sr], rpar, 1);
          if (++sr == S) { sr = 0; rpar ^= 1u; }
        }
        named_arrive(LAG_BAR_GAMMA + ((b - 1) & 1), bar_threads);
        if (b == nb) break;
      }
      wait.dead = wait.dead || *give_up != 0;
      named_barrier(LAG_BAR_SUM + (b & 1), sum_threads);
      float v = lag_sum_q<QROW>(qpart + (b & 1) * (B * QROW), n16);
      v += __shfl_xor_sync(0xffffffffu, v, 8);
      v += __shfl_xor_sync(0xffffffffu, v, 16);
      const uint32_t qb = (uint32_t)(b & (LAG_QBUF - 1));
      st_async_f32_if(q_dst0 + qb * 256u, v, q_bar0 + qb * 8u, !wait.dead && (uint32_t)(lane >> 3) < C);
      st_async_f32_if(q_dst1 + qb * 256u, v, q_bar1 + qb * 8u, !wait.dead && (uint32_t)(lane >> 3) + 4u < C);
    }
    wait.dead = __any_sync(0xffffffffu, wait.dead);
  } else if (place < pl_const) {
    // =========================== copy ======================================================================
    // One thread requests the slices of four rows at a time, one bulk copy each; they complete on the stage's barrier. (Copies
    // that a lane each issues cost the warp 52 cycles apiece, those of one elected thread 20: 508 and 267 for eight.)
    const int rows = lp.copy_warps == 2 ? B / 2 : B, row0 = (place - pl_copy) * rows;
    const int RS = REALIGN ? lp.raw_stages : S;
    unsigned long long* landed = REALIGN ? rfull : full;
    unsigned long long* free_ = REALIGN ? rempty : empty;
    unsigned char* dst0 = REALIGN ? smem + L.raw : ring;
    const uint32_t dst_stride = REALIGN ? (uint32_t)L.raw_stride : row_stride;
    // sample ids of four blocks at a time, the next four on their way (a load takes longer than a block)
    uint32_t ids = nb > 0 ? idx[lane] : 0u, ids_next = nb > LAG_GROUP ? idx[32 + lane] : 0u;
    // (Unaligned rows: every lane forms the address of its row with the ids, 48 bf16 chunks 1260 -> 1215 cycles per block. Aligned ones
    // below, where they are requested: formed ahead as well, 16 bf16 chunks took 813 instead of 781.)
    const char* row = nullptr;
    if constexpr (REALIGN) row = shard + ids * ld_bytes;
    int st = 0;
    uint32_t par = 1u;  // parity of the phase that frees the stage (the first pass over the ring needs none)
    int blk = 0;
#pragma unroll 1
    for (; blk < nb; ++blk) {
      if (blk >= RS) wait(&free_[st], par, 5);
      if (__any_sync(0xffffffffu, wait.dead)) break;
#pragma unroll 1
      for (int r0 = row0; r0 < row0 + rows; r0 += 4) {
        uint32_t id[4];
        const char* src[4];
#pragma unroll
        for (int m = 0; m < 4; ++m) {
          if constexpr (REALIGN) src[m] = (const char*)__shfl_sync(0xffffffffu, (unsigned long long)row, (blk & (LAG_GROUP - 1)) * B + r0 + m);
          else id[m] = __shfl_sync(0xffffffffu, ids, (blk & (LAG_GROUP - 1)) * B + r0 + m);
        }
        if (blk != bp.drop_block && elect_one()) {
          uint32_t bytes[4], all = 0u;
#pragma unroll
          for (int m = 0; m < 4; ++m) {  // whole 16-byte granules that hold at least one byte of the slice
            if constexpr (!REALIGN) src[m] = shard + id[m] * ld_bytes;
            const uint32_t lead = REALIGN ? (uint32_t)((uintptr_t)src[m] & 15u) : 0u;
            src[m] -= lead;
            bytes[m] = (lead + (uint32_t)ncols * (uint32_t)sizeof(XT) + 15u) & ~15u;
            all += bytes[m];
          }
          mbar_arrive_expect_tx(&landed[st], all);
#pragma unroll
          for (int m = 0; m < 4; ++m) bulk_copy_g2s(dst0 + (uint32_t)(st * B + r0 + m) * dst_stride, src[m], bytes[m], &landed[st]);
        }
        __syncwarp();
      }
      if ((blk & (LAG_GROUP - 1)) == LAG_GROUP - 1) {
        ids = ids_next;
        if constexpr (REALIGN) row = shard + ids * ld_bytes;
        if (blk + LAG_GROUP + 1 < nb) ids_next = idx[(long long)(blk + LAG_GROUP + 1) * B + lane];
      }
      if (++st == RS) { st = 0; par ^= 1u; }
    }
    if (blk < nb) {
      // giving up: leave no copy in flight into this CTA's shared memory (bounded)
      int s = blk >= RS ? st : 0;
      uint32_t pp = blk >= RS ? par : par ^ 1u;
#pragma unroll 1
      for (int r = blk >= RS ? blk - RS : 0; r < blk; ++r) {
        if (r != bp.drop_block) mbar_wait_bounded(&landed[s], pp, bp.spin_limit);
        if (++s == RS) { s = 0; pp ^= 1u; }
      }
    }
  } else if (place == pl_const) {
    // =========================== constants ================================================================
    // lane l: sample l & 7 of block 4 g + (l >> 3)
    const int n = lane & 7;
    const bool decaying = p.sched == LR_INV_SQRT;
    const long long first_j = p.first ? p.first[j] : 0;
    const int groups = (nb + LAG_GROUP - 1) / LAG_GROUP;
    auto label_id = [&](int g) -> uint32_t {
      const long long s = (long long)g * (LAG_GROUP * B) + lane;
      return s < (long long)nb * B ? idx[s] : 0u;
    };
    float y_nxt = 0.0f;
    uint32_t id_nxt = 0u;
    if (groups > 0) y_nxt = yshard[label_id(0)];
    if (groups > 1) id_nxt = label_id(1);
#pragma unroll 1
    for (int g = 0; g < groups; ++g) {
      const long long b = (long long)g * LAG_GROUP + (lane >> 3);
      const long long left = n_run - b * B;
      const int nv = left < 0 ? 0 : (left < B ? (int)left : B);
      const float y = y_nxt;
      if (g + 1 < groups) y_nxt = yshard[id_nxt];
      if (g + 2 < groups) id_nxt = label_id(g + 2);
      float a_nv = tab[nv], dl_nv = tab[32 + nv], apw = tab[n], cfac = tab[16 + n];
      if (decaying) lag_decaying_factors((double)p.eta0, (double)p.lambda, first_j + b * B, nv, apw, cfac, a_nv, dl_nv);
      if (n >= nv) cfac = 0.0f;  // samples beyond the chain's end take no step
      float ca, cb = 0.0f, sc = apw;
      if (p.loss == LOSS_SQUARED) {  // g = t - y, t = a^n r
        ca = cfac * apw;
        cb = -cfac * y;
      } else {                       // hinge: g = -y if t < 1, t = y a^n r; logistic: g = -y / (1 + 2^t), t = y a^n log2(e) r
        sc = y * apw;
        if (p.loss == LOSS_LOGISTIC) sc *= 1.4426950408889634f;
        ca = -y * cfac;
        if (p.loss == LOSS_HINGE) cb = -LAG_STEP * sc;
      }
      float sm = fabsf(sc);
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) sm = fmaxf(sm, __shfl_xor_sync(0xffffffffu, sm, o));
      const int slot = (int)(g & (LAG_GROUPS - 1));
      if (g >= LAG_GROUPS) wait(&cempty[slot], (uint32_t)((g / LAG_GROUPS - 1) & 1), 9);
      LagConst& K = cst[slot * LAG_GROUP + (lane >> 3)];
      K.a[n] = ca;
      K.b[n] = cb;
      K.sc[n] = sc;
      if (n == 0) { K.na_nv = -a_nv; K.ndl_nv = -dl_nv; K.sc_max = sm; }
      __syncwarp();
      if (lane == 0 && !wait.dead) mbar_arrive(&cfull[slot]);
    }
  } else if (place == pl_feed) {
    // =========================== feeder ===================================================================
    const int bar_threads = 32 * (2 + NM);
    int ts = 0, gs = 0;
    uint32_t par = 0u;
    auto take = [&](int t) __attribute__((always_inline)) {  // sums and constants of block t
      if (t >= nb) return;
      if ((t & (LAG_GROUP - 1)) == 0) wait(&cfull[(t / LAG_GROUP) & (LAG_GROUPS - 1)], (uint32_t)(t / (LAG_GROUP * LAG_GROUPS)) & 1u, 8);
      if (!MULTI) {
        wait(&tbar[ts], par, 3);
        if (++ts == TB) { ts = 0; par ^= 1u; }
      } else {
        if (lane == 0 && !wait.dead) mbar_arrive_expect_tx(&gbar[gs], C * (uint32_t)(LAG_SUMS * sizeof(float)));
        wait.cluster(&gbar[gs], par, 6);
        const float4* r4 = (const float4*)(red + (size_t)gs * C * LAG_SUMS) + lane;
        float4 s = r4[0];
        auto add = [&](const float4& v) __attribute__((always_inline)) { s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w; };
        add(r4[LAG_SUMS / 4]);
        if (C > 2) {
          const float4 v2 = r4[2 * (LAG_SUMS / 4)], v3 = r4[3 * (LAG_SUMS / 4)];
          add(v2); add(v3);
        }
        if (C > 4) {
          const float4 v4 = r4[4 * (LAG_SUMS / 4)], v5 = r4[5 * (LAG_SUMS / 4)], v6 = r4[6 * (LAG_SUMS / 4)], v7 = r4[7 * (LAG_SUMS / 4)];
          add(v4); add(v5); add(v6); add(v7);
        }
        *((float4*)(tabs + ts * LAG_SUMS) + lane) = s;
        if (++ts == TB) ts = 0;
        if (++gs == GB) { gs = 0; par ^= 1u; }
      }
    };
    take(0);
    named_arrive(LAG_BAR_START, 64);
    if (MULTI) {
#pragma unroll 1
      for (int t = 0; t < nb; ++t) {
        take(t + 1);
        named_barrier(LAG_BAR_Q + (t & 1), 64);
      }
    } else {
      // (here the feeder also lets gamma out behind the rows that the model warps read next, see the sums of q)
      int sr = S == 3 ? 0 : 3;
      uint32_t rpar = S == 3 ? 1u : 0u;
#pragma unroll 1
      for (int t = 0; t < nb + 2; ++t) {
        if (t >= 2) {
          if (t + 1 < nb) {
            wait(&full[sr], rpar, 1);
            if (++sr == S) { sr = 0; rpar ^= 1u; }
          }
          named_barrier(LAG_BAR_GAMMA + (t & 1), bar_threads);
        }
        take(t + 1);
        if (t < nb) named_arrive(LAG_BAR_Q + (t & 1), bar_threads);
      }
    }
  } else if (place < pl_realign) {
    // =========================== gram =====================================================================
    const int gw = place - pl_gram, team = (gw >= NW ? 1 : 0) + (gw >= 2 * NW ? 1 : 0) + (gw >= 3 * NW ? 1 : 0), tw = gw - team * NW;
    float* part = (float*)(smem + L.part) + (size_t)team * NW * LAG_SUMS;
    const size_t part_parity = (size_t)NT * NW * LAG_SUMS;
    const uint32_t ring_a = (uint32_t)__cvta_generic_to_shared(ring);
    int parity = 0;
    int st = team, gs = team, ts = team;  // (there are at least as many stages as teams)
    uint32_t par = 0u;
#pragma unroll 1
    for (int b = team; b < nb; b += NT) {
      const int stp = st == 0 ? S - 1 : st - 1;
      if (b > 0) wait(&full[stp], st == 0 ? par ^ 1u : par, 1);
      wait(&full[st], par, 1);
      const uint32_t xb = ring_a + (uint32_t)st * (B * row_stride);
      const uint32_t xp = b > 0 ? ring_a + (uint32_t)stp * (B * row_stride) : xb;  // block 0: gamma before it is zero
      float* sl = part + parity * part_parity + (size_t)tw * LAG_SUMS;
      if constexpr (sizeof(XT) == 2) {
        // A: rows 0..7 of X_b and of X_{b-1}; B: the X_b half again. Lanes 0..7 address rows 0..7 columns +0, 8..15 the
        // rows of X_{b-1} columns +0, 16..23 and 24..31 the same rows columns +8.
        float acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[a][e] = 0.0f;
        const uint32_t src = ((lane & 8) ? xp : xb) + (uint32_t)(lane & 7) * row_stride + (uint32_t)(lane >> 4) * 16u;
        const int ksteps = (my_chunks + 1) / 2;
        int ks = tw;
        for (; ks + 3 * NW < ksteps; ks += 4 * NW) {
          uint32_t x[4][4];
#pragma unroll
          for (int a = 0; a < 4; ++a) ldmatrix_x4(x[a], src + (uint32_t)(ks + a * NW) * 32u);
#pragma unroll
          for (int a = 0; a < 4; ++a) mma_bf16_m16n8k16(acc[a], x[a][0], x[a][1], x[a][2], x[a][3], x[a][0], x[a][2]);
        }
        for (; ks < ksteps; ks += NW) {
          uint32_t x[4];
          ldmatrix_x4(x, src + (uint32_t)ks * 32u);
          mma_bf16_m16n8k16(acc[0], x[0], x[1], x[2], x[3], x[0], x[2]);
        }
        const int g8 = lane >> 2, t4 = lane & 3;
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[0][e] = (acc[0][e] + acc[1][e]) + (acc[2][e] + acc[3][e]);
        *(float2*)(sl + g8 * 8 + 2 * t4) = make_float2(acc[0][0], acc[0][1]);
        sl[64 + 16 * t4 + g8] = acc[0][2];
        sl[64 + 16 * t4 + 8 + g8] = acc[0][3];
      } else {
        // 16 x 8 products as 4 x 4 tiles (rows ti + 4 q of [X_b; X_{b-1}], rows 4 tn + r of X_b): 8 lanes cover them on
        // the same 4 columns, the warp's four groups of 8 lanes take different chunks and meet by shuffles.
        const int ti = lane & 3, tn = (lane >> 2) & 1, cg = lane >> 3;
        float2 acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[a][e] = make_float2(0.0f, 0.0f);
        // rows of [X_b; X_{b-1}] of this lane's tile, and the first of its rows of X_b
        uint32_t a0 = xb + (uint32_t)ti * row_stride + (uint32_t)(tw * 4 + cg) * 16u, a1 = xp + (uint32_t)ti * row_stride + (uint32_t)(tw * 4 + cg) * 16u;
        uint32_t b0 = xb + (uint32_t)(4 * tn) * row_stride + (uint32_t)(tw * 4 + cg) * 16u;
#pragma unroll 1
        for (int ck = tw * 4 + cg; ck < my_chunks; ck += 4 * NW) {
          float4 xa[4], xn[4];
          xa[0] = lds_f32x4(a0);
          xa[1] = lds_f32x4(a0 + 4u * row_stride);
          xa[2] = lds_f32x4(a1);
          xa[3] = lds_f32x4(a1 + 4u * row_stride);
#pragma unroll
          for (int r = 0; r < 4; ++r) xn[r] = lds_f32x4(b0 + (uint32_t)r * row_stride);
          a0 += 64u * NW;
          a1 += 64u * NW;
          b0 += 64u * NW;
#pragma unroll
          for (int a = 0; a < 4; ++a)
#pragma unroll
            for (int r = 0; r < 4; ++r) {
              acc[a][r] = __ffma2_rn(make_float2(xa[a].x, xa[a].y), make_float2(xn[r].x, xn[r].y), acc[a][r]);
              acc[a][r] = __ffma2_rn(make_float2(xa[a].z, xa[a].w), make_float2(xn[r].z, xn[r].w), acc[a][r]);
            }
        }
        __syncwarp();
        float v[16];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int r = 0; r < 4; ++r) v[a * 4 + r] = acc[a][r].x + acc[a][r].y;
        const bool h8 = (lane & 8) != 0, h16 = (lane & 16) != 0;
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const float send = h8 ? v[i] : v[i + 8], keep = h8 ? v[i + 8] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 8);
        }
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float send = h16 ? v[i] : v[i + 4], keep = h16 ? v[i + 4] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, 16);
        }
        // this lane holds four products of row ti + 4 (h16 ? 1 : 0) of X_b, or of X_{b-1} (h8), with rows 4 tn .. of X_b
        const int row = ti + (h16 ? 4 : 0);
        float* dst = sl + (h8 ? 64 + tn * 32 + row : row * 8 + tn * 4);
        const int step = h8 ? 8 : 1;
#pragma unroll
        for (int i = 0; i < 4; ++i) dst[i * step] = v[i];
      }
      // the rows have been read
      __syncwarp();
      if (lane == 0 && !wait.dead) {
        if (b > 0) mbar_arrive(&empty[stp]);
        mbar_arrive(&empty[st]);
      }
      if (NW > 1) named_barrier(LAG_BAR_TEAM + team, NW * 32);
      if (tw == 0) {
        const float4* p4 = (const float4*)(part + parity * part_parity) + lane;
        float4 sum = p4[0];
#pragma unroll 1
        for (int w = 1; w < NW; ++w) {
          const float4 u = p4[w * (LAG_SUMS / 4)];
          sum.x += u.x; sum.y += u.y; sum.z += u.z; sum.w += u.w;
        }
        if (!MULTI) {
          *((float4*)(tabs + ts * LAG_SUMS) + lane) = sum;
          __syncwarp();
          if (lane == 0 && !wait.dead) mbar_arrive(&tbar[ts]);
        } else if (!wait.dead) {
          float* dst = red + ((size_t)gs * C + rank) * LAG_SUMS + 4 * lane;
#pragma unroll 1
          for (uint32_t rr = 0; rr < C; ++rr) st_async_f32x4(map_shared_rank(dst, rr), sum, map_shared_rank(&gbar[gs], rr));
        }
      }
      parity ^= 1;
      st += NT;
      if (st >= S) { st -= S; par ^= 1u; }
      gs += NT;
      if (gs >= GB) gs -= GB;
      ts += NT;
      if (ts >= TB) ts -= TB;
    }
  } else if (REALIGN && place < pl_realign + lp.realign_warps) {
    // =========================== realign =================================================================
    // Groups of warps take the blocks in turn, the warps of a group share the rows of a block. Groups of one warp move the most
    // bytes (no warp waits for the others at every block); groups of all warps need the fewest blocks in the rings. The number
    // of groups divides both ring depths: a stage then belongs to one group (a warp that waits for a phase of a barrier must have
    // seen the one before it, or the parity would stand for an older one). Word i of a ring row comes from two neighbouring words
    // of the fetched granules, shifted by the row's offset inside its first granule; words beyond the row become zero.
    const int RG = lp.realign_rows, RW = RG == 1 ? lp.realign_warps : 1;
    const int aw = place - pl_realign, RS = lp.raw_stages, row0 = RG == 1 ? 0 : aw, block0 = RG == 1 ? aw : 0;
    const unsigned char* raw = smem + L.raw;
    const uint32_t raw_stride = (uint32_t)L.raw_stride;
    const int words = my_chunks * 4, valid_bytes = ncols * (int)sizeof(XT);
    auto shift_of = [&](int blk) -> uint32_t {  // lane m & 7: of row m
      const uint32_t id = blk < nb ? idx[(long long)blk * B + (lane & 7)] : 0u;
      return ((uint32_t)(uintptr_t)shard + id * (uint32_t)ld_bytes) & 15u;
    };
    uint32_t sh_next = shift_of(block0);
    int rst = block0, st = block0;
    uint32_t rpar = 0u, epar = 1u;
#pragma unroll 1
    for (int b = block0; b < nb; b += RW) {
      const uint32_t sh_rows = sh_next;
      sh_next = shift_of(b + RW);
      if (b >= S) wait(&empty[st], epar, 5);
      wait(&rfull[rst], rpar, 1);
#pragma unroll 1
      for (int m = row0; m < B / 2; m += RG) {  // rows m and m + 4
        const uint32_t* src[2];
        uint32_t bits[2];
        uint32_t* dst = (uint32_t*)(ring + (uint32_t)(st * B + m) * row_stride);
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const uint32_t sh = __shfl_sync(0xffffffffu, sh_rows, m + 4 * h);
          bits[h] = 8u * (sh & 3u);
          src[h] = (const uint32_t*)(raw + (uint32_t)(rst * B + m + 4 * h) * raw_stride) + (sh >> 2);
        }
#pragma unroll 2
        for (int i = lane; i < words; i += 32) {
          const int left = valid_bytes - 4 * i;
          const uint32_t mask = left >= 4 ? 0xffffffffu : (left <= 0 ? 0u : (1u << (8 * left)) - 1u);
#pragma unroll
          for (int h = 0; h < 2; ++h) dst[i + (uint32_t)h * row_stride] = __funnelshift_r(src[h][i], src[h][i + 1], bits[h]) & mask;
        }
      }
      __syncwarp();
      if (lane == 0 && !wait.dead) {
        mbar_arrive(&full[st]);
        mbar_arrive(&rempty[rst]);
      }
      rst += RW;
      if (rst >= RS) { rst -= RS; rpar ^= 1u; }
      st += RW;
      if (st >= S) { st -= S; epar ^= 1u; }
    }
  }
  __syncwarp();
  if (wait.dead) {  // sums sent just now may still be on their way to a peer; let them land before anyone exits
    const long long t0 = clock64();
    while (clock64() - t0 < 100000) {}
  }
  __syncwarp();
  if (MULTI) cluster_barrier();
}

}  // namespace wpsgd
