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
//   copy         one or two warps that request the rows of a block (one cp.async.bulk per row, never multicast) into a ring
//                of stages (a warp needs about 100 cycles per bulk copy, 830 for the eight of a block)
//   constants    labels and step-size factors, four blocks at a time
//   feeder       does the waiting on mbarriers for the recurrence and the model warps: that the Gram sums of the next
//                blocks and the rows of block b + 3 are there (in clusters of more than one CTA it also adds up the CTAs' sums)
//   gram         [X_b; X_{b-1}] X_b^T over the slice: one mma.m16n8k16 per 16 columns for bf16 rows (A = the 16 rows,
//                B = the first 8 of them again), 4 x 4 register tiles on the fp32 pipes for fp32 rows. Teams of one or
//                more warps take the blocks in turn
//   model        own the model in registers: update with gamma_b, then the partial sums of q_{b+2}
//   realign      only when rows do not start on 16-byte boundaries or end inside a chunk: the copy warp then fetches the
//                16-byte granules that hold the row's slice, and these warps shift the bytes into the ring (bytes beyond
//                the row become zero)
// Recurrence, model and feeder warps, whose hand-offs are on the dependent path, meet on named barriers (about 25 cycles
// one way; a wait on an mbarrier costs about 100 even when its phase is complete); everything that runs ahead meets on
// mbarriers. Between CTAs of a
// cluster only sums travel: Gram sums (512 bytes) and q sums (128 bytes) of every CTA go to every CTA with st.async, and
// each CTA runs the recurrence redundantly.
//
// Code size. The loops of all roles run at the same time and share one instruction cache: straight-line code of about 2000
// instructions in all (32 KB) already runs at 2 to 3 cycles per instruction instead of 1 (measured with loops of
// independent FMAs). Loops are therefore kept rolled where they are off the dependent path, and one path serves all shapes.
//
// Buffers. Let g be the last block whose gamma a CTA has published. Its model warps hold rows up to block g + 3 in
// registers and have freed their stages, so it can have formed Gram sums up to block g + 3 + S (ring depth S) and q sums
// up to block g + 2. Publishing gamma_g took the q sums of block g from every CTA, which those sent after their own
// gamma_{g-2}: a peer may be two blocks behind. Tables read in the same CTA therefore have S + 4 entries, Gram sums from
// peers S + 6, q sums four.
//
// What bounds a block, and what it measured (B200, 1965 MHz; cycles per block of 8 samples of a chain that has its SMs to
// itself, logistic loss, fp32 rows): d = 64, one CTA, 890 (the warp-per-node kernel of chain_block.cuh: 1920); d = 1024,
// eight CTAs, 1270 (one CTA per node with the Gram block in the same warps: 2130; blocks of 16 over eight CTAs with the
// margins on the dependent path: 1700); d = 4096, eight CTAs, 2110 (one step at a time: 12500). bf16, squared: d = 1000,
// four CTAs, 1240 (1960); d = 2048, eight CTAs, 1310 (1970). d = 999, rows unaligned, eight CTAs: 1440 (one step at a time
// with scalar loads: 20000). The recurrence warp's own string (tables to registers 130, sums of q 130-180, steps 170
// (logistic 400), gamma out 140) is about 700 (1000) of these; the rest is waiting for q (update 80, dot products and
// their sum over lanes 240, exchange 100 to 400 with the cluster). From about 128 chunks per CTA on, the Gram block on the
// fp32 pipes (15 cycles per chunk), or the realigning of rows (21), bounds the block instead.
// Tried and taken back: rows by 16-byte copies of the threads instead of bulk copies (1900 against 1060 at d = 64), waits
// on mbarriers in the model and recurrence warps (1150 against 1060), roles pinned to schedulers (1140 against 1060).
//
// Leaving. Every wait on an mbarrier is bounded. One that runs out sets the status word and a flag in every CTA of the
// cluster; from then on a warp skips these waits and runs to the end of its loop, so that named barriers are still met by
// all their warps. Nobody exits before the cluster barrier at the end.
#pragma once

#include "chain_block.cuh"
#include "chain_mma16.cuh"

namespace wpsgd {

constexpr int LAG_B = 8;
constexpr int LAG_MAX_STAGES = 12;
constexpr int LAG_RAW_STAGES = 3;
constexpr int LAG_QBUF = 4;
constexpr int LAG_MAX_CLUSTER = 8;
constexpr int LAG_SUMS = 128;        // [16][8]: rows 0..7 G, rows 8..15 the transpose of C
constexpr int LAG_MAX_MODEL_WARPS = 8;
constexpr int LAG_GRAM_WARPS = 4;
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
  int realign;                 // 1: rows pass through the realigning warps
  int copy_warps;              // 1 or 2
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
  __host__ __device__ LagSmem(int stages, size_t slice_bytes, int C, int gram_warps_all, int realign) {
    // odd multiples of 16 bytes: tile loads of 8 (or 4) rows at the same column never meet in a bank
    row_stride = slice_bytes + 16;
    if (row_stride % 32 == 0) row_stride += 16;
    raw_stride = slice_bytes + 32;
    ring = 0;
    raw = ring + (size_t)stages * LAG_B * row_stride;
    red = raw + (realign ? (size_t)LAG_RAW_STAGES * LAG_B * raw_stride : 0);
    part = red + (C > 1 ? (size_t)(stages + 6) * C * LAG_SUMS * sizeof(float) : 0);  // [buffer][CTA][128]
    tabs = part + 2 * (size_t)gram_warps_all * LAG_SUMS * sizeof(float);             // [parity][gram warp][128]
    q = tabs + (size_t)(stages + 4) * LAG_SUMS * sizeof(float);
    qpart = q + (C > 1 ? LAG_QBUF * LAG_MAX_CLUSTER * 32 * sizeof(float) : 0);       // [LAG_QBUF][8][32]
    cst = qpart + 2 * LAG_MAX_MODEL_WARPS * 32 * sizeof(float);                      // [2][model warp][32]
    gam = cst + LAG_GROUPS * LAG_GROUP * sizeof(LagConst);
    tab = gam + 2 * LAG_GAM * sizeof(float);                                       // powers of 1 - eta lambda
    jet = tab + 3 * 16 * sizeof(float);
    full = jet + 8 * 4 * sizeof(float);
    empty = full + LAG_MAX_STAGES * 8;
    rfull = empty + LAG_MAX_STAGES * 8;
    rempty = rfull + 4 * 8;
    gbar = rempty + 4 * 8;
    tbar = gbar + (LAG_MAX_STAGES + 6) * 8;
    qbar = tbar + (LAG_MAX_STAGES + 4) * 8;
    cfull = qbar + LAG_QBUF * 8;
    cempty = cfull + LAG_GROUPS * 8;
    flag = cempty + LAG_GROUPS * 8;
    total = flag + 16;
  }
};

// Named barriers: 0 the CTA, then these
// (two of each where the arriving side can be a block ahead)
enum { LAG_BAR_GAMMA = 1, LAG_BAR_Q = 3, LAG_BAR_MODEL = 5, LAG_BAR_TEAM = 7, LAG_BAR_START = 15 };

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

// 16 or 8 bytes of a row as 32-bit words
template <int VB>
struct RowVec {
  uint32_t w[VB / 4];
  __device__ __forceinline__ void load(const unsigned char* p) {
    if constexpr (VB == 16) {
      const uint4 v = *(const uint4*)p;
      w[0] = v.x; w[1] = v.y; w[2] = v.z; w[3] = v.w;
    } else {
      const uint2 v = *(const uint2*)p;
      w[0] = v.x; w[1] = v.y;
    }
  }
};
// pair i of the vector's columns (bf16: one word holds a pair; fp32: words 2i and 2i + 1)
template <typename XT, int VB>
__device__ __forceinline__ float2 row_pair(const RowVec<VB>& v, int i) {
  if constexpr (sizeof(XT) == 2) return make_float2(__uint_as_float(v.w[i] << 16), __uint_as_float(v.w[i] & 0xffff0000u));
  else return make_float2(__uint_as_float(v.w[2 * i]), __uint_as_float(v.w[2 * i + 1]));
}

// The part of a bounded wait that is rarely reached: true when the phase has completed after all; false when the limit ran
// out (recorded in the status word and told to every CTA of the cluster) or another wait's had.
__device__ __noinline__ bool lag_wait_slow(uint32_t bar, uint32_t parity, int where, int polls, uint32_t C, uint32_t flag, DevStatus* status) {
  auto flagged = [&]() {
    int v;
    asm volatile("ld.volatile.shared.s32 %0, [%1];" : "=r"(v) : "r"(flag) : "memory");
    return v != 0;
  };
  for (int i = 0; i < polls; ++i) {
    if (flagged()) return false;
    if (mbar_sleep_wait(bar, parity)) return true;
  }
  if (!flagged()) {
    set_status(status, DEV_TIMEOUT, where, (long long)blockIdx.x);
    for (uint32_t rr = 0; rr < C; ++rr) {
      uint32_t a;
      asm volatile("mapa.shared::cluster.u32 %0, %1, %2;" : "=r"(a) : "r"(flag), "r"(rr));
      st_shared_cluster(a, 1);
    }
  }
  return false;
}
// Bounded waits on mbarriers; a warp that has seen one run out (its own or the cluster's) waits no more.
struct LagWait {
  DevStatus* status;
  uint32_t flag, C;
  int polls;  // a poll lasts up to 20 microseconds
  bool dead;
  __device__ __forceinline__ LagWait(DevStatus* st, long long spin_limit, volatile int* g, uint32_t C_)
      : status(st), flag((uint32_t)__cvta_generic_to_shared((const void*)g)), C(C_), dead(false) {
    polls = spin_limit < 64 ? 1 : (spin_limit > (1ll << 26) ? 1 << 20 : (int)(spin_limit >> 6));
  }
  // the answer of a poll taken earlier (`ok`) decides whether there is anything to wait for
  __device__ __forceinline__ void finish(bool ok, unsigned long long* bar, uint32_t parity, int where) {
    if (ok || dead) return;
    dead = !lag_wait_slow((uint32_t)__cvta_generic_to_shared(bar), parity, where, polls, C, flag, status);
  }
  __device__ __forceinline__ void operator()(unsigned long long* bar, uint32_t parity, int where) {
    if (dead) return;
    finish(mbar_sleep_wait((uint32_t)__cvta_generic_to_shared(bar), parity), bar, parity, where);
  }
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
    float acc0 = 0.0f, acc1 = 0.0f;
#pragma unroll
    for (int m = 0; m < LAG_B; m += 2) {
      acc0 = fmaf(ng[m], T[64 + m * 8 + n], acc0);
      acc1 = fmaf(ng[m + 1], T[64 + (m + 1) * 8 + n], acc1);
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

// The recurrence warp's loop. What is published and kept for the next block is -gamma_m.
template <int LOSS>
__device__ __forceinline__ void lag_recurrence(int nb, int TB, int C, int NM, const float* tabs, const LagConst* cst, const float* q,
                                               const float* qpart, float* gam, float4* jets, unsigned long long* qbar,
                                               unsigned long long* cempty, LagWait& wait) {
  constexpr int B = LAG_B;
  const int lane = threadIdx.x & 31, n = lane & 7;
  const int bar_threads = 32 * (2 + NM);
  // where this lane finds its share of the q sums: [slot][sample][4]; slots are the model warps of this CTA, or the CTAs, eight
  // in either case (absent ones are zero)
  const int q_stride = LAG_MAX_MODEL_WARPS * 32;
  const float* q_src = (C == 1 ? qpart : q) + (lane >> 3) * 32 + n * 4;
  const int q_mask = C == 1 ? 1 : LAG_QBUF - 1;
  float ng[B], ndl_prev = 0.0f;
#pragma unroll
  for (int m = 0; m < B; ++m) ng[m] = 0.0f;
  const float* T = tabs;
  const float* T_end = tabs + TB * LAG_SUMS;
  named_barrier(LAG_BAR_START, 64);  // sums and constants of block 0
#pragma unroll 1
  for (int b = 0; b < nb; ++b) {
    if (C > 1 && lane == 0 && !wait.dead) mbar_arrive_expect_tx(&qbar[b & (LAG_QBUF - 1)], C * 128u);
    const LagConst& K = cst[b & (LAG_GROUP * LAG_GROUPS - 1)];
    LagBlock<LOSS> blk;
    blk.load(T, K, n);
    const float acc = blk.correction(T, ng, n);
    const float na_nv = K.na_nv, ndl_nv = K.ndl_nv;
    named_barrier(LAG_BAR_Q + (b & 1), bar_threads);  // q_b is formed (and sent); sums and constants of block b + 1 are there
    if (C > 1) wait(&qbar[b & (LAG_QBUF - 1)], (uint32_t)(b / LAG_QBUF) & 1u, 4);
    const float* qs = q_src + (b & q_mask) * q_stride;
    const float4 s4 = *(const float4*)qs, t4 = *(const float4*)(qs + 4 * 32);
    float qv = ((s4.x + t4.x) + (s4.y + t4.y)) + ((s4.z + t4.z) + (s4.w + t4.w));
    qv += __shfl_xor_sync(0xffffffffu, qv, 8);
    qv += __shfl_xor_sync(0xffffffffu, qv, 16);
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
template <typename XT, int VB, int NC>
__global__ void __launch_bounds__(LAG_MAX_THREADS, 1) chain_lag_kernel(const LagParams lp) {
  constexpr int B = LAG_B;
  constexpr int V = 16 / (int)sizeof(XT);
  constexpr int VW = VB / (int)sizeof(XT);
  extern __shared__ __align__(16) unsigned char smem[];
  const BlockParams& bp = lp.b;
  const ChainParams& p = bp.c;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int S = bp.stages, TB = S + 4, GB = S + 6;
  const int NT = lp.gram_teams, NW = lp.gram_warps, NM = lp.model_warps;
  const uint32_t C = cluster_nctarank(), rank = cluster_ctarank();
  const long long d = p.d;
  const long long c_first = (long long)rank * lp.chunks_per_cta * V;  // first column of the slice
  const long long c_left = d - c_first;
  const int ncols = (int)(c_left < 0 ? 0 : (c_left < (long long)lp.chunks_per_cta * V ? c_left : (long long)lp.chunks_per_cta * V));
  const int my_chunks = (ncols + V - 1) / V;
  const size_t ld_bytes = (size_t)p.ld * sizeof(XT);
  const LagSmem L(S, (size_t)lp.chunks_per_cta * 16, (int)C, NT * NW, lp.realign);
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
      mbar_init(&full[s], lp.realign ? LAG_REALIGN_WARPS : lp.copy_warps);
      mbar_init(&empty[s], NM + 2 * NW);  // the block's own Gram team, the next block's, the model warps
    }
    for (int s = 0; s < LAG_RAW_STAGES; ++s) {
      mbar_init(&rfull[s], lp.copy_warps);
      mbar_init(&rempty[s], LAG_REALIGN_WARPS);
    }
    for (int s = 0; s < GB; ++s) mbar_init(&gbar[s], 1);
    for (int s = 0; s < TB; ++s) mbar_init(&tbar[s], 1);
    for (int s = 0; s < LAG_QBUF; ++s) mbar_init(&qbar[s], 1);
    for (int s = 0; s < LAG_GROUPS; ++s) {
      mbar_init(&cfull[s], 1);
      mbar_init(&cempty[s], 1);
    }
    *give_up = 0;
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
  const char* shard = (const char*)p.X + (size_t)p.shard_off[j] * ld_bytes + (size_t)c_first * sizeof(XT);
  const float* yshard = p.y + p.shard_off[j];
  const uint32_t* idx = p.idx + p.idx_off[j];  // padded to a multiple of 64 entries with the last step's row
  const int nb = (int)((n_run + B - 1) / B);  // the host sends chains of up to 2^33 steps here
  __syncthreads();
  cluster_barrier();  // every CTA of the cluster runs and has set up its shared memory

  LagWait wait(bp.c.status, bp.spin_limit, give_up, C);
  const int place = warp;  // recurrence, model warps, copy, constants, feeder, gram, realign
  const int first_part = 1 + NM;
  const int pl_copy = first_part, pl_const = pl_copy + lp.copy_warps, pl_feed = pl_const + 1, pl_gram = pl_feed + 1,
            pl_realign = pl_gram + NT * NW;

  if (place == 0) {
    // =========================== recurrence ==============================================================
    float4* jets = (float4*)(smem + L.jet);
    switch (p.loss) {
      case LOSS_HINGE: lag_recurrence<LOSS_HINGE>(nb, TB, (int)C, NM, tabs, cst, q, qpart, gam, jets, qbar, cempty, wait); break;
      case LOSS_LOGISTIC: lag_recurrence<LOSS_LOGISTIC>(nb, TB, (int)C, NM, tabs, cst, q, qpart, gam, jets, qbar, cempty, wait); break;
      default: lag_recurrence<LOSS_SQUARED>(nb, TB, (int)C, NM, tabs, cst, q, qpart, gam, jets, qbar, cempty, wait); break;
    }
  } else if (place < first_part) {
    // =========================== model ===================================================================
    const int mw = place - 1, mt = mw * 32 + lane, TM = NM * 32;
    const int bar_threads = 32 * (2 + NM);
    uint32_t off[NC];  // byte offset of the thread's vectors inside a staged row (threads without columns: its zero padding)
    float2 w[NC][VW / 2];
#pragma unroll
    for (int i = 0; i < NC; ++i) {
      const int v0 = (i * TM + mt) * VW;
      off[i] = v0 < my_chunks * V ? (uint32_t)(i * TM + mt) * VB : (uint32_t)lp.chunks_per_cta * 16u;
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
    // partial sums of q_blk: three rounds of a transposing sum leave lane l with value l >> 2 over its share of the lanes;
    // the last four lanes' worth is added up by the recurrence warp
    const uint32_t d0 = (uint32_t)(lane >> 3) < C ? (uint32_t)(lane >> 3) : rank, d1 = (uint32_t)(lane >> 3) + 4u < C ? (uint32_t)(lane >> 3) + 4u : rank;
    const uint32_t q_dst0 = map_shared_rank(q + rank * 32 + (lane & 7) * 4, d0), q_dst1 = map_shared_rank(q + rank * 32 + (lane & 7) * 4, d1);
    const uint32_t q_bar0 = map_shared_rank(qbar, d0), q_bar1 = map_shared_rank(qbar, d1);
    auto send_q = [&](float (&v)[B], int blk) __attribute__((always_inline)) {
#pragma unroll
      for (int half = 4; half >= 1; half >>= 1) {
        const int mask = half * 4;
        const bool hi = (lane & mask) != 0;
#pragma unroll
        for (int i = 0; i < half; ++i) {
          const float send = hi ? v[i] : v[i + half];
          const float keep = hi ? v[i + half] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, mask);
        }
      }
      float* qp = qpart + (blk & 1) * (LAG_MAX_MODEL_WARPS * 32);
      qp[mw * 32 + lane] = v[0];
      if (C > 1) {
        if (NM > 1) {
          if (mw != 0) named_arrive(LAG_BAR_MODEL + (blk & 1), TM);
          else named_barrier(LAG_BAR_MODEL + (blk & 1), TM);
        } else {
          __syncwarp();
        }
        if (mw == 0 && !wait.dead) {
          // lane l sends the four values of sample l & 7 to the CTAs l >> 3 and (l >> 3) + 4
          float4 t[4];  // (rows of absent warps stay zero)
#pragma unroll
          for (int k2 = 0; k2 < 4; ++k2) t[k2] = *(const float4*)(qp + k2 * 32 + (lane & 7) * 4);
          if (NM > 4) {
#pragma unroll
            for (int k2 = 0; k2 < 4; ++k2) {
              const float4 u = *(const float4*)(qp + (k2 + 4) * 32 + (lane & 7) * 4);
              t[k2].x += u.x; t[k2].y += u.y; t[k2].z += u.z; t[k2].w += u.w;
            }
          }
          const float4 s = make_float4((t[0].x + t[1].x) + (t[2].x + t[3].x), (t[0].y + t[1].y) + (t[2].y + t[3].y),
                                       (t[0].z + t[1].z) + (t[2].z + t[3].z), (t[0].w + t[1].w) + (t[2].w + t[3].w));
          const uint32_t qb = (uint32_t)(blk & (LAG_QBUF - 1));
          st_async_f32x4_if(q_dst0 + qb * 1024u, s, q_bar0 + qb * 8u, (uint32_t)(lane >> 3) < C);
          st_async_f32x4_if(q_dst1 + qb * 1024u, s, q_bar1 + qb * 8u, (uint32_t)(lane >> 3) + 4u < C);
        }
      }
      named_arrive(LAG_BAR_Q + (blk & 1), bar_threads);
    };
    auto dot = [&](const RowVec<VB>& x, int i) __attribute__((always_inline)) -> float {
      float2 s = make_float2(0.0f, 0.0f);
#pragma unroll
      for (int e = 0; e < VW / 2; ++e) s = __ffma2_rn(w[i][e], row_pair<XT, VB>(x, e), s);
      return s.x + s.y;
    };
    auto load_rows = [&](int stg, RowVec<VB> (&x)[NC][B]) __attribute__((always_inline)) {
      const unsigned char* stage = ring + (uint32_t)stg * (B * row_stride);
#pragma unroll
      for (int i = 0; i < NC; ++i)
#pragma unroll
        for (int m = 0; m < B; ++m) x[i][m].load(stage + (uint32_t)m * row_stride + off[i]);
    };
    // the q rows are read ahead too where registers allow, else when they are needed
    constexpr bool AHEAD = NC == 1;
    RowVec<VB> xb[NC][B], xq[AHEAD ? 1 : NC][AHEAD ? B : 1];
    auto load_q = [&](int stg) __attribute__((always_inline)) {
      if constexpr (AHEAD) load_rows(stg, xq);
    };
    auto q_now = [&](int stg, float (&qa)[B]) __attribute__((always_inline)) {
      const unsigned char* stage = ring + (uint32_t)stg * (B * row_stride);
#pragma unroll
      for (int m = 0; m < B; ++m) {
        if constexpr (AHEAD) {
          qa[m] = dot(xq[0][m], 0);
        } else {
          qa[m] = 0.0f;
#pragma unroll
          for (int i = 0; i < NC; ++i) {
            xq[i][0].load(stage + (uint32_t)m * row_stride + off[i]);
            qa[m] += dot(xq[i][0], i);
          }
        }
      }
    };
    int sb = 0, sq = 0;  // stages of the blocks whose rows the update and q read next
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
#pragma unroll
            for (int m = 1; m < B; ++m) s = __ffma2_rn(gm[m], row_pair<XT, VB>(xb[i][m], e), s);
            w[i][e] = __fadd2_rn(w[i][e], s);
          }
      }
      if (b + 2 < nb) {
        float qa[B];
        q_now(sq, qa);
        send_q(qa, b + 2);
      }
      if (b >= -1 && b + 1 < nb) {
        if (b >= 0) load_rows(sb, xb);
        __syncwarp();
        if (lane == 0 && !wait.dead) mbar_arrive(&empty[sb]);
        if (++sb == S) sb = 0;
      }
      if (++sq == S) sq = 0;
      if (b + 3 < nb) load_q(sq);
    }
#pragma unroll
    for (int i = 0; i < NC; ++i)
#pragma unroll
      for (int e = 0; e < VW; ++e) {
        const int v0 = (i * TM + mt) * VW + e;
        if (v0 < ncols) p.W[(size_t)j * d + c_first + v0] = (e & 1) ? w[i][e / 2].y : w[i][e / 2].x;
      }
  } else if (place < pl_const) {
    // =========================== copy ======================================================================
    // Lane m requests the slice of this warp's row m of a block as one bulk copy; the copies complete on the stage's barrier.
    const int rows = B / lp.copy_warps, row0 = (place - pl_copy) * rows;
    const int RS = lp.realign ? LAG_RAW_STAGES : S;
    unsigned long long* landed = lp.realign ? rfull : full;
    unsigned long long* free_ = lp.realign ? rempty : empty;
    unsigned char* dst0 = lp.realign ? smem + L.raw : ring;
    const uint32_t dst_stride = lp.realign ? (uint32_t)L.raw_stride : row_stride;
    // sample ids of four blocks at a time, the next four on their way (a load takes longer than a block)
    uint32_t ids = nb > 0 ? idx[lane] : 0u, ids_next = nb > LAG_GROUP ? idx[32 + lane] : 0u;
    int st = 0;
    uint32_t par = 1u;  // parity of the phase that frees the stage (the first pass over the ring needs none)
    int blk = 0;
#pragma unroll 1
    for (; blk < nb; ++blk) {
      if (blk >= RS) wait(&free_[st], par, 5);
      if (__any_sync(0xffffffffu, wait.dead)) break;
      const uint32_t id = __shfl_sync(0xffffffffu, ids, (blk & (LAG_GROUP - 1)) * B + row0 + (lane & (rows - 1)));
      if ((blk & (LAG_GROUP - 1)) == LAG_GROUP - 1) {
        ids = ids_next;
        if (blk + LAG_GROUP + 1 < nb) ids_next = idx[(long long)(blk + LAG_GROUP + 1) * B + lane];
      }
      if (blk != bp.drop_block) {
        const char* src = shard + (size_t)id * ld_bytes;
        // whole 16-byte granules that hold at least one byte of the slice
        const uint32_t lead = lp.realign ? (uint32_t)((uintptr_t)src & 15u) : 0u;
        const uint32_t bytes = (lead + (uint32_t)ncols * (uint32_t)sizeof(XT) + 15u) & ~15u;
        uint32_t all = bytes * (uint32_t)rows;
        if (lp.realign) {
          all = bytes;
          for (int o = rows / 2; o > 0; o >>= 1) all += __shfl_xor_sync(0xffffffffu, all, o);
        }
        if (lane == 0) mbar_arrive_expect_tx(&landed[st], all);
        __syncwarp();
        if (lane < rows) bulk_copy_g2s(dst0 + (uint32_t)(st * B + row0 + lane) * dst_stride, src - lead, bytes, &landed[st]);
      }
      if (++st == RS) { st = 0; par ^= 1u; }
    }
    if (blk < nb) {
      // giving up: leave no copy in flight into this CTA's shared memory (bounded)
      for (int r = blk > RS ? blk - RS : 0; r < blk; ++r)
        if (r != bp.drop_block) mbar_wait_bounded(&landed[r % RS], (uint32_t)((r / RS) & 1), bp.spin_limit);
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
    int ts = 0, gs = 0, sr = 3 % S;
    uint32_t par = 0u, rpar = (uint32_t)((3 / S) & 1);
    auto take = [&](int t) __attribute__((always_inline)) {  // sums and constants of block t
      if (t >= nb) return;
      if ((t & (LAG_GROUP - 1)) == 0) wait(&cfull[(t / LAG_GROUP) & (LAG_GROUPS - 1)], (uint32_t)(t / (LAG_GROUP * LAG_GROUPS)) & 1u, 8);
      if (C == 1) {
        wait(&tbar[ts], par, 3);
        if (++ts == TB) { ts = 0; par ^= 1u; }
      } else {
        if (lane == 0 && !wait.dead) mbar_arrive_expect_tx(&gbar[gs], C * (uint32_t)(LAG_SUMS * sizeof(float)));
        wait(&gbar[gs], par, 6);
        const float4* r4 = (const float4*)(red + (size_t)gs * C * LAG_SUMS) + lane;
        float4 s = r4[0];
#pragma unroll 1
        for (uint32_t w = 1; w < C; ++w) {
          const float4 v = r4[w * (LAG_SUMS / 4)];
          s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
        }
        *((float4*)(tabs + ts * LAG_SUMS) + lane) = s;
        if (++ts == TB) ts = 0;
        if (++gs == GB) { gs = 0; par ^= 1u; }
      }
    };
#pragma unroll 1
    for (int t = -1; t < nb + 2; ++t) {
      take(t + 1);
      if (t >= 2) {  // gamma of block t - 2 goes out behind the rows of block t + 1
        if (t + 1 < nb) {
          wait(&full[sr], rpar, 1);
          if (++sr == S) { sr = 0; rpar ^= 1u; }
        }
        named_barrier(LAG_BAR_GAMMA + (t & 1), bar_threads);
      }
      if (t < 0) named_arrive(LAG_BAR_START, 64);
      else if (t < nb) named_arrive(LAG_BAR_Q + (t & 1), bar_threads);
    }
  } else if (place < pl_realign) {
    // =========================== gram =====================================================================
    const int team = (place - pl_gram) / NW, tw = (place - pl_gram) % NW;
    float* part = (float*)(smem + L.part) + (size_t)team * NW * LAG_SUMS;
    const size_t part_parity = (size_t)NT * NW * LAG_SUMS;
    int parity = 0;
    int st = team % S, gs = team % GB, ts = team % TB;
    uint32_t par = (uint32_t)((team / S) & 1);
#pragma unroll 1
    for (int b = team; b < nb; b += NT) {
      const int stp = st == 0 ? S - 1 : st - 1;
      const bool ok = mbar_try_wait(&full[st], par);
      if (b > 0) wait(&full[stp], st == 0 ? par ^ 1u : par, 1);
      wait.finish(ok, &full[st], par, 1);
      const unsigned char* xb = ring + (size_t)st * B * row_stride;
      const unsigned char* xp = b > 0 ? ring + (size_t)stp * B * row_stride : xb;  // block 0: gamma before it is zero
      float* sl = part + parity * part_parity + (size_t)tw * LAG_SUMS;
      if constexpr (sizeof(XT) == 2) {
        // A: rows 0..7 of X_b and of X_{b-1}; B: the X_b half again. Lanes 0..7 address rows 0..7 columns +0, 8..15 the
        // rows of X_{b-1} columns +0, 16..23 and 24..31 the same rows columns +8.
        float acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[a][e] = 0.0f;
        const unsigned char* src = ((lane & 8) ? xp : xb) + (size_t)(lane & 7) * row_stride + (size_t)(lane >> 4) * 16;
        const int ksteps = (my_chunks + 1) / 2;
        int ks = tw;
        for (; ks + 3 * NW < ksteps; ks += 4 * NW) {
          uint32_t x[4][4];
#pragma unroll
          for (int a = 0; a < 4; ++a) ldmatrix_x4(x[a], src + (size_t)(ks + a * NW) * 32);
#pragma unroll
          for (int a = 0; a < 4; ++a) mma_bf16_m16n8k16(acc[a], x[a][0], x[a][1], x[a][2], x[a][3], x[a][0], x[a][2]);
        }
        for (; ks < ksteps; ks += NW) {
          uint32_t x[4];
          ldmatrix_x4(x, src + (size_t)ks * 32);
          mma_bf16_m16n8k16(acc[0], x[0], x[1], x[2], x[3], x[0], x[2]);
        }
        const int g8 = lane >> 2, t4 = lane & 3;
#pragma unroll
        for (int e = 0; e < 4; ++e) acc[0][e] = (acc[0][e] + acc[1][e]) + (acc[2][e] + acc[3][e]);
        *(float2*)(sl + g8 * 8 + 2 * t4) = make_float2(acc[0][0], acc[0][1]);
        *(float2*)(sl + 64 + g8 * 8 + 2 * t4) = make_float2(acc[0][2], acc[0][3]);
      } else {
        // 16 x 8 products as 4 x 4 tiles (rows ti + 4 q of [X_b; X_{b-1}], rows 4 tn + r of X_b): 8 lanes cover them on
        // the same 4 columns, the warp's four groups of 8 lanes take different chunks and meet by shuffles.
        const int ti = lane & 3, tn = (lane >> 2) & 1, cg = lane >> 3;
        float2 acc[4][4];
#pragma unroll
        for (int a = 0; a < 4; ++a)
#pragma unroll
          for (int e = 0; e < 4; ++e) acc[a][e] = make_float2(0.0f, 0.0f);
        const unsigned char* a0 = xb + (size_t)ti * row_stride;
        const unsigned char* a1 = xp + (size_t)ti * row_stride;
        const unsigned char* b0 = xb + (size_t)(4 * tn) * row_stride;
#pragma unroll 1
        for (int ck = tw * 4 + cg; ck < my_chunks; ck += 4 * NW) {
          float4 xa[4], xn[4];
          xa[0] = *(const float4*)(a0 + (size_t)ck * 16);
          xa[1] = *(const float4*)(a0 + 4 * (size_t)row_stride + (size_t)ck * 16);
          xa[2] = *(const float4*)(a1 + (size_t)ck * 16);
          xa[3] = *(const float4*)(a1 + 4 * (size_t)row_stride + (size_t)ck * 16);
#pragma unroll
          for (int r = 0; r < 4; ++r) xn[r] = *(const float4*)(b0 + r * (size_t)row_stride + (size_t)ck * 16);
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
        const int row = ti + 4 * ((h8 ? 2 : 0) + (h16 ? 1 : 0));
        *(float4*)(sl + row * 8 + tn * 4) = make_float4(v[0], v[1], v[2], v[3]);
      }
      // the rows have been read
      __syncwarp();
      if (lane == 0 && !wait.dead) {
        mbar_arrive(&empty[st]);
        if (b > 0) mbar_arrive(&empty[stp]);
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
        if (C == 1) {
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
  } else {
    // =========================== realign =================================================================
    // A warp takes rows aw and aw + 4 of every block. Word i of the ring row comes from two neighbouring words of the
    // fetched granules, shifted by the row's offset inside its first granule; words beyond the row become zero.
    const int aw = place - pl_realign;
    const unsigned char* raw = smem + L.raw;
    const uint32_t raw_stride = (uint32_t)L.raw_stride;
    const int words = my_chunks * 4, valid_bytes = ncols * (int)sizeof(XT);
    uint32_t ids = nb > 0 ? idx[lane] : 0u, ids_next = nb > LAG_GROUP ? idx[32 + lane] : 0u;
    int rst = 0, st = 0;
    uint32_t rpar = 0u, epar = 1u;
#pragma unroll 1
    for (int b = 0; b < nb; ++b) {
      uint32_t sh[2];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t id = __shfl_sync(0xffffffffu, ids, (b & (LAG_GROUP - 1)) * B + aw + 4 * h);
        sh[h] = (uint32_t)((uintptr_t)(shard + (size_t)id * ld_bytes) & 15u);
      }
      if ((b & (LAG_GROUP - 1)) == LAG_GROUP - 1) {
        ids = ids_next;
        if (b + LAG_GROUP + 1 < nb) ids_next = idx[(long long)(b + LAG_GROUP + 1) * B + lane];
      }
      if (b >= S) wait(&empty[st], epar, 5);
      wait(&rfull[rst], rpar, 1);
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int m = aw + 4 * h;
        const uint32_t* src = (const uint32_t*)(raw + ((size_t)rst * B + m) * raw_stride) + (sh[h] >> 2);
        uint32_t* dst = (uint32_t*)(ring + ((size_t)st * B + m) * row_stride);
        const uint32_t bits = 8u * (sh[h] & 3u);
#pragma unroll 2
        for (int i = lane; i < words; i += 32) {
          uint32_t v = __funnelshift_r(src[i], src[i + 1], bits);
          const int left = valid_bytes - 4 * i;
          if (left < 4) v = left <= 0 ? 0u : (v & ((1u << (8 * left)) - 1u));
          dst[i] = v;
        }
      }
      __syncwarp();
      if (lane == 0 && !wait.dead) {
        mbar_arrive(&full[st]);
        mbar_arrive(&rempty[rst]);
      }
      if (++rst == LAG_RAW_STAGES) { rst = 0; rpar ^= 1u; }
      if (++st == S) { st = 0; epar ^= 1u; }
    }
  }
  __syncwarp();
  if (wait.dead) {  // sums sent just now may still be on their way to a peer; let them land before anyone exits
    const long long t0 = clock64();
    while (clock64() - t0 < 100000) {}
  }
  __syncwarp();
  cluster_barrier();
}

}  // namespace wpsgd
