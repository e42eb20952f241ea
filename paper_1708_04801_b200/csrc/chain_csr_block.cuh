// Per-node SGD chains on CSR rows (Eq. 5), a block of steps at a time through a shared-memory cache of the
// model entries those steps touch. One CTA per node: warp 0 runs the chain, warp 1 plans, the others prepare blocks.
//
// As in chain_csr.cuh the model of node j is w = s * u with an fp64 scalar s (the regulariser's factor
// 1 - eta_n lambda multiplies s only), and a step is
//     z = s_{n-1} (u . x);  g = L'(y, z);  s_n = s_{n-1} (1 - eta_n lambda);  u_c <- u_c - (eta_n g / s_n) x_c
// on the row's nonzeros: the iterates of Eq. 5 in exact arithmetic, for any step-size schedule.
//
// Blocks. The sample stream does not depend on the model, so the rows of the next steps are known in advance. The helper
// warps take the next up to 64 steps (at most CSRB_EMAX nonzeros in all), give every distinct column among them a slot in a
// shared-memory hash table (linear probing, one compare-and-swap per probe), store per nonzero its slot and value, and
// read u at the block's columns into the block's cache, all while the chain warp runs the previous block.
//
// Groups of 8 inside a block. In u-space nothing decays, so with kappa_n = (eta_n / s_n) L'(y_n, s_{n-1} (u . x_n)) and the
// model u_0 before the group
//     u before step n . x_n = u_0 . x_n - sum_{m < n} kappa_m (x_m . x_n).
// The products x_m . x_n of a group's rows are formed ahead by helper warps: a row's values are scattered into a dense
// array over the block's slots (one per warp) and gathered at the slots of the seven other rows. The chain warp then pays
// once per 8 steps for the gather of the model entries and the sum over lanes (four lanes per sample), runs the 8 steps on
// registers (the recurrence of chain_lag.cuh) and applies the 8 updates one after the other (a column of several
// samples must see them in turn). All of it is in shared memory.
//
// Short form (blocks of at most 640 nonzeros in rows of at most 32). Most columns are held by one row of a group only. The
// helpers find the ones that several rows hold and give each a record with its value in all 8 rows; the products come from the
// records alone. After the 8 steps the lane that read a column's entry for the margins writes it back, and one lane per record
// applies all rows' updates in order: two passes where the long form makes eight. 640 is two nonzeros per helper thread: what
// it knows of them then stays in registers. Up to 10 nonzeros per row a block of 64 steps fits (a row of 12 takes 1590
// cycles per 8 steps in the long form, one of 10 takes 1270 in this); with as many nonzeros per thread as blocks of 40 per row
// need, this form was the slower one (see form_short). Blocks of fewer steps, which would let rows of 11 to 32 take it, were not measured.
//
// Blocks of long rows (more than 64 nonzeros per step on average) take their steps one at a time: the products cost their
// helpers time in proportion to eight times the nonzeros, and with rows of more than two chunks of 32 the group is the slower
// form (uniform columns, hinge, cycles per 8 steps, group against one at a time: 64 nonzeros 6470 / 7660, 72 nonzeros 10470 / 8210,
// 200 nonzeros 34500 / 21000).
//
// For the hinge loss a decision within 1e-4 of its threshold sends the group through one step at a time, so that the order of
// the sums never turns it.
//
// What bounds it, and what it measured (cycles per 8 steps of the longest chain, B200 at 1965 MHz): 40 Zipf-distributed
// nonzeros per row, d = 2^20, hinge, 64 chains: 2740 (11.43 ms for 65536 steps; 2685 before launches overlapped; one step after the other, each with a gather, a sum over 32 lanes and a
// scatter: 3840); 5 to 10 nonzeros, d = 100000, logistic, 10 chains: 1255 (3700). With short rows the chain warp's string is
// the longer side: margins 160, steps 500, updates 300, boundary 130 of 1500 before the short form. With long rows the chain (2400) and the
// helpers (insertion 700, products 1100, copies 400 per group) take about as long; the short form took 1615 to 1230 and, at 8
// Zipf-distributed nonzeros, 1480 to 1270. Tried and taken back: margins from
// the model one group back with a table per group and the model in L2 (5900 and 3300: everything that touches single
// nonzeros is latency, and a table per 8 rows pays it eight times as often as one per block).
//
// Block boundary. The values the helpers read for block b + 1 are stale exactly at the columns block b touches, so
// at the boundary every column of block b + 1 is looked up in block b's table and, when found, takes block b's
// cached value (shared memory to shared memory). No global-memory latency is left on the chain's path: block b's
// slots are written back to u by the helpers afterwards, before they reuse its tables for block b + 2. Tables and
// caches are double buffered, plans (row extents, labels, scale factors; two blocks ahead) are threefold.
//
// Slow boundaries (rare): a row with more than CSRB_EMAX nonzeros forms a block of its own that the chain warp runs
// on global memory, 16 loads of a lane in flight (rows of 2500 nonzeros: 32500 cycles a step, 162000 with single loads); when
// the scale has fallen below 1e-12 at the start of a block it is folded into u (u <- s u, s <- 1). In both cases, and for the
// first block, all threads write the previous block back, apply the fold, and
// read the block's columns again from global memory. A block also ends early before the scale would leave the fp32
// range of the per-step factors.
//
// Column indices are checked against d when they are inserted (a bad index sets the status word and the entry is
// dropped). The kernel has no wait on anything but CTA barriers that every thread reaches the same number of times.
#pragma once

#include <type_traits>

#include "chain_csr.cuh"
#include "chain_lag.cuh"

namespace wpsgd {

constexpr int CSRB_STEPS = 64;          // most steps per block, where all rows have at most 32 nonzeros
constexpr int CSRB_LONG_STEPS = 48;     // else: as many groups as there are warps for their products
constexpr int CSRB_GROUPS = CSRB_STEPS / LAG_B;
constexpr int CSRB_EMAX = 2048;         // most nonzeros per block
constexpr int CSRB_HASH = 4096;         // slots of the column table (power of two, > CSRB_EMAX)
constexpr int CSRB_HASH_BITS = 12;
constexpr int CSRB_THREADS = 384;       // warp 0: chain; warp 1: plans; warps 2..11: preparation
constexpr int CSRB_HELPERS = CSRB_THREADS - 64;
constexpr int CSRB_GRAM_WARPS = 6;      // helper warps that also form the products of a group's rows
constexpr int CSRB_SHORT_ENT = 2 * CSRB_HELPERS;  // blocks of at most that many nonzeros in rows of at most
constexpr int CSRB_SHORT_ROW = 32;      // these take the short form
constexpr int CSRB_SLOT = CSRB_HASH - 1;  // bits of a nonzero's slot entry: the slot,
constexpr int CSRB_SHARED = 0x8000;     // and (short form) whether another row of its group holds the column
constexpr int CSRB_APART = 64;          // blocks with more nonzeros per step on average take their steps one at a time
constexpr float CSRB_NEAR = 1e-4f;      // hinge decisions with |1 - t| below this are taken one step at a time
constexpr int CSRB_DIRECT = 16;         // the same of the chain warp on a row longer than the tables
constexpr int CSRB_BATCH = 8;           // independent global loads a thread keeps in flight

// Plan of a block
struct CsrPlan {
  int nsteps;    // steps in the block (0: the chain has ended)
  int nent;      // nonzeros of those steps
  int direct;    // 1: a single long row, run on global memory
  float fold;    // != 0: multiply u by it before the block (the scale was folded back)
  long long gbeg[CSRB_STEPS];          // first nonzero of the step's row in col_idx / val
  int4 step[CSRB_STEPS];               // per step: first nonzero within the block, nonzeros, label bits, scale-before bits
  float eos[CSRB_STEPS];               // eta_n / scale after the step
  LagConst k[CSRB_GROUPS];             // constants of a group of 8 steps
  int longest;                         // most nonzeros of a row of the block
  int brief;                           // the block takes the short form
  int apart;                           // its steps are run one at a time
  int pad[1];
};

// One buffer of a prepared block.
struct CsrBlockBuf {
  int keys[CSRB_HASH];                 // column of every slot, -1 = free
  float val[CSRB_EMAX];                // value of every nonzero, rows one after the other
  unsigned short slot[CSRB_EMAX];      // slot of every nonzero
  unsigned short uslot[CSRB_EMAX];     // the occupied slots, in order of first insertion
  float gram[CSRB_GROUPS][64];         // products of the rows of a group, [8][8], below the diagonal
  union {
    int col[CSRB_EMAX];                // columns of the nonzeros, until they have their slots
    float shared_x[CSRB_SHORT_ENT / 2][8];  // short form: value of every shared column in each of the 8 rows of its group,
  };
  unsigned short shared_slot[CSRB_SHORT_ENT / 2];  // its slot,
  int2 records[CSRB_GROUPS];           // first shared column of a group and how many
  int nuniq;                           // distinct columns (filled while inserting; 0 again once the block has been written back)
  int pad[3];
};

struct CsrBlockSmem {
  CsrBlockBuf buf[2];
  CsrPlan plan[3];
  float ucache[2][CSRB_HASH];          // u at the columns of a block, by slot
  float dense[CSRB_GRAM_WARPS][CSRB_HASH];  // one row at a time, by slot; zero in between
  unsigned votes[32];                  // per 32 nonzeros: which are the first of a shared column in their group
  int before[32];                      // how many there are before these
  float4 jets[8];
};

// Shared-memory accesses by 32-bit shared-window address. The block buffers are chosen at run time (b & 1), so the
// hot loops name the state space themselves instead of leaving it to address-space inference.
__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ float lds_f32(uint32_t a) {
  float v;
  asm volatile("ld.shared.f32 %0, [%1];" : "=f"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ int lds_s32(uint32_t a) {
  int v;
  asm volatile("ld.shared.s32 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ int lds_u16(uint32_t a) {
  unsigned short v;
  asm volatile("ld.shared.u16 %0, [%1];" : "=h"(v) : "r"(a));
  return (int)v;
}
__device__ __forceinline__ int lds_u8(uint32_t a) {
  int v;
  asm volatile("ld.shared.u8 %0, [%1];" : "=r"(v) : "r"(a));
  return v;
}
__device__ __forceinline__ int2 lds_s32x2(uint32_t a) {
  int2 v;
  asm volatile("ld.shared.v2.s32 {%0,%1}, [%2];" : "=r"(v.x), "=r"(v.y) : "r"(a));
  return v;
}
__device__ __forceinline__ int4 lds_s32x4(uint32_t a) {
  int4 v;
  asm volatile("ld.shared.v4.s32 {%0,%1,%2,%3}, [%4];" : "=r"(v.x), "=r"(v.y), "=r"(v.z), "=r"(v.w) : "r"(a));
  return v;
}
__device__ __forceinline__ void sts_u16(uint32_t a, int v) {
  asm volatile("st.shared.u16 [%0], %1;" ::"r"(a), "h"((unsigned short)v) : "memory");
}
// Where `yes`: a predicate, not a branch. (Branches around single accesses, even ones that all lanes take alike, cost more
// than the accesses: they end the stretch of code in which loads overlap.)
__device__ __forceinline__ void cp_async4_if(uint32_t smem_dst, const void* gmem_src, bool yes) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p cp.async.ca.shared.global [%0], [%1], 4;\n\t}" ::"r"(smem_dst), "l"(gmem_src), "r"((int)yes) : "memory");
}
__device__ __forceinline__ void atoms_cas_if(int& old, uint32_t a, int cmp, int val, bool yes) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %4, 0;\n\t@p atom.shared.cas.b32 %0, [%1], %2, %3;\n\t}" : "+r"(old) : "r"(a), "r"(cmp), "r"(val), "r"((int)yes) : "memory");
}
__device__ __forceinline__ void lds_s32_if(int& v, uint32_t a, bool yes) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p ld.shared.s32 %0, [%1];\n\t}" : "+r"(v) : "r"(a), "r"((int)yes) : "memory");
}
__device__ __forceinline__ void sts_u16_if(uint32_t a, int v, bool yes) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.shared.u16 [%0], %1;\n\t}" ::"r"(a), "h"((unsigned short)v), "r"((int)yes) : "memory");
}
__device__ __forceinline__ void reds_or_if(uint32_t a, uint32_t v, bool yes) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p red.shared.or.b32 [%0], %1;\n\t}" ::"r"(a), "r"(v), "r"((int)yes) : "memory");
}
__device__ __forceinline__ void sts_u8_if(uint32_t a, int v, bool yes) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.shared.u8 [%0], %1;\n\t}" ::"r"(a), "r"(v), "r"((int)yes) : "memory");
}
__device__ __forceinline__ void sts_zero32_if(uint32_t a, bool yes) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.shared.v4.f32 [%0], {%1, %1, %1, %1};\n\t@p st.shared.v4.f32 [%0+16], {%1, %1, %1, %1};\n\t}" ::"r"(a), "f"(0.0f), "r"((int)yes) : "memory");
}
__device__ __forceinline__ void prefetch_l2_if(const void* a, bool yes) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %1, 0;\n\t@p prefetch.global.L2 [%0];\n\t}" ::"l"(a), "r"((int)yes) : "memory");
}
__device__ __forceinline__ void sts_f32_if(uint32_t a, float v, bool yes) {
  asm volatile("{\n\t.reg .pred p;\n\tsetp.ne.s32 p, %2, 0;\n\t@p st.shared.f32 [%0], %1;\n\t}" ::"r"(a), "f"(v), "r"((int)yes) : "memory");
}
__device__ __forceinline__ int atoms_add(uint32_t a, int val) {
  int old;
  asm volatile("atom.shared.add.s32 %0, [%1], %2;" : "=r"(old) : "r"(a), "r"(val) : "memory");
  return old;
}

__device__ __forceinline__ int csrb_hash(int col) { return (int)(((uint32_t)col * 0x9E3779B1u) >> (32 - CSRB_HASH_BITS)); }

// cache[slot] <- u[column of slot] for the block's distinct columns i = t0, t0 + stride, ...; CSRB_BATCH loads in flight.
// (Beyond the list the first column is read and written again.)
__device__ __forceinline__ void csrb_gather(const CsrBlockBuf& B, float* cache, const float* u, int nuniq, int t0, int stride) {
  for (int base = t0; base < nuniq; base += stride * CSRB_BATCH) {
    int h[CSRB_BATCH], c[CSRB_BATCH];
    float v[CSRB_BATCH];
#pragma unroll
    for (int g = 0; g < CSRB_BATCH; ++g) h[g] = B.uslot[base + g * stride < nuniq ? base + g * stride : 0];
#pragma unroll
    for (int g = 0; g < CSRB_BATCH; ++g) c[g] = B.keys[h[g]];
#pragma unroll
    for (int g = 0; g < CSRB_BATCH; ++g) v[g] = __ldcg(u + c[g]);
#pragma unroll
    for (int g = 0; g < CSRB_BATCH; ++g) cache[h[g]] = v[g];
  }
}

// u[column of slot] <- cache[slot] for the block's distinct columns, and the table is emptied.
__device__ __forceinline__ void csrb_scatter(CsrBlockBuf& B, const float* cache, float* u, int nuniq, int t0, int stride) {
  for (int i = t0; i < nuniq; i += stride) {
    const int h = B.uslot[i];
    u[B.keys[h]] = cache[h];
    B.keys[h] = -1;
  }
}

// SHORT: the chain's blocks may take the short form
template <int LOSS, bool SHORT>
__device__ __forceinline__ void chain_csr_block(const CsrParams& p, CsrBlockSmem& sm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int j = p.order[blockIdx.x];
  const long long n_run = p.n_steps[j];
  const long long first = p.resume ? p.first[j] : 0;
  const long long* rp = p.row_ptr + p.shard_off[j];
  const float* yshard = p.y + p.shard_off[j];
  const uint32_t* idx = p.idx + p.idx_off[j];
  float* u = p.U + (size_t)j * p.d;

  for (int i = threadIdx.x; i < CSRB_HASH; i += CSRB_THREADS) {
    sm.buf[0].keys[i] = -1;
    sm.buf[1].keys[i] = -1;
    for (int w = 0; w < CSRB_GRAM_WARPS; ++w) sm.dense[w][i] = 0.0f;
  }
  if (threadIdx.x < 2) sm.buf[threadIdx.x].nuniq = 0;

  // ---- plan of the next block (planner warp) -----------------------------------------------------------------------
  long long s_next = 0;                          // first step of the next block to plan
  double sc = p.resume ? p.scale[j] : 1.0;       // scale after the last planned step
  const double lam = (double)p.lambda, eta0 = (double)p.eta0;
  auto plan_next = [&](CsrPlan& B) {
    float fold = 0.0f;
    if (sc < 1e-12 && s_next < n_run) {  // only ahead of a block that runs: the fold is applied at its start
      fold = (float)sc;
      sc = 1.0;
    }
    // row extents and labels of the next steps, all loads in flight together
    constexpr int PARTS = (CSRB_STEPS + 31) / 32;
    long long gb[PARTS], ge[PARTS];
    float yy[PARTS];
    uint32_t ri[PARTS];
#pragma unroll
    for (int part = 0; part < PARTS; ++part) {
      const long long s = s_next + part * 32 + lane;
      ri[part] = s < n_run ? idx[s] : 0u;
    }
#pragma unroll
    for (int part = 0; part < PARTS; ++part) {
      const long long s = s_next + part * 32 + lane;
      gb[part] = ge[part] = 0;
      yy[part] = 0.0f;
      if (s < n_run) {
        gb[part] = rp[ri[part]];
        ge[part] = rp[ri[part] + 1];
        yy[part] = yshard[ri[part]];
      }
    }
    bool lean = true;
#pragma unroll
    for (int part = 0; part < PARTS; ++part) lean = lean && ge[part] - gb[part] <= 32;
    const int limit = __all_sync(0xffffffffu, lean) ? CSRB_STEPS : CSRB_LONG_STEPS;
    int nsteps = 0, nent = 0, direct = 0, longest = 0;
    bool more = true;
#pragma unroll
    for (int part = 0; part < PARTS; ++part) {
      if (!more) break;
      const long long s = s_next + part * 32 + lane;
      const bool valid = s < n_run;
      const long long len = ge[part] - gb[part];
      const int cnt = len > (long long)CSRB_EMAX ? CSRB_EMAX + 1 : (len < 0 ? 0 : (int)len);
      const double eta = p.sched == LR_INV_SQRT ? eta0 / sqrt((double)(first + s + 1)) : eta0;
      const double a = valid ? 1.0 - eta * lam : 1.0;
      int icnt = cnt;
      double ia = a;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int c2 = __shfl_up_sync(0xffffffffu, icnt, o);
        const double a2 = __shfl_up_sync(0xffffffffu, ia, o);
        if (lane >= o) {
          icnt += c2;
          ia *= a2;
        }
      }
      double ea = __shfl_up_sync(0xffffffffu, ia, 1);
      if (lane == 0) ea = 1.0;
      const bool ok = valid && (part * 32 + lane < limit) && (nent + icnt <= CSRB_EMAX) && (sc * ea >= 1e-30);
      const unsigned mask = __ballot_sync(0xffffffffu, ok);
      const int n_ok = (mask == 0xffffffffu) ? 32 : (__ffs((int)~mask) - 1);
      if (lane < n_ok) {
        const int r = nsteps + lane;
        const float sb = (float)(sc * ea), eos = (float)(eta / (sc * ia)), y = yy[part];
        B.gbeg[r] = gb[part];
        B.step[r] = make_int4(nent + icnt - cnt, cnt, __float_as_int(y), __float_as_int(sb));
        B.eos[r] = eos;
        // kappa_n = a f(sc r_n), see LagConst
        LagConst& K = B.k[r >> 3];
        if (LOSS == LOSS_SQUARED) {  // loss derivative s r - y
          K.a[r & 7] = eos * sb;
          K.b[r & 7] = -eos * y;
          K.sc[r & 7] = sb;
        } else {                     // hinge: -y where y s r < 1; logistic: -y / (1 + 2^(y s log2(e) r))
          const float ks = LOSS == LOSS_LOGISTIC ? y * sb * 1.4426950408889634f : y * sb;
          K.a[r & 7] = -y * eos;
          K.b[r & 7] = -LAG_STEP * ks;
          K.sc[r & 7] = ks;
        }
        // the row's nonzeros are copied a block from now
        for (int o = 0; o < cnt; o += 32) {
          asm volatile("prefetch.global.L2 [%0];" ::"l"(p.col_idx + gb[part] + o));
          asm volatile("prefetch.global.L2 [%0];" ::"l"(p.val + gb[part] + o));
        }
      }
      longest = max(longest, (int)__reduce_max_sync(0xffffffffu, lane < n_ok ? (unsigned)cnt : 0u));
      // a first row that does not fit the tables: a block of its own, run on global memory
      const int lone = __shfl_sync(0xffffffffu, (part == 0 && n_ok == 0 && valid) ? 1 : 0, 0);
      if (lone) {
        if (lane == 0) {
          B.gbeg[0] = gb[part];
          B.gbeg[1] = ge[part];  // the row's end travels in the unused second entry
          B.step[0] = make_int4(0, 0, __float_as_int(yy[part]), __float_as_int((float)sc));
          B.eos[0] = (float)(eta / (sc * a));
        }
        direct = 1;
        nsteps = 1;
        nent = 0;
        sc *= __shfl_sync(0xffffffffu, a, 0);
        more = false;
      } else {
        if (n_ok > 0) {
          nent += __shfl_sync(0xffffffffu, icnt, n_ok - 1);
          sc *= __shfl_sync(0xffffffffu, ia, n_ok - 1);
          nsteps += n_ok;
        }
        if (n_ok < 32) more = false;
      }
    }
    if (!direct) {
      // steps that fill up the last group take no step
      const int r = nsteps + lane;
      if (lane < 8 && r < (nsteps + 7) / 8 * 8) {
        B.step[r] = make_int4(nent, 0, 0, 0);
        B.k[r >> 3].a[r & 7] = B.k[r >> 3].b[r & 7] = B.k[r >> 3].sc[r & 7] = 0.0f;
      }
      __syncwarp();
      if (lane < CSRB_GROUPS && 8 * lane < nsteps) {
        float mx = 0.0f;
        for (int m = 0; m < 8; ++m) mx = fmaxf(mx, fabsf(B.k[lane].sc[m]));
        B.k[lane].sc_max = mx;
      }
    }
    if (lane == 0) {
      B.nsteps = nsteps;
      B.nent = nent;
      B.longest = longest;
      B.brief = !direct && longest <= CSRB_SHORT_ROW && nent <= CSRB_SHORT_ENT;
      B.apart = nent > CSRB_APART * nsteps;
      B.direct = direct;
      B.fold = fold;
    }
    s_next += nsteps;
  };

  // ---- products of the rows of one group (a helper warp with a dense array of its own) -----------------------------------
  // CH: chunks of 32 nonzeros of a row in registers; REST: some row may have more. Compiled for each, so that the unrolled
  // code has no branches (with guards inside it the same loads took four times as long).
  auto form_gram = [&](const CsrBlockBuf& B, const CsrPlan& P, int gi, float* dense, float* out, auto ch_tag, auto rest_tag) {
    constexpr int CH = decltype(ch_tag)::value;
    constexpr bool REST = decltype(rest_tag)::value;
    const uint32_t dense_a = smem_addr(dense), slot_a = smem_addr(B.slot), val_a = smem_addr(B.val), step_a = smem_addr(P.step);
    int beg[8], cnt[8];
    uint32_t sl[CH][8];
    float v[CH][8], acc[32];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      const int4 st = lds_s32x4(step_a + 16u * (uint32_t)(8 * gi + m));
      beg[m] = st.x;
      cnt[m] = st.y;
    }
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        // lanes beyond the row read the block's first nonzero and take the value 0
        const int e = lane + 32 * c < cnt[m] ? beg[m] + lane + 32 * c : 0;
        sl[c][m] = (uint32_t)lds_u16(slot_a + 2u * (uint32_t)e);
        v[c][m] = lds_f32(val_a + 4u * (uint32_t)e);
      }
#pragma unroll
    for (int m = 0; m < 8; ++m)
#pragma unroll
      for (int c = 0; c < CH; ++c) {
        sl[c][m] = dense_a + 4u * sl[c][m];
        if (lane + 32 * c >= cnt[m]) v[c][m] = 0.0f;
      }
#pragma unroll
    for (int i = 0; i < 32; ++i) acc[i] = 0.0f;
#pragma unroll
    for (int m = 0; m < 7; ++m) {
#pragma unroll
      for (int c = 0; c < CH; ++c) sts_f32_if(sl[c][m], v[c][m], lane + 32 * c < cnt[m]);
      if constexpr (REST)
        for (int o = lane + 32 * CH; o < cnt[m]; o += 32) dense[B.slot[beg[m] + o]] = B.val[beg[m] + o];
      __syncwarp();
      float x[CH][8];
#pragma unroll
      for (int n = m + 1; n < 8; ++n)
#pragma unroll
        for (int c = 0; c < CH; ++c) x[c][n] = lds_f32(sl[c][n]);
#pragma unroll
      for (int n = m + 1; n < 8; ++n) {
        float t = x[0][n] * v[0][n];
#pragma unroll
        for (int c = 1; c < CH; ++c) t = fmaf(x[c][n], v[c][n], t);
        if constexpr (REST)
          for (int o = lane + 32 * CH; o < cnt[n]; o += 32) t = fmaf(dense[B.slot[beg[n] + o]], B.val[beg[n] + o], t);
        acc[n * (n - 1) / 2 + m] = t;
      }
      __syncwarp();
#pragma unroll
      for (int c = 0; c < CH; ++c) sts_f32_if(sl[c][m], 0.0f, lane + 32 * c < cnt[m]);
      if constexpr (REST)
        for (int o = lane + 32 * CH; o < cnt[m]; o += 32) dense[B.slot[beg[m] + o]] = 0.0f;
      __syncwarp();
    }
    const float tot = warp_transpose_sum32(acc);  // lane l: product number l
    int n2 = 1, m2 = lane;
    while (n2 < 8 && m2 >= n2) { m2 -= n2; ++n2; }
    if (n2 < 8) out[8 * n2 + m2] = tot;
  };

  // ---- short form of a block (few nonzeros, short rows; helper warps) -----------------------------------------------------
  // Slots, then the columns that rows of a group share: only these contribute to the products of its rows, and only these need
  // their updates one after the other. Thread ht takes the nonzeros ht + 320 i, i < F, whatever their rows, and keeps
  // what it knows of them in registers; a cell per group and slot collects the rows that hold the column and then the number
  // of its record. (For blocks of 2000 nonzeros the same form takes longer than form_gram, which leaves four warps to read
  // the model meanwhile: 3950 against 2950 cycles per 8 steps at 40 Zipf-distributed nonzeros per row.)
  auto form_short = [&](CsrBlockBuf& B, float* cache, const CsrPlan& P) __attribute__((always_inline)) {
    constexpr int F = CSRB_SHORT_ENT / CSRB_HELPERS;
    constexpr int W = CSRB_HELPERS / 32;
    static_assert(F * W <= 31, "one lane per 32 nonzeros, and one more");
    const int ht = (int)threadIdx.x - 64, hw = warp - 2;
    const int nsteps = P.nsteps, nent = P.nent;
    const unsigned below = (1u << lane) - 1u;
    const uint32_t keys_a = smem_addr(B.keys), slot_a = smem_addr(B.slot), uslot_a = smem_addr(B.uslot), val_a = smem_addr(B.val);
    const uint32_t col_a = smem_addr(B.col), nuniq_a = smem_addr(&B.nuniq), cell_a = smem_addr(sm.dense);
    const uint32_t rslot_a = smem_addr(B.shared_slot), rec_a = smem_addr(B.shared_x), cache_a = smem_addr(cache);
    int col[F], h[F], k2[F], r[F];
    bool in[F], seek[F], several[F], first[F];
    bool any_bad = false;
#pragma unroll
    for (int i = 0; i < F; ++i) {
      in[i] = seek[i] = ht + CSRB_HELPERS * i < nent;
      const uint32_t e = (uint32_t)(in[i] ? ht + CSRB_HELPERS * i : 0);
      col[i] = lds_s32(col_a + 4u * e);
      r[i] = lds_u16(slot_a + 2u * e) & (CSRB_STEPS - 1);  // the copies' note
      k2[i] = 0;
    }
#pragma unroll
    for (int i = 0; i < F; ++i) any_bad |= in[i] && (unsigned long long)(long long)col[i] >= (unsigned long long)p.d;
    if (any_bad) {
#pragma unroll
      for (int i = 0; i < F; ++i)
        if (in[i] && (unsigned long long)(long long)col[i] >= (unsigned long long)p.d) {
          set_status(p.status, DEV_BOUNDS, 21, (long long)col[i]);
          col[i] = 0;
          B.val[ht + CSRB_HELPERS * i] = 0.0f;
        }
    }
#pragma unroll
    for (int i = 0; i < F; ++i) h[i] = csrb_hash(col[i]);
    // until none of the warp's nonzeros has met another column
    for (int probe = 0; probe < CSRB_HASH; ++probe) {
#pragma unroll
      for (int i = 0; i < F; ++i) atoms_cas_if(k2[i], keys_a + 4u * (uint32_t)h[i], -1, col[i], seek[i]);
      bool any = false;
#pragma unroll
      for (int i = 0; i < F; ++i) {
        seek[i] = seek[i] && k2[i] != -1 && k2[i] != col[i];
        h[i] = seek[i] ? (h[i] + 1) & (CSRB_HASH - 1) : h[i];
        any |= seek[i];
      }
      if (!__any_sync(0xffffffffu, any)) break;
    }
    // which rows of its group hold a column: one bit per row in the cell of group and slot
    uint32_t ca[F];
#pragma unroll
    for (int i = 0; i < F; ++i) {
      ca[i] = cell_a + (uint32_t)((r[i] >> 3) * CSRB_HASH + h[i]);
      reds_or_if(ca[i] & ~3u, 1u << (8 * (ca[i] & 3u) + (r[i] & 7)), in[i]);
    }
    // one counter update per warp for the columns seen for the first time
    unsigned votes[F];
    int total = 0;
#pragma unroll
    for (int i = 0; i < F; ++i) {
      votes[i] = __ballot_sync(0xffffffffu, in[i] && k2[i] == -1);
      total += __popc(votes[i]);
    }
    int base = 0;
    if (lane == 0) base = atoms_add(nuniq_a, total);
    base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
    for (int i = 0; i < F; ++i) {
      const bool fresh = in[i] && k2[i] == -1;
      prefetch_l2_if(u + col[i], fresh);  // the block's read of u[col] follows soon
      sts_u16_if(uslot_a + 2u * (uint32_t)(base + __popc(votes[i] & below)), h[i], fresh);
      base += __popc(votes[i]);
    }
    named_barrier(1, CSRB_HELPERS);  // table, list of distinct columns and cells are complete
    int gh[F];
    float gu[F];
    const int nuniq = B.nuniq;
#pragma unroll
    for (int i = 0; i < F; ++i) gh[i] = lds_u16(uslot_a + 2u * (uint32_t)(ht + CSRB_HELPERS * i < nuniq ? ht + CSRB_HELPERS * i : 0)) & CSRB_SLOT;
#pragma unroll
    for (int i = 0; i < F; ++i) k2[i] = lds_s32(keys_a + 4u * (uint32_t)gh[i]);
#pragma unroll
    for (int i = 0; i < F; ++i) gu[i] = __ldcg(u + (ht + CSRB_HELPERS * i < nuniq ? k2[i] : 0));
    // the first row to hold a shared column gives it a record; records are numbered in the order of the nonzeros
#pragma unroll
    for (int i = 0; i < F; ++i) col[i] = lds_u8(ca[i]);
#pragma unroll
    for (int i = 0; i < F; ++i) {
      several[i] = in[i] && (col[i] & (col[i] - 1)) != 0;
      first[i] = several[i] && (col[i] & ((1 << (r[i] & 7)) - 1)) == 0;
      votes[i] = __ballot_sync(0xffffffffu, first[i]);
      if (lane == 0) sm.votes[i * W + hw] = votes[i];
    }
    named_barrier(1, CSRB_HELPERS);
    {  // (every warp writes the same numbers)
      const int n = lane < F * W ? __popc(sm.votes[lane]) : 0;
      int sum = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, sum, o);
        sum += lane >= o ? v : 0;
      }
      sm.before[lane] = sum - n;
    }
    __syncwarp();
    int rec0;  // lane g: the first record of group g
    {
      const int x = 8 * lane < nsteps && lane < CSRB_GROUPS ? P.step[8 * lane].x : nent;
      rec0 = min(sm.before[x >> 5] + __popc(sm.votes[x >> 5] & ((1u << (x & 31)) - 1u)), CSRB_SHORT_ENT / 2);
      const int next = __shfl_down_sync(0xffffffffu, rec0, 1);
      if (hw == 0 && lane < CSRB_GROUPS) B.records[lane] = make_int2(rec0, next - rec0);
    }
#pragma unroll
    for (int i = 0; i < F; ++i) {
      const int rec = sm.before[i * W + hw] + __popc(votes[i] & below);
      const int rel = rec - __shfl_sync(0xffffffffu, rec0, r[i] >> 3);
      const bool write = in[i] && first[i] == several[i];
      sts_u8_if(ca[i], first[i] ? rel : 0, write);
      const bool mine = first[i] && rec < CSRB_SHORT_ENT / 2;  // (more only where a row holds a column twice)
      sts_u16_if(rslot_a + 2u * (uint32_t)rec, h[i], mine);
      sts_zero32_if(rec_a + 32u * (uint32_t)rec, mine);
    }
    named_barrier(1, CSRB_HELPERS);
    float v[F];
#pragma unroll
    for (int i = 0; i < F; ++i) {
      col[i] = lds_u8(ca[i]);
      v[i] = lds_f32(val_a + 4u * (uint32_t)(in[i] ? ht + CSRB_HELPERS * i : 0));
    }
#pragma unroll
    for (int i = 0; i < F; ++i) {
      const int rec = __shfl_sync(0xffffffffu, rec0, r[i] >> 3) + col[i];
      sts_f32_if(rec_a + 32u * (uint32_t)rec + 4u * (uint32_t)(r[i] & 7), v[i], several[i] && rec < CSRB_SHORT_ENT / 2);
      sts_u16_if(slot_a + 2u * (uint32_t)(ht + CSRB_HELPERS * i), several[i] ? h[i] | CSRB_SHARED : h[i], in[i]);
      sts_f32_if(cache_a + 4u * (uint32_t)gh[i], gu[i], ht + CSRB_HELPERS * i < nuniq);
    }
    named_barrier(1, CSRB_HELPERS);  // records are complete
#pragma unroll
    for (int i = 0; i < F; ++i) sts_u8_if(ca[i], 0, several[i]);
    // products of the rows of a group: only shared columns contribute
    if (8 * hw < nsteps) {
      const int g0 = __shfl_sync(0xffffffffu, rec0, hw), n_rec = __shfl_sync(0xffffffffu, rec0, hw + 1) - g0;
      float acc[32];
#pragma unroll
      for (int i = 0; i < 32; ++i) acc[i] = 0.0f;
#pragma unroll 1
      for (int i = lane; i - lane < n_rec; i += 32) {
        const float4* r4 = (const float4*)B.shared_x[i < n_rec ? g0 + i : 0];
        const float in_f = i < n_rec ? 1.0f : 0.0f;
        const float4 lo = r4[0], hi = r4[1];
        const float x[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int n = 1; n < 8; ++n) {
          const float xn = in_f != 0.0f ? x[n] : 0.0f;
#pragma unroll
          for (int m = 0; m < n; ++m) acc[n * (n - 1) / 2 + m] = fmaf(xn, in_f != 0.0f ? x[m] : 0.0f, acc[n * (n - 1) / 2 + m]);
        }
      }
      const float tot = warp_transpose_sum32(acc);  // lane l: product number l
      int n2 = 1, m2 = lane;
      while (n2 < 8 && m2 >= n2) { m2 -= n2; ++n2; }
      if (n2 < 8) B.gram[hw][8 * n2 + m2] = tot;
    }
  };

  // ---- preparation of one block (helper warps only); writes the block that was in these tables back first ------------------
  auto prepare = [&](CsrBlockBuf& B, float* cache, const CsrPlan& P) {
    const int ht = (int)threadIdx.x - 64, hw = warp - 2;
    const int nsteps = P.nsteps, nent = P.nent, old = B.nuniq;
    const bool have = !P.direct && nsteps > 0;
    if (have) {
      // nonzeros of the block's rows: asynchronous 4-byte copies, all in flight together
      constexpr int W = CSRB_HELPERS / 32, ROWS = (CSRB_STEPS + W - 1) / W;
      int off[ROWS], cnt[ROWS];
      long long g0[ROWS];
#pragma unroll
      for (int i = 0; i < ROWS; ++i) {
        const int r = hw + W * i < nsteps ? hw + W * i : 0;
        off[i] = P.step[r].x;
        cnt[i] = hw + W * i < nsteps ? P.step[r].y : 0;
        g0[i] = P.gbeg[r];
      }
      const uint32_t col_a = smem_addr(B.col), val_a = smem_addr(B.val);
#pragma unroll
      for (int i = 0; i < ROWS; ++i)
#pragma unroll
        for (int o = 0; o < 64; o += 32) {
          cp_async4_if(col_a + 4u * (uint32_t)(off[i] + lane + o), p.col_idx + g0[i] + lane + o, lane + o < cnt[i]);
          cp_async4_if(val_a + 4u * (uint32_t)(off[i] + lane + o), p.val + g0[i] + lane + o, lane + o < cnt[i]);
        }
      if (SHORT && P.brief) {  // a nonzero's row, for form_short
#pragma unroll
        for (int i = 0; i < ROWS; ++i) sts_u16_if(smem_addr(B.slot) + 2u * (uint32_t)(off[i] + lane), hw + W * i, lane < cnt[i]);
      }
      if (P.longest > 64)
        for (int i = 0; i < ROWS; ++i)
          for (int o = lane + 64; o < cnt[i]; o += 32) {
            cp_async4(&B.col[off[i] + o], p.col_idx + g0[i] + o);
            cp_async4(&B.val[off[i] + o], p.val + g0[i] + o);
          }
    }
    cp_async_commit();
    csrb_scatter(B, cache, u, old, ht, CSRB_HELPERS);
    cp_async_wait(0);
    named_barrier(1, CSRB_HELPERS);  // every helper's copies have landed, the table is empty
    if (ht == 0) B.nuniq = 0;
    named_barrier(1, CSRB_HELPERS);
    if (!have) return;
    if (SHORT && P.brief) {
      form_short(B, cache, P);
      return;
    }
    const uint32_t keys_a = smem_addr(B.keys), slot_a = smem_addr(B.slot), uslot_a = smem_addr(B.uslot);
    const uint32_t col_a = smem_addr(B.col), nuniq_a = smem_addr(&B.nuniq);
    constexpr int F = 4;  // nonzeros of a thread that probe together
    for (int e0 = 0; e0 < nent; e0 += F * CSRB_HELPERS) {  // the same trip count for every lane of a warp
      int e[F], col[F], h[F], k2[F];
      bool in[F], seek[F];
      bool any_bad = false;
#pragma unroll
      for (int i = 0; i < F; ++i) {
        e[i] = e0 + ht + CSRB_HELPERS * i;
        in[i] = seek[i] = e[i] < nent;
        col[i] = lds_s32(col_a + 4u * (uint32_t)(in[i] ? e[i] : 0));
        k2[i] = 0;
      }
#pragma unroll
      for (int i = 0; i < F; ++i) any_bad |= in[i] && (unsigned long long)(long long)col[i] >= (unsigned long long)p.d;
      if (any_bad) {
#pragma unroll
        for (int i = 0; i < F; ++i)
          if (in[i] && (unsigned long long)(long long)col[i] >= (unsigned long long)p.d) {
            set_status(p.status, DEV_BOUNDS, 21, (long long)col[i]);
            col[i] = 0;
            B.val[e[i]] = 0.0f;
          }
      }
#pragma unroll
      for (int i = 0; i < F; ++i) h[i] = csrb_hash(col[i]);
      // until none of the warp's nonzeros has met another column
      for (int probe = 0; probe < CSRB_HASH; ++probe) {
#pragma unroll
        for (int i = 0; i < F; ++i) atoms_cas_if(k2[i], keys_a + 4u * (uint32_t)h[i], -1, col[i], seek[i]);
        bool any = false;
#pragma unroll
        for (int i = 0; i < F; ++i) {
          seek[i] = seek[i] && k2[i] != -1 && k2[i] != col[i];
          h[i] = seek[i] ? (h[i] + 1) & (CSRB_HASH - 1) : h[i];
          any |= seek[i];
        }
        if (!__any_sync(0xffffffffu, any)) break;
      }
      // one counter update per warp for the columns seen for the first time
      unsigned f[F];
      int total = 0;
#pragma unroll
      for (int i = 0; i < F; ++i) {
        f[i] = __ballot_sync(0xffffffffu, in[i] && k2[i] == -1);
        total += __popc(f[i]);
      }
      int base = 0;
      if (lane == 0) base = atoms_add(nuniq_a, total);
      base = __shfl_sync(0xffffffffu, base, 0);
#pragma unroll
      for (int i = 0; i < F; ++i) {
        if (in[i]) sts_u16(slot_a + 2u * (uint32_t)e[i], h[i]);
        if (in[i] && k2[i] == -1) {
          asm volatile("prefetch.global.L2 [%0];" ::"l"(u + col[i]));  // the block's read of u[col] follows soon
          sts_u16(uslot_a + 2u * (uint32_t)(base + __popc(f[i] & ((1u << lane) - 1u))), h[i]);
        }
        base += __popc(f[i]);
      }
    }
    named_barrier(1, CSRB_HELPERS);  // slots and the list of distinct columns are complete
    if (!SHORT && P.apart) {
      csrb_gather(B, cache, u, B.nuniq, ht, CSRB_HELPERS);
    } else if (hw < CSRB_GRAM_WARPS) {
      for (int gi = hw; 8 * gi < nsteps; gi += CSRB_GRAM_WARPS) {
        using std::integral_constant;
        if (P.longest <= 32) form_gram(B, P, gi, sm.dense[hw], B.gram[gi], integral_constant<int, 1>(), std::false_type());
        else if (SHORT) form_gram(B, P, gi, sm.dense[hw], B.gram[gi], integral_constant<int, 1>(), std::true_type());
        else if (P.longest <= 64) form_gram(B, P, gi, sm.dense[hw], B.gram[gi], integral_constant<int, 2>(), std::false_type());
        else form_gram(B, P, gi, sm.dense[hw], B.gram[gi], integral_constant<int, 2>(), std::true_type());
      }
    } else {
      // u at the block's columns (stale where the running block writes: see the boundary)
      csrb_gather(B, cache, u, B.nuniq, ht - 32 * CSRB_GRAM_WARPS, CSRB_HELPERS - 32 * CSRB_GRAM_WARPS);
    }
  };

  // ---- the steps of a block in groups of 8, chain warp, in shared memory --------------------------------------------------
  // Steps r0 .. r1 - 1 one at a time, each margin from the model as it then is: for a group in which a hinge decision comes so
  // near its threshold that the sums' order could turn it.
  auto one_by_one = [&](const CsrBlockBuf& B, const CsrPlan& P, float* cache, int r0, int r1) {
#pragma unroll 1
    for (int r = r0; r < r1; ++r) {
      const int4 st = P.step[r];
      const int beg = st.x, cnt = st.y;
      const bool in0 = lane < cnt, in1 = lane + 32 < cnt;
      const int h0 = in0 ? B.slot[beg + lane] & CSRB_SLOT : 0, h1 = in1 ? B.slot[beg + lane + 32] & CSRB_SLOT : 0;
      const float v0 = in0 ? B.val[beg + lane] : 0.0f, v1 = in1 ? B.val[beg + lane + 32] : 0.0f;
      const float u0 = in0 ? cache[h0] : 0.0f, u1 = in1 ? cache[h1] : 0.0f;
      float part = fmaf(u1, v1, u0 * v0);
      for (int o = lane + 64; o < cnt; o += 32) part = fmaf(cache[B.slot[beg + o] & CSRB_SLOT], B.val[beg + o], part);
      const float acc = warp_sum(part);
      const float coef = P.eos[r] * loss_derivative(LOSS, __int_as_float(st.z), __int_as_float(st.w) * acc);
      if (in0) cache[h0] = fmaf(-coef, v0, u0);
      if (in1) cache[h1] = fmaf(-coef, v1, u1);
      for (int o = lane + 64; o < cnt; o += 32) {
        const int h = B.slot[beg + o] & CSRB_SLOT;
        cache[h] = fmaf(-coef, B.val[beg + o], cache[h]);
      }
      __syncwarp();
    }
  };

  // Blocks of long rows: their steps one at a time, all lanes on a row. The first 128 nonzeros of a row and of the next one wait
  // in registers, the others are read again for the update.
  auto run_long = [&](const CsrBlockBuf& B, const CsrPlan& P, float* cache) __attribute__((always_inline)) {
    constexpr int U = 4;
    const uint32_t cache_a = smem_addr(cache), slot_a = smem_addr(B.slot), val_a = smem_addr(B.val), step_a = smem_addr(P.step);
    uint32_t c2[U];
    float v2[U];
    int4 st2;
    auto entries = [&](int r) __attribute__((always_inline)) {
      st2 = lds_s32x4(step_a + 16u * (uint32_t)r);
#pragma unroll
      for (int i = 0; i < U; ++i) {
        const int e = lane + 32 * i < st2.y ? st2.x + lane + 32 * i : 0;
        c2[i] = cache_a + 4u * (uint32_t)lds_u16(slot_a + 2u * (uint32_t)e);
        v2[i] = lds_f32(val_a + 4u * (uint32_t)e);
      }
    };
    entries(0);
#pragma unroll 1
    for (int r = 0; r < P.nsteps; ++r) {
      const int4 st = st2;
      uint32_t c[U];
      float v[U], x[U];
#pragma unroll
      for (int i = 0; i < U; ++i) {
        c[i] = c2[i];
        v[i] = lane + 32 * i < st.y ? v2[i] : 0.0f;
        x[i] = lds_f32(c[i]);
      }
      entries(r + 1 < P.nsteps ? r + 1 : r);
      const float eos = P.eos[r];
      float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
      for (int i = 0; i < U; i += 2) {
        a0 = lane + 32 * i < st.y ? fmaf(x[i], v[i], a0) : a0;
        a1 = lane + 32 * i + 32 < st.y ? fmaf(x[i + 1], v[i + 1], a1) : a1;
      }
      auto rest = [&](auto use) __attribute__((always_inline)) {
#pragma unroll 1
        for (int o = lane + 32 * U; o - lane < st.y; o += 32 * U) {
          uint32_t cr[U];
          float vr[U], xr[U];
#pragma unroll
          for (int i = 0; i < U; ++i) {
            const int e = o + 32 * i < st.y ? st.x + o + 32 * i : 0;
            cr[i] = cache_a + 4u * (uint32_t)lds_u16(slot_a + 2u * (uint32_t)e);
            vr[i] = lds_f32(val_a + 4u * (uint32_t)e);
          }
#pragma unroll
          for (int i = 0; i < U; ++i) xr[i] = lds_f32(cr[i]);
#pragma unroll
          for (int i = 0; i < U; ++i) use(cr[i], vr[i], xr[i], o + 32 * i < st.y);
        }
      };
      rest([&](uint32_t, float vv, float xx, bool in) { a0 = in ? fmaf(xx, vv, a0) : a0; });
      const float acc = warp_sum(a0 + a1);
      const float coef = eos * loss_derivative(LOSS, __int_as_float(st.z), __int_as_float(st.w) * acc);
#pragma unroll
      for (int i = 0; i < U; ++i) sts_f32_if(c[i], fmaf(-coef, v[i], x[i]), lane + 32 * i < st.y);
      rest([&](uint32_t a, float vv, float xx, bool in) { sts_f32_if(a, fmaf(-coef, vv, xx), in); });
      __syncwarp();
    }
  };

  // E: nonzeros per lane of a row whose slot and value wait in registers for the margins (four lanes per sample), CH: chunks
  // of 32 of them for the updates (all lanes on one sample); REST as above
  auto run_steps = [&](const CsrBlockBuf& B, const CsrPlan& P, float* cache, auto e_tag, auto ch_tag, auto rest_tag) {
    constexpr int E = decltype(e_tag)::value, CH = decltype(ch_tag)::value;
    constexpr bool REST = decltype(rest_tag)::value;
    const uint32_t cache_a = smem_addr(cache), slot_a = smem_addr(B.slot), val_a = smem_addr(B.val), step_a = smem_addr(P.step);
    const int n = lane >> 2, q = lane & 3, own = lane & 7;
    uint32_t ga[E];
    float gv[E];
    int gbeg = 0, gcnt = 0;
    const int groups = (P.nsteps + 7) / 8;
    // (lanes beyond a row read the slot of the block's first nonzero; what they read is not used)
    auto entries = [&](int gi) __attribute__((always_inline)) {
      const int4 st = lds_s32x4(step_a + 16u * (uint32_t)(8 * gi + n));
      gbeg = st.x;
      gcnt = st.y;
#pragma unroll
      for (int i = 0; i < E; ++i) {
        const int e = q + 4 * i < gcnt ? gbeg + q + 4 * i : 0;
        ga[i] = (uint32_t)lds_u16(slot_a + 2u * (uint32_t)e);
        gv[i] = lds_f32(val_a + 4u * (uint32_t)e);
      }
    };
    entries(0);
#pragma unroll 1
    for (int gi = 0; gi < groups; ++gi) {
      const float* T = B.gram[gi];
      const LagConst& K = P.k[gi];
      float uq[E];
#pragma unroll
      for (int i = 0; i < E; ++i) uq[i] = lds_f32(cache_a + 4u * ga[i]);
      // slots and values for the updates
      int ub[8], uc[8];
      uint32_t c[CH][8];
      float w[CH][8];
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int4 st = lds_s32x4(step_a + 16u * (uint32_t)(8 * gi + m));
        ub[m] = st.x;
        uc[m] = st.y;
      }
      LagBlock<LOSS> blk;
      blk.load(T, K, own);
      float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
      for (int i = 0; i < E; i += 2) {
        a0 = q + 4 * i < gcnt ? fmaf(uq[i], gv[i], a0) : a0;
        a1 = q + 4 * i + 4 < gcnt ? fmaf(uq[i + 1], gv[i + 1], a1) : a1;
      }
      if constexpr (REST)
        for (int e = q + 4 * E; e < gcnt; e += 4) a0 = fmaf(cache[B.slot[gbeg + e]], B.val[gbeg + e], a0);
      float r = a0 + a1;
      r += __shfl_xor_sync(0xffffffffu, r, 1);
#pragma unroll
      for (int m = 0; m < 8; ++m)
#pragma unroll
        for (int k2 = 0; k2 < CH; ++k2) {
          const int e = lane + 32 * k2 < uc[m] ? ub[m] + lane + 32 * k2 : 0;
          c[k2][m] = (uint32_t)lds_u16(slot_a + 2u * (uint32_t)e);
          w[k2][m] = lds_f32(val_a + 4u * (uint32_t)e);
        }
      r += __shfl_xor_sync(0xffffffffu, r, 2);
      float kappa[LAG_B], margin;
      blk.steps(__shfl_sync(0xffffffffu, r, 4 * own), T, K, sm.jets, kappa, margin);
      if (gi + 1 < groups) entries(gi + 1);  // on their way while the updates run
      if (LOSS == LOSS_HINGE && margin < CSRB_NEAR * LAG_STEP) {
        one_by_one(B, P, cache, 8 * gi, min(8 * gi + 8, P.nsteps));
        continue;
      }
      // u <- u - kappa_m x_m, m ascending
#pragma unroll
      for (int m = 0; m < LAG_B; ++m) {
        float um[CH];
#pragma unroll
        for (int k2 = 0; k2 < CH; ++k2) um[k2] = lds_f32(cache_a + 4u * c[k2][m]);
#pragma unroll
        for (int k2 = 0; k2 < CH; ++k2) sts_f32_if(cache_a + 4u * c[k2][m], fmaf(-kappa[m], w[k2][m], um[k2]), lane + 32 * k2 < uc[m]);
        if constexpr (REST)
          for (int o = lane + 32 * CH; o < uc[m]; o += 32) {
            const int h = B.slot[ub[m] + o];
            cache[h] = fmaf(-kappa[m], B.val[ub[m] + o], cache[h]);
          }
        __syncwarp();  // the next sample's loads see this sample's stores
      }
    }
  };

  // Four lanes per sample hold E nonzeros each in registers, from the margins to the updates (short form). A column that
  // only one row of the group holds is updated by the lane that read it; a shared one by a lane that takes all rows' values.
  auto run_short = [&](const CsrBlockBuf& B, const CsrPlan& P, float* cache, auto e_tag) {
    constexpr int E = decltype(e_tag)::value;
    const uint32_t cache_a = smem_addr(cache), slot_a = smem_addr(B.slot), val_a = smem_addr(B.val), step_a = smem_addr(P.step);
    const uint32_t rslot_a = smem_addr(B.shared_slot), records_a = smem_addr(B.records);
    const int n = lane >> 2, q = lane & 3, own = lane & 7;
    uint32_t ga[E], ga2[E];
    float gv[E];
    int gbeg, gcnt, gbeg2, gcnt2, rec0, rec02, n_rec, n_rec2;
    const int groups = (P.nsteps + 7) / 8;
    // (lanes beyond a row read the slot of the block's first nonzero; what they read is not used)
    auto entries = [&](int gi) __attribute__((always_inline)) {
      const int4 st = lds_s32x4(step_a + 16u * (uint32_t)(8 * gi + n));
      const int2 rr = lds_s32x2(records_a + 8u * (uint32_t)gi);
      rec02 = rr.x;
      n_rec2 = rr.y;
      gbeg2 = st.x;
      gcnt2 = st.y;
#pragma unroll
      for (int i = 0; i < E; ++i) ga2[i] = (uint32_t)lds_u16(slot_a + 2u * (uint32_t)(q + 4 * i < gcnt2 ? gbeg2 + q + 4 * i : 0));
    };
    entries(0);
#pragma unroll 1
    for (int gi = 0; gi < groups; ++gi) {
      const float* T = B.gram[gi];
      const LagConst& K = P.k[gi];
      gbeg = gbeg2;
      gcnt = gcnt2;
      rec0 = rec02;
      n_rec = n_rec2;
      float uq[E];
#pragma unroll
      for (int i = 0; i < E; ++i) {
        ga[i] = ga2[i];
        uq[i] = lds_f32(cache_a + 4u * (ga[i] & CSRB_SLOT));
        gv[i] = lds_f32(val_a + 4u * (uint32_t)(q + 4 * i < gcnt ? gbeg + q + 4 * i : 0));
      }
      // this lane's shared column: its value in each row, its model entry
      const int rec = lane < n_rec ? rec0 + lane : 0;
      const uint32_t rs = (uint32_t)lds_u16(rslot_a + 2u * (uint32_t)rec);
      const float4 xl = *(const float4*)B.shared_x[rec], xh = *(const float4*)(B.shared_x[rec] + 4);
      LagBlock<LOSS> blk;
      blk.load(T, K, own);
      float ru = lds_f32(cache_a + 4u * (rs & CSRB_SLOT));
      float a0 = 0.0f, a1 = 0.0f;
#pragma unroll
      for (int i = 0; i < E; i += 2) {
        a0 = q + 4 * i < gcnt ? fmaf(uq[i], gv[i], a0) : a0;
        a1 = q + 4 * i + 4 < gcnt ? fmaf(uq[i + 1], gv[i + 1], a1) : a1;
      }
      float r = a0 + a1;
      r += __shfl_xor_sync(0xffffffffu, r, 1);
      entries(gi + 1 < groups ? gi + 1 : gi);  // of the next group, on their way while the steps run
      r += __shfl_xor_sync(0xffffffffu, r, 2);
      float kappa[LAG_B], margin;
      blk.steps(__shfl_sync(0xffffffffu, r, 4 * own), T, K, sm.jets, kappa, margin);
      if (LOSS == LOSS_HINGE && margin < CSRB_NEAR * LAG_STEP) {
        one_by_one(B, P, cache, 8 * gi, min(8 * gi + 8, P.nsteps));
        continue;
      }
      // u <- u - kappa_m x_m, m ascending
      const float k01 = n & 1 ? kappa[1] : kappa[0], k23 = n & 1 ? kappa[3] : kappa[2];
      const float k45 = n & 1 ? kappa[5] : kappa[4], k67 = n & 1 ? kappa[7] : kappa[6];
      const float k03 = n & 2 ? k23 : k01, k47 = n & 2 ? k67 : k45;
      const float k_row = n & 4 ? k47 : k03;
#pragma unroll
      for (int i = 0; i < E; ++i)
        sts_f32_if(cache_a + 4u * (ga[i] & CSRB_SLOT), fmaf(-k_row, gv[i], uq[i]), q + 4 * i < gcnt && !(ga[i] & CSRB_SHARED));
      auto all_rows = [&](float v, const float4& lo, const float4& hi) __attribute__((always_inline)) {
        const float x[8] = {lo.x, lo.y, lo.z, lo.w, hi.x, hi.y, hi.z, hi.w};
#pragma unroll
        for (int m = 0; m < 8; ++m) v = x[m] != 0.0f ? fmaf(-kappa[m], x[m], v) : v;  // 0: not in this row
        return v;
      };
      ru = all_rows(ru, xl, xh);
      sts_f32_if(cache_a + 4u * (rs & CSRB_SLOT), ru, lane < n_rec);
      for (int i = lane + 32; i < n_rec; i += 32) {
        const int h = B.shared_slot[rec0 + i];
        const float4* x4 = (const float4*)B.shared_x[rec0 + i];
        cache[h] = all_rows(cache[h], x4[0], x4[1]);
      }
      __syncwarp();  // the next group's loads see these stores
    }
  };

  __syncthreads();
  if (warp == 1) plan_next(sm.plan[0]);
  __syncthreads();
  if (warp == 1) plan_next(sm.plan[1]);
  if (warp > 1) prepare(sm.buf[0], sm.ucache[0], sm.plan[0]);
  __syncthreads();

  int prev_direct = 0, cur = 0;  // cur = b mod 3
  for (long long b = 0;; ++b) {
    CsrBlockBuf& B = sm.buf[b & 1];
    CsrBlockBuf& Bp = sm.buf[(b + 1) & 1];  // the block that has just run (and the buffer of the next preparation)
    float* cache = sm.ucache[b & 1];
    float* cache_p = sm.ucache[(b + 1) & 1];
    const CsrPlan& P = sm.plan[cur];
    const CsrPlan& P1 = sm.plan[cur == 2 ? 0 : cur + 1];
    CsrPlan& P2 = sm.plan[cur == 0 ? 2 : cur - 1];
    const int nsteps = P.nsteps, nuniq = B.nuniq, direct = P.direct;
    const int nuniq_p = Bp.nuniq;
    const float fold = P.fold;
    const bool slow = b == 0 || nsteps == 0 || fold != 0.0f || direct || prev_direct;
    if (!slow) {
      // ---- boundary: columns that the block that has just run also holds take its values -----------------------------
      const uint32_t uslot_a = smem_addr(B.uslot), keys_a = smem_addr(B.keys), keysp_a = smem_addr(Bp.keys);
      const uint32_t cache_a = smem_addr(cache), cachep_a = smem_addr(cache_p);
      constexpr int F = 3;  // columns of a thread in flight
      for (int i0 = threadIdx.x; i0 - (int)threadIdx.x < nuniq; i0 += F * CSRB_THREADS) {
        int h2[F], col[F], h[F], k2[F];
        bool seek[F];
#pragma unroll
        for (int i = 0; i < F; ++i) {
          seek[i] = i0 + i * CSRB_THREADS < nuniq;
          h2[i] = lds_u16(uslot_a + 2u * (uint32_t)(seek[i] ? i0 + i * CSRB_THREADS : 0));
          k2[i] = -1;
        }
#pragma unroll
        for (int i = 0; i < F; ++i) col[i] = lds_s32(keys_a + 4u * (uint32_t)h2[i]);
#pragma unroll
        for (int i = 0; i < F; ++i) h[i] = csrb_hash(col[i]);
        for (int probe = 0; probe < CSRB_HASH; ++probe) {
#pragma unroll
          for (int i = 0; i < F; ++i) lds_s32_if(k2[i], keysp_a + 4u * (uint32_t)h[i], seek[i]);
          bool any = false;
#pragma unroll
          for (int i = 0; i < F; ++i) {
            seek[i] = seek[i] && k2[i] != col[i] && k2[i] != -1;
            h[i] = seek[i] ? (h[i] + 1) & (CSRB_HASH - 1) : h[i];
            any |= seek[i];
          }
          if (!__any_sync(0xffffffffu, any)) break;
        }
        float v[F];
#pragma unroll
        for (int i = 0; i < F; ++i) v[i] = lds_f32(cachep_a + 4u * (uint32_t)h[i]);
#pragma unroll
        for (int i = 0; i < F; ++i) sts_f32_if(cache_a + 4u * (uint32_t)h2[i], v[i], k2[i] == col[i]);
      }
      __syncthreads();
    } else {
      // ---- slow boundary: write back, fold, read again ------------------------------------------------------------------
      csrb_scatter(Bp, cache_p, u, nuniq_p, threadIdx.x, CSRB_THREADS);
      __syncthreads();
      if (threadIdx.x == 0) Bp.nuniq = 0;
      if (nsteps == 0) break;
      if (fold != 0.0f) {
        for (long long c = threadIdx.x; c < p.d; c += CSRB_THREADS) u[c] = __ldcg(u + c) * fold;
        __syncthreads();
      }
      csrb_gather(B, cache, u, nuniq, threadIdx.x, CSRB_THREADS);
      __syncthreads();
    }
    if (warp > 1) {
      // the block that has just run goes back to u (a slow boundary has done it already: nothing left to do), then its
      // tables and cache take the block after this one
      prepare(Bp, cache_p, P1);
    } else if (warp == 1) {
      plan_next(P2);
    } else if (direct) {
      // ---- a single long row, on global memory ---------------------------------------------------------------
      const long long g0 = P.gbeg[0], g1 = P.gbeg[1];
      // CSRB_DIRECT loads in flight per lane; lanes beyond the row take its first nonzero and the value 0
      auto batch = [&](long long o, long long (&e)[CSRB_DIRECT], int (&c)[CSRB_DIRECT], float (&v)[CSRB_DIRECT], float (&x)[CSRB_DIRECT]) __attribute__((always_inline)) {
#pragma unroll
        for (int i = 0; i < CSRB_DIRECT; ++i) {
          e[i] = o + 32 * i < g1 ? o + 32 * i : g0;
          c[i] = p.col_idx[e[i]];
          v[i] = o + 32 * i < g1 ? p.val[e[i]] : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < CSRB_DIRECT; ++i)
          if ((unsigned long long)(long long)c[i] >= (unsigned long long)p.d) {
            set_status(p.status, DEV_BOUNDS, 22, (long long)c[i]);
            c[i] = 0;
            v[i] = 0.0f;
          }
#pragma unroll
        for (int i = 0; i < CSRB_DIRECT; ++i) x[i] = __ldcg(u + c[i]);
      };
      long long e[CSRB_DIRECT];
      int c[CSRB_DIRECT];
      float v[CSRB_DIRECT], x[CSRB_DIRECT];
      float acc = 0.0f;
#pragma unroll 1
      for (long long o = g0 + lane; o - lane < g1; o += 32 * CSRB_DIRECT) {
        batch(o, e, c, v, x);
#pragma unroll
        for (int i = 0; i < CSRB_DIRECT; ++i) acc = v[i] != 0.0f ? fmaf(x[i], v[i], acc) : acc;
      }
      acc = warp_sum(acc);
      const float g = loss_derivative(LOSS, __int_as_float(P.step[0].z), __int_as_float(P.step[0].w) * acc);
      if (g != 0.0f) {
        const float coef = P.eos[0] * g;
#pragma unroll 1
        for (long long o = g0 + lane; o - lane < g1; o += 32 * CSRB_DIRECT) {
          batch(o, e, c, v, x);
#pragma unroll
          for (int i = 0; i < CSRB_DIRECT; ++i)
            if (v[i] != 0.0f) u[c[i]] = fmaf(-coef, v[i], x[i]);
        }
      }
    } else {
      using std::integral_constant;
      if (SHORT && P.brief && P.longest <= 16) run_short(B, P, cache, integral_constant<int, 4>());
      else if (SHORT && P.brief) run_short(B, P, cache, integral_constant<int, 8>());
      else if (P.longest <= 32) run_steps(B, P, cache, integral_constant<int, 8>(), integral_constant<int, 1>(), std::false_type());
      else if (SHORT) run_steps(B, P, cache, integral_constant<int, 8>(), integral_constant<int, 1>(), std::true_type());
      else if (P.apart) run_long(B, P, cache);
      else if (P.longest <= 64) run_steps(B, P, cache, integral_constant<int, 16>(), integral_constant<int, 2>(), std::false_type());
      else run_steps(B, P, cache, integral_constant<int, 16>(), integral_constant<int, 2>(), std::true_type());
    }
    prev_direct = direct;
    cur = cur == 2 ? 0 : cur + 1;
    __syncthreads();
  }
  if (warp == 1 && lane == 0) p.scale[j] = sc;
}

// The short form is compiled into a body of its own, for chains whose shard has at most 10 nonzeros per row on average (640
// nonzeros in 64 steps, the limit of that form). Code that a chain never runs costs it time all the same, through the registers
// and the schedule of the one body: 64 chains with 40 Zipf-distributed nonzeros per row take 11.55 ms with two bodies and 12.25 with
// one; 10 chains of 5 to 10 nonzeros take the same in both.
constexpr int CSRB_SHORT_MEAN = CSRB_SHORT_ENT / CSRB_STEPS;
template <int LOSS>
__global__ void __launch_bounds__(CSRB_THREADS, 1) chain_csr_block_kernel(const CsrParams p) {
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CsrBlockSmem& sm = *reinterpret_cast<CsrBlockSmem*>(smem_raw);
  const int j = p.order[blockIdx.x];
  const long long r0 = p.shard_off[j], r1 = p.shard_off[j + 1];
  if (p.row_ptr[r1] - p.row_ptr[r0] <= CSRB_SHORT_MEAN * (r1 - r0)) {
    chain_csr_block<LOSS, true>(p, sm);
    return;
  }
  chain_csr_block<LOSS, false>(p, sm);
}

}  // namespace wpsgd
