// C ABI of the WP-SGD library (see include/wpsgd.h): context, host-side planning (validation,
// delays and Eq. 6 / Eq. 8 weights in fp64, node ordering, kernel selection) and kernel launches.
#include "../../include/wpsgd.h"

#include <algorithm>
#include <atomic>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <functional>
#include <initializer_list>
#include <numeric>
#include <string>
#include <utility>
#include <vector>

#include "chain_block.cuh"
#include "chain_csr.cuh"
#include "chain_csr_block.cuh"
#include "chain_mma.cuh"
#include "chain_mma16.cuh"
#include "chain_dense.cuh"
#include "chain_lag.cuh"
#include "combine.cuh"
#include "philox.cuh"

using namespace wpsgd;

struct wpsgd_ctx {
  int device = 0;
  cudaStream_t stream = nullptr;
  int k = 0;
  long long d = 0;
  // models
  float* W = nullptr;       // [k, d]
  double* scale = nullptr;  // [k] (sparse path: w_j = scale_j * W[j])
  bool scaled = false;
  // per-launch tables on the device: one buffer laid out by TableLayout(k), and where its parts are
  unsigned char* tables = nullptr;
  long long *t_shard_off = nullptr, *t_steps = nullptr, *t_first = nullptr, *t_idx_off = nullptr;
  int* t_order = nullptr;
  std::vector<unsigned char> h_tables;
  double* t_weights = nullptr;       // [k]
  uint32_t* idx = nullptr;
  size_t idx_cap = 0;  // entries
  bool streams_read = false;  // every stream kernel so far has been followed by a launch of chains
  DevStatus* status = nullptr;
  double* part = nullptr;  // objective partial sums
  size_t part_cap = 0;     // doubles
  unsigned* ticket = nullptr;  // blocks of the running objective kernel that have finished (zero between launches)
  // staging of the host-buffer entry point
  void* st_X = nullptr;
  size_t st_X_cap = 0;
  float* st_y = nullptr;
  size_t st_y_cap = 0;
  float* st_v = nullptr;   // [d]
  long long* st_rp = nullptr;  // CSR staging of the host-buffer entry point
  size_t st_rp_cap = 0;
  int* st_ci = nullptr;
  size_t st_ci_cap = 0;
  float* st_va = nullptr;
  size_t st_va_cap = 0;
  float* st_w0 = nullptr;  // [d]
  // state of the chains
  bool have_run = false;
  std::vector<long long> steps_done;
  std::vector<int> node_ids;
  std::vector<long long> last_steps;    // step counts of the launch being prepared
  std::vector<long long> steps_sorted;  // step counts that the estimates of a launch go by, largest first (see estimate_for)
  double steps_sum = 0.0;
  float eta0 = 0.f, lambda = 0.f;
  int sched = 0, loss = 0;
  uint64_t seed = 0;
  // options
  int opt_stages = 0;
  int opt_variant = 0, opt_prefetch = 0, opt_threads = 0, opt_cluster = 0;
  int opt_block_samples = 0;   // tensor-core cluster kernel: samples per block (0: chosen here, 8 or 16)
  int opt_sparse_variant = 0;  // 0: chosen here, 1: one step per round trip, 2: blocks of steps through a shared-memory cache
  long long opt_spin_limit = 1ll << 20;
  long long opt_drop_block = -1;
  int opt_sampling = 0;  // 0: i.i.d. draws, 1: one shuffle per node, cycled
  int opt_timing = 0;
  int opt_host_pipeline = 1;  // host-buffer entry point: copy the shards in groups and start chains as they arrive
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t ev_fork = nullptr, ev_group[4] = {nullptr, nullptr, nullptr, nullptr};
  cudaEvent_t ev0 = nullptr, ev1 = nullptr;
  bool ev_valid = false;
  long long launches = 0;
  std::string err;
};

namespace {

std::string g_err;  // last error of context-free calls

struct DeviceGuard {
  int prev = -1;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) prev = -1;
    if (prev != dev) cudaSetDevice(dev);
    else prev = -1;
  }
  ~DeviceGuard() {
    if (prev >= 0) cudaSetDevice(prev);
  }
};

wpsgd_status fail(wpsgd_ctx* c, wpsgd_status s, const std::string& msg) {
  if (c) c->err = msg;
  else g_err = msg;
  return s;
}

#define CU_TRY(ctx, expr)                                                                          \
  do {                                                                                             \
    cudaError_t e_ = (expr);                                                                       \
    if (e_ != cudaSuccess) {                                                                       \
      cudaGetLastError(); /* reported here, and not by the next call's look at the last error too */ \
      const bool oom_ = (e_ == cudaErrorMemoryAllocation);                                         \
      return fail(ctx, oom_ ? WPSGD_ERR_ALLOC : WPSGD_ERR_CUDA,                                    \
                  std::string(#expr) + ": " + cudaGetErrorString(e_));                             \
    }                                                                                              \
  } while (0)

template <typename T>
wpsgd_status grow(wpsgd_ctx* c, T** p, size_t* cap, size_t need) {
  if (need <= *cap) return WPSGD_OK;
  if (*p) {
    CU_TRY(c, cudaStreamSynchronize(c->stream));
    CU_TRY(c, cudaFree(*p));
    *p = nullptr;
    *cap = 0;
  }
  const size_t want = need + need / 8;
  void* q = nullptr;
  CU_TRY(c, cudaMalloc(&q, want * sizeof(T)));
  *p = (T*)q;
  *cap = want;
  return WPSGD_OK;
}

// ---- Eq. 6 / Eq. 8 in fp64 -------------------------------------------------------------------------
// log of r^{T_j} (or of the product of skipped per-step factors for the decaying schedule)
wpsgd_status log_rates(const long long* n, int k, double eta0, int sched, double lambda, double r,
                       std::vector<double>* lg, std::string* why) {
  long long t = 0;
  for (int j = 0; j < k; ++j) {
    if (n[j] < 0) {
      *why = "negative step count";
      return WPSGD_ERR_INVALID_ARG;
    }
    t = std::max(t, n[j]);
  }
  lg->assign(k, 0.0);
  const bool given = r > 0.0;  // false for NaN
  if (given) {
    const double lr = std::log(r);
    for (int j = 0; j < k; ++j) (*lg)[j] = (double)(t - n[j]) * lr;
  } else if (sched == WPSGD_LR_CONST) {
    const double lr = std::log1p(-eta0 * lambda);
    for (int j = 0; j < k; ++j) (*lg)[j] = (double)(t - n[j]) * lr;
  } else {
    // sum_{s = n_j + 1}^{t} log(1 - c / sqrt(s)), c = eta0 lambda. From step 256 on by the Euler-Maclaurin formula: the sum over
    // (a, b] is T(b) - T(a), T the antiderivative plus f / 2 + f' / 12 - f''' / 720 (the next term is below 1e-16 c there); up to
    // step 256, and for the last few steps, term by term. All of it term by term took 25 ns a step: 32 chains averaged in 16
    // rounds of up to 250 steps spent more time here than on the GPU. The difference is formed part by part from sqrt(b) - sqrt(a):
    // T grows with sqrt(s), and two rounded values of it would leave nodes near t with errors of 5e-13 after 4e6 steps instead of 1e-15.
    const double c = eta0 * lambda;
    const long long head = 256, near = 32;
    auto term = [&](double s) { return std::log1p(-c / std::sqrt(s)); };
    auto tail = [&](double s, double u) {  // f' / 12 - f''' / 720, f''' = s^-3 / 2 sum_k (k / 2 + 1) (k / 2 + 2) (c / u)^k
      const double q = c / u, is = 1.0 / s;
      double f3 = 0.0;
      for (int k = 8; k >= 1; --k) f3 = (f3 + (0.5 * k + 1.0) * (0.5 * k + 2.0)) * q;
      return is * (c / (24.0 * (u - c)) - f3 * is * is * (1.0 / 1440.0));
    };
    const double u_end = std::sqrt((double)t), w_end = u_end - c, f_end = t > head ? term((double)t) : 0.0, tail_end = t > head ? tail((double)t, u_end) : 0.0;
    auto to_end = [&](long long a) {  // T(t) - T(a), T = s f - c u - c^2 log(u - c) + f / 2 + tail
      const double u = std::sqrt((double)a), w = u - c, n = (double)(t - a), du = n / (u + u_end), df = std::log1p(c * du / (u_end * w));
      return n * f_end + ((double)a + 0.5) * df - c * du - c * c * std::log(w_end / w) + (tail_end - tail((double)a, u));
    };
    const double from_head = t > head ? to_end(head) : 0.0;
    long long lo = t;
    for (int j = 0; j < k; ++j) lo = std::min(lo, n[j]);
    std::vector<double> suf;  // suf[i]: sum over s in (lo + i, min(t, head)]
    if (lo < head) {
      const long long end = std::min(t, head);
      suf.assign((size_t)(end - lo) + 1, 0.0);
      for (long long s = end; s > lo; --s) suf[(size_t)(s - 1 - lo)] = suf[(size_t)(s - lo)] + term((double)s);
    }
    for (int j = 0; j < k; ++j) {
      double v = 0.0;
      if (n[j] < head) v = suf[(size_t)(n[j] - lo)] + from_head;
      else if (t - n[j] > near) v = to_end(n[j]);
      else
        for (long long s = t; s > n[j]; --s) v += term((double)s);
      (*lg)[j] = v;
    }
  }
  return WPSGD_OK;
}

wpsgd_status weights_host(const long long* n, int k, float eta0, int sched, float lambda, double r, double* w,
                          int* cond, double* sum_rT, std::string* why) {
  if (!n || !w || k < 1) {
    *why = "weights: null argument or k < 1";
    return WPSGD_ERR_INVALID_ARG;
  }
  if (sched != WPSGD_LR_CONST && sched != WPSGD_LR_INV_SQRT) {
    *why = "weights: unknown schedule";
    return WPSGD_ERR_INVALID_ARG;
  }
  std::vector<double> lg;
  wpsgd_status s = log_rates(n, k, (double)eta0, sched, (double)lambda, r, &lg, why);
  if (s != WPSGD_OK) return s;
  const double mx = *std::max_element(lg.begin(), lg.end());
  double tot = 0.0, tot_raw = 0.0;
  for (int j = 0; j < k; ++j) {
    tot += std::exp(lg[j] - mx);
    tot_raw += std::exp(lg[j]);
  }
  for (int j = 0; j < k; ++j) w[j] = std::exp(lg[j] - mx) / tot;
  if (sum_rT) *sum_rT = tot_raw;
  if (cond) *cond = (2.0 * tot_raw > std::sqrt((double)k) + (double)k) ? 1 : 0;
  return WPSGD_OK;
}

// Waits for the stream, reads a device status word and maps it; a problem found is cleared after it has been reported.
wpsgd_status read_status(wpsgd_ctx* c, DevStatus* dev_status, cudaStream_t stream) {
  DevStatus h;
  CU_TRY(c, cudaMemcpyAsync(&h, dev_status, sizeof(h), cudaMemcpyDeviceToHost, stream));
  CU_TRY(c, cudaStreamSynchronize(stream));
  if (h.code == DEV_OK) return WPSGD_OK;
  char buf[200];
  const char* what = h.code == DEV_TIMEOUT ? "a bounded device-side wait gave up" : "a device-side check of the input failed";
  snprintf(buf, sizeof(buf), "%s: device status %d at %d (detail %lld)", what, h.code, h.where, h.detail);
  cudaMemsetAsync(dev_status, 0, sizeof(DevStatus), stream);
  return fail(c, h.code == DEV_TIMEOUT ? WPSGD_ERR_TIMEOUT : WPSGD_ERR_CUDA, buf);
}

// Kernel launch that may start while the kernel before it on the stream ends (see kernel_started in common.cuh).
template <typename... P, typename... A>
cudaError_t launch(void (*kern)(P...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream, A&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kern, std::forward<A>(args)...);
}

bool aligned16(const void* p) { return (uintptr_t)p % 16 == 0; }

int grid_for(long long work_items, int block, int cap = 148 * 16) {
  long long g = (work_items + block - 1) / block;
  return (int)std::max(1ll, std::min<long long>(g, cap));
}

// v_out = sum_j weights[j] scale_j W[j] (weights HOST)
template <int VEC, int N>
wpsgd_status launch_combine_form(wpsgd_ctx* c, const double* weights, float* v_out) {
  const double* scale = c->scaled ? c->scale : nullptr;
  InlineWeights<(N > 0 ? N : 1)> iw;
  if (N > 0) memcpy(iw.w, weights, c->k * sizeof(double));
  else CU_TRY(c, cudaMemcpyAsync(c->t_weights, weights, c->k * sizeof(double), cudaMemcpyHostToDevice, c->stream));
  const int warps = std::max(1, std::min(VEC == 4 ? 16 : 32, (c->k + 3) / 4));  // (32 warps of four columns were not measured)
  const unsigned blocks = (unsigned)((c->d + 32 * VEC - 1) / (32 * VEC));
  launch(combine_kernel<VEC, N>, blocks, 32 * warps, (size_t)warps * 32 * VEC * sizeof(double), c->stream, iw, c->W, c->t_weights, scale, c->k, c->d, v_out);
  CU_TRY(c, cudaGetLastError());
  c->launches++;
  return WPSGD_OK;
}
wpsgd_status launch_combine(wpsgd_ctx* c, const double* weights, float* v_out) {
  const bool few = c->k <= COMBINE_INLINE;
  // four columns per thread once that still gives every SM several blocks
  if (c->d % 4 == 0 && c->d >= 128 * 148 * 2 && aligned16(c->W))
    return few ? launch_combine_form<4, COMBINE_INLINE>(c, weights, v_out) : launch_combine_form<4, 0>(c, weights, v_out);
  return few ? launch_combine_form<1, COMBINE_INLINE>(c, weights, v_out) : launch_combine_form<1, 0>(c, weights, v_out);
}

// ---- common part of run / continue: tables, sample stream ---------------------------------------------
struct Plan {
  std::vector<long long> off, steps, first, idx_off;
  std::vector<int> order;
  long long total = 0;
};

wpsgd_status make_plan(wpsgd_ctx* c, const long long* shard_off, const long long* n_steps,
                       const std::vector<long long>& first, Plan* pl) {
  const int k = c->k;
  if (!shard_off || !n_steps) return fail(c, WPSGD_ERR_INVALID_ARG, "shard_off / n_steps is NULL");
  if (shard_off[0] < 0) return fail(c, WPSGD_ERR_INVALID_ARG, "shard_off[0] < 0");
  pl->off.assign(shard_off, shard_off + k + 1);
  pl->steps.assign(n_steps, n_steps + k);
  pl->first = first;
  pl->idx_off.assign(k + 1, 0);
  for (int j = 0; j < k; ++j) {
    const long long m = shard_off[j + 1] - shard_off[j];
    if (m < 0) return fail(c, WPSGD_ERR_INVALID_ARG, "shard_off is not non-decreasing");
    if (n_steps[j] < 0) return fail(c, WPSGD_ERR_INVALID_ARG, "negative step count");
    if (n_steps[j] > 0 && m < 1) return fail(c, WPSGD_ERR_INVALID_ARG, "a node with steps has an empty shard");
    if (m > 0xFFFFFFFFll) return fail(c, WPSGD_ERR_INVALID_ARG, "a shard has 2^32 rows or more");
    pl->idx_off[j + 1] = pl->idx_off[j] + stream_entries(n_steps[j]);
  }
  pl->total = pl->idx_off[k];
  pl->order.resize(k);
  std::iota(pl->order.begin(), pl->order.end(), 0);
  std::stable_sort(pl->order.begin(), pl->order.end(), [&](int a, int b) { return n_steps[a] > n_steps[b]; });
  return WPSGD_OK;
}

// Where the tables' parts are inside the device buffer
void bind_tables(wpsgd_ctx* c, unsigned char* base) {
  const TableLayout L(c->k);
  c->tables = base;
  c->t_shard_off = (long long*)(base + L.shard_off);
  c->t_steps = (long long*)(base + L.steps);
  c->t_first = (long long*)(base + L.first);
  c->t_idx_off = (long long*)(base + L.idx_off);
  c->t_order = (int*)(base + L.order);
}

template <int BYTES>
void launch_index_stream(wpsgd_ctx* c, dim3 grid, size_t bytes) {
  InlineTables<(BYTES > 0 ? BYTES : 16)> t;
  if (BYTES > 0) memcpy(t.b, c->h_tables.data(), bytes);
  launch(index_stream_kernel<BYTES>, grid, 256, 0, c->stream, t, c->streams_read ? 0 : 1, c->opt_sampling, c->seed, c->k, c->tables, c->idx);
}

wpsgd_status upload_plan_and_stream(wpsgd_ctx* c, const Plan& pl) {
  const int k = c->k;
  wpsgd_status s = grow(c, &c->idx, &c->idx_cap, (size_t)std::max(1ll, pl.total));
  if (s != WPSGD_OK) return s;
  const TableLayout L(k);
  c->h_tables.assign(L.total, 0);
  unsigned char* h = c->h_tables.data();
  memcpy(h + L.shard_off, pl.off.data(), (k + 1) * sizeof(long long));
  memcpy(h + L.steps, pl.steps.data(), k * sizeof(long long));
  memcpy(h + L.first, pl.first.data(), k * sizeof(long long));
  memcpy(h + L.idx_off, pl.idx_off.data(), (k + 1) * sizeof(long long));
  int* order = (int*)(h + L.order);
  std::copy(pl.order.begin(), pl.order.end(), order);
  std::fill(order + k, order + k + 8, -1);
  memcpy(h + L.ids, c->node_ids.data(), k * sizeof(int));
  // Up to 8 KB of tables (some 200 nodes) travel as an argument of the stream kernel, in one of two sizes; the eight copies
  // this replaces took 14 us of a 53 us round (32 nodes, 250 steps): 848 -> 622 us for 16 rounds.
  const bool as_argument = pl.total > 0 && L.total <= 8192;
  // pageable source: the copy has left the host buffer when cudaMemcpyAsync returns
  if (!as_argument) CU_TRY(c, cudaMemcpyAsync(c->tables, h, L.total, cudaMemcpyHostToDevice, c->stream));
  if (pl.total > 0) {
    const long long longest = *std::max_element(pl.steps.begin(), pl.steps.end());
    dim3 grid((unsigned)grid_for(c->opt_sampling ? longest + 8 : (longest + 3) / 4 + 3, 256, 1024), (unsigned)std::min(k, 65535));
    if (!as_argument) launch_index_stream<0>(c, grid, 0);
    else if (L.total <= 2048) launch_index_stream<2048>(c, grid, L.total);
    else launch_index_stream<8192>(c, grid, L.total);
    c->streams_read = false;
    CU_TRY(c, cudaGetLastError());
    c->launches++;
  }
  return WPSGD_OK;
}

wpsgd_status check_hyper(wpsgd_ctx* c, float eta0, int sched, float lambda, int loss) {
  if (!(eta0 >= 0.0f) || !std::isfinite(eta0)) return fail(c, WPSGD_ERR_INVALID_ARG, "eta0 must be finite and >= 0");
  if (!(lambda >= 0.0f) || !std::isfinite(lambda)) return fail(c, WPSGD_ERR_INVALID_ARG, "lambda must be finite and >= 0");
  if (!((double)eta0 * (double)lambda < 1.0)) return fail(c, WPSGD_ERR_INVALID_ARG, "eta * lambda must be < 1");
  if (sched != WPSGD_LR_CONST && sched != WPSGD_LR_INV_SQRT) return fail(c, WPSGD_ERR_INVALID_ARG, "unknown schedule");
  if (loss < 0 || loss > 2) return fail(c, WPSGD_ERR_INVALID_ARG, "unknown loss");
  return WPSGD_OK;
}

wpsgd_status timing_begin(wpsgd_ctx* c) {
  c->ev_valid = false;
  if (!c->opt_timing) return WPSGD_OK;
  if (!c->ev0) {
    CU_TRY(c, cudaEventCreate(&c->ev0));
    CU_TRY(c, cudaEventCreate(&c->ev1));
  }
  CU_TRY(c, cudaEventRecord(c->ev0, c->stream));
  return WPSGD_OK;
}

wpsgd_status timing_end(wpsgd_ctx* c) {
  if (!c->opt_timing) return WPSGD_OK;
  CU_TRY(c, cudaEventRecord(c->ev1, c->stream));
  c->ev_valid = true;
  return WPSGD_OK;
}

// Lets a kernel take up to all of an SM's shared memory. The limit belongs to the function and so to every thread and context of
// the process: set to the size of the launch at hand, a thread with a small ring lowered it between another's call and its
// launch, which was then refused. It is therefore only ever set to this one value; a launch names its own size.
constexpr size_t kSmemMax = 227 * 1024;
template <typename Kernel>
cudaError_t allow_all_smem(Kernel kern) {
  return cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmemMax);
}

// ---- dense chain launch ---------------------------------------------------------------------------------
template <typename XT, int R, int PF>
wpsgd_status launch_reg(wpsgd_ctx* c, const ChainParams& p, bool block_per_node, int threads) {
  if (block_per_node) {
    launch(chain_reg_kernel<XT, R, PF, true>, p.k, threads, 0, c->stream, p);
  } else {
    const int nodes_per_cta = 4;
    launch(chain_reg_kernel<XT, R, PF, false>, (p.k + nodes_per_cta - 1) / nodes_per_cta, 32 * nodes_per_cta, 0, c->stream, p);
  }
  CU_TRY(c, cudaGetLastError());
  c->launches++;
  return WPSGD_OK;
}

template <typename XT, int R>
wpsgd_status launch_reg_pf(wpsgd_ctx* c, const ChainParams& p, bool bpn, int threads, int pf) {
  switch (pf) {
    case 2: return launch_reg<XT, R, 2>(c, p, bpn, threads);
    case 4: return launch_reg<XT, R, 4>(c, p, bpn, threads);
    default: return launch_reg<XT, R, 8>(c, p, bpn, threads);
  }
}

// ---- blocked chain kernel: shapes it takes, ring depth, launch ------------------------------------------------
constexpr size_t kSmemBudget = 220 * 1024;

template <typename XT>
bool block_kernel_fits(const wpsgd_ctx* c, bool aligned, int* threads_out, int* R_out, int* stages_out) {
  constexpr int V = XVec<XT>::V;
  if (!aligned) return false;
  if ((double)c->eta0 * (double)c->lambda > 0.25) return false;  // keeps a^-8 harmless in fp32
  const long long chunks = c->d / V;
  // up to 8 math warps with one chunk per thread (two register copies of a block: Gram products overlap the
  // recurrence); wider rows take up to 16 math warps, then two chunks per thread
  int max_threads = chunks <= 256 ? 256 : 512;
  // fp32 rows of 129..256 chunks: four math warps with two chunks per thread (one register copy, Gram and p in one pass)
  // beat eight warps with the overlapped schedule: half as many cross-lane reductions per block, and the recurrence
  // warp runs while the math warps are idle (k = 16, d = 1024: 2.67 ms against 2.84 ms)
  if (sizeof(XT) == 4 && chunks > 128 && chunks <= 256) max_threads = 128;
  if (c->opt_threads >= 64 && c->opt_threads % 32 == 0) max_threads = std::min(512, c->opt_threads);
  const int math_threads = (int)std::min<long long>(max_threads, (chunks + 31) / 32 * 32);
  int R = (int)((chunks + math_threads - 1) / math_threads);
  if (R > 2) return false;  // beyond two chunks per thread the rows of a block no longer fit in registers
  const size_t row_bytes = (size_t)c->d * sizeof(XT) + (sizeof(XT) == 2 ? 16 : 0);  // bf16 rows are staged with padding
  int stages = c->opt_stages > 0 ? c->opt_stages : 4;
  if (stages > 8) stages = 8;
  while (stages >= 2 && BlockSmem(stages, row_bytes, math_threads / 32).total > kSmemBudget) --stages;
  if (stages < 2) return false;
  *threads_out = math_threads + 64;
  *R_out = R;
  *stages_out = stages;
  return true;
}

template <typename XT, int R, bool OVL, int MAXW>
wpsgd_status launch_block_r(wpsgd_ctx* c, const BlockParams& bp, int threads, size_t smem) {
  auto go = [&](auto kern) -> wpsgd_status {
    CU_TRY(c, allow_all_smem(kern));
    launch(kern, bp.c.k, threads, smem, c->stream, bp);
    CU_TRY(c, cudaGetLastError());
    c->launches++;
    return WPSGD_OK;
  };
  switch (c->loss) {
    // one 16-byte chunk per thread: room for two register copies of a block, so the Gram products of the
    // next block overlap the serial recurrence; more chunks: one copy, Gram and p in the same pass
    case WPSGD_LOSS_HINGE: return go(chain_block_kernel<XT, R, LOSS_HINGE, OVL, MAXW>);
    case WPSGD_LOSS_LOGISTIC: return go(chain_block_kernel<XT, R, LOSS_LOGISTIC, OVL, MAXW>);
    default: return go(chain_block_kernel<XT, R, LOSS_SQUARED, OVL, MAXW>);
  }
}

template <typename XT>
wpsgd_status launch_block(wpsgd_ctx* c, const ChainParams& p, int threads, int R, int stages) {
  BlockParams bp;
  bp.c = p;
  bp.stages = stages;
  bp.eta_lambda = (double)c->eta0 * (double)c->lambda;
  bp.spin_limit = c->opt_spin_limit;
  bp.drop_block = c->opt_drop_block;
  bp.group_order = nullptr;
  const size_t smem = BlockSmem(stages, (size_t)c->d * sizeof(XT) + (sizeof(XT) == 2 ? 16 : 0), threads / 32 - 2).total;
  const bool wide = threads > 64 + 32 * 8;  // more than 8 math warps: registers allow one copy of a block only
  // one register copy of a block, except fp32 rows of at most 8 math warps with one chunk per thread (two copies:
  // the Gram products of the next block overlap the recurrence)
  if (R == 1) {
    if (wide) return launch_block_r<XT, 1, false, 16>(c, bp, threads, smem);
    return sizeof(XT) == 2 ? launch_block_r<XT, 1, false, 8>(c, bp, threads, smem)
                           : launch_block_r<XT, 1, true, 8>(c, bp, threads, smem);
  }
  return wide ? launch_block_r<XT, 2, false, 16>(c, bp, threads, smem) : launch_block_r<XT, 2, false, 8>(c, bp, threads, smem);
}

// ---- bf16 rows: Gram block and margins on the tensor cores, columns split over a cluster -------------------------------
struct ClusterShape {
  int C = 1, cpc = 0, math_warps = 1, stages = 2;
  int block = 8;    // samples per block
  int stages16 = 0; // ring depth of the 16-sample form (0: it does not fit)
};

bool mma_kernel_fits(const wpsgd_ctx* c, bool aligned, ClusterShape* out) {
  if (!aligned) return false;
  if ((double)c->eta0 * (double)c->lambda > 0.25) return false;
  const long long chunks = c->d / 8;
  if (chunks < 1) return false;
  int C = c->opt_cluster;
  if (C <= 0) {
    // as few CTAs per chain as the row width allows (a CTA takes at most 8 math warps of 32 chunks): the kernel runs
    // one CTA per SM, and what a wider cluster gains in the tensor-core pass it loses in chains running at the same
    // time (measured on k = 128, d = 4096: 7.95 ms with two CTAs per chain, 9.9 ms with four, 14.0 ms with eight)
    C = 1;
    while ((chunks + C - 1) / C > 256 && C < 8) C *= 2;
  }
  if (C != 1 && C != 2 && C != 4 && C != 8) return false;
  const long long cpc = (chunks + C - 1) / C;
  if ((long long)(C - 1) * cpc >= chunks) return false;  // every CTA of the cluster owns at least one chunk
  // one 16-byte chunk of a row per lane, up to 8 math warps per CTA
  const long long mw = (cpc + 31) / 32;
  const int slots = MMA_SLOTS;
  if (mw > 8 || mw * C > slots) return false;
  // ring depth: as deep as asked for (default 2: a stage is free again as soon as its block has been through the
  // tensor-core pass, and a shallow ring lets more CTAs share an SM) while two CTAs still share an SM; else one per SM
  const size_t two_per_sm = (size_t)(227 * 1024) / 2 - 1024;
  int want = c->opt_stages > 0 ? std::min(c->opt_stages, 8) : 2;
  int stages = want;
  while (stages > 2 && MmaSmem(stages, (size_t)cpc * 16, slots).total > two_per_sm) --stages;
  if (MmaSmem(stages, (size_t)cpc * 16, slots).total > two_per_sm) {
    stages = want;
    while (stages >= 2 && MmaSmem(stages, (size_t)cpc * 16, slots).total > kSmemBudget) --stages;
    if (stages < 2) return false;
  }
  out->C = C;
  out->cpc = (int)cpc;
  out->math_warps = (int)mw;
  out->stages = stages;
  // 16 samples per block: half as many hand-offs per sample; one CTA per SM
  int s16 = c->opt_stages > 0 ? std::min(c->opt_stages, 8) : 2;
  while (s16 >= 2 && Mma16Smem(s16, (size_t)cpc * 16).total > kSmemBudget) --s16;
  out->stages16 = s16 >= 2 ? s16 : 0;
  const bool can16 = out->stages16 > 0;
  out->block = (c->opt_block_samples == 16 || (c->opt_block_samples == 0 && can16)) ? 16 : 8;
  if (out->block == 16 && !can16) return false;
  return true;
}

wpsgd_status launch_mma(wpsgd_ctx* c, const ChainParams& p, const ClusterShape& sh) {
  ClusterParams cp;
  cp.b.c = p;
  cp.b.stages = sh.stages;
  cp.b.eta_lambda = (double)c->eta0 * (double)c->lambda;
  cp.b.spin_limit = c->opt_spin_limit;
  cp.b.drop_block = c->opt_drop_block;
  cp.b.group_order = nullptr;
  cp.chunks_per_cta = sh.cpc;
  const bool b16 = sh.block == 16;
  if (b16) cp.b.stages = sh.stages16;
  const size_t smem = b16 ? Mma16Smem(sh.stages16, (size_t)sh.cpc * 16).total : MmaSmem(sh.stages, (size_t)sh.cpc * 16, MMA_SLOTS).total;
  auto go = [&](auto kern) -> wpsgd_status {
    CU_TRY(c, allow_all_smem(kern));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.k * sh.C));
    cfg.blockDim = dim3((unsigned)(64 + 32 * sh.math_warps));
    cfg.dynamicSmemBytes = smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)sh.C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    CU_TRY(c, cudaLaunchKernelEx(&cfg, kern, cp));
    c->launches++;
    return WPSGD_OK;
  };
  if (b16) {
    const bool full = sh.cpc % 32 == 0 && (long long)sh.cpc * sh.C * 8 == c->d;
    // Clusters of up to two CTAs have a form of their own where every warp is full (cycles per 16 samples, squared / logistic: 4096 columns
    // 3640 / 4660 in the form for up to eight, 3530 / 4570 in it; 2560: 3370 / 4296, 3289 / 4205; with guards the other way round, 3000
    // columns 3600 / 4500 and 3730 / 4620, 3328: 3670 / 4606 and 3780 / 4680).
    auto pick = [&](auto loss, auto is_full) -> wpsgd_status {
      if constexpr (is_full.value)
        if (sh.C <= 2) return go(chain_mma16_kernel<loss.value, true, 2>);
      return go(chain_mma16_kernel<loss.value, is_full.value, 8>);
    };
    auto with_loss = [&](auto is_full) -> wpsgd_status {
      switch (c->loss) {
        case WPSGD_LOSS_HINGE: return pick(std::integral_constant<int, LOSS_HINGE>(), is_full);
        case WPSGD_LOSS_LOGISTIC: return pick(std::integral_constant<int, LOSS_LOGISTIC>(), is_full);
        default: return pick(std::integral_constant<int, LOSS_SQUARED>(), is_full);
      }
    };
    return full ? with_loss(std::true_type()) : with_loss(std::false_type());
  }
  switch (c->loss) {
    case WPSGD_LOSS_HINGE: return go(chain_mma_kernel<LOSS_HINGE, 4>);
    case WPSGD_LOSS_LOGISTIC: return go(chain_mma_kernel<LOSS_LOGISTIC, 4>);
    default: return go(chain_mma_kernel<LOSS_SQUARED, 4>);
  }
}

// Warp-per-node kernel: one CTA of four warps per SM, or two? A warp alone on its scheduler takes about 1990 cycles
// per block of 8 samples, two warps sharing one about 3500 each (measured, d = 256 fp32). With one CTA per SM
// there are 148 CTA slots and the remaining CTAs queue behind, longest first; with two there are 296 slots. Which
// finishes first depends on the step counts (k = 1024: equal work is one wave of 3500 against two of 1990; with a speed
// ratio of 4 one CTA per SM is ahead), so both schedules are played through on the host: CTAs in launch order (a CTA lasts
// as long as its longest chain) onto the slot that frees first.
bool two_warp_ctas_per_sm_finish_first(const std::vector<long long>& steps, int warps) {
  std::vector<long long> sorted(steps);
  std::sort(sorted.begin(), sorted.end(), [](long long a, long long b) { return a > b; });
  std::vector<long long> cta_cost;
  for (size_t i = 0; i < sorted.size(); i += (size_t)warps) cta_cost.push_back(sorted[i]);
  auto makespan = [&](int slots, double cycles_per_block) {
    std::vector<double> free_at((size_t)std::min<size_t>((size_t)slots, cta_cost.size()), 0.0);
    if (free_at.empty()) return 0.0;
    std::make_heap(free_at.begin(), free_at.end(), std::greater<double>());
    double end = 0.0;
    for (long long cost : cta_cost) {
      std::pop_heap(free_at.begin(), free_at.end(), std::greater<double>());
      const double t = free_at.back() + (double)cost * cycles_per_block;
      free_at.back() = t;
      end = std::max(end, t);
      std::push_heap(free_at.begin(), free_at.end(), std::greater<double>());
    }
    return end;
  };
  return makespan(2 * 148, 3500.0) < makespan(148, 1990.0);
}

// ---- blocked kernel with lagged margins ---------------------------------------------------------------------------------
struct LagShape {
  int C = 1, cpc = 0, stages = 0, teams = 1, gram_warps = 1, model_warps = 1, vb = 8, nc = 1, raw_stages = 0, realign_warps = 0, realign_rows = 1, copy_warps = 2, warps = 0;
  size_t smem = 0;
};

template <typename XT>
bool lag_kernel_fits(const wpsgd_ctx* c, bool aligned, int C, LagShape* out) {
  constexpr int V = XVec<XT>::V;
  if ((double)c->eta0 * (double)c->lambda > 0.25) return false;  // keeps a^-8 harmless in fp32
  const long long chunks = (c->d + V - 1) / V;
  const long long cpc = (chunks + C - 1) / C;
  if ((long long)(C - 1) * cpc >= chunks) return false;  // every CTA of the cluster owns at least one chunk
  if (!c->steps_sorted.empty() && c->steps_sorted[0] > (1ll << 33)) return false;  // block numbers are ints
  LagShape sh;
  sh.C = C;
  sh.cpc = (int)cpc;
  // A model thread owns one vector of 8 bytes in narrow slices (the rows of two blocks then stay in registers), else one or two of
  // 16: 64 fp32 chunks 1143 cycles per block with 16-byte vectors, 1236 with 8-byte ones (twice as many warps); 63 bf16 chunks
  // 1106 and 1054.
  if (cpc > 2 * 32 * (aligned ? LAG_MAX_MODEL_WARPS : LAG_MAX_MODEL_WARPS_REALIGNED)) return false;
  sh.vb = cpc <= (sizeof(XT) == 4 ? 32 : 64) ? 8 : 16;
  // Two vectors where one would take so many warps that a Gram or copy warp had to go (fp32, unaligned rows, 8 CTAs of 65 / 97 / 128
  // chunks: 2090, 2700, 3090 cycles per block with one, 2030, 2550, 3000 with two; aligned, 4 CTAs of 204: 3230 and 3080, bf16 2010 and
  // 2700: those take one vector up to seven warps).
  const int most = aligned ? (C > 1 ? (sizeof(XT) == 4 ? 6 : 7) : LAG_MAX_MODEL_WARPS) : (sizeof(XT) == 4 && C > 1 ? 2 : LAG_MAX_MODEL_WARPS_REALIGNED);
  sh.nc = cpc <= 32 * most ? 1 : 2;
  const int per_warp = 32 * sh.vb * sh.nc;
  sh.model_warps = (int)((cpc * 16 + per_warp - 1) / per_warp);
  // As deep a ring as there is room for. Realigning warps: a block each and both rings in multiples of four up to 64 chunks (fp32,
  // 31 chunks, 12 chains: 1314 cycles per block, 1490 with all warps on every block), else all on a block (128 chunks: 3050, 5100).
  if (!aligned) {
    sh.realign_warps = LAG_REALIGN_WARPS;
    sh.realign_rows = cpc <= 64 && (c->opt_stages == 0 || c->opt_stages >= 4) ? 1 : LAG_REALIGN_WARPS;
  }
  int others = 3 + (C > 1 ? 1 : 0) + sh.model_warps + sh.realign_warps;
  const int gram = (others + LAG_GRAM_WARPS + 1) * 32 > LAG_MAX_THREADS ? LAG_GRAM_WARPS - 1 : LAG_GRAM_WARPS;
  others += gram;
  const int q_row = lag_q_row(sh.vb, sh.nc, !aligned);
  int want = c->opt_stages > 0 ? std::max(3, c->opt_stages) : LAG_MAX_STAGES;
  for (; want >= 3; --want) {
    if (!aligned && sh.realign_rows == 1 && want % LAG_REALIGN_WARPS != 0) continue;
    sh.raw_stages = aligned ? 0 : (sh.realign_rows > 1 ? 3 : (want >= 8 ? LAG_MAX_RAW_STAGES : 4));
    sh.smem = LagSmem(want, (size_t)cpc * 16, C, gram, sh.raw_stages, q_row).total;
    if (sh.smem <= kSmemMax) break;
  }
  if (want < 3 || (want < 4 && C < 8 && c->opt_stages == 0 && c->opt_cluster == 0)) return false;
  // Gram teams: four of one warp, two of two or one of all, as the ring feeds them (a team holds two stages while it works). With more
  // than two teams the ring is a multiple of their number, so that a team has seen every earlier block of the stages it
  // waits for (else a barrier's parity could stand for an older phase). Three warps, where no more fit: three teams from 6 stages
  // on, which costs up to two of the stages; a ring of 3 does not feed them (cycles per block, squared loss, three teams and one: fp32,
  // 2 CTAs of 449 / 512 chunks 10040 / 11230 and 7590 / 8330; 2 x 232 chunks of unaligned rows 7110 and 5840; 8 CTAs of 97
  // chunks, one team on 8 stages and three on 6: 3000 and 2700).
  if (gram < LAG_GRAM_WARPS) {
    if (want >= 6) want = sh.realign_rows == 1 && !aligned ? (want >= 12 ? 12 : want) : want - want % 3;
    sh.teams = want >= 6 && want % 3 == 0 ? 3 : 1;
  } else {
    if (want >= 8) want -= want % 4;
    sh.teams = want >= 8 ? 4 : (want >= 5 ? 2 : 1);
  }
  sh.gram_warps = gram / sh.teams;
  sh.stages = want;
  sh.smem = LagSmem(want, (size_t)cpc * 16, C, gram, sh.raw_stages, q_row).total;
  sh.copy_warps = (others + 2) * 32 <= LAG_MAX_THREADS ? 2 : 1;
  sh.warps = others + sh.copy_warps;
  if (sh.warps * 32 > LAG_MAX_THREADS) return false;
  *out = sh;
  return true;
}

template <typename XT>
wpsgd_status launch_lag(wpsgd_ctx* c, const ChainParams& p, const LagShape& sh) {
  LagParams lp;
  int launch_warps = 0;
  lp.b.c = p;
  lp.b.stages = sh.stages;
  lp.b.eta_lambda = (double)c->eta0 * (double)c->lambda;
  lp.b.spin_limit = c->opt_spin_limit;
  lp.b.drop_block = c->opt_drop_block;
  lp.b.group_order = nullptr;
  lp.chunks_per_cta = sh.cpc;
  lp.gram_teams = sh.teams;
  lp.gram_warps = sh.gram_warps;
  lp.model_warps = sh.model_warps;
  lp.raw_stages = sh.raw_stages;
  lp.realign_warps = sh.realign_warps;
  lp.realign_rows = sh.realign_rows;
  lp.copy_warps = sh.copy_warps;
  // Warp w runs on scheduler w mod 4. The scheduler of the recurrence warp gets only the two short loops beside it (sums of q,
  // constants); the others are dealt out over the other three (16 chains of 1024 fp32 columns, logistic: 1058 cycles per block
  // with the roles in plain order, 908 this way; all four gram warps on one scheduler: 1136).
  {
    const int sums = sh.C > 1 ? 1 : 0, constants = 1 + sh.model_warps + sums + sh.copy_warps, gram = constants + 2;
    int first[LAG_MAX_THREADS / 32], rest[LAG_MAX_THREADS / 32], nf = 0, nr = 0;
    first[nf++] = 0;
    if (sums) first[nf++] = 1 + sh.model_warps;
    // Wide fp32 slices: the Gram warps bound the block, one goes to every scheduler; 64 chunks 1143 cycles per block, 1285 without.
    // Wide aligned bf16 slices: the model warps do, and one of each goes there (the constants elsewhere); one CTA, 96 / 128 / 256 chunks
    // 1320, 1550, 2410 without, 1240, 1330, 2210 with them; 4 CTAs of 128 / 192 chunks 1510, 1990 and 1330, 1840
    // (up to 96 chunks clusters are 1 to 3 % slower with them).
    const int m0 = sizeof(XT) == 2 && sh.vb == 16 && !sh.raw_stages && (sh.C == 1 || sh.cpc > 96) ? 1 : 0, g0 = m0 || (sizeof(XT) == 4 && sh.cpc > 40) ? 1 : 0;
    first[nf++] = m0 ? sh.model_warps : constants;
    if (g0) first[nf++] = gram;
    for (int i = 0; i < sh.model_warps - m0; ++i) rest[nr++] = 1 + i;
    for (int i = g0; i < sh.teams * sh.gram_warps; ++i) rest[nr++] = gram + i;
    if (m0) rest[nr++] = constants;
    rest[nr++] = constants + 1;  // feeder
    for (int i = 0; i < sh.copy_warps; ++i) rest[nr++] = 1 + sh.model_warps + sums + i;
    for (int i = gram + sh.teams * sh.gram_warps; i < sh.warps; ++i) rest[nr++] = i;  // realign
    while (nr > 12) first[nf++] = rest[--nr];
    const int warps = 4 * std::max(nf, (nr + 2) / 3);
    int a = 0, b = 0;
    for (int w = 0; w < LAG_MAX_THREADS / 32; ++w) {
      if (w % 4 == 0) lp.role[w] = a < nf ? (unsigned char)first[a++] : 255;
      else lp.role[w] = b < nr ? (unsigned char)rest[b++] : 255;
    }
    launch_warps = warps;
  }
  auto go = [&](auto kern) -> wpsgd_status {
    CU_TRY(c, allow_all_smem(kern));
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)(p.k * sh.C));
    cfg.blockDim = dim3((unsigned)(32 * launch_warps));
    cfg.dynamicSmemBytes = sh.smem;
    cfg.stream = c->stream;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = (unsigned)sh.C;
    at[0].val.clusterDim.y = 1;
    at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
    CU_TRY(c, cudaLaunchKernelEx(&cfg, kern, lp));
    c->launches++;
    return WPSGD_OK;
  };
  auto pick = [&](auto multi, auto realign) -> wpsgd_status {
    if (sh.nc == 2) return go(chain_lag_kernel<XT, 16, 2, multi.value, realign.value>);
    if (sh.vb == 16) return go(chain_lag_kernel<XT, 16, 1, multi.value, realign.value>);
    return go(chain_lag_kernel<XT, 8, 1, multi.value, realign.value>);
  };
  if (sh.C > 1) return sh.raw_stages ? pick(std::true_type(), std::true_type()) : pick(std::true_type(), std::false_type());
  return sh.raw_stages ? pick(std::false_type(), std::true_type()) : pick(std::false_type(), std::false_type());
}

// blocked kernel, one warp per node (small d)
template <typename XT>
bool block_warp_kernel_fits(const wpsgd_ctx* c, int nk, bool aligned, int* R_out, int* stages_out, int* warps_out) {
  constexpr int V = XVec<XT>::V;
  if (!aligned) return false;
  if ((double)c->eta0 * (double)c->lambda > 0.25) return false;
  const long long chunks = c->d / V;
  const int R = (int)((chunks + 31) / 32);
  if (R > 2) return false;
  const size_t row_bytes = (size_t)c->d * sizeof(XT);
  // Four nodes per CTA and two CTAs per SM. Each chain is bound by its own dependent instruction stream, so what
  // a long chain needs is few co-runners late in the run, not an equal share of work per SM: with chains dealt out
  // longest first, the CTAs of the longest chains land on the SMs first and are paired with the shortest ones.
  // (Measured on k = 1024, d = 256, speed ratio 4: 4.9 ms this way, 6.9 ms with one balanced 7-warp CTA per SM.)
  if (nk != c->k) return false;  // its node-to-CTA table covers the whole node set
  int warps = (int)std::min<long long>(4, std::max<long long>(1, nk));
  if (c->opt_threads >= 32 && c->opt_threads % 32 == 0) warps = std::min(BLKW_MAX_WARPS, c->opt_threads / 32);
  // one CTA per SM (a ring of 4 stages per warp takes the shared memory of a second one) or two (3 stages): see above
  const bool one_cta_per_sm = c->opt_stages >= 4 || (c->opt_stages == 0 && !two_warp_ctas_per_sm_finish_first(c->last_steps, warps));
  int stages = c->opt_stages > 0 ? std::min(c->opt_stages, 4) : (one_cta_per_sm ? 4 : 3);
  while (BlockWarpSmem(stages, row_bytes, warps).total > ((warps <= 4 && !one_cta_per_sm) ? 100 * 1024 : kSmemBudget)) {
    if (stages > 2) --stages;
    else if (warps > 1) --warps;
    else return false;
  }
  *R_out = R;
  *stages_out = stages;
  *warps_out = warps;
  return true;
}

template <typename XT, int R>
wpsgd_status launch_block_warp_r(wpsgd_ctx* c, const BlockParams& bp, size_t smem, int ctas, int warps) {
  auto go = [&](auto kern) -> wpsgd_status {
    CU_TRY(c, allow_all_smem(kern));
    launch(kern, ctas, 32 * warps, smem, c->stream, bp);
    CU_TRY(c, cudaGetLastError());
    c->launches++;
    return WPSGD_OK;
  };
  const bool decay = c->sched == WPSGD_LR_INV_SQRT;
  switch (c->loss) {
    case WPSGD_LOSS_HINGE: return decay ? go(chain_block_warp_kernel<XT, R, LOSS_HINGE, true>) : go(chain_block_warp_kernel<XT, R, LOSS_HINGE, false>);
    case WPSGD_LOSS_LOGISTIC: return decay ? go(chain_block_warp_kernel<XT, R, LOSS_LOGISTIC, true>) : go(chain_block_warp_kernel<XT, R, LOSS_LOGISTIC, false>);
    default: return decay ? go(chain_block_warp_kernel<XT, R, LOSS_SQUARED, true>) : go(chain_block_warp_kernel<XT, R, LOSS_SQUARED, false>);
  }
}

template <typename XT>
wpsgd_status launch_block_warp(wpsgd_ctx* c, const ChainParams& p, int R, int stages, int warps) {
  BlockParams bp;
  bp.c = p;
  bp.stages = stages;
  bp.eta_lambda = (double)c->eta0 * (double)c->lambda;
  bp.spin_limit = c->opt_spin_limit;
  bp.drop_block = -1;
  bp.group_order = c->t_order;  // longest first, consecutive ranks share a CTA; -1 fills the last one
  const int ctas = (c->k + warps - 1) / warps;
  const size_t smem = BlockWarpSmem(stages, (size_t)c->d * sizeof(XT), warps).total;
  return R == 1 ? launch_block_warp_r<XT, 1>(c, bp, smem, ctas, warps) : launch_block_warp_r<XT, 2>(c, bp, smem, ctas, warps);
}

// ---- which dense kernel -------------------------------------------------------------------------------------------------
// Every chain is a serial string of blocks of 8 samples, so what decides is how long a block takes in a chain that has
// its SMs to itself (L cycles), how much of an SM's throughput it uses up when chains share one (I cycles), and how the
// chains queue for the slots. The estimate of a run:
//     max( longest queue of a slot x L,  all blocks x I / 148 )  +  start-up of the kernel per wave of chains,
// with the chains in launch order (longest first) on `slots` slots. The figures are device times of runs of 64 to 4000
// steps with k = 4 .. 2000 chains (1965 MHz); the estimates come out within about a tenth of the times measured, e.g.
// (measured, us, logistic, 2048 steps) fp32 d = 1024, k = 16: lagged form 160, one CTA per chain 242; k = 100: 475, 247; d = 256,
// k = 148: lagged 154, CTA per chain 178, warp per chain 275; k = 300: 445, 265, 275; d = 128, k = 200: 225, 202, 227.
double run_estimate(const wpsgd_ctx* c, int slots, double L, double I, double start, double restart) {
  const std::vector<long long>& n = c->steps_sorted;
  const size_t k = n.size(), m = (size_t)slots;
  double q = (double)n[0];
  // the t-th wave of a slot holds at best the (t m)-th longest chain
  for (size_t t = 1; t < 4 && t * m < k; ++t) q = std::max(q, (double)(t + 1) * (double)n[t * m]);
  q = std::max(q, c->steps_sum / (double)slots);
  const double waves = (double)((k + m - 1) / m);
  if (waves > 1.0) q *= 1.06;  // chains of a second wave do not fall into place perfectly
  return std::max(q * L, c->steps_sum * I / 148.0) / 8.0 + start + restart * (waves - 1.0);
}
// piecewise linear through (x_i, y_i), x ascending
double through(double x, std::initializer_list<std::pair<double, double>> pts) {
  const std::pair<double, double>* a = pts.begin();
  if (x <= a->first) return a->second;
  for (const std::pair<double, double>* b = a + 1; b != pts.end(); a = b, ++b)
    if (x <= b->first) return a->second + (b->second - a->second) * (x - a->first) / (b->first - a->first);
  return a->second * x / a->first;
}

// Clusters of C CTAs, one CTA per SM, that are resident at once. A cluster lies within one GPC and the GPCs differ in size from
// GPU to GPU, so the driver is asked, once per device: where 148 / 8 = 18 or 16 of 8 were taken for granted, 16 equally long
// chains over 8 CTAs each ran in two waves (measured: 15 of 8, 33 of 4, 74 of 2).
int cluster_slots(int device, int C, size_t chains) {
  if (C == 1) return 148;
  const int i = C == 2 ? 0 : (C == 4 ? 1 : 2);
  const int nominal = 148 / C;
  if (chains * (size_t)C <= 64) return nominal;  // these fit in any case
  static std::atomic<int> known[64][3];  // 0: not asked yet
  if (device < 64 && known[device][i] > 0) return known[device][i];
  auto kern = chain_lag_kernel<float, 8, 1, true, false>;
  const size_t smem = 200 * 1024;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(nominal * C));
  cfg.blockDim = dim3(LAG_MAX_THREADS);
  cfg.dynamicSmemBytes = smem;
  cudaLaunchAttribute at;
  at.id = cudaLaunchAttributeClusterDimension;
  at.val.clusterDim.x = (unsigned)C;
  at.val.clusterDim.y = 1;
  at.val.clusterDim.z = 1;
  cfg.attrs = &at;
  cfg.numAttrs = 1;
  int n = 0;
  if (allow_all_smem(kern) != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess || n < 1) {
    cudaGetLastError();
    n = C == 2 ? 74 : (C == 4 ? 32 : 14);
  }
  n = std::min(n, nominal);
  if (device < 64) known[device][i] = n;
  return n;
}

template <typename XT>
double lag_estimate(const wpsgd_ctx* c, const LagShape& sh) {
  constexpr bool F32 = sizeof(XT) == 4;
  const double x = (double)sh.cpc;
  double L;
  if (F32) L = sh.C == 1 ? through(x, {{8, 725}, {16, 740}, {32, 815}, {48, 920}, {64, 1090}, {96, 1430}, {128, 1875}, {256, 3490}, {512, 6850}})
                         : through(x, {{8, 790}, {16, 800}, {32, 840}, {48, 1000}, {64, 1130}, {96, 1500}, {128, 1940}, {256, 3560}, {384, 5560}, {448, 6290}, {456, 7680}, {512, 8330}});
  else L = sh.C == 1 ? through(x, {{16, 785}, {32, 885}, {64, 1015}, {96, 1245}, {128, 1330}, {192, 1740}, {256, 2205}, {336, 3040}, {420, 3320}, {448, 4550}, {512, 5470}})
                     : through(x, {{16, 865}, {48, 925}, {64, 1015}, {96, 1255}, {128, 1340}, {192, 1835}, {224, 2060}, {256, 2390}, {372, 3340}, {400, 4400}, {512, 4850}});
  if (sh.C == 8) L += 25.0;
  if (sh.realign_warps) L = std::max(L, through(x, {{8, 800}, {16, 850}, {32, 1000}, {48, 1350}, {64, 1550}, {72, 2000}, {96, 2500}, {128, 2950}, {224, 4850}, {232, 6000}, {256, 6700}}));
  return run_estimate(c, cluster_slots(c->device, sh.C, c->steps_sorted.size()), L, 0.0, 5000.0 + 40.0 * x, 10000.0);
}

// The lagged form's best cluster size (or the one asked for); the estimate, or a negative number when it does not fit.
template <typename XT>
double best_lag_shape(const wpsgd_ctx* c, bool aligned, LagShape* out) {
  double best = -1.0;
  for (int C = 1; C <= 8; C *= 2) {
    LagShape sh;
    if ((c->opt_cluster > 0 && C != c->opt_cluster) || !lag_kernel_fits<XT>(c, aligned, C, &sh)) continue;
    const double t = lag_estimate<XT>(c, sh);
    if (best < 0.0 || t < best) {
      best = t;
      *out = sh;
    }
  }
  return best;
}

template <typename XT>
wpsgd_status launch_dense(wpsgd_ctx* c, const ChainParams& p) {
  constexpr int V = XVec<XT>::V;
  constexpr bool F32 = sizeof(XT) == 4;
  const long long d = c->d;
  const bool aligned = ((uintptr_t)p.X % 16 == 0) && ((p.ld * (long long)sizeof(XT)) % 16 == 0) && (d % V == 0) &&
                       ((uintptr_t)c->W % 16 == 0);
  const long long chunks = d / V;
  int variant = c->opt_variant;
  int bthreads = 0, bR = 0, bstages = 0;
  const bool block_ok = block_kernel_fits<XT>(c, aligned, &bthreads, &bR, &bstages);
  int wR = 0, wstages = 0, wwarps = 0;
  const bool block_warp_ok = block_warp_kernel_fits<XT>(c, p.k, aligned, &wR, &wstages, &wwarps);
  ClusterShape mma_shape;
  const bool mma_ok = !F32 && mma_kernel_fits(c, aligned, &mma_shape);
  LagShape lag_shape;
  double lag_t = -1.0;
  if (variant == 0 || variant == 10) lag_t = best_lag_shape<XT>(c, aligned, &lag_shape);
  const double x = (double)chunks;
  // several CTAs share an SM (as many as their shared memory lets in): a chain then takes a fifth longer
  auto shared_estimate = [&](size_t smem, double L, double I) {
    const int per_sm = std::max(1, std::min(4, (int)(227 * 1024 / (smem + 1024))));
    return run_estimate(c, 148 * per_sm, c->steps_sorted.size() > 148 && per_sm > 1 ? 1.2 * L : L, I, 0.0, 6000.0);
  };
  const bool decay = c->sched == WPSGD_LR_INV_SQRT;
  double mma_t = -1.0;
  if (mma_ok) {
    // (guarded passes where some warp is not full; the decaying schedule's tables are formed on the chain's path)
    const bool full = mma_shape.cpc % 32 == 0 && (long long)mma_shape.cpc * mma_shape.C == chunks;
    const double w = (double)mma_shape.cpc;
    const double L = through(w, {{64, 1260}, {128, 1330}, {256, 1820}}) * (full || mma_shape.C > 1 ? 1.0 : 1.14) * (decay ? 1.1 : 1.0);
    if (mma_shape.C == 1) mma_t = shared_estimate(Mma16Smem(mma_shape.stages16, (size_t)mma_shape.cpc * 16).total, L, through(w, {{32, 620}, {64, 800}, {128, 1090}, {256, 1820}}));
    else mma_t = run_estimate(c, cluster_slots(c->device, mma_shape.C, c->steps_sorted.size()), L, 0.0, 0.0, 6000.0);
  }
  if (variant == 0) {
    double best = lag_t;
    if (best >= 0.0) variant = 10;
    auto offer = [&](bool ok, int v, double t) {
      if (ok && (best < 0.0 || t < best)) {
        best = t;
        variant = v;
      }
    };
    if (block_warp_ok) {
      // one chain per scheduler or two (see two_warp_ctas_per_sm_finish_first)
      const double L = (F32 ? (chunks <= 32 ? 1655.0 : 1990.0) : (chunks <= 32 ? 1700.0 : 2270.0)) * (decay ? 1.25 : 1.0);
      const double I = (F32 ? (chunks <= 32 ? 365.0 : 446.0) : (chunks <= 32 ? 440.0 : 655.0)) * (decay ? 1.25 : 1.0);
      offer(true, 5, std::min(run_estimate(c, 592, L, I, 0.0, 6000.0), run_estimate(c, 1184, 1.76 * L, I, 0.0, 6000.0)));
    }
    if (block_ok) {
      const double L = F32 ? through(x, {{32, 1310}, {64, 1320}, {128, 1655}, {256, 1825}, {512, 3140}})
                           : through(x, {{64, 1780}, {128, 1855}, {256, 2560}, {512, 4250}});
      const double I = F32 ? through(x, {{32, 530}, {64, 745}, {128, 1080}, {256, 1825}, {512, 3140}})
                           : through(x, {{32, 730}, {64, 1020}, {128, 1345}, {256, 2560}, {512, 4250}});
      offer(true, 4, shared_estimate(BlockSmem(bstages, (size_t)d * sizeof(XT) + (F32 ? 0 : 16), bthreads / 32 - 2).total, L, I));
    }
    // Rows of 2048 columns and more: the tensor-core kernel keeps the runs of up to about 16 blocks, whatever the start-up in the lagged
    // form's estimate (4 to 74 chains of 2048, 8 to 64 steps: 12 to 20 us there, 10 to 16; narrower rows 14 against 25 us after 128 steps).
    if (mma_ok && (best < 0.0 || mma_t < best + (variant == 10 && chunks >= 256 ? 7500.0 : 0.0))) {
      best = mma_t;
      variant = 8;
    }
    // rows wider than the blocked kernels take, many of them: the direct kernel keeps one chain per SM
    if (lag_t >= 0.0) offer(aligned && chunks > 512 && chunks <= 512 * 4, 2, run_estimate(c, 148, 7000.0 + 5.4 * x, 0.0, 0.0, 6000.0));
    if (best < 0.0) variant = !aligned || chunks > 512 * 4 ? 1 : (chunks <= 64 ? 3 : 2);
  }
  if (variant == 9) {
    // fp32 rows, at most 64 chunks of a row per CTA: with clusters of the size asked for, else the best one
    double best = -1.0;
    for (int C = 1; F32 && aligned && C <= 8; C *= 2) {
      LagShape sh;
      if ((c->opt_cluster > 0 && C != c->opt_cluster) || (chunks + C - 1) / C > 64 || !lag_kernel_fits<XT>(c, aligned, C, &sh)) continue;
      const double t = lag_estimate<XT>(c, sh);
      if (best < 0.0 || t < best) {
        best = t;
        lag_shape = sh;
      }
    }
    if (best < 0.0)
      return fail(c, WPSGD_ERR_UNSUPPORTED,
                  "cluster kernel for fp32 rows needs 16-byte aligned rows, eta*lambda <= 0.25 and a cluster of "
                  "1, 2, 4 or 8 CTAs with at most 64 chunks of a row each");
    return launch_lag<XT>(c, p, lag_shape);
  }
  if (variant == 10) {
    if (lag_t < 0.0)
      return fail(c, WPSGD_ERR_UNSUPPORTED,
                  "lagged kernel needs eta*lambda <= 0.25 and a cluster of 1, 2, 4 or 8 CTAs that each hold a share of the row");
    return launch_lag<XT>(c, p, lag_shape);
  }
  if (variant == 5) {
    if (!block_warp_ok)
      return fail(c, WPSGD_ERR_UNSUPPORTED,
                  "blocked warp kernel needs 16-byte aligned rows of at most 64 chunks, "
                  "eta*lambda <= 0.25");
    return launch_block_warp<XT>(c, p, wR, wstages, wwarps);
  }
  if (variant == 8) {
    ClusterShape sh;
    if (sizeof(XT) != 2 || !mma_kernel_fits(c, aligned, &sh))
      return fail(c, WPSGD_ERR_UNSUPPORTED,
                  "tensor-core cluster kernel needs bf16 rows, 16-byte aligned, eta*lambda <= 0.25, a "
                  "cluster of 1, 2, 4 or 8 CTAs with at most 256 chunks of a row each and at most 16 math warps in all");
    return launch_mma(c, p, sh);
  }
  if (variant == 4) {
    if (!block_ok)
      return fail(c, WPSGD_ERR_UNSUPPORTED,
                  "blocked kernel needs 16-byte aligned rows of at most 8 KiB and eta*lambda <= 0.25");
    return launch_block<XT>(c, p, bthreads, bR, bstages);
  }
  if ((variant == 2 || variant == 3) && !aligned)
    return fail(c, WPSGD_ERR_UNSUPPORTED, "register kernels need 16-byte aligned rows and d a multiple of 16 bytes");
  if (variant == 3 && chunks > 32 * 4) return fail(c, WPSGD_ERR_UNSUPPORTED, "warp-per-node kernel: d too large");
  if (variant == 2 && chunks > 512 * 4) return fail(c, WPSGD_ERR_UNSUPPORTED, "CTA-per-node kernel: d too large");
  if (variant == 1) {
    launch(chain_generic_kernel<XT>, p.k, 256, 0, c->stream, p);
    CU_TRY(c, cudaGetLastError());
    c->launches++;
    return WPSGD_OK;
  }
  if (variant != 2 && variant != 3) return fail(c, WPSGD_ERR_UNSUPPORTED, "dense_variant not available");
  int threads = 32, R = 1;
  if (variant == 3) {
    R = (int)((chunks + 31) / 32);
  } else {
    threads = c->opt_threads > 0 ? c->opt_threads : (int)std::min<long long>(512, ((chunks + 31) / 32) * 32);
    R = (int)((chunks + threads - 1) / threads);
  }
  if (R > 2) R = 4;  // instantiated: 1, 2, 4
  if ((long long)R * threads < chunks) return fail(c, WPSGD_ERR_UNSUPPORTED, "threads too few for d");
  int pf = c->opt_prefetch > 0 ? c->opt_prefetch : std::max(2, 8 / R);
  pf = pf >= 8 ? 8 : (pf >= 4 ? 4 : 2);
  const bool bpn = variant == 2;
  switch (R) {
    case 1: return launch_reg_pf<XT, 1>(c, p, bpn, threads, pf);
    case 2: return launch_reg_pf<XT, 2>(c, p, bpn, threads, pf);
    default: return launch_reg_pf<XT, 4>(c, p, bpn, threads, pf);
  }
}

// Nodes launched together (a run of `count` consecutive entries of the longest-first order) once `ready` has happened.
struct LaunchGroup {
  int count;
  cudaEvent_t ready;
};

wpsgd_status run_dense_common(wpsgd_ctx* c, const void* X, wpsgd_xtype xt, long long ld, const float* y,
                              const long long* shard_off, const long long* n_steps, const float* w0, bool resume,
                              const std::vector<LaunchGroup>* groups = nullptr) {
  if (xt != WPSGD_X_F32 && xt != WPSGD_X_BF16) return fail(c, WPSGD_ERR_INVALID_ARG, "unknown feature type");
  if (ld < c->d) return fail(c, WPSGD_ERR_INVALID_ARG, "ld_elems < d");
  Plan pl;
  std::vector<long long> first = resume ? c->steps_done : std::vector<long long>(c->k, 0);
  wpsgd_status s = make_plan(c, (const long long*)shard_off, (const long long*)n_steps, first, &pl);
  if (s != WPSGD_OK) return s;
  if (pl.total > 0 && (!X || !y)) return fail(c, WPSGD_ERR_INVALID_ARG, "X or y is NULL");
  s = upload_plan_and_stream(c, pl);
  if (s != WPSGD_OK) return s;
  c->last_steps = pl.steps;
  ChainParams p;
  p.X = X; p.ld = ld; p.y = y;
  p.shard_off = c->t_shard_off; p.n_steps = c->t_steps; p.first = c->t_first; p.idx_off = c->t_idx_off;
  p.idx = c->idx; p.order = c->t_order; p.W = c->W; p.w0 = w0; p.resume = resume ? 1 : 0;
  p.k = c->k; p.d = c->d; p.eta0 = c->eta0; p.sched = c->sched; p.lambda = c->lambda; p.loss = c->loss;
  p.status = c->status;
  s = timing_begin(c);
  if (s != WPSGD_OK) return s;
  // The estimates go by the chains of one launch. For groups of nodes that run one after another these are the group's, with its
  // step counts scaled to the longest chain of the run: groups of a run then differ in the number of chains only, and where all
  // of them fit the GPU at once anyway every group takes the kernel, and gives the bits, of a run on rows that lie on the device.
  auto estimate_for = [&](int first_slot, int count) {
    const long long longest = pl.steps[pl.order[0]], own = pl.steps[pl.order[first_slot]];
    c->steps_sorted.resize(count);
    c->steps_sum = 0.0;
    for (int i = 0; i < count; ++i) {
      const long long n = pl.steps[pl.order[first_slot + i]];
      c->steps_sorted[i] = own == longest ? n : (own > 0 ? (long long)((double)n / (double)own * (double)longest) : longest);
      c->steps_sum += (double)c->steps_sorted[i];
    }
  };
  if (!groups) {
    estimate_for(0, c->k);
    s = (xt == WPSGD_X_F32) ? launch_dense<float>(c, p) : launch_dense<__nv_bfloat16>(c, p);
    if (s != WPSGD_OK) return s;
  } else {
    // one launch per group of nodes, each behind the event that says its rows are on the device
    int first_slot = 0;
    for (const LaunchGroup& g : *groups) {
      CU_TRY(c, cudaStreamWaitEvent(c->stream, g.ready, 0));
      if (g.count > 0) {
        estimate_for(first_slot, g.count);
        ChainParams q = p;
        q.order = c->t_order + first_slot;
        q.k = g.count;
        s = (xt == WPSGD_X_F32) ? launch_dense<float>(c, q) : launch_dense<__nv_bfloat16>(c, q);  // grids follow q.k
        if (s != WPSGD_OK) return s;
      }
      first_slot += g.count;
    }
  }
  s = timing_end(c);
  if (s != WPSGD_OK) return s;
  for (int j = 0; j < c->k; ++j) c->steps_done[j] = first[j] + n_steps[j];
  c->have_run = c->streams_read = true;
  c->scaled = false;
  return WPSGD_OK;
}

// ---- sparse chain launch ---------------------------------------------------------------------------------
wpsgd_status run_csr_common(wpsgd_ctx* c, const long long* row_ptr, const int* col_idx, const float* val, const float* y,
                            const long long* shard_off, const long long* n_steps, const float* w0, bool resume) {
  Plan pl;
  std::vector<long long> first = resume ? c->steps_done : std::vector<long long>(c->k, 0);
  wpsgd_status s = make_plan(c, shard_off, n_steps, first, &pl);
  if (s != WPSGD_OK) return s;
  if (pl.total > 0 && (!row_ptr || !col_idx || !val || !y)) return fail(c, WPSGD_ERR_INVALID_ARG, "a CSR array or y is NULL");
  s = upload_plan_and_stream(c, pl);
  if (s != WPSGD_OK) return s;
  if (!resume || !c->scaled) {
    // fresh chains start from w0 with scale 1; chains continued from a dense run keep their models and get scale 1
    const long long n = (long long)c->k * c->d;
    if (c->d % 4 == 0 && aligned16(c->W) && aligned16(w0))
      launch(csr_init_kernel<4>, grid_for(n / 4, 256), 256, 0, c->stream, c->W, c->scale, w0, c->k, c->d, resume ? 1 : 0);
    else
      launch(csr_init_kernel<1>, grid_for(n, 256), 256, 0, c->stream, c->W, c->scale, w0, c->k, c->d, resume ? 1 : 0);
    CU_TRY(c, cudaGetLastError());
    c->launches++;
  }
  CsrParams p;
  p.row_ptr = row_ptr; p.col_idx = col_idx; p.val = val; p.y = y;
  p.shard_off = c->t_shard_off; p.n_steps = c->t_steps; p.first = c->t_first; p.idx_off = c->t_idx_off; p.idx = c->idx;
  p.order = c->t_order; p.U = c->W; p.scale = c->scale; p.k = c->k; p.d = c->d;
  p.eta0 = c->eta0; p.sched = c->sched; p.lambda = c->lambda; p.loss = c->loss; p.resume = resume ? 1 : 0;
  p.status = c->status;
  s = timing_begin(c);
  if (s != WPSGD_OK) return s;
  if (c->opt_sparse_variant == 1) {
    const int pf = c->opt_prefetch > 0 ? c->opt_prefetch : 4;
    if (pf >= 8) launch(chain_csr_kernel<8>, c->k, 32, 0, c->stream, p);
    else if (pf >= 4) launch(chain_csr_kernel<4>, c->k, 32, 0, c->stream, p);
    else launch(chain_csr_kernel<2>, c->k, 32, 0, c->stream, p);
    CU_TRY(c, cudaGetLastError());
  } else {
    const size_t smem = sizeof(CsrBlockSmem);
    auto go = [&](auto kern) -> wpsgd_status {
      CU_TRY(c, allow_all_smem(kern));
      // Launched after its predecessor, without the wait that an early start needs inside the kernel. With one body for all chains
      // the wait made no difference by itself (64 chains, 40 nonzeros per row: 12.18 ms with it and without; see
      // chain_csr_block_kernel for what did); the chains are long, so the plain launch costs nothing.
      kern<<<c->k, CSRB_THREADS, smem, c->stream>>>(p);
      CU_TRY(c, cudaGetLastError());
      return WPSGD_OK;
    };
    switch (c->loss) {
      case WPSGD_LOSS_HINGE: s = go(chain_csr_block_kernel<LOSS_HINGE>); break;
      case WPSGD_LOSS_LOGISTIC: s = go(chain_csr_block_kernel<LOSS_LOGISTIC>); break;
      default: s = go(chain_csr_block_kernel<LOSS_SQUARED>); break;
    }
    if (s != WPSGD_OK) return s;
  }
  c->launches++;
  s = timing_end(c);
  if (s != WPSGD_OK) return s;
  for (int j = 0; j < c->k; ++j) c->steps_done[j] = first[j] + n_steps[j];
  c->have_run = c->streams_read = true;
  c->scaled = true;
  return WPSGD_OK;
}

}  // namespace

// ---- built-in scratch of the entry point that allocates nothing ----------------------------------------
// Layout inside one file-scope device array (every section 256-byte aligned). The array exists once per
// GPU that loads this library and lives until the process exits.
namespace {
constexpr size_t align256(size_t x) { return (x + 255) / 256 * 256; }
struct StaticLayout {
  size_t W = 0;
  size_t idx = align256(W + sizeof(float) * (size_t)WPSGD_STATIC_MAX_MODEL_ELEMS);
  size_t tables = align256(idx + sizeof(uint32_t) * ((size_t)WPSGD_STATIC_MAX_STEPS + 64 * WPSGD_STATIC_MAX_NODES));
  size_t weights = align256(tables + TableLayout(WPSGD_STATIC_MAX_NODES).total);
  size_t scale = align256(weights + sizeof(double) * WPSGD_STATIC_MAX_NODES);
  size_t status = align256(scale + sizeof(double) * WPSGD_STATIC_MAX_NODES);
  size_t total = align256(status + sizeof(DevStatus));
};
constexpr size_t kStaticBytes = align256(sizeof(float) * (size_t)WPSGD_STATIC_MAX_MODEL_ELEMS) +
                                align256(sizeof(uint32_t) * ((size_t)WPSGD_STATIC_MAX_STEPS + 64 * WPSGD_STATIC_MAX_NODES)) +
                                13 * align256(sizeof(long long) * (WPSGD_STATIC_MAX_NODES + 1));
constexpr int kStaticMaxDevices = 64;
}  // namespace

static __device__ __align__(256) unsigned char g_static_scratch[kStaticBytes];

namespace {
// In host code the name g_static_scratch is only a handle of the symbol, not a device address; the address
// a kernel can use comes from cudaGetSymbolAddress, asked once per device with that device current.
unsigned char* g_static_base[kStaticMaxDevices] = {nullptr};

wpsgd_status static_scratch_base(int device, unsigned char** out) {
  static_assert(sizeof(DevStatus) <= 256, "status word must fit its section");
  if (StaticLayout().total > kStaticBytes) return fail(nullptr, WPSGD_ERR_STATE, "built-in scratch layout exceeds the array");
  if (!g_static_base[device]) {
    void* p = nullptr;
    cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      return fail(nullptr, WPSGD_ERR_CUDA, std::string("cudaGetSymbolAddress(built-in scratch): ") + cudaGetErrorString(e));
    }
    g_static_base[device] = (unsigned char*)p;
  }
  *out = g_static_base[device];
  return WPSGD_OK;
}
}  // namespace

extern "C" {

wpsgd_status wpsgd_create(int device, void* cuda_stream, int32_t k, int64_t d, wpsgd_ctx** out) {
  if (!out) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "out is NULL");
  *out = nullptr;
  if (k < 1 || d < 1) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "k and d must be >= 1");
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) {
    cudaGetLastError();
    return fail(nullptr, WPSGD_ERR_CUDA, "no CUDA device available");
  }
  if (device < 0 || device >= ndev) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "device index out of range");
  DeviceGuard guard(device);
  wpsgd_ctx* c = new wpsgd_ctx();
  c->device = device;
  c->stream = (cudaStream_t)cuda_stream;
  c->k = k;
  c->d = d;
  c->steps_done.assign(k, 0);
  c->node_ids.resize(k);
  std::iota(c->node_ids.begin(), c->node_ids.end(), 0);
  auto bail = [&](cudaError_t e, const char* what) {
    g_err = std::string(what) + ": " + cudaGetErrorString(e);
    const wpsgd_status s = (e == cudaErrorMemoryAllocation) ? WPSGD_ERR_ALLOC : WPSGD_ERR_CUDA;
    cudaGetLastError();
    wpsgd_destroy(c);
    return s;
  };
  cudaError_t e;
#define ALLOC(ptr, bytes)                                         \
  if ((e = cudaMalloc((void**)&(ptr), (bytes))) != cudaSuccess) return bail(e, "cudaMalloc(" #ptr ")");
  ALLOC(c->W, (size_t)k * (size_t)d * sizeof(float));
  ALLOC(c->scale, (size_t)k * sizeof(double));
  ALLOC(c->tables, TableLayout(k).total);
  bind_tables(c, c->tables);
  ALLOC(c->t_weights, (size_t)k * sizeof(double));
  ALLOC(c->status, sizeof(DevStatus));
  ALLOC(c->ticket, sizeof(unsigned));
#undef ALLOC
  if ((e = cudaMemsetAsync(c->status, 0, sizeof(DevStatus), c->stream)) != cudaSuccess) return bail(e, "cudaMemsetAsync");
  if ((e = cudaMemsetAsync(c->ticket, 0, sizeof(unsigned), c->stream)) != cudaSuccess) return bail(e, "cudaMemsetAsync");
  *out = c;
  return WPSGD_OK;
}

wpsgd_status wpsgd_destroy(wpsgd_ctx* c) {
  if (!c) return WPSGD_OK;
  DeviceGuard guard(c->device);
  cudaStreamSynchronize(c->stream);
  void* ptrs[] = {c->W, c->scale, c->tables, c->t_weights, c->idx, c->status, c->part, c->ticket, c->st_X, c->st_y, c->st_v, c->st_w0, c->st_rp, c->st_ci, c->st_va};
  for (void* p : ptrs)
    if (p) cudaFree(p);
  if (c->ev0) cudaEventDestroy(c->ev0);
  if (c->ev1) cudaEventDestroy(c->ev1);
  if (c->ev_fork) cudaEventDestroy(c->ev_fork);
  for (cudaEvent_t e : c->ev_group)
    if (e) cudaEventDestroy(e);
  if (c->copy_stream) cudaStreamDestroy(c->copy_stream);
  cudaGetLastError();
  delete c;
  return WPSGD_OK;
}

wpsgd_status wpsgd_set_option(wpsgd_ctx* c, const char* name, int64_t value) {
  if (!c || !name) return fail(c, WPSGD_ERR_INVALID_ARG, "ctx or name is NULL");
  const std::string n(name);
  if (n == "dense_variant") {
    if (value < 0 || value > 10 || value == 6 || value == 7) return fail(c, WPSGD_ERR_INVALID_ARG, "dense_variant must be 0..5 or 8..10");
    c->opt_variant = (int)value;
  } else if (n == "prefetch") {
    if (value < 0 || value > 64) return fail(c, WPSGD_ERR_INVALID_ARG, "prefetch must be 0..64");
    c->opt_prefetch = (int)value;
  } else if (n == "threads") {
    if (value != 0 && (value < 32 || value > 512 || value % 32)) return fail(c, WPSGD_ERR_INVALID_ARG, "threads must be 0 or a multiple of 32 in 32..512");
    c->opt_threads = (int)value;
  } else if (n == "cluster") {
    if (value != 0 && value != 1 && value != 2 && value != 4 && value != 8) return fail(c, WPSGD_ERR_INVALID_ARG, "cluster must be 0, 1, 2, 4 or 8");
    c->opt_cluster = (int)value;
  } else if (n == "host_pipeline") {
    if (value != 0 && value != 1) return fail(c, WPSGD_ERR_INVALID_ARG, "host_pipeline must be 0 or 1");
    c->opt_host_pipeline = (int)value;
  } else if (n == "block_samples") {
    if (value != 0 && value != 8 && value != 16) return fail(c, WPSGD_ERR_INVALID_ARG, "block_samples must be 0, 8 or 16");
    c->opt_block_samples = (int)value;
  } else if (n == "sparse_variant") {
    if (value < 0 || value > 2) return fail(c, WPSGD_ERR_INVALID_ARG, "sparse_variant must be 0, 1 or 2");
    c->opt_sparse_variant = (int)value;
  } else if (n == "stages") {
    if (value < 0 || value == 1 || value > 8) return fail(c, WPSGD_ERR_INVALID_ARG, "stages must be 0 or 2..8");
    c->opt_stages = (int)value;
  } else if (n == "timing") {
    if (value != 0 && value != 1) return fail(c, WPSGD_ERR_INVALID_ARG, "timing must be 0 or 1");
    c->opt_timing = (int)value;
  } else if (n == "sampling") {
    if (value != 0 && value != 1) return fail(c, WPSGD_ERR_INVALID_ARG, "sampling must be 0 (i.i.d. draws) or 1 (shuffled order)");
    c->opt_sampling = (int)value;
  } else if (n == "test_drop_block") {
    c->opt_drop_block = value;
  } else if (n == "spin_limit") {
    if (value < 1) return fail(c, WPSGD_ERR_INVALID_ARG, "spin_limit must be >= 1");
    c->opt_spin_limit = value;
  } else {
    return fail(c, WPSGD_ERR_INVALID_ARG, "unknown option: " + n);
  }
  return WPSGD_OK;
}

wpsgd_status wpsgd_set_node_ids(wpsgd_ctx* c, const int32_t* ids) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!ids) {
    std::iota(c->node_ids.begin(), c->node_ids.end(), 0);
    return WPSGD_OK;
  }
  for (int j = 0; j < c->k; ++j)
    if (ids[j] < 0) return fail(c, WPSGD_ERR_INVALID_ARG, "node ids must be >= 0");
  c->node_ids.assign(ids, ids + c->k);
  return WPSGD_OK;
}

wpsgd_status wpsgd_run(wpsgd_ctx* c, const void* X, wpsgd_xtype xt, int64_t ld_elems, const float* y,
                       const int64_t* shard_off, const int64_t* n_steps, float eta0, wpsgd_lr sched, float lambda,
                       wpsgd_loss loss, uint64_t seed, const float* w0) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  DeviceGuard guard(c->device);
  wpsgd_status s = check_hyper(c, eta0, (int)sched, lambda, (int)loss);
  if (s != WPSGD_OK) return s;
  c->eta0 = eta0; c->sched = (int)sched; c->lambda = lambda; c->loss = (int)loss; c->seed = seed;
  c->have_run = false;
  return run_dense_common(c, X, xt, ld_elems, y, (const long long*)shard_off, (const long long*)n_steps, w0, false);
}

wpsgd_status wpsgd_continue(wpsgd_ctx* c, const void* X, wpsgd_xtype xt, int64_t ld_elems, const float* y,
                            const int64_t* shard_off, const int64_t* n_more) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!c->have_run) return fail(c, WPSGD_ERR_STATE, "continue before run");
  if (c->scaled) return fail(c, WPSGD_ERR_UNSUPPORTED, "chains started on CSR rows continue with wpsgd_continue_csr");
  DeviceGuard guard(c->device);
  return run_dense_common(c, X, xt, ld_elems, y, (const long long*)shard_off, (const long long*)n_more, nullptr, true);
}

wpsgd_status wpsgd_run_csr(wpsgd_ctx* c, const int64_t* row_ptr, const int32_t* col_idx, const float* val,
                           const float* y, const int64_t* shard_off, const int64_t* n_steps, float eta0,
                           wpsgd_lr sched, float lambda, wpsgd_loss loss, uint64_t seed, const float* w0) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  DeviceGuard guard(c->device);
  wpsgd_status s = check_hyper(c, eta0, (int)sched, lambda, (int)loss);
  if (s != WPSGD_OK) return s;
  c->eta0 = eta0; c->sched = (int)sched; c->lambda = lambda; c->loss = (int)loss; c->seed = seed;
  c->have_run = false;
  return run_csr_common(c, (const long long*)row_ptr, col_idx, val, y, (const long long*)shard_off,
                        (const long long*)n_steps, w0, false);
}

wpsgd_status wpsgd_continue_csr(wpsgd_ctx* c, const int64_t* row_ptr, const int32_t* col_idx, const float* val,
                                const float* y, const int64_t* shard_off, const int64_t* n_more) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!c->have_run) return fail(c, WPSGD_ERR_STATE, "continue before run");
  DeviceGuard guard(c->device);
  return run_csr_common(c, (const long long*)row_ptr, col_idx, val, y, (const long long*)shard_off,
                        (const long long*)n_more, nullptr, true);
}

wpsgd_status wpsgd_get_weights(wpsgd_ctx* c, double r, double* weights, int* cond_holds) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!c->have_run) return fail(c, WPSGD_ERR_STATE, "weights before run");
  std::string why;
  wpsgd_status s = weights_host(c->steps_done.data(), c->k, c->eta0, c->sched, c->lambda, r, weights, cond_holds, nullptr, &why);
  return s == WPSGD_OK ? s : fail(c, s, why);
}

wpsgd_status wpsgd_weights(const int64_t* n_steps, int32_t k, float eta0, wpsgd_lr sched, float lambda, double r,
                           double* weights, int* cond_holds, double* sum_rT) {
  std::string why;
  wpsgd_status s = weights_host((const long long*)n_steps, k, eta0, (int)sched, lambda, r, weights, cond_holds, sum_rT, &why);
  return s == WPSGD_OK ? s : fail(nullptr, s, why);
}

wpsgd_status wpsgd_span_valid(const int64_t* n_steps, int32_t k, float eta0, float lambda, double r, int64_t span,
                              double* lhs, int* holds) {
  if (span < 0) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "span_valid: span must be >= 0");
  if (!((double)eta0 * (double)lambda < 1.0) || !(eta0 >= 0.0f) || !(lambda >= 0.0f))
    return fail(nullptr, WPSGD_ERR_INVALID_ARG, "span_valid: need eta0 >= 0, lambda >= 0, eta0 * lambda < 1");
  if (!n_steps || k < 1) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "span_valid: null argument or k < 1");
  std::string why;
  std::vector<double> lg;
  wpsgd_status s = log_rates((const long long*)n_steps, k, (double)eta0, WPSGD_LR_CONST, (double)lambda, r, &lg, &why);
  if (s != WPSGD_OK) return fail(nullptr, s, why);
  // log of sum_j r^{T_j}, summed from the largest term
  const double mx = *std::max_element(lg.begin(), lg.end());
  double tot = 0.0;
  for (int j = 0; j < k; ++j) tot += std::exp(lg[j] - mx);
  const double log_lhs = std::log((double)k) - (mx + std::log(tot)) + (double)span * std::log1p(-(double)eta0 * (double)lambda);
  const double v = std::exp(log_lhs);
  if (lhs) *lhs = v;
  if (holds) *holds = log_lhs < 0.0 ? 1 : 0;
  return WPSGD_OK;
}

wpsgd_status wpsgd_sample_indices_host(uint64_t seed, int32_t node, int64_t m, int64_t n_begin, int64_t count,
                                       int32_t sampling, uint32_t* out) {
  if (node < 0 || m < 1 || m > 0xFFFFFFFFll || n_begin < 0 || count < 0 || (sampling != 0 && sampling != 1))
    return fail(nullptr, WPSGD_ERR_INVALID_ARG,
                "sample_indices_host: need node >= 0, 1 <= m < 2^32, n_begin >= 0, count >= 0, sampling 0 or 1");
  if (count == 0) return WPSGD_OK;
  if (!out) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "out is NULL");
  emit_indices(sampling, seed, (uint32_t)node, n_begin, count, count, (uint32_t)m, out, 0, 1);  // the kernels' own function
  return WPSGD_OK;
}

wpsgd_status wpsgd_validate_csr(wpsgd_ctx* c, const int64_t* row_ptr, const int32_t* col_idx, int64_t n_rows, int64_t nnz) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (n_rows < 0 || nnz < 0 || !row_ptr || (nnz > 0 && !col_idx)) return fail(c, WPSGD_ERR_INVALID_ARG, "validate_csr: bad argument");
  if (n_rows == 0) return WPSGD_OK;
  DeviceGuard guard(c->device);
  launch(validate_csr_kernel, grid_for(n_rows, 8), 256, 0, c->stream, (const long long*)row_ptr, col_idx, n_rows, nnz, c->d, c->status);
  CU_TRY(c, cudaGetLastError());
  c->launches++;
  return WPSGD_OK;
}

wpsgd_status wpsgd_combine(wpsgd_ctx* c, double r, float* v_out) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!c->have_run) return fail(c, WPSGD_ERR_STATE, "combine before run");
  if (!v_out) return fail(c, WPSGD_ERR_INVALID_ARG, "v_out is NULL");
  DeviceGuard guard(c->device);
  std::vector<double> w(c->k);
  std::string why;
  wpsgd_status s = weights_host(c->steps_done.data(), c->k, c->eta0, c->sched, c->lambda, r, w.data(), nullptr, nullptr, &why);
  if (s != WPSGD_OK) return fail(c, s, why);
  return launch_combine(c, w.data(), v_out);
}

wpsgd_status wpsgd_combine_weighted(wpsgd_ctx* c, const double* weights, float* v_out) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!c->have_run) return fail(c, WPSGD_ERR_STATE, "combine before run");
  if (!v_out || !weights) return fail(c, WPSGD_ERR_INVALID_ARG, "weights or v_out is NULL");
  for (int j = 0; j < c->k; ++j)
    if (!std::isfinite(weights[j])) return fail(c, WPSGD_ERR_INVALID_ARG, "a weight is not finite");
  DeviceGuard guard(c->device);
  return launch_combine(c, weights, v_out);
}

wpsgd_status wpsgd_last_chain_ms(wpsgd_ctx* c, float* ms) {
  if (!c || !ms) return fail(c, WPSGD_ERR_INVALID_ARG, "ctx or ms is NULL");
  if (!c->ev_valid) return fail(c, WPSGD_ERR_STATE, "no timed chain launch (set option \"timing\" to 1 before the run)");
  DeviceGuard guard(c->device);
  CU_TRY(c, cudaEventSynchronize(c->ev1));
  CU_TRY(c, cudaEventElapsedTime(ms, c->ev0, c->ev1));
  return WPSGD_OK;
}

wpsgd_status wpsgd_get_models(wpsgd_ctx* c, float* W_out) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!c->have_run) return fail(c, WPSGD_ERR_STATE, "get_models before run");
  if (!W_out) return fail(c, WPSGD_ERR_INVALID_ARG, "W_out is NULL");
  DeviceGuard guard(c->device);
  const double* scale = c->scaled ? c->scale : nullptr;
  const long long n = (long long)c->k * c->d;
  if (c->d % 4 == 0 && aligned16(c->W) && aligned16(W_out))
    launch(export_models_kernel<4>, grid_for(n / 4, 256), 256, 0, c->stream, c->W, scale, c->k, c->d, W_out);
  else
    launch(export_models_kernel<1>, grid_for(n, 256), 256, 0, c->stream, c->W, scale, c->k, c->d, W_out);
  CU_TRY(c, cudaGetLastError());
  c->launches++;
  return WPSGD_OK;
}

wpsgd_status wpsgd_set_models(wpsgd_ctx* c, const float* v) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!c->have_run) return fail(c, WPSGD_ERR_STATE, "set_models before run");
  if (!v) return fail(c, WPSGD_ERR_INVALID_ARG, "v is NULL");
  DeviceGuard guard(c->device);
  const long long n = (long long)c->k * c->d;
  if (c->d % 4 == 0 && aligned16(c->W) && aligned16(v))
    launch(broadcast_model_kernel<4>, grid_for(n / 4, 256), 256, 0, c->stream, c->W, c->scale, v, c->k, c->d);
  else
    launch(broadcast_model_kernel<1>, grid_for(n, 256), 256, 0, c->stream, c->W, c->scale, v, c->k, c->d);
  CU_TRY(c, cudaGetLastError());
  c->launches++;
  return WPSGD_OK;
}

wpsgd_status wpsgd_sample_indices(wpsgd_ctx* c, uint64_t seed, int32_t node, int64_t m, int64_t n_begin, int64_t count,
                                  uint32_t* out) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (node < 0 || m < 1 || m > 0xFFFFFFFFll || n_begin < 0 || count < 0)
    return fail(c, WPSGD_ERR_INVALID_ARG, "sample_indices: need node >= 0, 1 <= m < 2^32, n_begin >= 0, count >= 0");
  if (count == 0) return WPSGD_OK;
  if (!out) return fail(c, WPSGD_ERR_INVALID_ARG, "out is NULL");
  DeviceGuard guard(c->device);
  launch(index_single_kernel, grid_for(c->opt_sampling ? count : (count + 3) / 4 + 1, 256), 256, 0, c->stream, c->opt_sampling, seed, node, m, n_begin, count, out);
  CU_TRY(c, cudaGetLastError());
  c->launches++;
  return WPSGD_OK;
}

wpsgd_status wpsgd_objective(wpsgd_ctx* c, const void* X, wpsgd_xtype xt, int64_t ld_elems, const float* y,
                             int64_t n_rows, const float* w, float lambda, wpsgd_loss loss, double* out) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!w || !out || n_rows < 0 || ld_elems < c->d || (int)loss < 0 || (int)loss > 2 || (n_rows > 0 && (!X || !y)))
    return fail(c, WPSGD_ERR_INVALID_ARG, "objective: bad argument");
  if (xt != WPSGD_X_F32 && xt != WPSGD_X_BF16) return fail(c, WPSGD_ERR_INVALID_ARG, "unknown feature type");
  DeviceGuard guard(c->device);
  const int nblk = grid_for((n_rows + 7) / 8, 1, 148 * 8);
  wpsgd_status s = grow(c, &c->part, &c->part_cap, (size_t)nblk * 3);
  if (s != WPSGD_OK) return s;
  auto go = [&](auto kern, const auto* rows) {
    launch(kern, nblk, 256, 0, c->stream, rows, ld_elems, y, n_rows, w, c->d, (int)loss, lambda, c->part, c->ticket, out);
  };
  const size_t es = xt == WPSGD_X_F32 ? 4 : 2;
  const bool vec = aligned16(X) && aligned16(w) && ((size_t)ld_elems * es) % 16 == 0 && ((size_t)c->d * es) % 16 == 0;
  const bool narrow = (size_t)c->d * es <= 32 * (vec ? 16 : 2 * es);  // at most one load (two where they are of single elements) per lane
  auto pick = [&](auto vec_tag, auto narrow_tag) {
    if (xt == WPSGD_X_F32) go(objective_rows_kernel<float, vec_tag.value, narrow_tag.value>, (const float*)X);
    else go(objective_rows_kernel<__nv_bfloat16, vec_tag.value, narrow_tag.value>, (const __nv_bfloat16*)X);
  };
  if (vec) narrow ? pick(std::true_type(), std::true_type()) : pick(std::true_type(), std::false_type());
  else narrow ? pick(std::false_type(), std::true_type()) : pick(std::false_type(), std::false_type());
  CU_TRY(c, cudaGetLastError());
  c->launches++;
  return WPSGD_OK;
}

wpsgd_status wpsgd_objective_csr(wpsgd_ctx* c, const int64_t* row_ptr, const int32_t* col_idx, const float* val,
                                 const float* y, int64_t n_rows, const float* w, float lambda, wpsgd_loss loss,
                                 double* out) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!w || !out || n_rows < 0 || (int)loss < 0 || (int)loss > 2 || (n_rows > 0 && (!row_ptr || !col_idx || !val || !y)))
    return fail(c, WPSGD_ERR_INVALID_ARG, "objective_csr: bad argument");
  DeviceGuard guard(c->device);
  const bool few = n_rows <= 148 * 8 * 4;  // half the warps that the GPU holds
  const int nblk = grid_for(few ? (n_rows + 7) / 8 : (n_rows + 31) / 32, 1, 148 * 8);
  wpsgd_status s = grow(c, &c->part, &c->part_cap, (size_t)nblk * 3);
  if (s != WPSGD_OK) return s;
  launch(few ? objective_rows_csr_kernel<32> : objective_rows_csr_kernel<8>, nblk, 256, 0, c->stream, (const long long*)row_ptr, col_idx, val, y, n_rows, w,
         c->d, (int)loss, lambda, c->part, c->ticket, out);
  CU_TRY(c, cudaGetLastError());
  c->launches++;
  return WPSGD_OK;
}

wpsgd_status wpsgd_solve_host(wpsgd_ctx* c, const void* X, wpsgd_xtype xt, const float* y, const int64_t* shard_off,
                              const int64_t* n_steps, float eta0, wpsgd_lr sched, float lambda, wpsgd_loss loss,
                              uint64_t seed, const float* w0, double r, float* v_out) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!shard_off || !v_out) return fail(c, WPSGD_ERR_INVALID_ARG, "shard_off or v_out is NULL");
  if (xt != WPSGD_X_F32 && xt != WPSGD_X_BF16) return fail(c, WPSGD_ERR_INVALID_ARG, "unknown feature type");
  DeviceGuard guard(c->device);
  const long long N = shard_off[c->k];
  if (N < 0) return fail(c, WPSGD_ERR_INVALID_ARG, "shard_off[k] < 0");
  if (N > 0 && (!X || !y)) return fail(c, WPSGD_ERR_INVALID_ARG, "X or y is NULL");
  const size_t es = xt == WPSGD_X_F32 ? 4 : 2;
  const size_t xbytes = (size_t)N * (size_t)c->d * es;
  char* sx = (char*)c->st_X;
  wpsgd_status s = grow(c, &sx, &c->st_X_cap, std::max<size_t>(xbytes, 16));
  c->st_X = sx;
  if (s != WPSGD_OK) return s;
  s = grow(c, &c->st_y, &c->st_y_cap, (size_t)std::max(1ll, N));
  if (s != WPSGD_OK) return s;
  if (!c->st_v) CU_TRY(c, cudaMalloc((void**)&c->st_v, (size_t)c->d * sizeof(float)));
  if (w0 && !c->st_w0) CU_TRY(c, cudaMalloc((void**)&c->st_w0, (size_t)c->d * sizeof(float)));
  // Pipelined form: the shards go to the device longest chain first on a copy stream of the context, in up to four
  // groups of nodes, and the chains of a group start as soon as its rows have arrived, so all but the shortest chains
  // run under the remaining copies. Not for rows of at most 64 chunks (their kernel packs nodes into CTAs over the
  // whole node set) and not with fewer than two nodes.
  const long long chunks = c->d / (long long)(16 / es);
  const bool pipelined = c->opt_host_pipeline && N > 0 && c->k >= 2 && n_steps && chunks > 64;
  if (!pipelined) {
    if (N > 0) {
      CU_TRY(c, cudaMemcpyAsync(c->st_X, X, xbytes, cudaMemcpyHostToDevice, c->stream));
      CU_TRY(c, cudaMemcpyAsync(c->st_y, y, (size_t)N * sizeof(float), cudaMemcpyHostToDevice, c->stream));
    }
    if (w0) CU_TRY(c, cudaMemcpyAsync(c->st_w0, w0, (size_t)c->d * sizeof(float), cudaMemcpyHostToDevice, c->stream));
    s = wpsgd_run(c, c->st_X, xt, c->d, c->st_y, shard_off, n_steps, eta0, sched, lambda, loss, seed, w0 ? c->st_w0 : nullptr);
    if (s != WPSGD_OK) return s;
  } else {
    s = check_hyper(c, eta0, (int)sched, lambda, (int)loss);
    if (s != WPSGD_OK) return s;
    for (int j = 0; j < c->k; ++j)
      if (shard_off[j + 1] < shard_off[j] || shard_off[j] < 0) return fail(c, WPSGD_ERR_INVALID_ARG, "shard_off is not non-decreasing");
    if (!c->copy_stream) {
      CU_TRY(c, cudaStreamCreateWithFlags(&c->copy_stream, cudaStreamNonBlocking));
      CU_TRY(c, cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming));
      for (cudaEvent_t& e : c->ev_group) CU_TRY(c, cudaEventCreateWithFlags(&e, cudaEventDisableTiming));
    }
    // the copies start after whatever the caller's stream still does with the staging buffers
    CU_TRY(c, cudaEventRecord(c->ev_fork, c->stream));
    CU_TRY(c, cudaStreamWaitEvent(c->copy_stream, c->ev_fork, 0));
    CU_TRY(c, cudaMemcpyAsync(c->st_y, y, (size_t)N * sizeof(float), cudaMemcpyHostToDevice, c->copy_stream));
    if (w0) CU_TRY(c, cudaMemcpyAsync(c->st_w0, w0, (size_t)c->d * sizeof(float), cudaMemcpyHostToDevice, c->copy_stream));
    std::vector<int> order(c->k);
    std::iota(order.begin(), order.end(), 0);
    std::stable_sort(order.begin(), order.end(), [&](int a, int b) { return n_steps[a] > n_steps[b]; });  // as make_plan
    const int n_groups = std::min(4, c->k);
    std::vector<LaunchGroup> groups;
    const size_t row_bytes = (size_t)c->d * es;
    int slot = 0;
    for (int g = 0; g < n_groups; ++g) {
      const int count = (c->k - slot + (n_groups - g) - 1) / (n_groups - g);
      for (int q = slot; q < slot + count; ++q) {
        const int j = order[q];
        const size_t off = (size_t)shard_off[j] * row_bytes, len = (size_t)(shard_off[j + 1] - shard_off[j]) * row_bytes;
        if (len > 0)
          CU_TRY(c, cudaMemcpyAsync((char*)c->st_X + off, (const char*)X + off, len, cudaMemcpyHostToDevice, c->copy_stream));
      }
      CU_TRY(c, cudaEventRecord(c->ev_group[g], c->copy_stream));
      groups.push_back({count, c->ev_group[g]});
      slot += count;
    }
    c->eta0 = eta0; c->sched = (int)sched; c->lambda = lambda; c->loss = (int)loss; c->seed = seed;
    c->have_run = false;
    s = run_dense_common(c, c->st_X, xt, c->d, c->st_y, (const long long*)shard_off, (const long long*)n_steps,
                         w0 ? c->st_w0 : nullptr, false, &groups);
    if (s != WPSGD_OK) return s;
  }
  s = wpsgd_combine(c, r, c->st_v);
  if (s != WPSGD_OK) return s;
  CU_TRY(c, cudaMemcpyAsync(v_out, c->st_v, (size_t)c->d * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
  CU_TRY(c, cudaStreamSynchronize(c->stream));
  return WPSGD_OK;
}

wpsgd_status wpsgd_solve_host_csr(wpsgd_ctx* c, const int64_t* row_ptr, const int32_t* col_idx, const float* val, const float* y,
                                  const int64_t* shard_off, const int64_t* n_steps, float eta0, wpsgd_lr sched, float lambda,
                                  wpsgd_loss loss, uint64_t seed, const float* w0, double r, float* v_out) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  if (!shard_off || !v_out) return fail(c, WPSGD_ERR_INVALID_ARG, "shard_off or v_out is NULL");
  DeviceGuard guard(c->device);
  const long long N = shard_off[c->k];
  if (N < 0) return fail(c, WPSGD_ERR_INVALID_ARG, "shard_off[k] < 0");
  if (N > 0 && (!row_ptr || !y)) return fail(c, WPSGD_ERR_INVALID_ARG, "row_ptr or y is NULL");
  const long long nnz = N > 0 ? row_ptr[N] : 0;
  if (nnz < 0 || (nnz > 0 && (!col_idx || !val))) return fail(c, WPSGD_ERR_INVALID_ARG, "row_ptr[N] < 0, or col_idx / val is NULL");
  wpsgd_status s = grow(c, &c->st_rp, &c->st_rp_cap, (size_t)N + 1);
  if (s != WPSGD_OK) return s;
  s = grow(c, &c->st_ci, &c->st_ci_cap, (size_t)std::max(1ll, nnz));
  if (s != WPSGD_OK) return s;
  s = grow(c, &c->st_va, &c->st_va_cap, (size_t)std::max(1ll, nnz));
  if (s != WPSGD_OK) return s;
  s = grow(c, &c->st_y, &c->st_y_cap, (size_t)std::max(1ll, N));
  if (s != WPSGD_OK) return s;
  if (!c->st_v) CU_TRY(c, cudaMalloc((void**)&c->st_v, (size_t)c->d * sizeof(float)));
  if (w0 && !c->st_w0) CU_TRY(c, cudaMalloc((void**)&c->st_w0, (size_t)c->d * sizeof(float)));
  if (N > 0) {
    CU_TRY(c, cudaMemcpyAsync(c->st_rp, row_ptr, ((size_t)N + 1) * sizeof(long long), cudaMemcpyHostToDevice, c->stream));
    CU_TRY(c, cudaMemcpyAsync(c->st_y, y, (size_t)N * sizeof(float), cudaMemcpyHostToDevice, c->stream));
  }
  if (nnz > 0) {
    CU_TRY(c, cudaMemcpyAsync(c->st_ci, col_idx, (size_t)nnz * sizeof(int), cudaMemcpyHostToDevice, c->stream));
    CU_TRY(c, cudaMemcpyAsync(c->st_va, val, (size_t)nnz * sizeof(float), cudaMemcpyHostToDevice, c->stream));
  }
  if (w0) CU_TRY(c, cudaMemcpyAsync(c->st_w0, w0, (size_t)c->d * sizeof(float), cudaMemcpyHostToDevice, c->stream));
  s = wpsgd_run_csr(c, (const int64_t*)c->st_rp, c->st_ci, c->st_va, c->st_y, shard_off, n_steps, eta0, sched, lambda, loss, seed,
                    w0 ? c->st_w0 : nullptr);
  if (s != WPSGD_OK) return s;
  s = wpsgd_combine(c, r, c->st_v);
  if (s != WPSGD_OK) return s;
  CU_TRY(c, cudaMemcpyAsync(v_out, c->st_v, (size_t)c->d * sizeof(float), cudaMemcpyDeviceToHost, c->stream));
  CU_TRY(c, cudaStreamSynchronize(c->stream));
  return WPSGD_OK;
}

wpsgd_status wpsgd_solve_static(int device, void* cuda_stream, const void* X, wpsgd_xtype xt, int64_t ld_elems,
                                const float* y, const int64_t* shard_off, const int64_t* n_steps, int32_t k, int64_t d,
                                float eta0, wpsgd_lr sched, float lambda, wpsgd_loss loss, uint64_t seed,
                                const float* w0, double r, float* v_out) {
  if (k < 1 || d < 1) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "solve_static: k and d must be >= 1");
  if (!shard_off || !n_steps || !v_out) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "solve_static: shard_off, n_steps or v_out is NULL");
  char msg[200];
  if (k > WPSGD_STATIC_MAX_NODES) {
    snprintf(msg, sizeof(msg), "solve_static: k = %d exceeds the built-in maximum of %d nodes", (int)k, WPSGD_STATIC_MAX_NODES);
    return fail(nullptr, WPSGD_ERR_UNSUPPORTED, msg);
  }
  if ((long long)k * (long long)d > WPSGD_STATIC_MAX_MODEL_ELEMS) {
    snprintf(msg, sizeof(msg), "solve_static: k * d = %lld exceeds the built-in maximum of %lld model elements",
             (long long)k * (long long)d, (long long)WPSGD_STATIC_MAX_MODEL_ELEMS);
    return fail(nullptr, WPSGD_ERR_UNSUPPORTED, msg);
  }
  long long total = 0;
  for (int j = 0; j < k; ++j) {
    if (n_steps[j] < 0) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "solve_static: negative step count");
    total += n_steps[j];
    if (total > WPSGD_STATIC_MAX_STEPS) {
      snprintf(msg, sizeof(msg), "solve_static: the step counts add up to more than the built-in maximum of %lld",
               (long long)WPSGD_STATIC_MAX_STEPS);
      return fail(nullptr, WPSGD_ERR_UNSUPPORTED, msg);
    }
  }
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) {
    cudaGetLastError();
    return fail(nullptr, WPSGD_ERR_CUDA, "no CUDA device available");
  }
  if (device < 0 || device >= ndev || device >= kStaticMaxDevices)
    return fail(nullptr, WPSGD_ERR_INVALID_ARG, "solve_static: device index out of range");
  DeviceGuard guard(device);
  unsigned char* base = nullptr;
  wpsgd_status s = static_scratch_base(device, &base);
  if (s != WPSGD_OK) return s;

  // A context on the host stack whose device pointers all lie inside the built-in array. It is never
  // handed to wpsgd_destroy: nothing in it was allocated, so nothing is freed.
  wpsgd_ctx c;
  c.device = device;
  c.stream = (cudaStream_t)cuda_stream;
  c.k = k;
  c.d = d;
  c.steps_done.assign(k, 0);
  c.node_ids.resize(k);
  std::iota(c.node_ids.begin(), c.node_ids.end(), 0);
  const StaticLayout L;
  c.W = (float*)(base + L.W);
  c.idx = (uint32_t*)(base + L.idx);
  c.idx_cap = (size_t)WPSGD_STATIC_MAX_STEPS + 64 * WPSGD_STATIC_MAX_NODES;  // never regrown: padding included
  bind_tables(&c, base + L.tables);
  c.t_weights = (double*)(base + L.weights);
  c.scale = (double*)(base + L.scale);
  c.status = (DevStatus*)(base + L.status);
  // the array keeps what the previous call left: the status word is the one thing that must start at zero
  // (models, tables and the sample stream are fully rewritten for the sizes of this call)
  cudaError_t e = cudaMemsetAsync(c.status, 0, sizeof(DevStatus), c.stream);
  if (e != cudaSuccess) return fail(nullptr, WPSGD_ERR_CUDA, std::string("solve_static: cudaMemsetAsync: ") + cudaGetErrorString(e));
  s = wpsgd_run(&c, X, xt, ld_elems, y, shard_off, n_steps, eta0, sched, lambda, loss, seed, w0);
  if (s == WPSGD_OK) s = wpsgd_combine(&c, r, v_out);
  if (s != WPSGD_OK) g_err = "solve_static: " + c.err;
  return s;
}

wpsgd_status wpsgd_check(wpsgd_ctx* c) {
  if (!c) return fail(nullptr, WPSGD_ERR_INVALID_ARG, "ctx is NULL");
  DeviceGuard guard(c->device);
  return read_status(c, c->status, c->stream);
}

wpsgd_status wpsgd_check_static(int device, void* cuda_stream) {
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || ndev < 1) {
    cudaGetLastError();
    return fail(nullptr, WPSGD_ERR_CUDA, "no CUDA device available");
  }
  if (device < 0 || device >= ndev || device >= kStaticMaxDevices)
    return fail(nullptr, WPSGD_ERR_INVALID_ARG, "check_static: device index out of range");
  DeviceGuard guard(device);
  unsigned char* base = nullptr;
  wpsgd_status s = static_scratch_base(device, &base);
  if (s != WPSGD_OK) return s;
  return read_status(nullptr, (DevStatus*)(base + StaticLayout().status), (cudaStream_t)cuda_stream);
}

int64_t wpsgd_launch_count(const wpsgd_ctx* c) { return c ? c->launches : 0; }

const char* wpsgd_last_error(const wpsgd_ctx* c) { return c ? c->err.c_str() : g_err.c_str(); }

}  // extern "C"
