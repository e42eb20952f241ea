// Aggregation step of Algorithm 1 (v = sum_j weight_j w_j with the weights of Eq. 6 / Eq. 8), model
// export, model broadcast, and the evaluation measures of the paper's experiments.
#pragma once

#include "common.cuh"

namespace wpsgd {

// v[c] = sum_j (weight_j * scale_j) * W[j][c] in fp64. scale may be null. Bound by the read of W. A block owns 32 VEC
// columns and its warps split the nodes (every fourth, eighth, .. one each, j ascending), so that few columns with many
// nodes still fill the machine; the warps' sums are added in warp order, so the result does not depend on timing. The host
// launches up to 32 warps, four nodes or more each, and takes VEC = 4 when the column count fills the SMs with it.
// k = 1024, d = 256: 226 us with one thread per column over all nodes, 7 us this way.
// N > 0: the weights are the argument `iw` (no copy is enqueued for them), else they lie at `far_weights`.
template <int N>
struct InlineWeights {
  double w[N];
};
constexpr int COMBINE_INLINE = 256;
template <int VEC, int N>
__global__ void __launch_bounds__(1024) combine_kernel(const __grid_constant__ InlineWeights<(N > 0 ? N : 1)> iw,
                                                       const float* __restrict__ W, const double* __restrict__ far_weights,
                                                       const double* __restrict__ scale, int k, long long d, float* __restrict__ v) {
  extern __shared__ __align__(16) double sums[];  // [warp][32 VEC]
  const double* weights = N > 0 ? iw.w : far_weights;
  kernel_started();
  kernel_inputs_ready();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, warps = blockDim.x >> 5;
  const long long c = ((long long)blockIdx.x * 32 + lane) * VEC;
  double a[VEC];
#pragma unroll
  for (int e = 0; e < VEC; ++e) a[e] = 0.0;
  if (c < d) {
#pragma unroll 4
    for (int j = warp; j < k; j += warps) {
      float f[VEC];
      const float* src = W + (size_t)j * d + c;
      if constexpr (VEC == 4) {
        const float4 q = __ldg((const float4*)src);
        f[0] = q.x; f[1] = q.y; f[2] = q.z; f[3] = q.w;
      } else {
        f[0] = __ldg(src);
      }
      const double wj = weights[j] * (scale ? scale[j] : 1.0);
#pragma unroll
      for (int e = 0; e < VEC; ++e) a[e] = fma(wj, (double)f[e], a[e]);
    }
  }
#pragma unroll
  for (int e = 0; e < VEC; ++e) sums[(warp * VEC + e) * 32 + lane] = a[e];
  __syncthreads();
  for (int e = warp; e < VEC; e += warps) {
    double t = 0.0;
    for (int w = 0; w < warps; ++w) t += sums[(w * VEC + e) * 32 + lane];
    if (c < d) v[c + e] = (float)t;
  }
}

// W_out[j][c] = scale_j * W[j][c], VEC columns at a time (VEC = 4: d a multiple of 4 and both matrices 16-byte aligned)
template <int VEC>
__global__ void export_models_kernel(const float* __restrict__ W, const double* __restrict__ scale, int k, long long d,
                                     float* __restrict__ out) {
  kernel_started();
  kernel_inputs_ready();
  const long long per_row = d / VEC, total = (long long)k * per_row;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const double s = scale ? scale[row_of(i, per_row)] : 1.0;
    if constexpr (VEC == 4) {
      float4 q = ((const float4*)W)[i];
      if (scale) q = make_float4((float)(s * (double)q.x), (float)(s * (double)q.y), (float)(s * (double)q.z), (float)(s * (double)q.w));
      ((float4*)out)[i] = q;
    } else {
      out[i] = scale ? (float)(s * (double)W[i]) : W[i];
    }
  }
}

// W[j][:] = v for every node; scale_j = 1
template <int VEC>
__global__ void broadcast_model_kernel(float* __restrict__ W, double* __restrict__ scale, const float* __restrict__ v,
                                       int k, long long d) {
  kernel_started();
  kernel_inputs_ready();
  const long long per_row = d / VEC, total = (long long)k * per_row;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < total; i += (long long)gridDim.x * blockDim.x) {
    const long long c = i - row_of(i, per_row) * per_row;
    if constexpr (VEC == 4) ((float4*)W)[i] = ((const float4*)v)[c];
    else W[i] = v[c];
  }
  if (blockIdx.x == 0)
    for (int j = threadIdx.x; j < k; j += blockDim.x) scale[j] = 1.0;
}

// ---- objective of Eq. 3-4 and 0/1 error ----------------------------------------------------------------------------------
__device__ __forceinline__ double loss_value(int loss, float yy, float z) {
  if (loss == LOSS_HINGE) return fmax(0.0, 1.0 - (double)yy * (double)z);
  if (loss == LOSS_LOGISTIC) {
    const double t = (double)yy * (double)z;
    return t > 0 ? log1p(exp(-t)) : -t + log1p(exp(t));
  }
  return 0.5 * ((double)z - (double)yy) * ((double)z - (double)yy);
}
__device__ __forceinline__ double warp_sum_f64(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// The end of both objective kernels: sums of the block (loss, error count, its share of |w|^2) go to part[3 blockIdx.x ..];
// the block that finishes last adds all of them up in block order and writes out (so the result does not depend on which
// block that is) and resets the ticket for the next launch.
__device__ __forceinline__ void objective_finish(double lsum, double esum, const float* __restrict__ w, long long d, float lambda,
                                                 long long n_rows, double* __restrict__ part, unsigned* ticket, double* __restrict__ out) {
  __shared__ double sh[3][8];
  __shared__ bool last;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double r = 0.0;
  for (long long c = (long long)blockIdx.x * 256 + threadIdx.x; c < d; c += (long long)gridDim.x * 256) r += (double)w[c] * (double)w[c];
  auto block_sums = [&](double a, double b, double c) {  // to sh[.][0], for thread 0
    a = warp_sum_f64(a); b = warp_sum_f64(b); c = warp_sum_f64(c);
    if (lane == 0) { sh[0][warp] = a; sh[1][warp] = b; sh[2][warp] = c; }
    __syncthreads();
    if (threadIdx.x < 3) {
      double t = 0.0;
      for (int i = 0; i < 8; ++i) t += sh[threadIdx.x][i];
      sh[threadIdx.x][0] = t;
    }
    __syncthreads();
  };
  block_sums(lsum, esum, r);
  if (threadIdx.x == 0) {
    for (int q = 0; q < 3; ++q) __stcg(&part[3 * blockIdx.x + q], sh[q][0]);
    __threadfence();
    last = atomicAdd(ticket, 1u) == gridDim.x - 1;
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  double a = 0.0, b = 0.0, c = 0.0;
  for (unsigned i = threadIdx.x; i < gridDim.x; i += 256) {
    a += __ldcg(&part[3 * i]);
    b += __ldcg(&part[3 * i + 1]);
    c += __ldcg(&part[3 * i + 2]);
  }
  block_sums(a, b, c);
  if (threadIdx.x == 0) {
    const double n = n_rows > 0 ? (double)n_rows : 1.0;
    out[0] = 0.5 * (double)lambda * sh[2][0] + sh[0][0] / n;
    out[1] = sh[1][0] / n;
    *ticket = 0u;
  }
}

// Dense rows, one warp per row. Bound by the read of X: 16 bytes per lane and load, four loads in flight per lane (VEC; rows
// that are not 16-byte aligned go element by element, four or eight in flight), the model from L1. The end of such a row is a matter of predicates,
// not of a loop of its own, in which each load would be waited for; rows of at most 32 chunks (64 elements), NARROW, go four at a time. A
// warp keeps the margins of up to 32 of its rows, one per lane, and then evaluates their fp64 losses side by side. 262144 rows of
// 1024 fp32 columns: 231 us with single 4-byte loads, a loss evaluation per row on all lanes and a second launch for the sums;
// 177 us this way (6.1 TB/s). 300000 fp32 rows of 166 columns: 179 us with a loop for the row's
// end, 98 without; 300000 bf16 rows of 8 columns: 63 us one at a time, 42 four at a time. Four or five blocks per SM: with six (40
// registers) the rows that do not start on 16 bytes lose the cache lines that neighbouring loads share (30000 rows of 4673 fp32
// columns: 181 us against 111).
template <typename XT, bool VEC, bool NARROW>
__global__ void __launch_bounds__(256, sizeof(XT) == 2 ? 5 : 4) objective_rows_kernel(const XT* __restrict__ X, long long ld, const float* __restrict__ y,
                                                             long long n_rows, const float* __restrict__ w, long long d,
                                                             int loss, float lambda, double* __restrict__ part, unsigned* ticket,
                                                             double* __restrict__ out) {
  kernel_started();
  kernel_inputs_ready();
  constexpr int V = XVec<XT>::V;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double lsum = 0.0, esum = 0.0;
  float z_own = 0.0f, y_own = 0.0f;
  int held = 0;
  auto evaluate = [&]() {
    if (lane < held) {
      lsum += loss_value(loss, y_own, z_own);
      esum += ((z_own >= 0.0f) != (y_own >= 0.0f)) ? 1.0 : 0.0;
    }
    held = 0;
  };
  auto hold = [&](float z, float yy) {
    if (lane == held) { z_own = z; y_own = yy; }
    if (++held == 32) evaluate();
  };
  auto add = [&](const uint4& raw, long long c, float& acc) {
    float x[V];
    XVec<XT>::widen(raw, x);
#pragma unroll
    for (int e = 0; e < V; e += 4) {
      const float4 q = __ldg((const float4*)(w + c * V + e));
      acc = fmaf(q.x, x[e], acc); acc = fmaf(q.y, x[e + 1], acc); acc = fmaf(q.z, x[e + 2], acc); acc = fmaf(q.w, x[e + 3], acc);
    }
  };
  const long long warps = (long long)gridDim.x * 8, units = VEC ? d / V : d;
  long long i = (long long)blockIdx.x * 8 + warp;
  if constexpr (NARROW) {
    constexpr int R = 4, U = VEC ? 1 : 2;
    for (; i < n_rows; i += R * warps) {
      float yy[R], acc[R];
      uint4 raw[R];
      float x[R][U];
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const bool in = i + r * warps < n_rows;
        const XT* row = X + (size_t)(in ? i + r * warps : i) * ld;
        yy[r] = y[in ? i + r * warps : i];
        if constexpr (VEC) {
          raw[r] = ld_stream16_if(row + lane * V, lane < units);
        } else {
#pragma unroll
          for (int u = 0; u < U; ++u) x[r][u] = lane + 32 * u < units ? widen_scalar<XT>(row[lane + 32 * u]) : 0.0f;
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) {
        acc[r] = 0.0f;
        if constexpr (VEC) {
          if (lane < units) add(raw[r], lane, acc[r]);
        } else {
#pragma unroll
          for (int u = 0; u < U; ++u)
            if (lane + 32 * u < units) acc[r] = fmaf(w[lane + 32 * u], x[r][u], acc[r]);
        }
      }
#pragma unroll
      for (int r = 0; r < R; ++r) acc[r] = warp_sum(acc[r]);
#pragma unroll
      for (int r = 0; r < R; ++r)
        if (i + r * warps < n_rows) hold(acc[r], yy[r]);
    }
  } else {
    for (; i < n_rows; i += warps) {
      const XT* row = X + (size_t)i * ld;
      const float yy = y[i];
      float acc = 0.0f;
      long long c = lane;
      if constexpr (VEC) {
        for (; c + 96 < units; c += 128) {
          uint4 raw[4];
#pragma unroll
          for (int u = 0; u < 4; ++u) raw[u] = ld_stream16(row + (c + 32 * u) * V);
#pragma unroll
          for (int u = 0; u < 4; ++u) add(raw[u], c + 32 * u, acc);
        }
        for (; c < units; c += 32) add(ld_stream16(row + c * V), c, acc);
      } else {
        float x[4], q[4];
#pragma unroll 2
        for (; c + 96 < units; c += 128) {
#pragma unroll
          for (int u = 0; u < 4; ++u) { x[u] = widen_scalar<XT>(row[c + 32 * u]); q[u] = w[c + 32 * u]; }
#pragma unroll
          for (int u = 0; u < 4; ++u) acc = fmaf(q[u], x[u], acc);
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          x[u] = c + 32 * u < units ? widen_scalar<XT>(row[c + 32 * u]) : 0.0f;
          q[u] = c + 32 * u < units ? w[c + 32 * u] : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) acc = fmaf(q[u], x[u], acc);
      }
      hold(warp_sum(acc), yy);
    }
  }
  evaluate();
  objective_finish(lsum, esum, w, d, lambda, n_rows, part, ticket, out);
}

// Lane l of L: its share of w . x over the nonzeros b .. e - 1 of a row
template <int L>
__device__ __forceinline__ float csr_margin_part(const int* __restrict__ col_idx, const float* __restrict__ val, const float* __restrict__ w,
                                                 long long b, long long e, int l) {
  float acc = 0.0f;
  if constexpr (L == 8) {  // (short rows: predicated batches as below cost them 3 to 6 %)
#pragma unroll 4
    for (long long q = b + l; q < e; q += 8) acc = fmaf(w[col_idx[q]], val[q], acc);
  } else {
    for (long long q = b + l; q - l < e; q += 4 * L) {
      int c[4];
      float v[4];
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        c[u] = q + L * u < e ? col_idx[q + L * u] : 0;
        v[u] = q + L * u < e ? val[q + L * u] : 0.0f;
      }
#pragma unroll
      for (int u = 0; u < 4; ++u)
        if (q + L * u < e) acc = fmaf(w[c[u]], v[u], acc);
    }
  }
  return acc;
}

// CSR rows. LANES = 8: four rows per warp (rows of a few tens of nonzeros), except that a warp with a row of more than 512 takes
// its rows in turn with all lanes. LANES = 32: for so few rows that every warp has one at most, whatever their length (the host
// decides by the row count: 100 rows of 10000 nonzeros take 62 us with all lanes of a warp, 206 with eight; 9000 rows of 30 take
// 22.1 and 20.7).
template <int LANES>
__global__ void __launch_bounds__(256) objective_rows_csr_kernel(const long long* __restrict__ row_ptr, const int* __restrict__ col_idx,
                                                                 const float* __restrict__ val, const float* __restrict__ y,
                                                                 long long n_rows, const float* __restrict__ w, long long d,
                                                                 int loss, float lambda, double* __restrict__ part, unsigned* ticket,
                                                                 double* __restrict__ out) {
  kernel_started();
  kernel_inputs_ready();
  constexpr int ROWS = 256 / LANES;  // of a block
  const int lane = threadIdx.x & 31, sub = threadIdx.x & (LANES - 1);
  double lsum = 0.0, esum = 0.0;
  // the same trip count for all rows of a warp (shuffles)
  for (long long i0 = (long long)blockIdx.x * ROWS; i0 < n_rows; i0 += (long long)gridDim.x * ROWS) {
    const long long i = i0 + threadIdx.x / LANES;
    const bool in = i < n_rows;
    const long long b = in ? row_ptr[i] : 0, e = in ? row_ptr[i + 1] : 0;
    float acc = 0.0f;
    if (LANES < 32 && __any_sync(0xffffffffu, e - b > 512)) {
#pragma unroll 1
      for (int r = 0; r < 32 / LANES; ++r) {
        const long long rb = __shfl_sync(0xffffffffu, b, r * LANES), re = __shfl_sync(0xffffffffu, e, r * LANES);
        const float z = warp_sum(csr_margin_part<32>(col_idx, val, w, rb, re, lane));
        if (lane / LANES == r) acc = z;
      }
    } else {
      acc = csr_margin_part<LANES>(col_idx, val, w, b, e, sub);
#pragma unroll
      for (int o = LANES / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
    }
    if (in && sub == 0) {
      const float yy = y[i];
      lsum += loss_value(loss, yy, acc);
      esum += ((acc >= 0.0f) != (yy >= 0.0f)) ? 1.0 : 0.0;
    }
  }
  objective_finish(lsum, esum, w, d, lambda, n_rows, part, ticket, out);
}

// Read-only check of a CSR matrix before it is handed to the chains: row_ptr within [0, nnz] and non-decreasing,
// every column in [0, d), columns strictly increasing within a row (so no column occurs twice: the sparse update
// writes every nonzero's model entry once). The first problem found goes to the status word (where = 31 row extents,
// 32 column range, 33 column order; detail = the row). Nothing is read outside [0, nnz).
__global__ void validate_csr_kernel(const long long* __restrict__ row_ptr, const int* __restrict__ col_idx, long long n_rows,
                                    long long nnz, long long d, DevStatus* status) {
  kernel_started();
  kernel_inputs_ready();
  const int lane = threadIdx.x & 31;
  const long long warp0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nwarps = ((long long)gridDim.x * blockDim.x) >> 5;
  for (long long i = warp0; i < n_rows; i += nwarps) {
    const long long b = row_ptr[i], e = row_ptr[i + 1];
    if (b < 0 || e < b || e > nnz) {
      if (lane == 0) set_status(status, DEV_BOUNDS, 31, i);
      continue;
    }
    for (long long q = b + lane; q < e; q += 32) {
      const long long c = col_idx[q];
      if (c < 0 || c >= d) set_status(status, DEV_BOUNDS, 32, i);
      else if (q > b && (long long)col_idx[q - 1] >= c) set_status(status, DEV_BOUNDS, 33, i);
    }
  }
}

}  // namespace wpsgd
