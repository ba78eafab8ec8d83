// Learned Newton warm start: a per-node MLP 28 -> 256 -> 256 -> 256 -> 12 with GELU, BF16 weights
// and activations, FP32 accumulation on the tensor cores (tcgen05.mma kind::f16 with TMEM
// accumulators, operands staged by TMA; tc_gemm.cuh, gemm_split.cuh), trained with an MSE loss and Adam by the
// kernels of this file. The paper has no learning component; the implicit-Euler Newton solve of
// Sec. 6.1 stays the judge of every step.
//
// One kernel (k_mlp_rows) takes 128 rows through all layers without leaving the SM, for the warm start, for
// inference and, with the loss and the back-propagation, for training; a second one (k_gemm_split) forms
// every weight gradient.
//
// Node features (28, FP32): the node's 12 DOFs relative to rest (u = q - q_rest), its 12 velocity
// DOFs, and 4 means over its present edge neighbours: of u_nb - u_i for the position DOFs (a
// discrete Laplacian of the displacement, 3 values), and of the neighbours' position speed |v_nb|
// (their previous step's |dq| over dt, 1 value).
// Output (12): the node's update beyond the inertial predictor, q^{n+1} - q^n - dt v^n.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <string>
#include <vector>

#include "common.cuh"
#include "gemm_split.cuh"

namespace bhem {
namespace mlp {

constexpr int kIn = 28, kInPad = 32, kHid = 256, kOut = 12, kOutPad = 16, kLayers = 4;
constexpr int kDin[kLayers] = {kInPad, kHid, kHid, kHid};   // padded fan-in
constexpr int kDout[kLayers] = {kHid, kHid, kHid, kOutPad};  // padded fan-out
constexpr int kRin[kLayers] = {kIn, kHid, kHid, kHid};       // fan-in
constexpr int kRout[kLayers] = {kHid, kHid, kHid, kOut};     // fan-out
// normalisation vector: in_mean[28] in_istd[28] out_mean[12] out_std[12] out_istd[12]
constexpr int kNormInMean = 0, kNormInIstd = 28, kNormOutMean = 56, kNormOutStd = 68, kNormOutIstd = 80;
constexpr int kNormSize = 96;

using bf16 = __nv_bfloat16;

constexpr int kErrIndex = 1, kErrTimeout = 2;   // bits of the network's error word

// ------------------------------------------------------------------------------------------
// Element-wise kernels
// ------------------------------------------------------------------------------------------
// Adam (Kingma and Ba) on the FP32 master parameters of every tensor of the network in one launch,
// refreshing a tensor's BF16 copy and its transpose (a [rows x cols] matrix stored [cols][rows])
// where given. Padded entries see zero gradients and stay zero.
constexpr int kAdamTensors = 2 * kLayers;
struct AdamSet {
  float* w[kAdamTensors];
  const float* g[kAdamTensors];
  float* m[kAdamTensors];
  float* v[kAdamTensors];
  bf16* wb[kAdamTensors];
  bf16* wbT[kAdamTensors];
  int rows[kAdamTensors], cols[kAdamTensors];
  long long end[kAdamTensors];   // cumulative element counts
};

__global__ void k_adam(AdamSet S, float lr, float b1, float b2, float eps, float c1, float c2) {
  const long long total = S.end[kAdamTensors - 1];
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < total;
       e += (long long)gridDim.x * blockDim.x) {
    int t = 0;
    while (e >= S.end[t]) ++t;
    const long long i = e - (t ? S.end[t - 1] : 0);
    const float gr = S.g[t][i];
    const float mm = b1 * S.m[t][i] + (1.f - b1) * gr;
    const float vv = b2 * S.v[t][i] + (1.f - b2) * gr * gr;
    S.m[t][i] = mm;
    S.v[t][i] = vv;
    const float wn = S.w[t][i] - lr * (mm / c1) / (sqrtf(vv / c2) + eps);
    S.w[t][i] = wn;
    if (S.wb[t]) S.wb[t][i] = __float2bfloat16(wn);
    if (S.wbT[t]) S.wbT[t][(i % S.cols[t]) * S.rows[t] + i / S.cols[t]] = __float2bfloat16(wn);
  }
}

// BF16 copy of a [rows x cols] FP32 matrix, and its transpose [cols][rows] when bT is given
__global__ void k_to_bf16(int rows, int cols, const float* __restrict__ a, bf16* __restrict__ b,
                          bf16* __restrict__ bT) {
  const long long count = (long long)rows * cols;
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < count;
       e += (long long)gridDim.x * blockDim.x) {
    const bf16 h = __float2bfloat16(a[e]);
    b[e] = h;
    if (bT) bT[(e % cols) * rows + e / cols] = h;
  }
}

// per-column sum and sum of squares (FP64) of a [rows x cols] FP32 matrix; one CTA per column
__global__ void k_colstats(long long rows, int cols, const float* __restrict__ X, double* __restrict__ acc) {
  const int c = blockIdx.x;
  __shared__ double s1[256], s2[256];
  double a = 0.0, b = 0.0;
  for (long long r = threadIdx.x; r < rows; r += blockDim.x) {
    const double x = X[r * cols + c];
    a += x;
    b += x * x;
  }
  s1[threadIdx.x] = a;
  s2[threadIdx.x] = b;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (threadIdx.x < o) {
      s1[threadIdx.x] += s1[threadIdx.x + o];
      s2[threadIdx.x] += s2[threadIdx.x + o];
    }
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    acc[2 * c] = s1[0];
    acc[2 * c + 1] = s2[0];
  }
}

// ------------------------------------------------------------------------------------------
// Shell-side kernels: node features, training targets, warm start
// ------------------------------------------------------------------------------------------
// the 28 features of node i (shared by the feature kernel and the fused warm start)
__device__ __forceinline__ void node_features_of(int i, int n1, int n2, int per_u, int per_v,
                                                 const double* __restrict__ q, const double* __restrict__ rest,
                                                 const double* __restrict__ v, float* out) {
  double ui[3];
  for (int k = 0; k < 12; ++k) {
    const double u = q[(size_t)i * 12 + k] - rest[(size_t)i * 12 + k];
    if (k < 3) ui[k] = u;
    out[k] = (float)u;
    out[12 + k] = (float)v[(size_t)i * 12 + k];
  }
  const int ii = i % n1, jj = i / n1;
  const int di[4] = {-1, 1, 0, 0}, dj[4] = {0, 0, -1, 1};
  double lap[3] = {0.0, 0.0, 0.0}, speed = 0.0;
  int cnt = 0;
  for (int e = 0; e < 4; ++e) {
    int a = ii + di[e], b = jj + dj[e];
    if (per_u) a = (a + n1) % n1;
    if (per_v) b = (b + n2) % n2;
    if (a < 0 || a >= n1 || b < 0 || b >= n2 || (a == ii && b == jj)) continue;
    const size_t o = ((size_t)b * n1 + a) * 12;
    for (int c = 0; c < 3; ++c) lap[c] += (q[o + c] - rest[o + c]) - ui[c];
    speed += sqrt(v[o] * v[o] + v[o + 1] * v[o + 1] + v[o + 2] * v[o + 2]);
    ++cnt;
  }
  for (int c = 0; c < 3; ++c) out[24 + c] = cnt ? (float)(lap[c] / cnt) : 0.f;
  out[27] = cnt ? (float)(speed / cnt) : 0.f;
}

__global__ void k_node_features(int n1, int n2, int per_u, int per_v, const double* __restrict__ q,
                                const double* __restrict__ rest, const double* __restrict__ v,
                                float* __restrict__ X) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n1 * n2) return;
  node_features_of(i, n1, n2, per_u, per_v, q, rest, v, X + (size_t)i * kIn);
}

__global__ void k_targets(long long n_dof, const double* __restrict__ q_next, const double* __restrict__ q,
                          const double* __restrict__ v, double dt, float* __restrict__ T) {
  for (long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x; e < n_dof;
       e += (long long)gridDim.x * blockDim.x)
    T[e] = (float)(q_next[e] - q[e] - dt * v[e]);
}

// warm = q + dt v, the inertial predictor alone
__global__ void k_predict(int n_dof, const double* __restrict__ q, const double* __restrict__ v, double dt,
                          double* __restrict__ warm) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < n_dof; e += gridDim.x * blockDim.x) warm[e] = q[e] + dt * v[e];
}

// ------------------------------------------------------------------------------------------
// The rows kernel: 128 rows (one per TMEM lane) through the network in one CTA. The activations stay in
// shared memory as the next product's A operand (128-byte swizzled K-major tiles, written by the
// epilogue); each product's weights arrive by TMA into one shared buffer as soon as the previous product's
// MMAs are done, and one thread issues the tcgen05.mma into a 128 x 256 FP32 TMEM accumulator.
//   kWarm:  node features -> network -> q + dt v + output
//   kInfer: rows of X -> de-normalised output
//   kTrain: rows of X (through an index) -> loss, then back through the layers: dZ of every layer, transposed,
//           and the transposed activations (the operands of the weight-gradient GEMMs), and the bias
//           gradients (column sums of the FP32 dZ).
// What bounds it: the epilogues, 64 accumulators a thread and product with an erff each (4 us a hidden layer
// against 0.5 us of MMAs). So GELU' is formed beside GELU from the same erff, in the forward epilogue,
// and waits in global memory (FP32, written and read by the same thread, 512 B per warp access) for the
// back-propagation; its loads are issued before the wait for the product. One launch per product, with FP32
// copies of every Z and dZ and a column-sum launch per layer, took 230 us for the gradients of 16,384
// rows; this and k_gemm_split take 77 us.
// ------------------------------------------------------------------------------------------
enum RowsMode { kWarm, kInfer, kTrain };
constexpr int kRowThreads = 512;                  // 16 warps: TMEM lane quarter w % 4, column part w / 4
constexpr int kActBytes = 4 * tc::kBM * 128;      // 4 K chunks of 128 rows x 128 bytes
constexpr int kWgtBytes = 4 * kHid * 128;         // 4 K chunks of 256 rows x 128 bytes
constexpr size_t kRowsSmem = (size_t)kActBytes + kWgtBytes + 1024;
constexpr int kPhases = 2 * kLayers - 1;          // products of a training pass: 4 forward, 3 back

// W[l] as [fan_out][fan_in] (forward) and its transpose (back, l >= 1), in boxes of 64 columns x all rows
struct RowsMaps {
  CUtensorMap w[kLayers], wt[kLayers];
};

struct RowsArgs {
  int rows;
  // kWarm
  int n1, n2, per_u, per_v;
  const double *q, *rest, *v;
  double dt;
  double* warm;
  // kInfer, kTrain
  const float* X;
  float* Y;
  // kTrain
  const float* T;
  long long data_rows;
  const int* idx;
  double* loss;
  long long ldt;
  bf16 *XbT, *AbT[kLayers - 1], *dZbT[kLayers];
  float4* G[kLayers - 1];   // GELU'(Z): [tile of 128 rows][64 groups of 4 columns][128 rows]
  float* gb[kLayers];
  const float* bias[kLayers];
  const float* norm;
  int* err;
  unsigned polls;
};

__device__ __forceinline__ uint4 pack_bf16x8(const float* x) {
  unsigned w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j)
    w[j] = (unsigned)__bfloat16_as_ushort(__float2bfloat16(x[2 * j])) |
           ((unsigned)__bfloat16_as_ushort(__float2bfloat16(x[2 * j + 1])) << 16);
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// 16 activations of a row (columns c0 .. c0 + 15) into the A tiles
__device__ __forceinline__ void store_act16(unsigned char* act, int row, int c0, const float* a) {
  unsigned char* rp = act + (c0 / tc::kBK) * (tc::kBM * 128) + row * 128;
  const int p = (c0 % tc::kBK) / 8;
  *reinterpret_cast<uint4*>(rp + ((p ^ (row & 7)) * 16)) = pack_bf16x8(a);
  *reinterpret_cast<uint4*>(rp + (((p + 1) ^ (row & 7)) * 16)) = pack_bf16x8(a + 8);
}

// sum over the warp's 32 rows of column lane / 2 of t[16] (each exchange halves the columns a lane keeps)
__device__ __forceinline__ float column_sum16(const float (&v)[16], int lane) {
  float t[16];
#pragma unroll
  for (int j = 0; j < 16; ++j) t[j] = v[j];
#pragma unroll
  for (int o = 16, n = 8; n > 0; o >>= 1, n >>= 1) {
    const bool hi = lane & o;
#pragma unroll
    for (int j = 0; j < n; ++j) {
      const float send = hi ? t[j] : t[j + n], keep = hi ? t[j + n] : t[j];
      t[j] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return t[0] + __shfl_xor_sync(0xffffffffu, t[0], 1);
}

template <RowsMode MODE>
__global__ void __launch_bounds__(kRowThreads, 1)
k_mlp_rows(const __grid_constant__ RowsMaps maps, const __grid_constant__ RowsArgs A) {
  extern __shared__ unsigned char rows_smem_raw[];
  __shared__ __align__(8) uint64_t bar_w, bar_mma;
  __shared__ uint32_t tmem_slot;
  __shared__ int s_abort;
  __shared__ __align__(16) float s_bias[kLayers][kHid];
  __shared__ float s_sum[MODE == kTrain ? 4 : 1][kHid];   // column sums per TMEM lane quarter
  volatile int* abort_flag = &s_abort;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t raw = tc::smem_addr(rows_smem_raw);
  const uint32_t act = (raw + 1023u) & ~1023u, wgt = act + kActBytes;
  unsigned char* act_g = rows_smem_raw + (act - raw);   // generic pointer to the activation tiles
  const uint32_t bw = tc::smem_addr(&bar_w), bm = tc::smem_addr(&bar_mma);
  const int r0 = blockIdx.x * tc::kBM;
  if (tid == 0) {
    tc::mbar_init(bw, 1);
    tc::mbar_init(bm, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    s_abort = 0;
  }
  if (warp == 0) tc::tmem_alloc<kHid>(tc::smem_addr(&tmem_slot));
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const uint32_t tmem = tmem_slot;
  if (tid == 0) {   // layer-0 weights (K = 32: one 64-column chunk, the rest read as zeros)
    tc::mbar_arrive_expect_tx(bw, kHid * 128);
    tc::tma_load_2d(wgt, &maps.w[0], bw, 0, 0);
  }
  for (int e = tid; e < kLayers * kHid; e += kRowThreads)
    s_bias[e / kHid][e % kHid] = e % kHid < (e / kHid < kLayers - 1 ? kHid : kOutPad) ? A.bias[e / kHid][e % kHid] : 0.f;
  // layer-0 input rows: K chunk 0, columns 32..63 zero
  if (MODE == kWarm) {
    if (tid < tc::kBM) {
      const int i = r0 + tid;
      float f[kIn];
      if (i < A.rows) node_features_of(i, A.n1, A.n2, A.per_u, A.per_v, A.q, A.rest, A.v, f);
      float x[kInPad];
#pragma unroll
      for (int c = 0; c < kInPad; ++c)
        x[c] = (i < A.rows && c < kIn) ? (f[c] - A.norm[kNormInMean + c]) * A.norm[kNormInIstd + c] : 0.f;
      uint4* row = reinterpret_cast<uint4*>(act_g + tid * 128);
#pragma unroll
      for (int p = 0; p < 8; ++p) row[p ^ (tid & 7)] = p < 4 ? pack_bf16x8(x + 8 * p) : make_uint4(0u, 0u, 0u, 0u);
    }
  } else {
    // four threads per row, 8 columns each; an index outside [0, data_rows) gives a zero row and raises the
    // error flag
    const int lr = tid & 127, part = tid >> 7, i = r0 + lr;
    float x[8];
    long long src = -1;
    if (i < A.rows) {
      src = MODE == kTrain && A.idx ? (long long)A.idx[i] : i;
      if (MODE == kTrain && (src < 0 || src >= A.data_rows)) {
        src = -1;
        if (part == 0) atomicOr(A.err, kErrIndex);
      }
    }
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int c = 8 * part + j;
      x[j] = 0.f;
      if (src >= 0 && c < kIn) x[j] = (A.X[src * kIn + c] - A.norm[kNormInMean + c]) * A.norm[kNormInIstd + c];
    }
    uint4* row = reinterpret_cast<uint4*>(act_g + lr * 128);
    row[part ^ (lr & 7)] = pack_bf16x8(x);
    row[(4 + part) ^ (lr & 7)] = make_uint4(0u, 0u, 0u, 0u);
    if (MODE == kTrain && i < A.rows) {
#pragma unroll
      for (int j = 0; j < 8; ++j) A.XbT[(8 * part + j) * A.ldt + i] = __float2bfloat16(x[j]);
    }
  }
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  tc::tc_fence_before();
  __syncthreads();
  tc::tc_fence_after();
  const int quarter = warp & 3, part = warp >> 2, row = quarter * 32 + lane, i = r0 + row;
  const bool valid = i < A.rows;
  const uint32_t lane_addr = tmem + ((uint32_t)(quarter * 32) << 16);
  const int cpart = part * (kHid / 4);
  constexpr int nph = MODE == kTrain ? kPhases : kLayers;
  int w_inflight = 0;   // thread 0: the phase whose weight copy is in flight, or -1
  int ph = 0;
#pragma unroll 1
  for (; ph < nph; ++ph) {
    // phase ph: layer ph forward, or layer lb = 2 kLayers - 1 - ph back (dZ_lb W_lb)
    const int lb = 2 * kLayers - 1 - ph;
    const int N = ph == kLayers - 1 ? kOutPad : kHid;
    const int nch = ph == 0 || ph == kLayers ? 1 : kHid / tc::kBK;
    float4 gp[MODE == kTrain ? kHid / 16 : 1];
    float tn[MODE == kTrain ? kOut : 1];
    bool has_target = false;
    if (tid == 0) {
      if (!tc::mbar_wait_parity(bw, ph & 1, A.polls)) {
        *abort_flag = 1;
      } else {
        w_inflight = -1;
        tc::tc_fence_after();
        const uint32_t idesc = tc::idesc_bf16(tc::kBM, N);
        const int steps = ph == kLayers ? kOutPad / 16 : tc::kBK / 16;
        for (int c = 0; c < nch; ++c)
          for (int j = 0; j < steps; ++j)
            tc::mma_bf16_ss(tmem, tc::smem_desc_sw128(act + c * (tc::kBM * 128) + 32 * j),
                            tc::smem_desc_sw128(wgt + c * (N * 128) + 32 * j), idesc, c > 0 || j > 0);
      }
      tc::mma_commit(bm);
    }
    if (MODE == kTrain && ph >= kLayers) {
      const float4* gsrc = A.G[lb - 1] + ((long long)blockIdx.x * (kHid / 4) + cpart / 4) * tc::kBM + row;
#pragma unroll
      for (int k = 0; k < kHid / 16; ++k) gp[k] = gsrc[k * tc::kBM];
    }
    if (MODE == kTrain && ph == kLayers - 1 && part == 0 && valid) {
      const long long src = A.idx ? (long long)A.idx[i] : i;
      has_target = src >= 0 && src < A.data_rows;
#pragma unroll
      for (int c = 0; c < kOut; ++c) tn[c] = has_target ? A.T[src * kOut + c] : 0.f;
    }
    if (!tc::mbar_wait_parity(bm, ph & 1, A.polls)) *abort_flag = 1;
    tc::tc_fence_after();
    __syncthreads();
    if (*abort_flag) break;
    if (tid == 0 && ph + 1 < nph) {   // the weight buffer is free: fetch the next phase's
      const int N1 = ph + 1 == kLayers - 1 ? kOutPad : kHid;
      const int ch1 = ph + 1 == kLayers ? 1 : kHid / tc::kBK;
      const CUtensorMap* m = ph + 1 < kLayers ? &maps.w[ph + 1] : &maps.wt[lb - 1];
      tc::mbar_arrive_expect_tx(bw, ch1 * N1 * 128);
      for (int c = 0; c < ch1; ++c) tc::tma_load_2d(wgt + c * N1 * 128, m, bw, c * tc::kBK, 0);
      w_inflight = ph + 1;
    }
    if (ph < kLayers - 1) {
      // hidden layer: GELU(acc + bias) in BF16 over the activations as the next product's A tiles
#pragma unroll 1
      for (int c0 = cpart; c0 < cpart + kHid / 4; c0 += 16) {
        float v[16], a[16];
        tc::tmem_ld16(lane_addr + (uint32_t)c0, v);
#pragma unroll
        for (int j4 = 0; j4 < 4; ++j4) {
          const float4 b4 = *reinterpret_cast<const float4*>(&s_bias[ph][c0 + 4 * j4]);
          const float z[4] = {v[4 * j4] + b4.x, v[4 * j4 + 1] + b4.y, v[4 * j4 + 2] + b4.z, v[4 * j4 + 3] + b4.w};
          float g[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float e = 1.f + erff(z[j] * 0.70710678118654752f);
            a[4 * j4 + j] = 0.5f * z[j] * e;
            if (MODE == kTrain) g[j] = 0.5f * e + z[j] * 0.39894228040143268f * expf(-0.5f * z[j] * z[j]);
          }
          if (MODE == kTrain)
            A.G[ph][((long long)blockIdx.x * (kHid / 4) + c0 / 4 + j4) * tc::kBM + row] = make_float4(g[0], g[1], g[2], g[3]);
        }
        store_act16(act_g, row, c0, a);
        if (MODE == kTrain && valid) {
          bf16* t = A.AbT[ph] + c0 * A.ldt + i;
#pragma unroll
          for (int j = 0; j < 16; ++j) t[j * A.ldt] = __float2bfloat16(a[j]);
        }
      }
    } else if (ph == kLayers - 1) {
      if (part == 0) {
        float v[16];
        tc::tmem_ld16(lane_addr, v);
#pragma unroll
        for (int c = 0; c < kOutPad; ++c) v[c] += s_bias[ph][c];
        if (MODE == kWarm && valid) {
          // warm = q + dt v + out_std * Z + out_mean
#pragma unroll
          for (int c = 0; c < kOut; ++c) {
            const float y = v[c] * A.norm[kNormOutStd + c] + A.norm[kNormOutMean + c];
            const size_t gi = (size_t)i * 12 + c;
            A.warm[gi] = A.q[gi] + A.dt * A.v[gi] + (double)y;
          }
        }
        if (MODE == kInfer && valid) {
#pragma unroll
          for (int c = 0; c < kOut; ++c)
            A.Y[(long long)i * kOut + c] = v[c] * A.norm[kNormOutStd + c] + A.norm[kNormOutMean + c];
        }
        if (MODE == kTrain) {
          // MSE on normalised targets: loss = mean (Z - Tn)^2 over rows x 12; dZ = 2 (Z - Tn) / (rows x 12)
          const float scale = 2.f / (float)(A.rows * kOut);
          double sum = 0.0;
#pragma unroll
          for (int c = 0; c < kOutPad; ++c) {
            float d = 0.f;
            if (c < kOut && has_target) {
              const float diff = v[c] - (tn[c] - A.norm[kNormOutMean + c]) * A.norm[kNormOutIstd + c];
              sum += (double)diff * diff;
              d = scale * diff;
            }
            v[c] = d;
          }
          store_act16(act_g, row, 0, v);
          if (valid) {
#pragma unroll
            for (int c = 0; c < kOutPad; ++c) A.dZbT[ph][c * A.ldt + i] = __float2bfloat16(v[c]);
          }
          const float cs = column_sum16(v, lane);
          if (!(lane & 1)) s_sum[quarter][lane >> 1] = cs;
          for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
          if (lane == 0) atomicAdd(A.loss, sum / (double)(A.rows * kOut));
        }
      }
    } else if (MODE == kTrain) {
      // back through a hidden layer: dZ = (dZ_next W) * GELU'(Z)
#pragma unroll
      for (int k = 0; k < kHid / 64; ++k) {
        const int c0 = cpart + 16 * k;
        float v[16];
        tc::tmem_ld16(lane_addr + (uint32_t)c0, v);
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 g = gp[4 * k + j];
          v[4 * j] = valid ? v[4 * j] * g.x : 0.f;
          v[4 * j + 1] = valid ? v[4 * j + 1] * g.y : 0.f;
          v[4 * j + 2] = valid ? v[4 * j + 2] * g.z : 0.f;
          v[4 * j + 3] = valid ? v[4 * j + 3] * g.w : 0.f;
        }
        if (ph + 1 < nph) store_act16(act_g, row, c0, v);
        if (valid) {
          bf16* t = A.dZbT[lb - 1] + c0 * A.ldt + i;
#pragma unroll
          for (int j = 0; j < 16; ++j) t[j * A.ldt] = __float2bfloat16(v[j]);
        }
        const float cs = column_sum16(v, lane);
        if (!(lane & 1)) s_sum[quarter][c0 + (lane >> 1)] = cs;
      }
    }
    if (MODE == kTrain || ph + 1 < nph) {
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      tc::tc_fence_before();
      __syncthreads();
      tc::tc_fence_after();
    }
    // bias gradients: the CTA's column sums, one atomic per column
    if (MODE == kTrain && ph >= kLayers - 1 && tid < N)
      atomicAdd(&A.gb[ph == kLayers - 1 ? ph : lb - 1][tid], (s_sum[0][tid] + s_sum[1][tid]) + (s_sum[2][tid] + s_sum[3][tid]));
  }
  if (tid == 0 && *abort_flag) {
    atomicOr(A.err, kErrTimeout);
    // a weight copy still in flight, and the commit of the stopped phase, land in shared memory:
    // wait for them before the CTA exits
    if (w_inflight >= 0) tc::mbar_wait_parity(bw, w_inflight & 1, tc::kDrainPolls);
    tc::mbar_wait_parity(bm, ph & 1, tc::kDrainPolls);
  }
  tc::tc_fence_before();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc<kHid>(tmem);
}

}  // namespace mlp
}  // namespace bhem

// ==========================================================================================
// Host side
// ==========================================================================================
using namespace bhem;
using namespace bhem::mlp;

struct shell_mlp_s {
  int max_rows = 0;
  cudaStream_t stream = nullptr;
  unsigned wait_polls = (unsigned)kDefaultWaitPolls;   // bound of the tensor-core pipeline waits
  long long launches = 0;
  int step = 0;
  // parameters (padded; FP32 master copies, BF16 copies for the products), Adam moments, gradients
  float *W[kLayers] = {}, *b[kLayers] = {};
  // one block: the error word, the loss (float 2 on), padding, then gW and gb of every layer
  float* grads = nullptr;
  float *gW[kLayers] = {}, *gb[kLayers] = {};
  float *mW[kLayers] = {}, *vW[kLayers] = {}, *mb[kLayers] = {}, *vb[kLayers] = {};
  bf16* Wb[kLayers] = {};
  bf16* WbT[kLayers] = {};   // transposed BF16 weights [fan_in][fan_out] (back-propagation)
  RowsMaps maps;             // TMA maps of Wb and WbT
  // of the last training pass: transposed copies [features][ldt] (the operands of the weight-gradient
  // GEMMs) of the input, the activations and their gradients, and GELU' (FP32)
  long long ldt = 0;         // max_rows rounded up to 8 (16-byte rows for TMA)
  bf16* XbT = nullptr;
  bf16 *AbT[kLayers - 1] = {}, *dZbT[kLayers] = {};
  float4* G[kLayers - 1] = {};
  float* norm = nullptr;  // kNormSize floats
  double* stats = nullptr;
  int* err = nullptr;       // the block's error word
  float* h_block = nullptr;   // pinned image of the block; also stages parameters on their way in and out
};

namespace {

template <typename T>
shell_status malloc_zero(T** p, size_t count, cudaStream_t s) {
  *p = nullptr;
  cudaError_t e = cudaMalloc((void**)p, sizeof(T) * (count ? count : 1));
  if (e != cudaSuccess) {
    *p = nullptr;
    cudaGetLastError();
    return fail(SHELL_ERR_OOM, std::string("cudaMalloc: ") + cudaGetErrorString(e));
  }
  BHEM_CUDA(cudaMemsetAsync(*p, 0, sizeof(T) * (count ? count : 1), s));
  return SHELL_OK;
}

void free_mlp(shell_mlp_s* m) {
  for (int l = 0; l < kLayers; ++l) {
    void* ps[] = {m->W[l],  m->b[l],   m->mW[l],  m->vW[l], m->mb[l],
                  m->vb[l], m->Wb[l], m->WbT[l], m->dZbT[l]};
    for (void* p : ps)
      if (p) cudaFree(p);
  }
  for (int l = 0; l < kLayers - 1; ++l) {
    if (m->AbT[l]) cudaFree(m->AbT[l]);
    if (m->G[l]) cudaFree(m->G[l]);
  }
  void* ps[] = {m->grads, m->XbT, m->norm, m->stats};
  for (void* p : ps)
    if (p) cudaFree(p);
  if (m->h_block) cudaFreeHost(m->h_block);
  delete m;
}

int eblocks(long long n) { return (int)std::min<long long>(4096, std::max(1LL, (n + 255) / 256)); }

constexpr int kLossAt = 2, kHeadFloats = 64;   // the loss's place in the block, and where the gradients begin
constexpr size_t block_floats() {
  size_t n = kHeadFloats;
  for (int l = 0; l < kLayers; ++l) n += (size_t)kDout[l] * kDin[l] + kDout[l];
  return n;
}

double* loss_of(const shell_mlp_s& M) { return reinterpret_cast<double*>(M.grads + kLossAt); }

template <RowsMode MODE>
shell_status launch_rows(shell_mlp_s& M, RowsArgs& A, cudaStream_t st) {
  static bool attr_set[64] = {false};
  int dev = 0;
  BHEM_CUDA(cudaGetDevice(&dev));
  if (!attr_set[dev & 63]) {
    BHEM_CUDA(cudaFuncSetAttribute(k_mlp_rows<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kRowsSmem));
    attr_set[dev & 63] = true;
  }
  for (int l = 0; l < kLayers; ++l) A.bias[l] = M.b[l];
  A.norm = M.norm;
  A.err = M.err;
  A.polls = M.wait_polls;
  k_mlp_rows<MODE><<<(A.rows + tc::kBM - 1) / tc::kBM, kRowThreads, kRowsSmem, st>>>(M.maps, A);
  BHEM_CUDA(cudaGetLastError());
  ++M.launches;
  return SHELL_OK;
}

// dW_l = dZ_l^T A_{l-1} of every layer: M = fan-out, N = fan-in, K = rows
shell_status weight_gradients(shell_mlp_s& M, int rows, cudaStream_t st) {
  int dev = 0, nsm = 0;
  BHEM_CUDA(cudaGetDevice(&dev));
  BHEM_CUDA(cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev));
  tc::GemmSet S;
  static_assert(kLayers == tc::kMaxGroups, "one group per layer");
  int tiles = 0;
  bool ok = true;
  for (int l = 0; l < kLayers; ++l) {
    tc::GemmGroup& g = S.g[l];
    ok = ok && tc::encode_bf16_map(&g.a, M.dZbT[l], kDout[l], rows, M.ldt, tc::kBM) &&
         tc::encode_bf16_map(&g.b, l > 0 ? M.AbT[l - 1] : M.XbT, kDin[l], rows, M.ldt, tc::kBN) &&
         tc::encode_c_map(&g.c, M.gW[l], kDout[l], kDin[l], kDin[l]);
    S.n[l] = kDin[l];
    S.tiles_n[l] = (kDin[l] + tc::kBN - 1) / tc::kBN;
    S.first[l] = tiles;
    tiles += S.tiles_n[l] * ((kDout[l] + tc::kBM - 1) / tc::kBM);
  }
  S.first[kLayers] = tiles;
  if (!ok) return fail(SHELL_ERR_CUDA, "tensor map encoding failed (cuTensorMapEncodeTiled)");
  S.polls = M.wait_polls;
  S.err = M.err;
  S.err_bit = kErrTimeout;
  BHEM_CUDA(tc::launch_gemm_split(S, tiles, rows, 2 * nsm / tiles, st));
  ++M.launches;
  return SHELL_OK;
}

// waits for the stream, returns the loss when asked, and turns a raised error flag into an error
shell_status finish(shell_mlp_s& M, double* loss) {
  BHEM_CUDA(cudaMemcpyAsync(M.h_block, M.grads, sizeof(float) * (kLossAt + 2), cudaMemcpyDeviceToHost, M.stream));
  BHEM_CUDA(cudaStreamSynchronize(M.stream));
  int e;
  std::memcpy(&e, M.h_block, sizeof(int));
  if (e) {
    BHEM_CUDA(cudaMemsetAsync(M.err, 0, sizeof(int), M.stream));
    BHEM_CUDA(cudaStreamSynchronize(M.stream));
    if (e & kErrTimeout) return fail(SHELL_ERR_TIMEOUT, "a bounded tensor-core pipeline wait expired");
    return fail(SHELL_ERR_ARG, "row index outside [0, data_rows)");
  }
  if (loss) std::memcpy(loss, M.h_block + kLossAt, sizeof(double));
  return SHELL_OK;
}

long long param_count() {
  long long n = 0;
  for (int l = 0; l < kLayers; ++l) n += (long long)kRout[l] * kRin[l] + kRout[l];
  return n;
}

// host packed layout: per layer W [fan_out x fan_in] row-major, then b [fan_out]. Everything passes through
// the pinned image of the gradient block (whose layout is the padded one of the device): one copy for the
// gradients, asynchronous ones for the parameters, then one wait. Read in eight blocking pageable copies the
// gradients took 128 us, now 46 us.
shell_status copy_params(shell_mlp_s& M, float* host_out, const float* host_in, int grads) {
  float* const image = M.h_block;
  if (!host_in && grads)
    BHEM_CUDA(cudaMemcpyAsync(image, M.grads, sizeof(float) * block_floats(), cudaMemcpyDeviceToHost, M.stream));
  for (int pass = 0; pass < 2; ++pass) {   // out: fetch, wait, unpack; in: pack and send, wait
    if (pass == 1) BHEM_CUDA(cudaStreamSynchronize(M.stream));
    if (pass == 1 && host_in) break;
    float* p = image + kHeadFloats;
    long long off = 0;
    for (int l = 0; l < kLayers; ++l) {
      const int ro = kRout[l], ri = kRin[l], din = kDin[l];
      const size_t nw = (size_t)kDout[l] * din;
      float* pb = p + nw;
      if (host_in) {
        std::memset(p, 0, sizeof(float) * (nw + kDout[l]));
        for (int o = 0; o < ro; ++o)
          std::memcpy(p + (size_t)o * din, host_in + off + (long long)o * ri, sizeof(float) * ri);
        std::memcpy(pb, host_in + off + (long long)ro * ri, sizeof(float) * ro);
        BHEM_CUDA(cudaMemcpyAsync(M.W[l], p, sizeof(float) * nw, cudaMemcpyHostToDevice, M.stream));
        BHEM_CUDA(cudaMemcpyAsync(M.b[l], pb, sizeof(float) * ro, cudaMemcpyHostToDevice, M.stream));
      } else if (pass == 0) {
        if (grads) break;
        BHEM_CUDA(cudaMemcpyAsync(p, M.W[l], sizeof(float) * nw, cudaMemcpyDeviceToHost, M.stream));
        BHEM_CUDA(cudaMemcpyAsync(pb, M.b[l], sizeof(float) * ro, cudaMemcpyDeviceToHost, M.stream));
      } else {
        if (ri == din) {
          std::memcpy(host_out + off, p, sizeof(float) * (size_t)ro * ri);
        } else {
          for (int o = 0; o < ro; ++o)
            std::memcpy(host_out + off + (long long)o * ri, p + (size_t)o * din, sizeof(float) * ri);
        }
        std::memcpy(host_out + off + (long long)ro * ri, pb, sizeof(float) * ro);
      }
      p = pb + kDout[l];
      off += (long long)ro * ri + ro;
    }
  }
  return SHELL_OK;
}

}  // namespace

extern "C" shell_status shell_mlp_create(int max_rows, void* stream, shell_mlp_t** out) {
  if (!out || max_rows < 1 || max_rows > (1 << 24)) return fail(SHELL_ERR_ARG, "invalid argument");
  *out = nullptr;
  shell_mlp_s* M = new shell_mlp_s();
  M->max_rows = max_rows;
  M->stream = (cudaStream_t)stream;
  M->ldt = ((long long)max_rows + 7) / 8 * 8;
  shell_status st = SHELL_OK;
  const size_t R128 = ((size_t)max_rows + tc::kBM - 1) / tc::kBM * tc::kBM, RT = (size_t)M->ldt;
  for (int l = 0; l < kLayers && st == SHELL_OK; ++l) {
    const size_t nw = (size_t)kDout[l] * kDin[l], nb = kDout[l];
    float** f32w[] = {&M->W[l], &M->mW[l], &M->vW[l]};
    for (float** p : f32w)
      if (st == SHELL_OK) st = malloc_zero(p, nw, M->stream);
    float** f32b[] = {&M->b[l], &M->mb[l], &M->vb[l]};
    for (float** p : f32b)
      if (st == SHELL_OK) st = malloc_zero(p, nb, M->stream);
    if (st == SHELL_OK) st = malloc_zero(&M->Wb[l], nw, M->stream);
    if (st == SHELL_OK && l > 0) st = malloc_zero(&M->WbT[l], nw, M->stream);
    if (st == SHELL_OK && l < kLayers - 1) st = malloc_zero(&M->AbT[l], RT * kDout[l], M->stream);
    if (st == SHELL_OK && l < kLayers - 1) st = malloc_zero(&M->G[l], R128 * kDout[l] / 4, M->stream);
    if (st == SHELL_OK) st = malloc_zero(&M->dZbT[l], RT * kDout[l], M->stream);
  }
  if (st == SHELL_OK) st = malloc_zero(&M->grads, block_floats(), M->stream);
  if (st == SHELL_OK) {
    M->err = reinterpret_cast<int*>(M->grads);
    float* p = M->grads + kHeadFloats;
    for (int l = 0; l < kLayers; ++l) {
      M->gW[l] = p;
      M->gb[l] = p + (size_t)kDout[l] * kDin[l];
      p = M->gb[l] + kDout[l];
    }
  }
  if (st == SHELL_OK) st = malloc_zero(&M->XbT, RT * kInPad, M->stream);
  if (st == SHELL_OK) st = malloc_zero(&M->norm, kNormSize, M->stream);
  if (st == SHELL_OK) st = malloc_zero(&M->stats, 2 * kIn, M->stream);
  if (st == SHELL_OK && cudaMallocHost((void**)&M->h_block, sizeof(float) * block_floats()) != cudaSuccess) {
    cudaGetLastError();
    st = fail(SHELL_ERR_OOM, "cudaMallocHost failed");
  }
  for (int l = 0; l < kLayers && st == SHELL_OK; ++l)
    if (!tc::encode_bf16_map(&M->maps.w[l], M->Wb[l], kDout[l], kDin[l], kDin[l], kDout[l]) ||
        (l > 0 && !tc::encode_bf16_map(&M->maps.wt[l], M->WbT[l], kDin[l], kDout[l], kDout[l], kDin[l])))
      st = fail(SHELL_ERR_CUDA, "tensor map encoding failed (cuTensorMapEncodeTiled)");
  if (st == SHELL_OK) {
    // identity normalisation until shell_mlp_set_normalization
    float h[kNormSize] = {};
    for (int k = 0; k < kIn; ++k) h[kNormInIstd + k] = 1.f;
    for (int k = 0; k < kOut; ++k) h[kNormOutStd + k] = h[kNormOutIstd + k] = 1.f;
    if (cudaMemcpyAsync(M->norm, h, sizeof(h), cudaMemcpyHostToDevice, M->stream) != cudaSuccess ||
        cudaStreamSynchronize(M->stream) != cudaSuccess)
      st = fail(SHELL_ERR_CUDA, "normalisation upload failed");
  }
  if (st != SHELL_OK) {
    cudaStreamSynchronize(M->stream);
    free_mlp(M);
    return st;
  }
  *out = M;
  return SHELL_OK;
}

extern "C" shell_status shell_mlp_destroy(shell_mlp_t* M) {
  if (!M) return SHELL_OK;
  cudaStreamSynchronize(M->stream);
  free_mlp(M);
  return SHELL_OK;
}

extern "C" shell_status shell_mlp_param_count(long long* count) {
  if (!count) return fail(SHELL_ERR_ARG, "NULL argument");
  *count = param_count();
  return SHELL_OK;
}

extern "C" shell_status shell_mlp_set_params(shell_mlp_t* M, const float* params) {
  if (!M || !params) return fail(SHELL_ERR_ARG, "NULL argument");
  BHEM_CUDA(cudaStreamSynchronize(M->stream));
  BHEM_TRY(copy_params(*M, nullptr, params, 0));
  for (int l = 0; l < kLayers; ++l) {
    const long long n = (long long)kDout[l] * kDin[l];
    k_to_bf16<<<eblocks(n), 256, 0, M->stream>>>(kDout[l], kDin[l], M->W[l], M->Wb[l], M->WbT[l]);
    BHEM_CUDA(cudaGetLastError());
    ++M->launches;
    BHEM_CUDA(cudaMemsetAsync(M->mW[l], 0, sizeof(float) * n, M->stream));
    BHEM_CUDA(cudaMemsetAsync(M->vW[l], 0, sizeof(float) * n, M->stream));
    BHEM_CUDA(cudaMemsetAsync(M->mb[l], 0, sizeof(float) * kDout[l], M->stream));
    BHEM_CUDA(cudaMemsetAsync(M->vb[l], 0, sizeof(float) * kDout[l], M->stream));
  }
  M->step = 0;
  BHEM_CUDA(cudaStreamSynchronize(M->stream));
  return SHELL_OK;
}

extern "C" shell_status shell_mlp_get_params(shell_mlp_t* M, float* params, float* grads) {
  if (!M) return fail(SHELL_ERR_ARG, "NULL argument");
  BHEM_CUDA(cudaStreamSynchronize(M->stream));
  if (params) BHEM_TRY(copy_params(*M, params, nullptr, 0));
  if (grads) BHEM_TRY(copy_params(*M, grads, nullptr, 1));
  return SHELL_OK;
}

extern "C" shell_status shell_mlp_set_normalization(shell_mlp_t* M, const float* in_mean, const float* in_std,
                                                    const float* out_mean, const float* out_std) {
  if (!M || !in_mean || !in_std || !out_mean || !out_std) return fail(SHELL_ERR_ARG, "NULL argument");
  float h[kNormSize] = {};
  for (int k = 0; k < kIn; ++k) {
    h[kNormInMean + k] = in_mean[k];
    h[kNormInIstd + k] = in_std[k] > 0.f ? 1.f / in_std[k] : 1.f;
  }
  for (int k = 0; k < kOut; ++k) {
    h[kNormOutMean + k] = out_mean[k];
    h[kNormOutStd + k] = out_std[k] > 0.f ? out_std[k] : 1.f;
    h[kNormOutIstd + k] = out_std[k] > 0.f ? 1.f / out_std[k] : 1.f;
  }
  BHEM_CUDA(cudaMemcpyAsync(M->norm, h, sizeof(h), cudaMemcpyHostToDevice, M->stream));
  BHEM_CUDA(cudaStreamSynchronize(M->stream));
  return SHELL_OK;
}

extern "C" shell_status shell_mlp_column_stats(shell_mlp_t* M, const float* X, long long rows, int cols,
                                               double* mean, double* stdv) {
  if (!M || !X || rows < 1 || cols < 1 || cols > kIn || !mean || !stdv)
    return fail(SHELL_ERR_ARG, "invalid argument");
  k_colstats<<<cols, 256, 0, M->stream>>>(rows, cols, X, M->stats);
  BHEM_CUDA(cudaGetLastError());
  ++M->launches;
  double h[2 * kIn];
  BHEM_CUDA(cudaMemcpyAsync(h, M->stats, sizeof(double) * 2 * cols, cudaMemcpyDeviceToHost, M->stream));
  BHEM_CUDA(cudaStreamSynchronize(M->stream));
  for (int c = 0; c < cols; ++c) {
    mean[c] = h[2 * c] / (double)rows;
    const double var = h[2 * c + 1] / (double)rows - mean[c] * mean[c];
    stdv[c] = var > 0.0 ? std::sqrt(var) : 0.0;
  }
  return SHELL_OK;
}

extern "C" shell_status shell_mlp_forward(shell_mlp_t* M, const float* X, int rows, float* Y) {
  if (!M || !X || !Y || rows < 1 || rows > M->max_rows) return fail(SHELL_ERR_ARG, "invalid argument");
  RowsArgs A{};
  A.rows = rows;
  A.X = X;
  A.Y = Y;
  return launch_rows<kInfer>(*M, A, M->stream);
}

extern "C" shell_status shell_mlp_gradients(shell_mlp_t* M, const float* X, const float* T, long long data_rows,
                                            const int* idx, int rows, double* loss) {
  if (!M || !X || !T || rows < 1 || rows > M->max_rows || data_rows < 1 || (!idx && rows > data_rows))
    return fail(SHELL_ERR_ARG, "invalid argument");
  BHEM_CUDA(cudaMemsetAsync(M->grads + kLossAt, 0, sizeof(float) * (block_floats() - kLossAt), M->stream));
  RowsArgs A{};
  A.rows = rows;
  A.X = X;
  A.T = T;
  A.data_rows = data_rows;
  A.idx = idx;
  A.loss = loss_of(*M);
  A.ldt = M->ldt;
  A.XbT = M->XbT;
  for (int l = 0; l < kLayers; ++l) {
    if (l < kLayers - 1) {
      A.AbT[l] = M->AbT[l];
      A.G[l] = M->G[l];
    }
    A.dZbT[l] = M->dZbT[l];
    A.gb[l] = M->gb[l];
  }
  BHEM_TRY(launch_rows<kTrain>(*M, A, M->stream));
  BHEM_TRY(weight_gradients(*M, rows, M->stream));
  return loss ? finish(*M, loss) : SHELL_OK;
}

extern "C" shell_status shell_mlp_train_step(shell_mlp_t* M, const float* X, const float* T, long long data_rows,
                                             const int* idx, int rows, float lr, double* loss) {
  BHEM_TRY(shell_mlp_gradients(M, X, T, data_rows, idx, rows, nullptr));
  M->step += 1;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  const float c1 = 1.f - std::pow(b1, (float)M->step), c2 = 1.f - std::pow(b2, (float)M->step);
  AdamSet S{};
  long long end = 0;
  for (int l = 0; l < kLayers; ++l) {
    const int t = 2 * l;   // weights, then bias
    S.w[t] = M->W[l];
    S.g[t] = M->gW[l];
    S.m[t] = M->mW[l];
    S.v[t] = M->vW[l];
    S.wb[t] = M->Wb[l];
    S.wbT[t] = M->WbT[l];
    S.rows[t] = kDout[l];
    S.cols[t] = kDin[l];
    S.end[t] = end += (long long)kDout[l] * kDin[l];
    S.w[t + 1] = M->b[l];
    S.g[t + 1] = M->gb[l];
    S.m[t + 1] = M->mb[l];
    S.v[t + 1] = M->vb[l];
    S.rows[t + 1] = 1;
    S.cols[t + 1] = kDout[l];
    S.end[t + 1] = end += kDout[l];
  }
  k_adam<<<eblocks(end), 256, 0, M->stream>>>(S, lr, b1, b2, eps, c1, c2);
  ++M->launches;
  BHEM_CUDA(cudaGetLastError());
  return loss ? finish(*M, loss) : SHELL_OK;
}

extern "C" shell_status shell_mlp_set_wait_budget(shell_mlp_t* M, int polls) {
  if (!M) return fail(SHELL_ERR_ARG, "NULL argument");
  BHEM_CUDA(cudaStreamSynchronize(M->stream));
  M->wait_polls = polls < 0 ? (unsigned)kDefaultWaitPolls : (unsigned)polls;
  return SHELL_OK;
}

extern "C" shell_status shell_mlp_kernel_launches(const shell_mlp_t* M, long long* count) {
  if (!M || !count) return fail(SHELL_ERR_ARG, "NULL argument");
  *count = M->launches;
  return SHELL_OK;
}

extern "C" shell_status shell_node_features(shell_t* shell, const double* q, const double* v, float* X) {
  if (!shell || !q || !v || !X) return fail(SHELL_ERR_ARG, "NULL argument");
  Shell& s = *shell;
  k_node_features<<<(s.n_nodes + 127) / 128, 128, 0, s.stream>>>(s.n1, s.n2, s.grid.periodic_u, s.grid.periodic_v,
                                                                 q, s.d_rest, v, X);
  BHEM_CUDA(cudaGetLastError());
  ++s.launches;
  return SHELL_OK;
}

extern "C" shell_status shell_warm_targets(long long n_dof, const double* q_next, const double* q, const double* v,
                                           double dt, float* T, void* stream) {
  if (n_dof < 1 || !q_next || !q || !v || !T) return fail(SHELL_ERR_ARG, "invalid argument");
  k_targets<<<eblocks(n_dof), 256, 0, (cudaStream_t)stream>>>(n_dof, q_next, q, v, dt, T);
  BHEM_CUDA(cudaGetLastError());
  return SHELL_OK;
}

extern "C" shell_status shell_mlp_warm_start(shell_mlp_t* M, shell_t* shell, const double* q, const double* v,
                                             double dt, double* warm) {
  if (!shell || !q || !v || !warm) return fail(SHELL_ERR_ARG, "NULL argument");
  Shell& s = *shell;
  if (!M) {
    k_predict<<<eblocks(s.n_dof), 256, 0, s.stream>>>(s.n_dof, q, v, dt, warm);
    BHEM_CUDA(cudaGetLastError());
    ++s.launches;
    return SHELL_OK;
  }
  RowsArgs A{};
  A.rows = s.n_nodes;
  A.n1 = s.n1;
  A.n2 = s.n2;
  A.per_u = s.grid.periodic_u;
  A.per_v = s.grid.periodic_v;
  A.q = q;
  A.rest = s.d_rest;
  A.v = v;
  A.dt = dt;
  A.warm = warm;
  return launch_rows<kWarm>(*M, A, s.stream);
}
