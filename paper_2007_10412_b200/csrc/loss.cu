// Softmax cross-entropy and its Jacobian (exact; Sec. 4.2: the loss Jacobian is never sampled).
#include <algorithm>

#include "common.cuh"

namespace rad {
namespace {

// One warp per row: loss_b = logsumexp(z_b) - z_b[label]; dZ = (softmax - onehot) / B.  Returns loss_b in lane 0.
// NV > 0: the row's logits and exponentials stay in NV registers a lane (C <= 32 NV), so the row is read once, all
// its loads in flight together, and each exponential is taken once; NV = 0: rows of any length, read three times.
template <typename T, int NV>
__device__ __forceinline__ float xent_row(const float* z, int32_t y, int64_t C, T* dz, float invB, int lane) {
  float v[NV > 0 ? NV : 1];
  float mx = -INFINITY, sum = 0.0f;
  if (NV > 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) v[i] = lane + 32 * i < C ? z[lane + 32 * i] : -INFINITY;
#pragma unroll
    for (int i = 0; i < NV; ++i) mx = fmaxf(mx, v[i]);
  } else {
    for (int64_t c = lane; c < C; c += 32) mx = fmaxf(mx, z[c]);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
  if (NV > 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i)
      if (lane + 32 * i < C) sum += (v[i] = expf(v[i] - mx));
  } else {
    for (int64_t c = lane; c < C; c += 32) sum += expf(z[c] - mx);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  const float inv = 1.0f / sum;
  if (NV > 0) {
#pragma unroll
    for (int i = 0; i < NV; ++i) {
      const int c = lane + 32 * i;
      float g = v[i] * inv;
      if (c == y) g -= 1.0f;
      if (c < C) dz[c] = from_float<T>(g * invB);
    }
  } else {
    for (int64_t c = lane; c < C; c += 32) {
      float g = expf(z[c] - mx) * inv;
      if (c == y) g -= 1.0f;
      dz[c] = from_float<T>(g * invB);
    }
  }
  return lane == 0 && y >= 0 && y < C ? (logf(sum) + mx - z[y]) : 0.0f;
}

template <typename T, int NV>
__global__ void __launch_bounds__(256) xent_rows_kernel(const float* logits, int64_t ldl, const int32_t* labels,
                                                        int64_t B, int64_t C, T* dZ, int64_t ldz,
                                                        float* row_loss) {
  begin_after_previous();
  const int lane = threadIdx.x & 31;
  const int64_t b = (int64_t)blockIdx.x * 8 + (threadIdx.x >> 5);
  if (b >= B) return;
  const float l = xent_row<T, NV>(logits + b * ldl, labels[b], C, dZ + b * ldz, 1.0f / (float)B, lane);
  if (lane == 0) row_loss[b] = l;
}

// Rows and mean in one launch for small batches (the small nets are bound by their launch count): a cluster of up to
// eight CTAs, a warp takes rows w, w + W, ... of the cluster's W warps and leaves their losses in the first CTA's
// shared memory, which takes the same fixed-order mean as below.  What bounds it is the chain of one row (load,
// two warp reductions, exponentials); with all rows in one CTA a warp walked up to 64 of them: 150 x 10 logits
// 15 us, 328 x 200 38 us; a cluster 8 and 11 us.
constexpr int kXentSmallRows = 2048;
constexpr int kXentCluster = 8;            // portable cluster size
template <typename T, int NV>
__global__ void __launch_bounds__(1024) xent_small_kernel(const float* logits, int64_t ldl, const int32_t* labels, int64_t B,
                                                          int64_t C, T* dZ, int64_t ldz, float* loss) {
  begin_after_previous();
  __shared__ float s_row[kXentSmallRows];
  __shared__ float s[1024];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  cluster_barrier();                       // the first CTA has started before anyone writes to its shared memory
  for (int64_t b = (int64_t)blockIdx.x * 32 + warp; b < B; b += (int64_t)gridDim.x * 32) {
    const float l = xent_row<T, NV>(logits + b * ldl, labels[b], C, dZ + b * ldz, 1.0f / (float)B, lane);
    if (lane == 0) st_cluster_f32(&s_row[b], 0, l);
  }
  cluster_barrier();
  if (blockIdx.x != 0) return;
  float acc = 0.0f;
  for (int64_t i = threadIdx.x; i < B; i += 1024) acc += s_row[i];
  s[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 512; o >= 32; o >>= 1) {
    if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
    __syncthreads();
  }
  if (warp == 0) {
    float t = s[lane];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) t += __shfl_down_sync(0xffffffffu, t, o);
    if (lane == 0) *loss = t / (float)B;
  }
}

// Fixed-order mean of the per-row losses (one CTA).
__global__ void __launch_bounds__(1024) mean_kernel(const float* row_loss, int64_t B, float* loss) {
  begin_after_previous();
  __shared__ float s[1024];
  float acc = 0.0f;
  for (int64_t i = threadIdx.x; i < B; i += 1024) acc += row_loss[i];
  s[threadIdx.x] = acc;
  __syncthreads();
  for (int o = 512; o > 0; o >>= 1) {
    if ((int)threadIdx.x < o) s[threadIdx.x] += s[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *loss = s[0] / (float)B;
}

template <typename T, int NV>
int launch_xent(const float* logits, int64_t ldl, const int32_t* labels, int64_t B, int64_t C, T* dZ, int64_t ldz, float* loss,
                float* rows, cudaStream_t s) {
  if (B <= kXentSmallRows) {
    const unsigned ctas = (unsigned)std::min<int64_t>(kXentCluster, ceil_div(B, 32));
    count_launch();
    return launch_with_cluster(xent_small_kernel<T, NV>, dim3(ctas), 1024, 0, dim3(ctas), s, logits, ldl, labels, B, C, dZ, ldz, loss);
  }
  count_launch(2);
  RAD_TRY(launch_kernel(xent_rows_kernel<T, NV>, (unsigned)ceil_div(B, 8), 256, 0, s, logits, ldl, labels, B, C, dZ, ldz, rows));
  RAD_TRY(launch_kernel(mean_kernel, 1, 1024, 0, s, rows, B, loss));
  return RAD_OK;
}
template <typename T>
int launch_xent_of(const float* logits, int64_t ldl, const int32_t* labels, int64_t B, int64_t C, T* dZ, int64_t ldz, float* loss,
                   float* rows, cudaStream_t s) {
  if (C <= 32) return launch_xent<T, 1>(logits, ldl, labels, B, C, dZ, ldz, loss, rows, s);
  if (C <= 256) return launch_xent<T, 8>(logits, ldl, labels, B, C, dZ, ldz, loss, rows, s);
  if (C <= 1024) return launch_xent<T, 32>(logits, ldl, labels, B, C, dZ, ldz, loss, rows, s);
  return launch_xent<T, 0>(logits, ldl, labels, B, C, dZ, ldz, loss, rows, s);
}

}  // namespace
}  // namespace rad

using namespace rad;

extern "C" int rad_softmax_xent(int32_t dtype, int64_t B, int64_t C, const float* logits, int64_t ldl,
                                const int32_t* labels, float* loss, void* dZ, int64_t ldz, void* workspace,
                                int64_t workspace_bytes, void* stream) {
  if (B <= 0 || C <= 0 || logits == nullptr || labels == nullptr || loss == nullptr || dZ == nullptr)
    return RAD_EINVAL;
  if (ldl < C || ldz < C) return RAD_EINVAL;
  if (dtype != RAD_F32 && dtype != RAD_BF16) return RAD_EINVAL;
  if (workspace == nullptr || workspace_bytes < B * 4) return RAD_EWORKSPACE;
  int rc = check_device();
  if (rc != RAD_OK) return rc;
  cudaStream_t s = static_cast<cudaStream_t>(stream);
  float* rows = static_cast<float*>(workspace);
  if (dtype == RAD_BF16) return launch_xent_of(logits, ldl, labels, B, C, static_cast<bf16*>(dZ), ldz, loss, rows, s);
  return launch_xent_of(logits, ldl, labels, B, C, static_cast<float*>(dZ), ldz, loss, rows, s);
}
