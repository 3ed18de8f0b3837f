// Second-stage reductions of the backward pass, in a fixed order so results repeat bit for bit
// (the paper's Algorithm 2 uses atomic adds for these sums).
#include "device_common.cuh"
#include "internal.h"

namespace m2rnn {
namespace {

// dW[n] = sum_b dW_part[b][n]   (Algorithm 2 sums dW over the batch with an atomic add)
__global__ void reduce_dW_kernel(const float *__restrict__ part, float *__restrict__ dW, int B, size_t NVV) {
  begin_dependent();
  const size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= NVV) return;
  float s = 0.f;
  for (int b = 0; b < B; ++b) s += part[(size_t)b * NVV + x];
  dW[x] = s;
}

// out[bt][g][:] = sum over the heads n of group g of part[bt][n][:]
// (Algorithm 2 sums dq and dk over the heads that share them with atomic adds).  Four entries of a row a thread (K is a
// multiple of 16), eight heads' loads in flight: HBM-bound (one entry and load after another read 71 MB in 19 us, now 14).
template <typename TIO>
__global__ void __launch_bounds__(256) reduce_heads_kernel(const float4 *__restrict__ part, TIO *__restrict__ out, size_t rows, int per, int K4) {
  begin_dependent();
  const size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= rows * K4) return;
  const size_t row = x / K4, at = row * per * K4 + x % K4;      // row: (bt, g)
  float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
  for (int h0 = 0; h0 < per; h0 += 8) {
    float4 p[8];
#pragma unroll
    for (int h = 0; h < 8; ++h)
      if (h0 + h < per) p[h] = __ldcs(part + at + (size_t)(h0 + h) * K4);
#pragma unroll
    for (int h = 0; h < 8; ++h)
      if (h0 + h < per) { s.x += p[h].x; s.y += p[h].y; s.z += p[h].z; s.w += p[h].w; }
  }
  if constexpr (sizeof(TIO) == 4) {
    reinterpret_cast<float4 *>(out)[x] = s;
  } else {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(s.x, s.y), hi = __floats2bfloat162_rn(s.z, s.w);
    reinterpret_cast<uint2 *>(out)[x] = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
  }
}

// out[x] = sum_r part[r][x]: sums over the row slabs of a state that were handled by different CTAs
// (dv and dgate are sums over all K rows).  Four adjacent elements per thread where rows of the parts stay
// 16-byte aligned, up to four slabs' loads in flight: HBM-bound (one element per thread and load left
// it at 2.2 TB/s: 22 M elements of two slabs 100 us, now 36).
template <typename TIO>
__global__ void reduce_slabs_kernel(const float *__restrict__ part, TIO *__restrict__ out, int R, size_t n) {
  begin_dependent();
  const size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= n) return;
  float s = 0.f;
  for (int r = 0; r < R; ++r) s += part[(size_t)r * n + x];
  out[x] = from_f32<TIO>(s);
}
template <typename TIO>
__global__ void __launch_bounds__(256) reduce_slabs4_kernel(const float4 *__restrict__ part, TIO *__restrict__ out, int R, size_t n4) {
  begin_dependent();
  for (size_t x = (size_t)blockIdx.x * blockDim.x + threadIdx.x; x < n4; x += (size_t)gridDim.x * blockDim.x) {
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int r0 = 0; r0 < R; r0 += 4) {
      float4 p[4];
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (r0 + r < R) p[r] = __ldcs(part + (size_t)(r0 + r) * n4 + x);
#pragma unroll
      for (int r = 0; r < 4; ++r)
        if (r0 + r < R) { s.x += p[r].x; s.y += p[r].y; s.z += p[r].z; s.w += p[r].w; }
    }
    if constexpr (sizeof(TIO) == 4) {
      reinterpret_cast<float4 *>(out)[x] = s;
    } else {
      const __nv_bfloat162 lo = __floats2bfloat162_rn(s.x, s.y), hi = __floats2bfloat162_rn(s.z, s.w);
      reinterpret_cast<uint2 *>(out)[x] = make_uint2(*reinterpret_cast<const uint32_t *>(&lo), *reinterpret_cast<const uint32_t *>(&hi));
    }
  }
}

}  // namespace

cudaError_t launch_reduce_slabs(const float *part, void *out, int io_dtype, int R, size_t n, cudaStream_t s) {
  if (n % 4 == 0) {
    const size_t n4 = n / 4, need = (n4 + 255) / 256, most = (size_t)sm_count() * 32;
    const unsigned grid = (unsigned)(need < most ? need : most);
    const float4 *p = reinterpret_cast<const float4 *>(part);
    if (io_dtype == M2RNN_F32) (void)launch_early(reduce_slabs4_kernel<float>, grid, 256, 0, s, p, static_cast<float *>(out), R, n4);
    else (void)launch_early(reduce_slabs4_kernel<__nv_bfloat16>, grid, 256, 0, s, p, static_cast<__nv_bfloat16 *>(out), R, n4);
    return cudaGetLastError();
  }
  const unsigned grid = (unsigned)((n + 255) / 256);
  if (io_dtype == M2RNN_F32)
    (void)launch_early(reduce_slabs_kernel<float>, grid, 256, 0, s, part, static_cast<float *>(out), R, n);
  else
    (void)launch_early(reduce_slabs_kernel<__nv_bfloat16>, grid, 256, 0, s, part, static_cast<__nv_bfloat16 *>(out), R, n);
  return cudaGetLastError();
}

cudaError_t launch_reduce_dW(const float *dW_part, float *dW, int B, int N, int V, cudaStream_t s) {
  const size_t NVV = (size_t)N * V * V;
  (void)launch_early(reduce_dW_kernel, (unsigned)((NVV + 255) / 256), 256, 0, s, dW_part, dW, B, NVV);
  return cudaGetLastError();
}

cudaError_t launch_reduce_heads(const float *part, void *out, int io_dtype, size_t BT, int N, int Ng,
                                int K, cudaStream_t s) {
  const size_t rows = BT * Ng;
  const int per = N / Ng, K4 = K / 4;
  const unsigned grid = (unsigned)((rows * K4 + 255) / 256);
  const float4 *p = reinterpret_cast<const float4 *>(part);
  if (io_dtype == M2RNN_F32) (void)launch_early(reduce_heads_kernel<float>, grid, 256, 0, s, p, static_cast<float *>(out), rows, per, K4);
  else (void)launch_early(reduce_heads_kernel<__nv_bfloat16>, grid, 256, 0, s, p, static_cast<__nv_bfloat16 *>(out), rows, per, K4);
  return cudaGetLastError();
}

}  // namespace m2rnn
