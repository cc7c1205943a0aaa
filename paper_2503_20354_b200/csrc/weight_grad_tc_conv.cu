// Conversion of the output gradient to bf16, as streaming pre-passes of the weight-gradient kernels.
#include <cuda.h>

#include "surgeon_internal.cuh"
#include "tc_common.cuh"
#include "weight_grad_tc_conv.cuh"

namespace surgeon {

namespace {

using namespace tc;

// fp32 -> bf16 (round to nearest even), 8 elements per thread.
__global__ void __launch_bounds__(256)
grad_to_bf16_kernel(const float* __restrict__ g, long long n, unsigned short* __restrict__ out,
                    uint32_t* __restrict__ status) {
  prepass_begin(status);
  const long long n8 = n >> 3;
  const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < n8;
       i += stride) {
    const float4 a = __ldg(reinterpret_cast<const float4*>(g) + 2 * i);
    const float4 b = __ldg(reinterpret_cast<const float4*>(g) + 2 * i + 1);
    uint4 o;
    o.x = pack_bf16x2(a.x, a.y); o.y = pack_bf16x2(a.z, a.w);
    o.z = pack_bf16x2(b.x, b.y); o.w = pack_bf16x2(b.z, b.w);
    reinterpret_cast<uint4*>(out)[i] = o;
  }
  if (blockIdx.x == 0)
    for (long long j = (n8 << 3) + threadIdx.x; j < n; j += blockDim.x)
      out[j] = static_cast<unsigned short>(pack_bf16x2(g[j], 0.0f) & 0xFFFFu);
}

// rows of `len` floats -> rows of `pitch` bf16 (pitch a multiple of 8, padding zero)
__global__ void __launch_bounds__(256)
grad_to_bf16_rows_kernel(const float* __restrict__ g, long long rows, int len, int pitch,
                         unsigned short* __restrict__ out, uint32_t* __restrict__ status) {
  prepass_begin(status);
  const int per_row = pitch >> 3;
  const long long total = rows * per_row;
  const long long stride = static_cast<long long>(gridDim.x) * blockDim.x;
  for (long long i = static_cast<long long>(blockIdx.x) * blockDim.x + threadIdx.x; i < total;
       i += stride) {
    const long long r = i / per_row;
    const int c0 = static_cast<int>(i - r * per_row) * 8;
    const float* src = g + r * len + c0;
    float v[8];
    if ((len & 3) == 0 && c0 + 8 <= len) {         // rows start on 16-byte boundaries
      const float4 a = __ldg(reinterpret_cast<const float4*>(src));
      const float4 b = __ldg(reinterpret_cast<const float4*>(src) + 1);
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
      v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
    } else {
#pragma unroll
      for (int e = 0; e < 8; ++e) v[e] = (c0 + e < len) ? __ldg(src + e) : 0.0f;
    }
    uint4 o;
    o.x = pack_bf16x2(v[0], v[1]); o.y = pack_bf16x2(v[2], v[3]);
    o.z = pack_bf16x2(v[4], v[5]); o.w = pack_bf16x2(v[6], v[7]);
    reinterpret_cast<uint4*>(out)[i] = o;
  }
}

}  // namespace

cudaError_t launch_grad_to_bf16(const float* g, long long n, void* out_bf16, uint32_t* status, cudaStream_t stream) {
  const long long want = (n / 8 + 255) / 256;
  const long long cap = 16LL * sm_count();
  const int grid = static_cast<int>(want < 1 ? 1 : (want > cap ? cap : want));
  note_launches(1);
  return launch_kernel(grad_to_bf16_kernel, dim3(grid), dim3(256), 0, stream, true, g, n,
                       static_cast<unsigned short*>(out_bf16), status);
}

cudaError_t launch_grad_to_bf16_rows(const float* g, long long rows, int len, int pitch,
                                     void* out_bf16, uint32_t* status, cudaStream_t stream) {
  const long long want = (rows * (pitch >> 3) + 255) / 256;
  const long long cap = 16LL * sm_count();
  const int grid = static_cast<int>(want < 1 ? 1 : (want > cap ? cap : want));
  note_launches(1);
  return launch_kernel(grad_to_bf16_rows_kernel, dim3(grid), dim3(256), 0, stream, true, g, rows, len, pitch,
                       static_cast<unsigned short*>(out_bf16), status);
}

}  // namespace surgeon
