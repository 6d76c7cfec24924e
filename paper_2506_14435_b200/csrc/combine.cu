// Gate-weighted combine and un-permute (Eq. 2, Eq. 4), gather form (no atomics, deterministic):
//   out[t,:] = bf16( [residual[t,:] +] s[t,:] + sum_{j<k} w[t,j] * y[perm[t*k+j], :] )
// (s may arrive as the partial sums of a K-split down projection, added here in ascending order)
// fp32 arithmetic, slots added in ascending j, one bf16 rounding at the end.
// HBM-bound: per output element 4 B (s) + 4k B (y) [+ 2 B residual] read, 2 B written.
#include "mote_common.cuh"
#include "mote_internal.h"

namespace mote {

// Short prefills (many partial sums of few rows) are bound by the latency of the loads and by how many are in flight: a
// thread owns four columns (twice the CTAs of eight) and asks for kBatch partial sums at a time and for two expert rows
// ahead of them.  The CUDA-core path (one sum, any number of rows) and the longer of the short prefills (two to four) are
// bound by HBM and need the warps instead, so kBatch is no larger than the number of sums: 40, 56, 76 and 99 registers.
// One kernel of eight for all (99 registers, two CTAs per SM): 44 -> 107 us for 8192 x 2048, one sum, k = 2; with kBatch 1: 46.
// Two sums of 1024 rows at 2048 x 5632, 16 experts (the whole layer): 219 us with batches of eight, 211 with this.
__device__ __forceinline__ void add4(float (&acc)[4], const float4& a) { acc[0] += a.x; acc[1] += a.y; acc[2] += a.z; acc[3] += a.w; }
__device__ __forceinline__ void fma4(float (&acc)[4], float w, const float4& a) {
  acc[0] = fmaf(w, a.x, acc[0]); acc[1] = fmaf(w, a.y, acc[1]); acc[2] = fmaf(w, a.z, acc[2]); acc[3] = fmaf(w, a.w, acc[3]);
}

template <int kBatch>
__global__ void __launch_bounds__(256) combine_kernel(const float* __restrict__ s, const float* __restrict__ y,
                                                      const float* __restrict__ w, const int32_t* __restrict__ perm,
                                                      const uint16_t* residual, int64_t T, int d, int k,
                                                      uint16_t* out, int n_partials) {
  constexpr int kEarly = 2;
  const int vec_per_row = d / 4;
  const int64_t total = T * vec_per_row;
  pdl_wait();                            // no-op unless launched as a programmatic dependent
  const int64_t stride = int64_t(gridDim.x) * blockDim.x;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < total; i += stride) {
    const int64_t t = i / vec_per_row;
    const int v = (int)(i - t * vec_per_row);
    float wj[kEarly];
    float4 yj[kEarly];
#pragma unroll
    for (int j = 0; j < kEarly; ++j)
      if (j < k) {
        wj[j] = w[t * k + j];
        yj[j] = *reinterpret_cast<const float4*>(y + int64_t(perm[t * k + j]) * d + v * 4);
      }
    float acc[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    const float* sp = s + t * d + v * 4;
#pragma unroll 1
    for (int p0 = 0; p0 < n_partials; p0 += kBatch) {   // partial sums of a K-split projection, in order
      float4 sv[kBatch];
#pragma unroll
      for (int p = 0; p < kBatch; ++p)
        if (p0 + p < n_partials) sv[p] = *reinterpret_cast<const float4*>(sp + int64_t(p0 + p) * T * d);
#pragma unroll
      for (int p = 0; p < kBatch; ++p) {
        if (p0 + p == 0) { acc[0] = sv[0].x; acc[1] = sv[0].y; acc[2] = sv[0].z; acc[3] = sv[0].w; }
        else if (p0 + p < n_partials) add4(acc, sv[p]);
      }
    }
#pragma unroll
    for (int j = 0; j < kEarly; ++j)
      if (j < k) fma4(acc, wj[j], yj[j]);
    for (int j = kEarly; j < k; ++j) fma4(acc, w[t * k + j], *reinterpret_cast<const float4*>(y + int64_t(perm[t * k + j]) * d + v * 4));
    if (residual) {
      const uint2 r = *reinterpret_cast<const uint2*>(residual + t * d + v * 4);
      acc[0] += bf16_lo(r.x); acc[1] += bf16_hi(r.x); acc[2] += bf16_lo(r.y); acc[3] += bf16_hi(r.y);
    }
    *reinterpret_cast<uint2*>(out + t * d + v * 4) =
        make_uint2(f32_to_bf16_bits(acc[0]) | (f32_to_bf16_bits(acc[1]) << 16), f32_to_bf16_bits(acc[2]) | (f32_to_bf16_bits(acc[3]) << 16));
  }
}

mote_status_t launch_combine(const float* s, const float* y, const float* w, const int32_t* perm,
                             const void* residual, int64_t T, int d, int k, void* out_bf16, cudaStream_t stream,
                             bool pdl, int n_partials) {
  if (T == 0) return MOTE_OK;
  const int64_t total = T * (d / 4);
  const unsigned blocks = (unsigned)std::min<int64_t>((total + 255) / 256, 148 * 16);
#define MOTE_COMBINE_LAUNCH(B_)                                                                                       \
  do {                                                                                                               \
    if (pdl)                                                                                                         \
      MOTE_CUDA_OK(launch_pdl(combine_kernel<B_>, dim3(blocks), dim3(256), 0, stream, s, y, w, perm,                 \
                              static_cast<const uint16_t*>(residual), T, d, k, static_cast<uint16_t*>(out_bf16),     \
                              n_partials));                                                                          \
    else                                                                                                             \
      combine_kernel<B_><<<blocks, 256, 0, stream>>>(s, y, w, perm, static_cast<const uint16_t*>(residual), T, d, k, \
                                                     static_cast<uint16_t*>(out_bf16), n_partials);                  \
  } while (0)
  if (n_partials <= 1) MOTE_COMBINE_LAUNCH(1);
  else if (n_partials <= 2) MOTE_COMBINE_LAUNCH(2);
  else if (n_partials <= 4) MOTE_COMBINE_LAUNCH(4);
  else MOTE_COMBINE_LAUNCH(8);
#undef MOTE_COMBINE_LAUNCH
  ++g_launch_count;
  MOTE_LAUNCH_OK();
  return MOTE_OK;
}

}  // namespace mote
