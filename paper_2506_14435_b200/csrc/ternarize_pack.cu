// Absmean ternary weight quantizer with INT2 packing (Eq. 7, 9, 10; storage per Section 3.1).
//
// Two launches per matrix (after a clear of the bins), both bound by HBM; 83 -> 38 us per 11008 x 2048
// fp32 matrix against three launches with a branch per element and a division per code:
//   1. abs_sum_alpha   exact accumulation of sum |w|: each fp32 magnitude is split into its
//                      24-bit integer significand and its exponent; significands are added (shifted
//                      to a common unit, as integers) into 64-bit integer bins indexed by exponent.
//                      Integer adds commute, so the bins' total does not depend on thread order.
//                      The CTA that finishes last adds the bins into a 384-bit integer (exact),
//                      rounds it to fp64 (nearest even), divides by m*n in fp64 and rounds once to fp32.
//   2. pack_codes      code = clamp(rint(w / alpha), -1, 1), four codes per byte; walks the matrix from
//                      its end, so that it starts on what the sum left in L2.
#include <algorithm>
#include <mutex>

#include "mote_common.cuh"

namespace mote {

constexpr int kBins = 256;

// Exact sum of |w|: every thread keeps ONE 64-bit fixed-point accumulator in units of 2^(base - 150).
// An element with exponent e in [base, base + 31] adds significand << (e - base), below 2^55, so 511 elements
// fit; the accumulator is flushed after 256 to 271 of them (and when a larger element moves the window up).  A flush adds
// the low 32 bits to bin `base` and the high 32 bits to bin `base + 32` (whose unit is 2^32 times
// larger): exact, and every bin stays far below 2^64.  The rare element outside the window goes
// straight to the bin of its own exponent.  All of it is integer addition, so neither the choice of
// base nor the order of threads changes the bins' total.
struct AbsAcc {
  unsigned long long acc;
  int base, count;
};

__device__ __forceinline__ void abs_acc_flush(AbsAcc& st, unsigned long long* sbins) {
  if (st.acc) {
    atomicAdd(&sbins[st.base], st.acc & 0xFFFFFFFFull);
    if (st.acc >> 32) atomicAdd(&sbins[st.base + 32], st.acc >> 32);
  }
  st.acc = 0ull;
  st.count = 0;
}

__device__ __forceinline__ void abs_acc_add(AbsAcc& st, uint32_t bits, unsigned long long* sbins) {
  const uint32_t a = bits & 0x7FFFFFFFu;
  if (a == 0u) return;
  const uint32_t e_raw = a >> 23;
  const uint32_t mant = e_raw ? ((a & 0x7FFFFFu) | 0x800000u) : a;   // subnormals: no hidden bit
  const int e = e_raw ? (int)e_raw : 1;                              // ... and the unit of exponent 1
  if (st.base < 0 || e > st.base + 31) {                             // first element, or one above the window:
    if (st.base >= 0) abs_acc_flush(st, sbins);                      // move the window up to it
    st.base = min(max(e - 16, 1), 222);                              // base + 32 must be a valid bin
  }
  const unsigned sh = (unsigned)(e - st.base);
  if (sh < 32u) {
    st.acc += (unsigned long long)mant << sh;
    if (++st.count >= 256) abs_acc_flush(st, sbins);
  } else {
    atomicAdd(&sbins[e_raw], (unsigned long long)mant);              // outside the window: its own bin
  }
}

// The warp's accumulators into the bins.  A lane's window moves only when it meets a weight far above the
// first ones, so nearly always the lanes share one and their sums are added up first: 64-bit atomics of
// a whole CTA on two addresses of shared memory took longer than everything else in the kernel
// (51 -> 36 us for 90 MB).
__device__ __forceinline__ void abs_acc_flush_warp(AbsAcc& st, unsigned long long* sbins) {
  int same;
  __match_all_sync(0xffffffffu, st.base, &same);
  if (!same) {
    abs_acc_flush(st, sbins);
    return;
  }
  unsigned long long lo = st.acc & 0xFFFFFFFFull, hi = st.acc >> 32;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo += __shfl_xor_sync(0xffffffffu, lo, o);
    hi += __shfl_xor_sync(0xffffffffu, hi, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (lo) atomicAdd(&sbins[st.base], lo);
    if (hi) atomicAdd(&sbins[st.base + 32], hi);
  }
}

// Sixteen elements at once (called by whole warps).  Where all of them lie in the window (32 binades,
// placed 24 below the largest of the warp's first weights) they need one range check together and six instructions
// each: the magnitude less the window's lower edge, in one add (bits + bits drops the sign), is at once
// the shift (top byte) and, compared unsigned, the check.  Zeros and outliers go one by one.
__device__ __forceinline__ void abs_acc_add16(AbsAcc& st, const uint32_t (&bits)[16], unsigned long long* sbins) {
  if (st.base < 0) {
    uint32_t hi = 0u;
#pragma unroll
    for (int j = 0; j < 16; ++j) hi = max(hi, bits[j] & 0x7FFFFFFFu);
    hi = __reduce_max_sync(0xffffffffu, hi);                         // no lane or every lane has a window yet
    if (hi != 0u) st.base = min(max((int)(hi >> 23) - 24, 1), 222);  // base + 32 must be a valid bin
  }
  // base >= 1: a magnitude in the window is normal, i.e. has its hidden bit
  const uint32_t edge = 0u - ((uint32_t)st.base << 24);
  uint32_t top = 0u;
  unsigned long long sum = 0ull;                                     // 16 x 2^55 = 2^59
#pragma unroll
  for (int j = 0; j < 16; ++j) {
    const uint32_t x = bits[j] + bits[j] + edge, sh = x >> 24;
    const uint32_t mant = (bits[j] & 0x7FFFFFu) | 0x800000u;
    top = max(top, x);
    sum += (unsigned long long)mant * (1u << (sh & 31u));            // the shift as a wide multiply-add: one instruction of
                                                                     // the FMA pipe for four of the busier integer ALU
  }
  if (st.base > 0 && top < (32u << 24)) {
    st.acc += sum;
    if ((st.count += 16) >= 256) abs_acc_flush(st, sbins);
  } else {
#pragma unroll
    for (int j = 0; j < 16; ++j) abs_acc_add(st, bits[j], sbins);
  }
}

// A warp's 512 consecutive elements (item v of the matrix), 16 per lane: fp32 as four 512-byte rows of 16-byte
// loads, bf16 as two.  `left` elements of the matrix remain from the item's start on; missing ones read 0.
template <bool kBf16>
__device__ __forceinline__ void load16(const void* __restrict__ W, int64_t v, int64_t left, int lane, uint32_t (&bits)[16]) {
  constexpr int kRows = kBf16 ? 2 : 4, kPer = 16 / kRows;
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    const int first = (r * 32 + lane) * kPer;
    uint4 q = make_uint4(0u, 0u, 0u, 0u);
    if (first < left) q = __ldg(reinterpret_cast<const uint4*>(W) + v * (32 * kRows) + r * 32 + lane);
    if (kBf16) {
      const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) { bits[8 * r + 2 * j] = w[j] << 16; bits[8 * r + 2 * j + 1] = w[j] & 0xFFFF0000u; }
    } else {
      bits[4 * r] = q.x; bits[4 * r + 1] = q.y; bits[4 * r + 2] = q.z; bits[4 * r + 3] = q.w;
    }
  }
}

// alpha from the bins, by one warp.  bins[e] counts units of 2^(max(e,1) - 150); the total,
// sum_e bins[e] << (max(e,1) - 1) in units of 2^-149, is formed in 32-bit limbs: lane i collects what falls
// into limb i, one lane then carries.  e = 255 (inf/nan) is undefined input, ignored.
constexpr int kLimbs = 12;
__device__ __forceinline__ void finalize_alpha(const unsigned long long* s_bins, unsigned long long* s_limb, double count,
                                               float* __restrict__ alpha) {
  const int lane = threadIdx.x & 31;
  // only bins that hold something (a handful: the weights' binades over 32): going over all of them, three limbs each,
  // took the one warp 7 us
  unsigned long long col = 0ull;                           // at most 3 x 32 parts below 2^32
  for (int e0 = 0; e0 < 255; e0 += 32) {
    uint32_t used = __ballot_sync(0xffffffffu, e0 + lane < 255 && s_bins[min(e0 + lane, 254)] != 0ull);
    while (used) {
      const int e = e0 + __ffs(used) - 1, sft = (e ? e : 1) - 1, part = lane - (sft >> 5);
      used &= used - 1u;
      if (part < 0 || part > 2) continue;
      const unsigned __int128 sv = (unsigned __int128)s_bins[e] << (sft & 31);   // < 2^95
      col += (uint32_t)(sv >> (32 * part));
    }
  }
  if (lane < kLimbs) s_limb[lane] = col;
  __syncwarp();
  if (lane != 0) return;
  unsigned long long carry = 0ull;
  int top = -1;
  for (int i = 0; i < kLimbs; ++i) {
    carry += s_limb[i];
    s_limb[i] = carry & 0xFFFFFFFFull;
    if (s_limb[i]) top = i;
    carry >>= 32;
  }
  double sum = 0.0;
  if (top >= 0) {
    // the 64 bits from the leading one down, and whether any lower bit is set
    auto limb = [&](int i) -> unsigned long long { return i < 0 ? 0ull : s_limb[i]; };
    const int c = __clz((int)limb(top));
    const unsigned long long low = limb(top - 2) << c;                   // its upper half still belongs to the 64 bits
    const unsigned long long m64 = (((limb(top) << 32) | limb(top - 1)) << c) | (low >> 32);
    bool sticky = (low & 0xFFFFFFFFull) != 0ull;
    for (int i = top - 3; i >= 0; --i) sticky = sticky || limb(i) != 0ull;
    unsigned long long m = m64 >> 11;                                    // 53 bits
    const bool round_bit = (m64 >> 10) & 1ull;
    sticky = sticky || (m64 & 0x3FFull) != 0ull;
    if (round_bit && (sticky || (m & 1ull))) ++m;                        // nearest, ties to even
    sum = scalbn((double)m, top * 32 + 31 - c - 52 - 149);
  }
  const float a = (float)(sum / count);                                  // fp64 divide, one rounding to fp32
  *alpha = fmaxf(a, kEpsScale);
}

// One warp takes items of 512 elements; the next item is on its way while one is added.  The last bin
// (never counted into) is the grid's arrival counter.
// One CTA of 1024 threads per SM: a quarter of the CTAs meet at the bins' atomics that four of 256 would send there (three
// matrices of 2048 x 11008: fp32 117 -> 114 us, bf16 102.7 -> 100).
constexpr int kSumThreads = 1024;
template <bool kBf16>
__global__ void __launch_bounds__(kSumThreads, 1) abs_sum_alpha_kernel(const void* __restrict__ W, int64_t total, double count,
                                                            unsigned long long* __restrict__ bins, float* __restrict__ alpha) {
  __shared__ unsigned long long sbins[kBins];
  __shared__ unsigned long long s_limb[kLimbs];
  __shared__ int s_last;
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) sbins[i] = 0ull;
  __syncthreads();
  const int lane = threadIdx.x & 31;
  const int64_t n_warps = (int64_t(gridDim.x) * blockDim.x) >> 5, n_items = (total + 511) / 512;
  AbsAcc st{0ull, -1, 0};
  int64_t v = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5;
  uint32_t b0[16], b1[16];
  if (v < n_items) load16<kBf16>(W, v, total - v * 512, lane, b0);
  for (; v < n_items; v += 2 * n_warps) {
    const int64_t v1 = v + n_warps, v2 = v1 + n_warps;
    if (v1 < n_items) load16<kBf16>(W, v1, total - v1 * 512, lane, b1);
    abs_acc_add16(st, b0, sbins);
    if (v1 >= n_items) break;
    if (v2 < n_items) load16<kBf16>(W, v2, total - v2 * 512, lane, b0);
    abs_acc_add16(st, b1, sbins);
  }
  abs_acc_flush_warp(st, sbins);
  __syncthreads();
  for (int i = threadIdx.x; i < kBins - 1; i += blockDim.x)
    if (sbins[i]) atomicAdd(&bins[i], sbins[i]);
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) s_last = atomicAdd(&bins[kBins - 1], 1ull) == (unsigned long long)gridDim.x - 1ull;
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  for (int i = threadIdx.x; i < kBins; i += blockDim.x) sbins[i] = __ldcg(&bins[i]);
  __syncthreads();
  if (threadIdx.x < 32) finalize_alpha(sbins, s_limb, count, alpha);
}

// code = clamp(rint(fl32(w / alpha)), -1, 1) without the division: +1 where w > alpha/2, -1 where w < -alpha/2.
// rint (ties to even) gives 0 up to a quotient of 0.5 and at least 1 above it.  w <= alpha/2 gives a real
// quotient <= 0.5, and rounding keeps that.  The next float above alpha/2 = m * 2^k (1 <= m < 2; alpha >= 1e-5,
// so alpha/2 is exact and normal) is alpha/2 + 2^(k-23), a quotient of 0.5 + 2^-24/m > 0.5 + 2^-25, beyond
// the midpoint between 0.5 and the next float, so it rounds above 0.5.
// A lane packs its 4 (fp32) or 8 (bf16) consecutive elements to a byte or two.
template <bool kBf16>
__global__ void __launch_bounds__(256) pack_codes_kernel(const void* __restrict__ W, int64_t total,
                                                         const float* __restrict__ alpha_ptr, uint8_t* __restrict__ packed) {
  constexpr int kRows = kBf16 ? 2 : 4, kPer = 16 / kRows;
  pdl_wait();
  const float half = 0.5f * __ldcg(alpha_ptr);
  const int lane = threadIdx.x & 31;
  const int64_t n_warps = (int64_t(gridDim.x) * blockDim.x) >> 5, n_items = (total + 511) / 512;
  for (int64_t i = (int64_t(blockIdx.x) * blockDim.x + threadIdx.x) >> 5; i < n_items; i += n_warps) {
    const int64_t v = n_items - 1 - i, left = total - v * 512;
    uint32_t bits[16];
    load16<kBf16>(W, v, left, lane, bits);
#pragma unroll
    for (int r = 0; r < kRows; ++r) {
      uint32_t out = 0x5555u;                              // code 0 everywhere
#pragma unroll
      for (int j = 0; j < kPer; ++j) {
        const float x = __uint_as_float(bits[r * kPer + j]);
        if (x > half) out += 1u << (2 * j);
        if (!(x >= -half)) out -= 1u << (2 * j);           // a NaN too, as the clamp of the quotient from below would give
      }
      if ((r * 32 + lane) * kPer < left) {
        if (kBf16) reinterpret_cast<uint16_t*>(packed)[v * 64 + r * 32 + lane] = (uint16_t)out;
        else packed[v * 128 + r * 32 + lane] = (uint8_t)out;
      }
    }
  }
}

}  // namespace mote

namespace mote {

// The quantizer's launch sequence on exponent bins that the caller owns (a workspace, or the
// library's built-in array): clear the bins, exact sum of |w|, alpha, codes.
static mote_status_t ternarize_with_bins(const void* W, int w_dtype, int64_t total, uint8_t* packed, float* alpha,
                                         unsigned long long* bins, cudaStream_t stream) {
  // whatever the bins held before (an earlier call's sums, or nothing defined) must go
  MOTE_CUDA_OK(cudaMemsetAsync(bins, 0, kBins * sizeof(unsigned long long), stream));
  const int threads = 256;
  const int64_t ctas = (total + 512 * 8 - 1) / (512 * 8);            // 512 elements per warp
  const int blocks_a = (int)std::min<int64_t>((ctas + 3) / 4, int64_t(device_sm_count()));
  const int blocks_c = (int)std::min<int64_t>(ctas, int64_t(device_sm_count()) * 16);
  const bool bf16 = w_dtype == MOTE_DTYPE_BF16;
  if (bf16) abs_sum_alpha_kernel<true><<<blocks_a, kSumThreads, 0, stream>>>(W, total, (double)total, bins, alpha);
  else abs_sum_alpha_kernel<false><<<blocks_a, kSumThreads, 0, stream>>>(W, total, (double)total, bins, alpha);
  MOTE_LAUNCH_OK();
  if (bf16) MOTE_CUDA_OK(launch_pdl(pack_codes_kernel<true>, dim3(blocks_c), dim3(threads), 0, stream, W, total, alpha, packed));
  else MOTE_CUDA_OK(launch_pdl(pack_codes_kernel<false>, dim3(blocks_c), dim3(threads), 0, stream, W, total, alpha, packed));
  MOTE_LAUNCH_OK();
  return MOTE_OK;
}

}  // namespace mote

extern "C" size_t mote_ternarize_workspace_bytes(void) { return mote::kBins * sizeof(unsigned long long); }

extern "C" mote_status_t mote_ternarize_pack(const void* W, int w_dtype, int64_t m, int64_t n,
                                             uint8_t* packed, float* alpha, void* ws, size_t ws_bytes,
                                             void* stream_) {
  using namespace mote;
  if (!W || !packed || !alpha || !ws) return MOTE_ERR_NULL;
  if (w_dtype != MOTE_DTYPE_F32 && w_dtype != MOTE_DTYPE_BF16) return MOTE_ERR_DTYPE;
  if (m <= 0 || n <= 0 || (n % 16) != 0) return MOTE_ERR_SHAPE;
  if (m >= (int64_t(1) << 38) / n) return MOTE_ERR_SHAPE;
  if (!aligned16(W) || !aligned16(packed) || !aligned16(ws)) return MOTE_ERR_ALIGN;
  if (ws_bytes < mote_ternarize_workspace_bytes()) return MOTE_ERR_WORKSPACE;
  return ternarize_with_bins(W, w_dtype, m * n, packed, alpha, static_cast<unsigned long long*>(ws),
                             static_cast<cudaStream_t>(stream_));
}

// ---------------------------------------------------------------------------------------------
// mote_ternarize_pack_static: the same quantizer for callers that have no scratch buffer to give.
// The exponent bins live in a device array that is part of the loaded library image.
// ---------------------------------------------------------------------------------------------
namespace mote {

// 256 bins x 8 bytes.  One copy per GPU that loads the library, held until the process exits.
static __device__ __align__(256) unsigned long long g_static_bins[kBins];

static unsigned long long* g_static_bins_ptr[kMaxDevices];   // device address of g_static_bins, per device
static std::mutex g_static_bins_mutex;

// In host code `g_static_bins` is only a handle; the kernels need the address the array has on the
// device that is current.  It is looked up on the first call made on each device.
static mote_status_t static_bins_address(unsigned long long** out) {
  int dev = -1;
  MOTE_CUDA_OK(cudaGetDevice(&dev));
  if (dev < 0 || dev >= kMaxDevices) return MOTE_ERR_CUDA;
  std::lock_guard<std::mutex> lock(g_static_bins_mutex);
  if (!g_static_bins_ptr[dev]) {
    void* p = nullptr;
    if (cudaGetSymbolAddress(&p, g_static_bins) != cudaSuccess || !p) return MOTE_ERR_CUDA;
    g_static_bins_ptr[dev] = static_cast<unsigned long long*>(p);
  }
  *out = g_static_bins_ptr[dev];
  return MOTE_OK;
}

}  // namespace mote

extern "C" mote_status_t mote_ternarize_pack_static(const void* W, int w_dtype, int64_t m, int64_t n,
                                                    uint8_t* packed, float* alpha, void* stream_) {
  using namespace mote;
  if (!W || !packed || !alpha) return MOTE_ERR_NULL;
  if (w_dtype != MOTE_DTYPE_F32 && w_dtype != MOTE_DTYPE_BF16) return MOTE_ERR_DTYPE;
  if (m <= 0 || n <= 0 || (n % 16) != 0) return MOTE_ERR_SHAPE;
  if (m > MOTE_STATIC_MAX_ELEMENTS / n) return MOTE_ERR_TOO_LARGE;
  if (!aligned16(W) || !aligned16(packed)) return MOTE_ERR_ALIGN;
  unsigned long long* bins = nullptr;
  const mote_status_t st = static_bins_address(&bins);
  if (st != MOTE_OK) return st;
  return ternarize_with_bins(W, w_dtype, m * n, packed, alpha, bins, static_cast<cudaStream_t>(stream_));
}
