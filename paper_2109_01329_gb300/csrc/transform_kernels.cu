// Distribution transform of caller-supplied words (grng_transform_words), the
// same transforms as the fused fill kernels: 4 words make 16 output bytes, so
// where the units line up with the output's 16-byte groups a thread takes
// whole groups, else one unit (one output, or one Box-Muller pair).
#include <cuda_runtime.h>

#include <cstdint>

#include "device_common.cuh"
#include "grng_internal.h"

namespace grng {
namespace {

using namespace dev;

constexpr int kThreads = 256;

// Unit k: its words, transformed, to its place in the output.
template <int V>
__device__ __forceinline__ void transform_unit(const TransformParams& t, const uint32_t* words,
                                               int64_t k, int64_t out_words, uint32_t* out) {
  using I = VInfo<V>;
  uint32_t w[I::wpu];
#pragma unroll
  for (int i = 0; i < I::wpu; ++i) w[i] = words[k * I::wpu + i];
  uint32_t o[I::wpu];
  // odd units take the other pipe's form as in the fill kernels (the same
  // bits), so this kernel checks both forms
  unit_outputs<V>(w, o, t, (k & 1) != 0);
#pragma unroll
  for (int i = 0; i < I::wpu; ++i) {
    const int64_t ow = k * I::wpu + i;  // 4 output bytes per word
    if (ow < out_words) out[ow] = o[i];
  }
}

// Units at any alignment.
template <int V>
__global__ void __launch_bounds__(kThreads) transform_kernel(TransformParams t, const uint32_t* words,
                                                             int64_t n, uint32_t* out) {
  using I = VInfo<V>;
  const int64_t units = (n + I::epu - 1) / I::epu;
  const int64_t out_words = n * I::ow_per_elem;
  for (int64_t k = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; k < units;
       k += (int64_t)gridDim.x * blockDim.x)
    transform_unit<V>(t, words, k, out_words, out);
}

// Whole 16-byte groups: units [head, head + groups upg) of the call, the output
// 16-byte aligned from unit head on.  kVec: the words there are too; else a
// thread's four words come in four loads, each coalesced across the warp in
// 16-byte strides.  The few units before and after go to the first CTA's
// first threads.
struct TransformParts {
  TransformParams t;
  const uint32_t* words;  // of unit 0
  uint32_t* out;
  int64_t units, out_words;
  int64_t head, groups;
};

// Groups in flight per thread.  Bound by the two passes over memory (10^8
// words in, 10^8 out: 118 us at the copy peak) up to the FP64 fixed-point
// transforms.  10^8 outputs, one unit per thread with 4-byte accesses -> now:
// bits 192 -> 118 us, FP32 gaussians 151 -> 118, FP32 inverse CDFs 209 -> 118, FP64
// uniforms 283 -> 232, FP64 gaussians 627 -> 532.  With one group per thread 122
// to 128 us, with one wave of CTAs 126 to 136.
template <int V>
constexpr int kGroups = VInfo<V>::weight == 0 ? 4 : VInfo<V>::weight == 1 ? 2 : 1;
constexpr int64_t kMaxCtasPerSm = 128;

template <int V, bool kVec>
__global__ void __launch_bounds__(kThreads) transform_groups_kernel(const __grid_constant__ TransformParts p) {
  using I = VInfo<V>;
  constexpr int U = kGroups<V>;
  constexpr int kUpg = 4 / I::wpu;
  if (blockIdx.x == 0) {
    const int64_t k = threadIdx.x < p.head ? threadIdx.x : p.groups * kUpg + threadIdx.x;
    if (threadIdx.x < p.head + kUpg && k < p.units)
      transform_unit<V>(p.t, p.words, k, p.out_words, p.out);
  }
  const uint32_t* words = p.words + p.head * I::wpu;
  uint4* out = reinterpret_cast<uint4*>(p.out + p.head * I::wpu);
  auto load = [&](int64_t g) {
    if constexpr (kVec) return __ldcs(reinterpret_cast<const uint4*>(words) + g);
    return make_uint4(words[4 * g], words[4 * g + 1], words[4 * g + 2], words[4 * g + 3]);
  };
  const int64_t step = (int64_t)gridDim.x * (kThreads * U);
  int64_t g = (int64_t)blockIdx.x * (kThreads * U) + threadIdx.x;
  for (; g + (U - 1) * kThreads < p.groups; g += step) {
    uint4 w[U];
#pragma unroll
    for (int u = 0; u < U; ++u) w[u] = load(g + u * kThreads);
#pragma unroll
    for (int u = 0; u < U; ++u) out[g + u * kThreads] = block_outputs<V>(w[u], p.t);
  }
  if constexpr (U > 1) {
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
      if (g + u * kThreads < p.groups) out[g + u * kThreads] = block_outputs<V>(load(g + u * kThreads), p.t);
  }
}

template <int V>
grng_status launch_v(const TransformParams& t, const uint32_t* words, int64_t n, void* out,
                     cudaStream_t stream) {
  using I = VInfo<V>;
  const int64_t units = (n + I::epu - 1) / I::epu;
  int dev = 0;
  const int sms = current_device_sms(&dev);
  const uint32_t phase = (uint32_t)(((uintptr_t)out & 15u) / 4u);  // output words past a group
  if (phase % (uint32_t)I::wpu == 0) {
    TransformParts p;
    p.t = t;
    p.words = words;
    p.out = reinterpret_cast<uint32_t*>(out);
    p.units = units;
    p.out_words = n * I::ow_per_elem;
    p.head = phase == 0 ? 0 : (int64_t)((4u - phase) / (uint32_t)I::wpu);
    const int64_t whole = n / I::epu;  // units all of whose outputs are wanted
    if (p.head > whole) p.head = whole;
    p.groups = (whole - p.head) / (4 / I::wpu);
    constexpr int64_t kTile = (int64_t)kThreads * kGroups<V>;
    int64_t grid = (p.groups + kTile - 1) / kTile;
    if (grid < 1) grid = 1;
    if (grid > sms * kMaxCtasPerSm) grid = sms * kMaxCtasPerSm;
    if (((uintptr_t)(words + p.head * I::wpu) & 15u) == 0) {
      transform_groups_kernel<V, true><<<(unsigned)grid, kThreads, 0, stream>>>(p);
    } else {
      transform_groups_kernel<V, false><<<(unsigned)grid, kThreads, 0, stream>>>(p);
    }
  } else {
    int64_t grid = (units + kThreads - 1) / kThreads;
    if (grid > (int64_t)sms * 8) grid = (int64_t)sms * 8;
    transform_kernel<V><<<(unsigned)grid, kThreads, 0, stream>>>(t, words, n,
                                                                 reinterpret_cast<uint32_t*>(out));
  }
  const cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) {
    set_error("transform launch failed: %s", cudaGetErrorString(err));
    return GRNG_ERR_CUDA;
  }
  return GRNG_OK;
}

}  // namespace

grng_status launch_transform(int variant, const TransformParams& t, const uint32_t* words,
                             int64_t n, void* out, CUstream_st* stream) {
  switch (variant) {
    case V_BITS: return launch_v<V_BITS>(t, words, n, out, stream);
    case V_U01_F32: return launch_v<V_U01_F32>(t, words, n, out, stream);
    case V_UNI_F32: return launch_v<V_UNI_F32>(t, words, n, out, stream);
    case V_U01_F64: return launch_v<V_U01_F64>(t, words, n, out, stream);
    case V_AFF_F64: return launch_v<V_AFF_F64>(t, words, n, out, stream);
    case V_UNI_F64: return launch_v<V_UNI_F64>(t, words, n, out, stream);
    case V_GAUSS_F32: return launch_v<V_GAUSS_F32>(t, words, n, out, stream);
    case V_LOGN_F32: return launch_v<V_LOGN_F32>(t, words, n, out, stream);
    case V_GAUSS_F64: return launch_v<V_GAUSS_F64>(t, words, n, out, stream);
    case V_LOGN_F64: return launch_v<V_LOGN_F64>(t, words, n, out, stream);
    case V_ICDF_GAUSS_F32: return launch_v<V_ICDF_GAUSS_F32>(t, words, n, out, stream);
    case V_ICDF_LOGN_F32: return launch_v<V_ICDF_LOGN_F32>(t, words, n, out, stream);
    case V_ICDF_GAUSS_F64: return launch_v<V_ICDF_GAUSS_F64>(t, words, n, out, stream);
    case V_ICDF_LOGN_F64: return launch_v<V_ICDF_LOGN_F64>(t, words, n, out, stream);
    case V_STDGAUSS_F64: return launch_v<V_STDGAUSS_F64>(t, words, n, out, stream);
    default: set_error("unknown variant %d", variant); return GRNG_ERR_INVALID_ARG;
  }
}

}  // namespace grng
