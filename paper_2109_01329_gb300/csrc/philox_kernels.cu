// Philox4x32-10 fill kernels with the distribution transform fused in.
//
// The paper's path is two kernels: the vendor generator writes raw uniforms,
// then a SYCL kernel re-reads and rewrites the buffer to apply the range
// (Sec. 4.3, Listings 1 and 2; profiled as separate kernels in Sec. 7, Fig. 4).
// Here one kernel computes each counter block in registers, transforms it and
// stores it once: 4 output bytes per word and no reads.
//
// Output is cut into 16-byte groups at 16-byte aligned addresses.  Every
// variant consumes exactly 4 words per 16 output bytes, so:
//   * stream / multi kernels: when the word phase of the first group matches
//     its block boundary (and Box-Muller pairs do not straddle groups), group
//     j is exactly Philox block base + j: one block, one transform, one
//     st.v4.  Only the first and the last group of a stream may be partial.
//   * shift kernel (one stream at any other phase): group j is the tail of
//     block base + j and the head of block base + j + 1; a warp computes 32
//     consecutive blocks and emits 31 groups, exchanging the words between
//     neighbouring lanes by shuffle.  When the output's start splits a
//     Box-Muller pair, lanes transform pair-aligned groups one element
//     earlier and exchange the straddling element too (30 groups per warp).
//   * pieces kernel (one stream of 2- or 4-word units at a word offset that
//     keeps them inside blocks, the output start at another 16-byte phase):
//     each lane transforms its own block and stores it in 4- and 8-byte
//     pieces; the FP64 uniforms, near the write roof, rotate their outputs into
//     whole groups by shuffle instead (rotate kernel).
//   * multi-shift kernel: substreams at another phase or alignment, the
//     shift kernel's exchange applied per stream (a warp works on 30 groups
//     of one stream).
// Both write every output exactly once; results do not depend on the launch
// geometry (each output is a function of its word index only).
#include <cuda_runtime.h>

#include <atomic>

#include <cstdint>

#include "device_common.cuh"
#include "grng_internal.h"

namespace grng {
namespace {

using namespace dev;

constexpr int kThreads = 256;

__device__ __forceinline__ void add128(uint64_t& lo, uint64_t& hi, uint64_t vlo, uint64_t vhi) {
  const uint64_t s = lo + vlo;
  hi += vhi + ((s < lo) ? 1u : 0u);
  lo = s;
}

// Stores the in-range elements of a partial group whose first element is e0.
template <int V>
__device__ __forceinline__ void store_partial(char* stream_base, int64_t e0, int64_t n, uint4 o) {
  using I = VInfo<V>;
  constexpr int kEpg = 16 / I::es;
  const uint32_t ow[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
  for (int i = 0; i < kEpg; ++i) {
    const int64_t e = e0 + i;
    if (e >= 0 && e < n) {
      if constexpr (I::es == 4) {
        reinterpret_cast<uint32_t*>(stream_base)[e] = ow[i];
      } else {
        reinterpret_cast<uint2*>(stream_base)[e] = make_uint2(ow[2 * i], ow[2 * i + 1]);
      }
    }
  }
}

// ------------------------------------------------------------ single stream
// Full 16-byte groups [jf, jl) in the main loop, U independent counter blocks
// per thread per iteration (stores of the U blocks are each coalesced across
// the warp).  The at most two partial groups (the first and the last) are done
// by the grid's first two threads before the loop.
//
// Bound by the FMA-heavy pipe (the products) until it meets the write roof:
// with 18 products, each one wide multiply, a bits block costs 44 instructions
// of 55 before, and the contiguous tiles keep a CTA's stores together (grid-
// strided: bits 0.541 ms).  10^9 outputs, before -> now: bits 0.602 -> 0.531 ms
// (7.53 TB/s), FP32 uniforms 0.665 -> 0.594, FP64 uniforms 1.650 -> 1.41, FP32
// gaussians 1.351 -> 1.10 (1.22 with the f32x2 polynomials alone), FP64
// gaussians 6.26 -> 6.10 (5.69 with the pair reworked after it).
struct StreamParams {
  TransformParams t;
  uint4* gbase;       // 16-byte aligned address of group 0 (may precede out)
  void* out;
  int64_t n;          // elements
  int64_t head;       // elements of group 0 that lie before out
  uint32_t jf, jl;    // full groups [jf, jl)
  int64_t edge[2];    // partial groups, or -1
  PhiloxStream ctr;   // block 0: that of group 0
};

template <int V, int U, bool kCross>
__device__ __forceinline__ void philox_stream_body(const StreamParams& p) {
  using I = VInfo<V>;
  constexpr int kEpg = 16 / I::es;
  const uint32_t tid = blockIdx.x * kThreads + threadIdx.x;
  if (tid < 2 && p.edge[tid] >= 0) {
    const int64_t j = p.edge[tid];
    const uint4 o = block_outputs<V>(philox_block<true>((uint32_t)j, p.ctr), p.t);
    store_partial<V>(reinterpret_cast<char*>(p.out), j * kEpg - p.head, p.n, o);
  }
  // a CTA's tile is U x kThreads consecutive groups, thread t's at t, t +
  // kThreads, ...: constant store offsets and counter steps
  const uint32_t step = gridDim.x * (kThreads * U);
  uint32_t j = p.jf + blockIdx.x * (kThreads * U) + threadIdx.x;
  uint4* dst = p.gbase + j;
  for (; j + (U - 1) * kThreads < p.jl; j += step, dst += step) {
    uint4 o[U];
#pragma unroll
    for (int u = 0; u < U; ++u) o[u] = block_outputs<V>(philox_block<kCross>(j + u * kThreads, p.ctr), p.t);
#pragma unroll
    for (int u = 0; u < U; ++u) dst[u * kThreads] = o[u];
  }
  if constexpr (U > 1) {
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
      if (j + u * kThreads < p.jl)
        dst[u * kThreads] = block_outputs<V>(philox_block<kCross>(j + u * kThreads, p.ctr), p.t);
  }
}

// Counter blocks per thread per loop iteration: six for bits and the FP32
// uniforms, near the write roof (10^9 uniforms at 1, 2, 4, 6, 8: 0.642, 0.607,
// 0.605, 0.594, 0.590 ms), two for the FP32 Box-Muller and inverse CDF (10^9
// gaussians 1.095 ms; 1: 1.111), one for the 8-byte outputs, whose transform is
// long enough by itself (10^9 FP64 uniforms 1.405 ms; 2: 1.449).
template <int V>
constexpr int blocks_per_thread() {
  return (V == V_BITS || V == V_U01_F32 || V == V_UNI_F32) ? 6 : VInfo<V>::es == 8 ? 1 : 2;
}

// Substream tiles: eight for bits and the FP32 uniforms (16384 x 16384 uniforms
// at 4, 6, 8: 169.2, 170.9, 168.8 us), the others as above.
template <int V>
constexpr int multi_blocks_per_thread() {
  return (V == V_BITS || V == V_U01_F32 || V == V_UNI_F32) ? 8 : blocks_per_thread<V>();
}
constexpr int64_t kMultiTile = 16 * kThreads;  // groups; at most (8: 5 % slower, 32: idle SMs)

// In the kernels that exchange between lanes the [0, 1) and exact FP64 uniforms
// take two (10^8 at word offset 1: 0.223 ms against 0.226 with one).
template <int V>
constexpr int exchange_blocks_per_thread() {
  return V == V_U01_F64 || V == V_AFF_F64 ? 2 : blocks_per_thread<V>();
}

// The Box-Muller and FP32 inverse-CDF variants gain from a fifth resident CTA
// per SM (registers capped near 51: 1-5 % faster); the light variants keep
// the compiler's own register choice, which a CTA minimum would change.
template <int V>
constexpr bool stream_wants_5_ctas() {
  return V == V_GAUSS_F32 || V == V_LOGN_F32 || V == V_ICDF_GAUSS_F32 || V == V_GAUSS_F64 ||
         V == V_STDGAUSS_F64 || V == V_LOGN_F64 || V == V_ICDF_GAUSS_F64 || V == V_ICDF_LOGN_F64;
}

template <int V, int U, bool kCross>
__global__ void __launch_bounds__(kThreads) philox_stream_kernel(const __grid_constant__ StreamParams p) {
  philox_stream_body<V, U, kCross>(p);
}

template <int V, int U, bool kCross>
__global__ void __launch_bounds__(kThreads, 5) philox_stream_kernel_5(const __grid_constant__ StreamParams p) {
  philox_stream_body<V, U, kCross>(p);
}

// ------------------------------------------------------ single stream, shifted
// The same groups when the word offset is not on a block boundary (phase
// ph = 1..3 after removing the head words): group j is the last 4 - ph words
// of block base + j and the first ph words of block base + j + 1.  Each warp
// computes 32 consecutive blocks and emits the 31 groups that start in its
// lanes 0..30, taking the next block's words from lane + 1 by shuffle, so a
// group still costs 32/31 of a block and no shared memory or barrier.  U
// chunks of groups per warp per iteration, as U blocks per thread above.
//
// kSplit: the output's start splits a Box-Muller pair (odd head).  Lane l
// then transforms the pair-aligned "virtual" group that starts one element
// earlier (its words found as above, for any phase), and output group j is
// virtual group j without its first element plus the first element of
// virtual group j + 1, taken from lane + 1: 30 groups per warp, every pair
// transformed once.
struct ShiftParams {
  TransformParams t;
  uint4* gbase;       // 16-byte aligned address of group 0 (may precede out)
  void* out;
  int64_t n;          // elements
  int64_t head;       // elements of group 0 that lie before out
  int64_t groups;
  int64_t jf, jl;     // groups [jf, jl) lie wholly inside the output
  int64_t chunks;     // ceil(groups / groups per warp chunk)
  PhiloxStream ctr;   // block 0: that of the first word of (virtual) group 0
  uint32_t ph;        // its word phase: 1..3, or 0..3 with kSplit
};

template <bool kSplit>
__host__ __device__ constexpr int shift_per_warp() {
  return kSplit ? 30 : 31;
}

// The 4 words of a group whose first word is at phase kPh (1..3) of block b
// (this lane's), the rest from the next lane's block; kPh a constant, so only
// the kPh words needed cross lanes.
template <int kPh>
__device__ __forceinline__ uint4 shift_words_c(uint4 b) {
  const uint32_t n0 = __shfl_down_sync(0xFFFFFFFFu, b.x, 1);
  if constexpr (kPh == 1) {
    return make_uint4(b.y, b.z, b.w, n0);
  } else {
    const uint32_t n1 = __shfl_down_sync(0xFFFFFFFFu, b.y, 1);
    if constexpr (kPh == 2) {
      return make_uint4(b.z, b.w, n0, n1);
    } else {
      const uint32_t n2 = __shfl_down_sync(0xFFFFFFFFu, b.z, 1);
      return make_uint4(b.w, n0, n1, n2);
    }
  }
}

// The same with the phase ph known only at run time (warp-uniform).
__device__ __forceinline__ uint4 shift_words(uint4 b, uint32_t ph) {
  const uint32_t n0 = __shfl_down_sync(0xFFFFFFFFu, b.x, 1);
  const uint32_t n1 = __shfl_down_sync(0xFFFFFFFFu, b.y, 1);
  const uint32_t n2 = __shfl_down_sync(0xFFFFFFFFu, b.z, 1);
  if (ph == 1) return make_uint4(b.y, b.z, b.w, n0);
  if (ph == 2) return make_uint4(b.z, b.w, n0, n1);
  if (ph == 3) return make_uint4(b.w, n0, n1, n2);
  return b;
}

// Output group from this lane's transformed virtual group v and the next
// lane's first element (a Box-Muller pair split by the output's start).
template <int V>
__device__ __forceinline__ uint4 split_group(uint4 v) {
  const uint32_t m0 = __shfl_down_sync(0xFFFFFFFFu, v.x, 1);
  const uint32_t m1 = __shfl_down_sync(0xFFFFFFFFu, v.y, 1);
  return VInfo<V>::es == 4 ? make_uint4(v.y, v.z, v.w, m0) : make_uint4(v.z, v.w, m0, m1);
}

// kPh: the word phase as a constant (1..3), or -1 to read it from p.ph.
template <int V, int U, bool kCross, bool kSplit, int kPh>
__device__ __forceinline__ void philox_shift_body(const ShiftParams& p) {
  using I = VInfo<V>;
  constexpr int kEpg = 16 / I::es;
  constexpr int kPer = shift_per_warp<kSplit>();
  const int lane = threadIdx.x & 31;
  const int64_t TW = (int64_t)gridDim.x * (kThreads / 32);
  const int64_t c0 = ((int64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * U;
  // a warp takes U consecutive chunks; this lane's group of chunk c is j =
  // c kPer + lane, and those of the U chunks lie at constant offsets
  const int64_t dj = TW * kPer;
  int64_t j = c0 * kPer + lane;
  uint4* dst = p.gbase + j;
  // the loop bound depends only on the warp: every shuffle has all 32 lanes
  for (int64_t c = c0; c < p.chunks; c += U * TW, j += U * dj, dst += U * dj) {
    uint4 b[U];
#pragma unroll
    for (int u = 0; u < U; ++u) b[u] = philox_block<kCross>((uint32_t)j + u * kPer, p.ctr);
    // every group of this iteration lies wholly inside the output (uniform)
    const bool interior = c * kPer >= p.jf && (c + U) * kPer <= p.jl;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      uint4 w;
      if constexpr (kPh < 0) {
        w = shift_words(b[u], p.ph);
      } else {
        w = shift_words_c<kPh>(b[u]);
      }
      // every lane transforms its (virtual) group; in split mode lane l + 1's
      // first element is needed by lane l
      uint4 o = block_outputs<V>(w, p.t);
      if constexpr (kSplit) o = split_group<V>(o);
      if (interior) {
        if (lane < kPer) dst[u * kPer] = o;
      } else {
        const int64_t ju = j + u * kPer;
        if (lane < kPer && ju < p.groups) {
          const int64_t e0 = ju * kEpg - p.head;
          if (e0 >= 0 && e0 + kEpg <= p.n) {
            dst[u * kPer] = o;
          } else {
            store_partial<V>(reinterpret_cast<char*>(p.out), e0, p.n, o);
          }
        }
      }
    }
  }
}

// The phase is the same for the whole grid.  Raw bits take one loop per
// phase, each with the phase a constant (n = 10^9 at phases 1, 2, 3: 0.638,
// 0.630, 0.640 ms against 0.682, 0.677, 0.746 with the phase a variable).  The
// FP32 uniforms take the constant form for phases 2 and 3 (0.706, 0.715 ms
// against 0.761, 0.814).  Their phase 1 keeps the variable form, from loops with
// 64-bit counters, where the constant one was 10 % slower; in the present ones it
// would be the faster (0.706 ms against 0.743).  The other variants keep the
// variable phase.
template <int V, int U, bool kCross, bool kSplit>
__device__ __forceinline__ void philox_shift_phases(const ShiftParams& p) {
  if constexpr (V == V_BITS && !kSplit) {
    switch (p.ph) {
      case 1: philox_shift_body<V, U, kCross, kSplit, 1>(p); break;
      case 2: philox_shift_body<V, U, kCross, kSplit, 2>(p); break;
      default: philox_shift_body<V, U, kCross, kSplit, 3>(p); break;
    }
  } else if constexpr ((V == V_U01_F32 || V == V_UNI_F32) && !kSplit) {
    switch (p.ph) {
      case 2: philox_shift_body<V, U, kCross, kSplit, 2>(p); break;
      case 3: philox_shift_body<V, U, kCross, kSplit, 3>(p); break;
      default: philox_shift_body<V, U, kCross, kSplit, -1>(p); break;
    }
  } else {
    philox_shift_body<V, U, kCross, kSplit, -1>(p);
  }
}

template <int V, int U, bool kCross, bool kSplit>
__global__ void __launch_bounds__(kThreads) philox_shift_kernel(const __grid_constant__ ShiftParams p) {
  philox_shift_phases<V, U, kCross, kSplit>(p);
}

template <int V, int U, bool kCross, bool kSplit>
__global__ void __launch_bounds__(kThreads, 5) philox_shift_kernel_5(const __grid_constant__ ShiftParams p) {
  philox_shift_phases<V, U, kCross, kSplit>(p);
}

// ----------------------------------- single stream, whole units, another phase
// One stream whose units lie inside counter blocks (the word offset a multiple
// of the words per unit) while its output start is not at the blocks' 16-byte
// phase.  Block j's four output words are then output words 4 j - r .. 4 j -
// r + 3 (r = word offset mod 4).
struct PiecesParams {
  TransformParams t;
  uint4* gbase;       // out's 16-byte group
  char* out;          // element 0
  int64_t nw;         // output words: n es / 4
  int64_t h;          // output words of out's group before out
  int64_t r;          // word offset mod 4
  int64_t gofs;       // the group lane l completes is out's group + j + gofs (0 or -1)
  int64_t chunks;     // ceil(blocks / 32)
  PhiloxStream ctr;   // block 0: that of the stream's first word
};

__device__ __forceinline__ uint32_t word_of(uint4 v, int q) {
  return q == 0 ? v.x : q == 1 ? v.y : q == 2 ? v.z : v.w;
}

// Each lane stores its own block in pieces of 8 (kOdd: 4, 8, 4) bytes, back to
// back, and the pieces of a sector meet in L2.  Blocks [jf, jl) lie wholly inside
// the output; the at most two others are checked word by word.  10^8 FP32
// gaussians 117 to 119 us at the three phases against 114 aligned, where
// rotating them into whole groups by shuffle took 131 and 136; FP64 gaussians 574
// against 660.
template <bool kOdd>
__device__ __forceinline__ void store_pieces(uint32_t* d, uint4 o) {
  if constexpr (kOdd) {
    d[0] = o.x;
    *reinterpret_cast<uint2*>(d + 1) = make_uint2(o.y, o.z);
    d[3] = o.w;
  } else {
    *reinterpret_cast<uint2*>(d) = make_uint2(o.x, o.y);
    *reinterpret_cast<uint2*>(d + 2) = make_uint2(o.z, o.w);
  }
}

template <int V, int U, bool kCross, bool kOdd>
__device__ __forceinline__ void philox_pieces_body(const PiecesParams& p) {
  uint32_t* out = reinterpret_cast<uint32_t*>(p.out) - p.r;  // block j's words at 4 j
  const uint32_t jf = p.r > 0 ? 1u : 0u, jl = (uint32_t)((p.nw + p.r) / 4);
  const uint32_t tid = blockIdx.x * kThreads + threadIdx.x;
  if (tid < 2) {
    const uint32_t j = tid == 0 ? 0u : jl;
    if ((tid == 0 ? jf > 0 : 4 * (int64_t)jl - p.r < p.nw) && (tid == 0 || jl > 0 || jf == 0)) {
      const uint4 o = block_outputs<V>(philox_block<true>(j, p.ctr), p.t);
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int64_t i = 4 * (int64_t)j + q - p.r;
        if (i >= 0 && i < p.nw) out[4 * (int64_t)j + q] = word_of(o, q);
      }
    }
  }
  const uint32_t step = gridDim.x * (kThreads * U);
  uint32_t j = jf + blockIdx.x * (kThreads * U) + threadIdx.x;
  uint32_t* dst = out + 4 * (int64_t)j;
  for (; j + (U - 1) * kThreads < jl; j += step, dst += 4 * (int64_t)step) {
    uint4 o[U];
#pragma unroll
    for (int u = 0; u < U; ++u) o[u] = block_outputs<V>(philox_block<kCross>(j + u * kThreads, p.ctr), p.t);
#pragma unroll
    for (int u = 0; u < U; ++u) store_pieces<kOdd>(dst + 4 * u * kThreads, o[u]);
  }
  if constexpr (U > 1) {
#pragma unroll
    for (int u = 0; u < U - 1; ++u)
      if (j + u * kThreads < jl)
        store_pieces<kOdd>(dst + 4 * u * kThreads,
                           block_outputs<V>(philox_block<kCross>(j + u * kThreads, p.ctr), p.t));
  }
}

template <int V, int U, bool kCross>
__device__ __forceinline__ void philox_pieces_phases(const PiecesParams& p) {
  if (VInfo<V>::es == 8 || ((p.h - p.r) & 1) == 0) {
    philox_pieces_body<V, U, kCross, false>(p);
  } else {
    philox_pieces_body<V, U, kCross, true>(p);
  }
}

template <int V, int U, bool kCross>
__global__ void __launch_bounds__(kThreads) philox_pieces_kernel(const __grid_constant__ PiecesParams p) {
  philox_pieces_phases<V, U, kCross>(p);
}

template <int V, int U, bool kCross>
__global__ void __launch_bounds__(kThreads, 5) philox_pieces_kernel_5(const __grid_constant__ PiecesParams p) {
  philox_pieces_phases<V, U, kCross>(p);
}

// The FP64 uniforms: a block's second double opens the next 16-byte group, so
// each lane completes its group from lane - 1's by shuffle; lane 0 stores only
// its own half of its group and lane 31 the opening half of the next, so a warp
// writes 32 groups per 32 blocks (10^8 172 us; in 8-byte pieces 188).
template <int V, int U, bool kCross>
__global__ void __launch_bounds__(kThreads) philox_rotate_kernel(const __grid_constant__ PiecesParams p) {
  static_assert(VInfo<V>::es == 8 && VInfo<V>::wpu == 2);
  const int lane = threadIdx.x & 31;
  const int64_t TW = (int64_t)gridDim.x * (kThreads / 32);
  const int64_t c0 = ((int64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5)) * U;
  // a warp takes U consecutive chunks; lane l of chunk c holds block j =
  // 32 c + l, and those of the U chunks lie at constant offsets
  const int64_t dj = TW * 32;
  int64_t j = c0 * 32 + lane;
  uint4* dst = p.gbase + (j + p.gofs);
  // the loop bound depends only on the warp: every shuffle has all 32 lanes
  for (int64_t c = c0; c < p.chunks; c += U * TW, j += U * dj, dst += U * dj) {
    uint4 b[U];
#pragma unroll
    for (int u = 0; u < U; ++u) b[u] = philox_block<kCross>((uint32_t)j + u * 32, p.ctr);
    // every output word of this iteration's chunks lies inside the output
    // (uniform): words 128 c - r .. 128 (c + U) - 1 - r
    const bool interior = c * 128 - p.r >= 0 && (c + U) * 128 - 1 - p.r < p.nw;
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint4 o = block_outputs<V>(b[u], p.t);
      const uint32_t n2 = __shfl_up_sync(0xFFFFFFFFu, o.z, 1);
      const uint32_t n3 = __shfl_up_sync(0xFFFFFFFFu, o.w, 1);
      if (interior) {
        uint4* gp = dst + u * 32;
        if (lane > 0) {
          *gp = make_uint4(n2, n3, o.x, o.y);
        } else {
          reinterpret_cast<uint2*>(gp)[1] = make_uint2(o.x, o.y);
        }
        if (lane == 31) *reinterpret_cast<uint2*>(gp + 1) = make_uint2(o.z, o.w);
      } else {  // each of the block's two doubles checked
        const int64_t e = (4 * (j + u * 32) - p.r) >> 1;
        uint2* out = reinterpret_cast<uint2*>(p.out);
        if (e >= 0 && 2 * e < p.nw) out[e] = make_uint2(o.x, o.y);
        if (e + 1 >= 0 && 2 * (e + 1) < p.nw) out[e + 1] = make_uint2(o.z, o.w);
      }
    }
  }
}

// ------------------------------------------------------------ substreams
// num_streams streams whose every group is full (16-byte aligned streams of
// whole groups); stream s, group j is block base + s * sb + j.
struct MultiParams {
  TransformParams t;
  uint4* out;
  int64_t groups;     // groups per stream
  int64_t total;      // groups * num_streams
  uint64_t base_lo, base_hi;
  uint64_t sb_lo, sb_hi;      // block-counter stride between streams
  int64_t tq, tr;             // grid stride = tq * groups + tr
  uint64_t tqsb_lo, tqsb_hi;  // tq * sb
  PhiloxRoundKeys rk;
};

template <int V>
__global__ void __launch_bounds__(kThreads) philox_multi_kernel(const __grid_constant__ MultiParams p) {
  const int64_t T = (int64_t)gridDim.x * kThreads;
  int64_t idx = (int64_t)blockIdx.x * kThreads + threadIdx.x;
  if (idx >= p.total) return;
  int64_t s = idx / p.groups;
  int64_t j = idx - s * p.groups;
  uint64_t sb_lo = p.base_lo, sb_hi = p.base_hi;  // block counter of group 0 of stream s
  {
    const uint64_t us = (uint64_t)s;
    add128(sb_lo, sb_hi, us * p.sb_lo, __umul64hi(us, p.sb_lo) + us * p.sb_hi);
  }
  for (; idx < p.total; idx += T) {
    uint64_t c_lo = sb_lo, c_hi = sb_hi;
    add128(c_lo, c_hi, (uint64_t)j, 0);
    p.out[idx] = block_outputs<V>(philox4x32_10(ctr_from(c_lo, c_hi), p.rk), p.t);
    j += p.tr;
    add128(sb_lo, sb_hi, p.tqsb_lo, p.tqsb_hi);
    if (j >= p.groups) {
      j -= p.groups;
      add128(sb_lo, sb_hi, p.sb_lo, p.sb_hi);
    }
  }
}

// The same for streams of 256 groups or more (512 for the light transforms:
// 16384 x 1024 FP32 uniforms, 256 groups, take 27.2 us here and 25.5 above): a CTA takes a tile of one stream,
// so that the stream's counter base (a 128-bit product), its upper words'
// constants and the position are found once per tile, and its groups go as
// in the single-stream kernel (one group at a time with 128-bit counters took
// 90 instructions a block against 64 there).  16384 x 16384: FP32 uniforms
// 258 -> 169 us (159 in one stream), bits 230 -> 147, FP64 uniforms 540 -> 402,
// FP32 gaussians 428 -> 311, FP64 gaussians 1791 -> 1656 (1560 with the pair reworked).
struct MultiTileParams {
  TransformParams t;
  uint4* out;
  uint32_t groups;    // groups per stream
  uint32_t tile;      // groups per tile
  uint32_t tps;       // tiles per stream
  uint32_t tiles;     // of all streams
  uint64_t base_lo, base_hi;
  uint64_t sb_lo, sb_hi;  // block-counter stride between streams
  PhiloxRoundKeys rk;
};

template <int V, int U>
__device__ __forceinline__ void philox_multi_tile(const MultiTileParams& p, uint32_t tile) {
  const uint32_t s = tile / p.tps, first = (tile - s * p.tps) * p.tile;
  uint64_t lo = p.base_lo, hi = p.base_hi;  // block counter of group 0 of stream s
  add128(lo, hi, (uint64_t)s * p.sb_lo, __umul64hi((uint64_t)s, p.sb_lo) + (uint64_t)s * p.sb_hi);
  const uint32_t x0 = (uint32_t)lo;
  const PhiloxUpper up = philox_upper(p.rk.k[0], p.rk.k[1], (uint32_t)(lo >> 32), (uint32_t)hi,
                                      (uint32_t)(hi >> 32) & 0x3FFFFFFFu);
  // the low word carries inside the stream (the same for the whole CTA)
  const bool cross = x0 + p.groups < x0;
  const uint32_t end = p.groups - first < p.tile ? p.groups : first + p.tile;
  uint32_t j = first + threadIdx.x;
  uint4* dst = p.out + ((uint64_t)s * p.groups + j);
  if (cross) {
    for (; j < end; j += kThreads, dst += kThreads) {
      uint64_t c_lo = lo, c_hi = hi;
      add128(c_lo, c_hi, j, 0);
      *dst = block_outputs<V>(philox4x32_10(ctr_from(c_lo, c_hi), p.rk), p.t);
    }
    return;
  }
  for (; j + (U - 1) * kThreads < end; j += U * kThreads, dst += U * kThreads) {
    uint4 o[U];
#pragma unroll
    for (int u = 0; u < U; ++u)
      o[u] = block_outputs<V>(philox_block(x0 + j + u * kThreads, up, p.rk), p.t);
#pragma unroll
    for (int u = 0; u < U; ++u) dst[u * kThreads] = o[u];
  }
  if constexpr (U > 1)
    for (; j < end; j += kThreads, dst += kThreads)
      *dst = block_outputs<V>(philox_block(x0 + j, up, p.rk), p.t);
}

// kWalk: fewer CTAs, as a tuned geometry asks, walk the tiles with a grid stride;
// else one tile a CTA.  In one kernel the loop cost the built-in geometry 2-3 %
// (16384 x 16384 bits 153 -> 158 us, FP32 gaussians 318 -> 325).
template <int V, int U, bool kWalk>
__device__ __forceinline__ void philox_multi_tile_body(const MultiTileParams& p) {
  if constexpr (kWalk) {
    for (uint32_t tile = blockIdx.x; tile < p.tiles; tile += gridDim.x) philox_multi_tile<V, U>(p, tile);
  } else {
    philox_multi_tile<V, U>(p, blockIdx.x);
  }
}

template <int V, int U, bool kWalk>
__global__ void __launch_bounds__(kThreads) philox_multi_tile_kernel(const __grid_constant__ MultiTileParams p) {
  philox_multi_tile_body<V, U, kWalk>(p);
}

template <int V, int U, bool kWalk>
__global__ void __launch_bounds__(kThreads, 5) philox_multi_tile_kernel_5(const __grid_constant__ MultiTileParams p) {
  philox_multi_tile_body<V, U, kWalk>(p);
}

// Substreams at any word phase and pointer alignment: stream s writes
// out + s n elements from word offset off + s stride, and its 16-byte groups
// are found as in the shift kernel, per stream.  A warp takes one chunk of
// 30 groups of one stream, so the stream's phase, head and pair split are
// uniform across the warp: lanes compute 32 consecutive blocks, take the
// next block's first words from lane + 1, and, when the stream's start
// splits a Box-Muller pair, transform pair-aligned virtual groups one
// element earlier and exchange the straddling element (as kSplit above).
struct MultiShiftParams {
  TransformParams t;
  char* out;                 // element 0 of stream 0
  int64_t n;                 // elements per stream
  int64_t cps;               // warp chunks per stream
  int64_t total;             // cps * num_streams
  uint64_t off_lo, off_hi;   // word offset of stream 0
  uint64_t stride_lo, stride_hi;
  PhiloxRoundKeys rk;
};

constexpr int kMultiShiftPer = 30;

// Where stream s's (virtual) groups start, per stream of a multi-shift fill.
struct ShiftStream {
  char* sbase;      // element 0 of the stream
  uint4* gbase;     // its 16-byte aligned group 0
  int64_t head;     // elements of group 0 before sbase
  int64_t groups, jf, jl;
  uint64_t b_lo, b_hi;  // block of the first word of (virtual) group 0
  PhiloxUpper up;       // its upper words' constants
  uint32_t ph;
  bool split;
  bool cross;           // the low counter word may carry inside the stream
};

template <int V, bool kLong>
__device__ __forceinline__ ShiftStream shift_stream(const MultiShiftParams& p, int64_t s) {
  using I = VInfo<V>;
  constexpr int kEpg = 16 / I::es;
  constexpr uint32_t kWpe = (uint32_t)(I::es / 4);  // words per element
  ShiftStream t;
  t.sbase = p.out + s * p.n * I::es;
  t.head = (int64_t)(((uintptr_t)t.sbase & 15u) / (uint32_t)I::es);
  t.gbase = reinterpret_cast<uint4*>((uintptr_t)t.sbase & ~(uintptr_t)15);
  t.split = I::epu == 2 && (t.head & 1) != 0;
  // first word of (virtual) group 0: off + s stride - head es/4 (one element
  // earlier when split), 128-bit
  uint64_t a_lo = p.off_lo, a_hi = p.off_hi;
  const uint64_t us = (uint64_t)s;
  add128(a_lo, a_hi, us * p.stride_lo, __umul64hi(us, p.stride_lo) + us * p.stride_hi);
  const uint64_t back = (uint64_t)t.head * kWpe + (t.split ? kWpe : 0u);
  a_hi -= (a_lo < back) ? 1u : 0u;
  a_lo -= back;
  t.b_lo = (a_lo >> 2) | (a_hi << 62);
  t.b_hi = a_hi >> 2;
  t.ph = (uint32_t)a_lo & 3u;
  t.groups = (t.head + p.n + kEpg - 1) / kEpg;
  t.cross = !kLong || (uint64_t)(uint32_t)t.b_lo + (uint64_t)t.groups + 32u >= kPhiloxMaxBlocks;
  if (!t.cross)
    t.up = philox_upper(p.rk.k[0], p.rk.k[1], (uint32_t)(t.b_lo >> 32), (uint32_t)t.b_hi,
                        (uint32_t)(t.b_hi >> 32) & 0x3FFFFFFFu);
  t.jf = t.head > 0 ? 1 : 0;
  t.jl = ((t.head + p.n) % kEpg) != 0 ? t.groups - 1 : t.groups;
  return t;
}

// kLong: warps take four chunks or more, so that making the upper counter
// words' constants per stream pays; the short form, whole counters throughout,
// is also the smaller program (1000 x 1023 FP64 uniforms 9.1 us against 10.8).
template <int V, bool kLong>
__global__ void __launch_bounds__(kThreads) philox_multishift_kernel(
    const __grid_constant__ MultiShiftParams p) {
  using I = VInfo<V>;
  constexpr int kEpg = 16 / I::es;
  constexpr int kPer = kMultiShiftPer;
  const int lane = threadIdx.x & 31;
  // each warp takes a run of consecutive chunks (chunk c = stream c / cps,
  // chunk c mod cps of it), so a stream's set-up is redone only when the run
  // enters the next stream; the loop bound depends only on the warp
  const int64_t W = (int64_t)gridDim.x * (kThreads / 32);
  const int64_t w = (int64_t)blockIdx.x * (kThreads / 32) + (threadIdx.x >> 5);
  const int64_t L = (p.total + W - 1) / W;
  int64_t c = w * L;
  const int64_t c_end = (c + L) < p.total ? (c + L) : p.total;
  if (c >= c_end) return;
  int64_t s = c / p.cps;
  int64_t k = c - s * p.cps;
  ShiftStream t = shift_stream<V, kLong>(p, s);
  // groups [k kPer, (k + 1) kPer) of the stream, from this lane's block
  auto emit = [&](int64_t k, int64_t j, uint4 b) {
    // the stream's phase and split are the same for the whole warp, so the
    // exchanges run on all 32 lanes or on none: a stream at phase 0 skips the
    // word exchange
    uint4 w = b;
    if (t.ph != 0) w = shift_words(b, t.ph);
    uint4 o = block_outputs<V>(w, p.t);
    if constexpr (I::epu == 2) {
      if (t.split) o = split_group<V>(o);
    }
    if (k * kPer >= t.jf && k * kPer + kPer <= t.jl) {  // whole groups (uniform)
      if (lane < kPer) t.gbase[j] = o;
    } else if (lane < kPer && j < t.groups) {
      const int64_t e0 = j * kEpg - t.head;
      if (e0 >= 0 && e0 + kEpg <= p.n) {
        t.gbase[j] = o;
      } else {
        store_partial<V>(t.sbase, e0, p.n, o);
      }
    }
  };
  while (true) {
    // the run's chunks in this stream, in a loop of their own where the upper
    // counter words are fixed (16384 x 16385 at a stride of 2^40 + 1: FP32
    // uniforms 302 -> 263 us, FP32 gaussians 518 -> 446)
    const int64_t k_end = k + (c_end - c) < p.cps ? k + (c_end - c) : p.cps;
    c += k_end - k;
    if (!t.cross) {
      for (; k < k_end; ++k) {
        const int64_t j = k * kPer + lane;
        emit(k, j, philox_block((uint32_t)t.b_lo + (uint32_t)j, t.up, p.rk));
      }
    } else {
      for (; k < k_end; ++k) {
        const int64_t j = k * kPer + lane;
        uint64_t c_lo = t.b_lo, c_hi = t.b_hi;
        add128(c_lo, c_hi, (uint64_t)j, 0);
        emit(k, j, philox4x32_10(ctr_from(c_lo, c_hi), p.rk));
      }
    }
    if (c >= c_end) return;
    k = 0;
    t = shift_stream<V, kLong>(p, ++s);
  }
}

// CTAs per SM a launch may use, from the tuned geometry: 1..16 a cap on the
// resident CTAs; 17 and above (geom - 16) waves of resident CTAs, each CTA
// taking that fraction of a resident CTA's share of the grid-stride loop, so
// that the hardware refills an SM as its CTAs finish instead of the SM
// emptying out as the faster warps of long-lived CTAs finish first (ncu: a
// single persistent wave kept 33 of 48 possible warps active); 0, the
// built-in choice, is 8 waves (within 1 % of the best wave count for every
// fill at n = 10^9; one wave was up to 6 % slower).
int ctas_cap(int occ, int32_t geom) {
  if (geom == 0) return occ * 8;
  if (geom > 16) return occ * (geom - 16);
  return geom < occ ? (int)geom : occ;
}

template <typename K>
int blocks_per_sm(K kernel) {
  int b = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, kThreads, 0) != cudaSuccess ||
      b < 1) {
    cudaGetLastError();
    b = 1;
  }
  return b;
}

// The same kept in a slot of the kernel's own, 0 until it is known: launches may
// come from several host threads, and each finds its slot filled or fills it.
template <typename K>
int resident_ctas(std::atomic<int>& slot, K kernel) {
  int o = slot.load(std::memory_order_relaxed);
  if (o == 0) {
    o = blocks_per_sm(kernel);
    slot.store(o, std::memory_order_relaxed);
  }
  return o;
}

// Launches the shift kernel: words of (virtual) group 0 start at word a of
// the stream (128-bit, a = off - head words, one element earlier for kSplit).
template <int V, bool kSplit>
void launch_shift(ShiftParams& p, const uint32_t* key, uint64_t a_lo, uint64_t a_hi, int sms,
                  int32_t geom, cudaStream_t stream) {
  constexpr int kPer = shift_per_warp<kSplit>();
  constexpr int kU = exchange_blocks_per_thread<V>();
  p.ctr = philox_stream(key[0], key[1], (a_lo >> 2) | (a_hi << 62), a_hi >> 2);
  p.ph = (uint32_t)(a_lo & 3u);
  p.chunks = (p.groups + kPer - 1) / kPer;
  // a warp's turn starts below chunk `chunks` and takes kU of them: the blocks lie
  // below (chunks + kU) kPer + 32 past base
  const uint64_t reach = (uint64_t)(p.chunks + kU) * (uint64_t)kPer + 32u;
  const bool cross = p.ctr.x0 + reach >= kPhiloxMaxBlocks;
  void (*kernel)(const ShiftParams);
  if constexpr (stream_wants_5_ctas<V>()) {
    kernel = cross ? philox_shift_kernel_5<V, kU, true, kSplit> : philox_shift_kernel_5<V, kU, false, kSplit>;
  } else {
    kernel = cross ? philox_shift_kernel<V, kU, true, kSplit> : philox_shift_kernel<V, kU, false, kSplit>;
  }
  static std::atomic<int> occ[2] = {{0}, {0}};
  const int o = resident_ctas(occ[cross ? 1 : 0], kernel);
  const int64_t warps = (p.chunks + kU - 1) / kU;
  int64_t grid = (warps + (kThreads / 32) - 1) / (kThreads / 32);
  if (grid < 1) grid = 1;
  const int64_t cap = (int64_t)sms * ctas_cap(o, geom);
  if (grid > cap) grid = cap;
  kernel<<<(unsigned)grid, kThreads, 0, stream>>>(p);
}

// Launches the pieces or the rotate kernel (units inside blocks, output start at
// another phase); p.t, p.out, p.gbase, p.nw, p.h are set by the caller.
template <int V>
void launch_pieces(PiecesParams& p, const uint32_t* key, uint64_t off_lo, uint64_t off_hi, int sms,
                   int32_t geom, cudaStream_t stream) {
  constexpr bool kRotate = VInfo<V>::weight == 0;
  constexpr int kU = exchange_blocks_per_thread<V>();
  p.r = (int64_t)(off_lo & 3u);
  p.gofs = p.h - p.r < 0 ? -1 : 0;
  p.ctr = philox_stream(key[0], key[1], (off_lo >> 2) | (off_hi << 62), off_hi >> 2);
  const int64_t blocks = (p.nw - 1 + p.r) / 4 + 1;
  p.chunks = (blocks + 31) / 32;
  // as in launch_shift
  const uint64_t reach = (uint64_t)(p.chunks + kU) * 32u + 32u;
  const bool cross = p.ctr.x0 + reach >= kPhiloxMaxBlocks;
  void (*kernel)(const PiecesParams);
  if constexpr (kRotate) {
    kernel = cross ? philox_rotate_kernel<V, kU, true> : philox_rotate_kernel<V, kU, false>;
  } else if constexpr (stream_wants_5_ctas<V>()) {
    kernel = cross ? philox_pieces_kernel_5<V, kU, true> : philox_pieces_kernel_5<V, kU, false>;
  } else {
    kernel = cross ? philox_pieces_kernel<V, kU, true> : philox_pieces_kernel<V, kU, false>;
  }
  static std::atomic<int> occ[2] = {{0}, {0}};
  const int o = resident_ctas(occ[cross ? 1 : 0], kernel);
  const int64_t warps = (p.chunks + kU - 1) / kU;
  int64_t grid = (warps + (kThreads / 32) - 1) / (kThreads / 32);
  if (grid < 1) grid = 1;
  const int64_t cap = (int64_t)sms * ctas_cap(o, geom);
  if (grid > cap) grid = cap;
  kernel<<<(unsigned)grid, kThreads, 0, stream>>>(p);
}

template <int V>
grng_status launch_variant(const FillRequest& r, cudaStream_t stream) {
  using I = VInfo<V>;
  constexpr int kEpg = 16 / I::es;
  int dev = 0;
  const int sms = current_device_sms(&dev);
  const int32_t geom = fill_geometry(GRNG_PHILOX4X32X10, V, r.asked);
  const uintptr_t addr = (uintptr_t)r.out;
  const uint32_t phase_w = (uint32_t)((addr & 15u) / 4u);  // output words before out in group 0
  const uint64_t stream_bytes = (uint64_t)r.n * I::es;
  // same alignment phase for every stream, and a block-multiple stride
  const bool uniform_streams =
      r.num_streams == 1 || ((stream_bytes % 16u) == 0 && (r.stride_lo & 3u) == 0);
  const bool fast = uniform_streams && ((r.off_lo - phase_w) & 3u) == 0 &&
                    (phase_w % (uint32_t)I::wpu) == 0;

  // base block counter = (off - phase_w) / 4 with a 128-bit borrow
  const uint64_t lo0 = r.off_lo - phase_w;
  const uint64_t hi0 = r.off_hi - ((r.off_lo < phase_w) ? 1u : 0u);
  const uint64_t base_lo = (lo0 >> 2) | (hi0 << 62);
  const uint64_t base_hi = hi0 >> 2;
  const int64_t head = (int64_t)(phase_w * 4u / I::es);
  const int64_t groups = (head + r.n + kEpg - 1) / kEpg;
  if (fast && r.num_streams == 1) {
    StreamParams p;
    p.t = r.t;
    p.out = r.out;
    p.gbase = reinterpret_cast<uint4*>(addr - phase_w * 4u);
    p.n = r.n;
    p.head = head;
    p.ctr = philox_stream(r.key[0], r.key[1], base_lo, base_hi);
    // full groups: the first group is partial when head > 0, the last one
    // when the end is not on a group boundary (or both are the same group)
    int64_t jf = head > 0 ? 1 : 0;
    int64_t jl = ((head + r.n) % kEpg) != 0 ? groups - 1 : groups;
    p.edge[0] = p.edge[1] = -1;
    if (jf > jl) {  // a single partial group
      p.edge[0] = 0;
      jf = jl = 0;
    } else {
      if (head > 0) p.edge[0] = 0;
      if (jl < groups) p.edge[1] = groups - 1;
    }
    p.jf = (uint32_t)jf;
    p.jl = (uint32_t)jl;
    constexpr int kU = blocks_per_thread<V>();
    const bool cross = p.ctr.x0 + (uint64_t)groups >= kPhiloxMaxBlocks;
    void (*kernel)(const StreamParams);
    if constexpr (stream_wants_5_ctas<V>()) {
      kernel = cross ? philox_stream_kernel_5<V, kU, true> : philox_stream_kernel_5<V, kU, false>;
    } else {
      kernel = cross ? philox_stream_kernel<V, kU, true> : philox_stream_kernel<V, kU, false>;
    }
    static std::atomic<int> occ[2] = {{0}, {0}};
    const int o = resident_ctas(occ[cross ? 1 : 0], kernel);
    const int64_t work = (jl - jf + (int64_t)kU - 1) / kU;
    int64_t grid = (work + kThreads - 1) / kThreads;
    if (grid < 1) grid = 1;
    const int64_t cap = (int64_t)sms * ctas_cap(o, geom);
    if (grid > cap) grid = cap;
    kernel<<<(unsigned)grid, kThreads, 0, stream>>>(p);
  } else if (fast && head == 0 && (stream_bytes % 16u) == 0 && groups >= (I::weight == 0 ? 2 : 1) * kThreads &&
             groups <= (int64_t(1) << 31)) {
    MultiTileParams p;
    p.t = r.t;
    p.out = reinterpret_cast<uint4*>(r.out);
    p.groups = (uint32_t)groups;
    p.base_lo = base_lo;
    p.base_hi = base_hi;
    p.sb_lo = (r.stride_lo >> 2) | (r.stride_hi << 62);
    p.sb_hi = r.stride_hi >> 2;
    p.rk = philox_round_keys(r.key[0], r.key[1]);
    constexpr int kU = multi_blocks_per_thread<V>();
    // at most kMultiTile, less where the fill is small (8 CTAs per SM at least,
    // 32 for the longer transforms, whose last wave weighs more), and a
    // stream's tiles alike
    const int64_t ctas = (int64_t)sms * (I::weight == 0 ? 8 : 32);
    int64_t cap = groups * r.num_streams / (ctas * kThreads) * kThreads;
    if (cap > kMultiTile) cap = kMultiTile;
    if (cap < kThreads) cap = kThreads;
    const int64_t tiles = (groups + cap - 1) / cap;
    const int64_t tile = ((groups + tiles - 1) / tiles + kThreads - 1) / kThreads * kThreads;
    p.tile = (uint32_t)tile;
    const int64_t tps = (groups + tile - 1) / tile;
    p.tps = (uint32_t)tps;
    int64_t grid = tps * r.num_streams;
    p.tiles = (uint32_t)grid;
    void (*kernel)(const MultiTileParams);
    if constexpr (stream_wants_5_ctas<V>()) {
      kernel = geom == 0 ? philox_multi_tile_kernel_5<V, kU, false> : philox_multi_tile_kernel_5<V, kU, true>;
    } else {
      kernel = geom == 0 ? philox_multi_tile_kernel<V, kU, false> : philox_multi_tile_kernel<V, kU, true>;
    }
    if (geom != 0) {
      static std::atomic<int> occ_cache{0};
      const int64_t cap = (int64_t)sms * ctas_cap(resident_ctas(occ_cache, kernel), geom);
      if (grid > cap) grid = cap;
    }
    kernel<<<(unsigned)grid, kThreads, 0, stream>>>(p);
  } else if (fast && head == 0 && (stream_bytes % 16u) == 0) {
    MultiParams p;
    p.t = r.t;
    p.out = reinterpret_cast<uint4*>(r.out);
    p.groups = groups;
    p.total = groups * r.num_streams;
    p.base_lo = base_lo;
    p.base_hi = base_hi;
    p.sb_lo = (r.stride_lo >> 2) | (r.stride_hi << 62);
    p.sb_hi = r.stride_hi >> 2;
    p.rk = philox_round_keys(r.key[0], r.key[1]);
    static std::atomic<int> occ_cache{0};
    const int occ = resident_ctas(occ_cache, philox_multi_kernel<V>);
    int64_t grid = (p.total + kThreads - 1) / kThreads;
    const int64_t cap = (int64_t)sms * ctas_cap(occ, geom);
    if (grid > cap) grid = cap;
    const int64_t gstride = grid * kThreads;
    p.tq = gstride / p.groups;
    p.tr = gstride - p.tq * p.groups;
    const unsigned __int128 tqsb =
        (unsigned __int128)(uint64_t)p.tq *
        (((unsigned __int128)p.sb_hi << 64) | (unsigned __int128)p.sb_lo);
    p.tqsb_lo = (uint64_t)tqsb;
    p.tqsb_hi = (uint64_t)(tqsb >> 64);
    philox_multi_kernel<V><<<(unsigned)grid, kThreads, 0, stream>>>(p);
  } else if (I::wpu >= 2 && r.num_streams == 1 && (r.off_lo % (uint64_t)I::wpu) == 0) {
    // one stream whose units lie inside counter blocks, the output start at
    // another phase (e.g. a Box-Muller pair split by the pointer)
    if constexpr (I::wpu >= 2) {
      PiecesParams p;
      p.t = r.t;
      p.out = reinterpret_cast<char*>(r.out);
      p.gbase = reinterpret_cast<uint4*>(addr - phase_w * 4u);
      p.nw = r.n * (I::es / 4);
      p.h = (int64_t)phase_w;
      launch_pieces<V>(p, r.key, r.off_lo, r.off_hi, sms, geom, stream);
    }
  } else if (r.num_streams == 1 &&
             ((phase_w % (uint32_t)I::wpu) == 0 || (I::epu == 2 && (head & 1) != 0))) {
    // one stream at another word phase, or a pair split by the output's start
    ShiftParams p;
    p.t = r.t;
    p.out = r.out;
    p.gbase = reinterpret_cast<uint4*>(addr - phase_w * 4u);
    p.n = r.n;
    p.head = head;
    p.groups = groups;
    p.jf = head > 0 ? 1 : 0;
    p.jl = ((head + r.n) % kEpg) != 0 ? groups - 1 : groups;
    if ((phase_w % (uint32_t)I::wpu) == 0) {
      launch_shift<V, false>(p, r.key, lo0, hi0, sms, geom, stream);
    } else if constexpr (I::epu == 2) {
      // the virtual groups start one element (es / 4 words) earlier
      const uint32_t pv = phase_w + (uint32_t)(I::es / 4);
      const uint64_t a_lo = r.off_lo - pv;
      const uint64_t a_hi = r.off_hi - ((r.off_lo < pv) ? 1u : 0u);
      launch_shift<V, true>(p, r.key, a_lo, a_hi, sms, geom, stream);
    }
  } else {
    // substreams at any other phase or alignment
    MultiShiftParams p;
    p.t = r.t;
    p.out = reinterpret_cast<char*>(r.out);
    p.n = r.n;
    // groups of a stream with the largest head (16 / es - 1 elements)
    const int64_t max_groups = (r.n + (kEpg - 1) + kEpg - 1) / kEpg;
    p.cps = (max_groups + kMultiShiftPer - 1) / kMultiShiftPer;
    p.total = p.cps * r.num_streams;
    p.off_lo = r.off_lo;
    p.off_hi = r.off_hi;
    p.stride_lo = r.stride_lo;
    p.stride_hi = r.stride_hi;
    p.rk = philox_round_keys(r.key[0], r.key[1]);
    static std::atomic<int> occ_cache{0};
    const int occ = resident_ctas(occ_cache, philox_multishift_kernel<V, true>);
    int64_t grid = (p.total + (kThreads / 32) - 1) / (kThreads / 32);
    const int64_t cap = (int64_t)sms * ctas_cap(occ, geom);
    if (grid > cap) grid = cap;
    if (grid < 1) grid = 1;
    const bool is_long = p.total >= 4 * grid * (kThreads / 32);
    (is_long ? philox_multishift_kernel<V, true> : philox_multishift_kernel<V, false>)<<<(unsigned)grid, kThreads, 0, stream>>>(p);
  }
  const cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) {
    set_error("Philox fill launch failed: %s", cudaGetErrorString(err));
    return GRNG_ERR_CUDA;
  }
  return GRNG_OK;
}

grng_status launch_by_variant(const FillRequest& r, cudaStream_t stream) {
  switch (r.variant) {
    case V_BITS: return launch_variant<V_BITS>(r, stream);
    case V_U01_F32: return launch_variant<V_U01_F32>(r, stream);
    case V_UNI_F32: return launch_variant<V_UNI_F32>(r, stream);
    case V_U01_F64: return launch_variant<V_U01_F64>(r, stream);
    case V_AFF_F64: return launch_variant<V_AFF_F64>(r, stream);
    case V_UNI_F64: return launch_variant<V_UNI_F64>(r, stream);
    case V_GAUSS_F32: return launch_variant<V_GAUSS_F32>(r, stream);
    case V_LOGN_F32: return launch_variant<V_LOGN_F32>(r, stream);
    case V_GAUSS_F64: return launch_variant<V_GAUSS_F64>(r, stream);
    case V_LOGN_F64: return launch_variant<V_LOGN_F64>(r, stream);
    case V_ICDF_GAUSS_F32: return launch_variant<V_ICDF_GAUSS_F32>(r, stream);
    case V_ICDF_LOGN_F32: return launch_variant<V_ICDF_LOGN_F32>(r, stream);
    case V_ICDF_GAUSS_F64: return launch_variant<V_ICDF_GAUSS_F64>(r, stream);
    case V_ICDF_LOGN_F64: return launch_variant<V_ICDF_LOGN_F64>(r, stream);
    case V_STDGAUSS_F64: return launch_variant<V_STDGAUSS_F64>(r, stream);
    default: set_error("unknown variant %d", r.variant); return GRNG_ERR_INVALID_ARG;
  }
}

}  // namespace

// A single-stream fill counts its blocks in 32 bits: a longer one is launched
// in pieces of 2^32 elements (at most 2^31 blocks), each a fill of its own at
// its own word offset, with the geometry of the whole.
grng_status launch_philox(const FillRequest& r, CUstream_st* stream) {
  constexpr int64_t kPiece = int64_t(1) << 32;
  if (r.num_streams != 1 || r.n <= kPiece) return launch_by_variant(r, stream);
  const VariantInfo v = variant_info(r.variant);
  FillRequest piece = r;
  for (int64_t at = 0; at < r.n; at += kPiece) {
    piece.n = (r.n - at) < kPiece ? (r.n - at) : kPiece;
    piece.out = reinterpret_cast<char*>(r.out) + at * v.es;
    const uint64_t words = (uint64_t)(at / v.epu) * (uint64_t)v.wpu;
    piece.off_lo = r.off_lo + words;
    piece.off_hi = r.off_hi + ((piece.off_lo < words) ? 1u : 0u);
    const grng_status st = launch_by_variant(piece, stream);
    if (st != GRNG_OK) return st;
  }
  return GRNG_OK;
}

}  // namespace grng
