// Batched generation: many independent Philox requests in one persistent
// launch (the event batching the paper leaves as future work, Sec. 7, and the
// small-batch latency it measures, Sec. 7 / Fig. 2-4).
//
// A batch is planned once on the host (grng_batch_create): per request its
// variant, parameters, output pointer, 16-byte group count and starting word
// offset; a tile -> request map; and per request the words its engine
// advances per launch.  The tables live in a caller-provided device
// workspace.  grng_batch_launch then enqueues one kernel: CTAs walk the tiles (a
// tile is kThreads * ipt 16-byte groups of one request) with a static grid
// stride, up to eight at a time, and count the launch in the workspace as they
// finish.  A request's offset is its start plus the launches so far times its
// advance, so launching again (or replaying a CUDA graph of the launch)
// continues every generator's sequence with no host work.  grng_batch_commit
// reads the count and moves the engines.
//
// A request whose word offset matches its pointer's 16-byte phase maps each
// 16-byte group to one Philox block; at any other phase a warp computes 32
// consecutive blocks and exchanges the straddling words by shuffle (no
// shared memory anywhere).
#include <cuda_runtime.h>

#include <cstdint>
#include <cstring>
#include <new>
#include <unordered_map>
#include <vector>

#include "device_common.cuh"
#include "grng.h"
#include "grng_internal.h"

namespace grng {

namespace {

using namespace dev;

constexpr int kThreads = 256;

// Workspace layout (each part 256-byte aligned):
//   BatchReq reqs[count] | uint64_t off[count][2] | uint64_t arrivals | int32_t tile_req[tiles]
size_t align256(size_t x) { return (x + 255u) & ~(size_t)255u; }

// Stores the elements of group (first element e0) that lie in [0, n).
template <int V>
__device__ __forceinline__ void store_group(char* base, int64_t e0, int64_t n, uint4 o) {
  using I = VInfo<V>;
  constexpr int kEpg = 16 / I::es;
  if (e0 >= 0 && e0 + kEpg <= n) {
    store16(base + e0 * I::es, o);
    return;
  }
  const uint32_t ow[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
  for (int i = 0; i < kEpg; ++i) {
    const int64_t e = e0 + i;
    if (e >= 0 && e < n) {
      if constexpr (I::es == 4) {
        reinterpret_cast<uint32_t*>(base)[e] = ow[i];
      } else {
        reinterpret_cast<uint2*>(base)[e] = make_uint2(ow[2 * i], ow[2 * i + 1]);
      }
    }
  }
}

// Blocks per thread at once in a tile whose groups are blocks.
template <int V>
constexpr int kTileBlocks = VInfo<V>::es == 8 ? 1 : VInfo<V>::weight == 0 ? 4 : 2;

// The blocks of a tile from block (b_lo, b_hi) on: the round keys and, where
// the low counter word does not carry inside the tile, the upper words'
// constants, made once per tile.
struct TileBlocks {
  PhiloxRoundKeys rk;
  PhiloxUpper up;
  uint64_t b_lo, b_hi;
  __device__ __forceinline__ TileBlocks(uint32_t k0, uint32_t k1, uint64_t lo, uint64_t hi)
      : rk(philox_round_keys(k0, k1)),
        up(philox_upper(k0, k1, (uint32_t)(lo >> 32), (uint32_t)hi,
                        (uint32_t)(hi >> 32) & 0x3FFFFFFFu)),
        b_lo(lo),
        b_hi(hi) {}
  template <bool kCross>
  __device__ __forceinline__ uint4 at(uint32_t i) const {
    if constexpr (!kCross) return philox_block((uint32_t)b_lo + i, up, rk);
    const uint64_t lo = b_lo + i;
    return philox4x32_10(ctr_from(lo, b_hi + ((lo < b_lo) ? 1u : 0u)), rk);
  }
};

// A tile's groups: `count` from group 0 at dst, those of [wf, wl) whole inside the
// request, at most the first and the last not; the first element of group 0 is
// element e0 of the request.
struct TileOut {
  uint4* dst;
  uint32_t count, wf, wl;
  char* base;
  int64_t e0, n;
};

template <int V>
__device__ __forceinline__ void tile_store(const TileOut& o, uint32_t i, uint4 v) {
  if (i >= o.wf && i < o.wl) {
    o.dst[i] = v;
  } else {
    store_group<V>(o.base, o.e0 + (int64_t)i * (16 / VInfo<V>::es), o.n, v);
  }
}

// Group i is block i.
template <int V>
__device__ __forceinline__ void tile_blocks_loop(const TransformParams& t, const TileBlocks& q,
                                                 const TileOut& out) {
  constexpr uint32_t U = kTileBlocks<V>;
  if (threadIdx.x < 2) {  // the groups that are not whole
    const uint32_t i = threadIdx.x == 0 ? 0u : out.count - 1u;
    if ((i < out.wf || i >= out.wl) && (threadIdx.x == 0 || out.count > 1))
      tile_store<V>(out, i, block_outputs<V>(q.at<false>(i), t));
  }
  uint32_t i = out.wf + threadIdx.x;
  uint4* dst = out.dst + i;
  for (; i + (U - 1) * kThreads < out.wl; i += U * kThreads, dst += U * kThreads) {
    uint4 o[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) o[u] = block_outputs<V>(q.at<false>(i + u * kThreads), t);
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) dst[u * kThreads] = o[u];
  }
  if constexpr (U > 1)
    for (; i < out.wl; i += kThreads, dst += kThreads) *dst = block_outputs<V>(q.at<false>(i), t);
}

// The same where a group straddles two blocks (word phase ph), where the low
// counter word carries (kCross; any ph) or, kSplit, where the output's start
// splits a Box-Muller pair (an odd head; any ph): a warp computes 32
// consecutive blocks and emits 31 or 30 groups, exchanging the straddling
// words, and elements, between neighbouring lanes as in the single-stream
// shift kernel.  The loop bound depends only on the warp, so every shuffle has
// all 32 lanes.
//
// kPh: the word phase as a constant (only the words needed cross lanes), or -1
// to read it from ph; two chunks per warp at once with a constant phase.  Bits
// and the uniforms, whose share the exchange is largest of, take it: with
// tile_halves_loop below the table of 4096 requests 568 -> 541 us a launch, three
// in four of its requests at another phase.
template <int V, bool kCross, bool kSplit, int kPh = -1>
__device__ __forceinline__ void tile_shift_loop(const TransformParams& t, const TileBlocks& q,
                                                uint32_t ph, const TileOut& out) {
  using I = VInfo<V>;
  constexpr uint32_t kPerWarp = kSplit ? 30 : 31;
  constexpr uint32_t U = kPh > 0 && I::es == 4 ? 2 : 1;
  const uint32_t lane = threadIdx.x & 31u;
  for (uint32_t c = (threadIdx.x >> 5) * (kPerWarp * U); c < out.count;
       c += kPerWarp * U * (kThreads / 32)) {
    const uint32_t i = c + lane;
    uint4 b[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) b[u] = q.at<kCross>(i + u * kPerWarp);
    const bool whole = c >= out.wf && c + kPerWarp * U <= out.wl;  // (uniform)
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      uint4 w = b[u];
      if constexpr (kPh > 0) {
        const uint32_t n0 = __shfl_down_sync(0xFFFFFFFFu, b[u].x, 1);
        if constexpr (kPh == 1) {
          w = make_uint4(b[u].y, b[u].z, b[u].w, n0);
        } else {
          const uint32_t n1 = __shfl_down_sync(0xFFFFFFFFu, b[u].y, 1);
          if constexpr (kPh == 2) {
            w = make_uint4(b[u].z, b[u].w, n0, n1);
          } else {
            w = make_uint4(b[u].w, n0, n1, __shfl_down_sync(0xFFFFFFFFu, b[u].z, 1));
          }
        }
      } else if ((!kSplit && !kCross) || ph != 0) {
        const uint32_t n0 = __shfl_down_sync(0xFFFFFFFFu, b[u].x, 1);
        const uint32_t n1 = __shfl_down_sync(0xFFFFFFFFu, b[u].y, 1);
        const uint32_t n2 = __shfl_down_sync(0xFFFFFFFFu, b[u].z, 1);
        if (ph == 1) {
          w = make_uint4(b[u].y, b[u].z, b[u].w, n0);
        } else if (ph == 2) {
          w = make_uint4(b[u].z, b[u].w, n0, n1);
        } else {
          w = make_uint4(b[u].w, n0, n1, n2);
        }
      }
      uint4 o = block_outputs<V>(w, t);
      if constexpr (kSplit) {
        const uint32_t m0 = __shfl_down_sync(0xFFFFFFFFu, o.x, 1);
        const uint32_t m1 = __shfl_down_sync(0xFFFFFFFFu, o.y, 1);
        o = I::es == 4 ? make_uint4(o.y, o.z, o.w, m0) : make_uint4(o.z, o.w, m0, m1);
      }
      if (lane < kPerWarp) {
        const uint32_t g = i + u * kPerWarp;
        if (whole) {
          out.dst[g] = o;
        } else if (g < out.count) {
          tile_store<V>(out, g, o);
        }
      }
    }
  }
}

// FP32 Box-Muller pairs at word phase 2: block i holds the last pair of group
// i - 1 and the first of group i, so each lane stores its own block as two
// 8-byte pieces.  A tile takes the blocks 0 .. count, of the first and the last
// one only the half that lies in it.
template <int V>
__device__ __forceinline__ void tile_halves_loop(const TransformParams& t, const TileBlocks& q,
                                                 const TileOut& out) {
  static_assert(VInfo<V>::es == 4 && VInfo<V>::wpu == 2);
  constexpr uint32_t U = 2;
  // blocks [wf + 1, wl) lie wholly in whole groups; at most two before them and
  // two after them, each element checked
  const uint32_t before = out.wf + 1 < out.count + 1 ? out.wf + 1 : out.count + 1;
  const uint32_t after = out.wl > before ? out.wl : before;
  if (threadIdx.x < 4) {
    const uint32_t i = threadIdx.x < 2 ? threadIdx.x : after + threadIdx.x - 2;
    if (threadIdx.x < 2 ? i < before : i <= out.count) {
      const uint4 o = block_outputs<V>(q.at<false>(i), t);
      const uint32_t ow[4] = {o.x, o.y, o.z, o.w};
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        const int64_t m = 4 * (int64_t)i - 2 + k, e = out.e0 + m;  // in the tile, in the request
        if (m >= 0 && m < 4 * (int64_t)out.count && e >= 0 && e < out.n)
          reinterpret_cast<uint32_t*>(out.base)[e] = ow[k];
      }
    }
  }
  uint32_t i = before + threadIdx.x;
  uint2* dst = reinterpret_cast<uint2*>(out.dst) + 2 * (int64_t)i;
  for (; i + (U - 1) * kThreads < after; i += U * kThreads, dst += 2 * U * kThreads) {
    uint4 o[U];
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) o[u] = block_outputs<V>(q.at<false>(i + u * kThreads), t);
#pragma unroll
    for (uint32_t u = 0; u < U; ++u) {
      uint2* d = dst + 2 * u * kThreads;
      d[-1] = make_uint2(o[u].x, o[u].y);
      d[0] = make_uint2(o[u].z, o[u].w);
    }
  }
  for (; i < after; i += kThreads, dst += 2 * kThreads) {
    const uint4 o = block_outputs<V>(q.at<false>(i), t);
    dst[-1] = make_uint2(o.x, o.y);
    dst[0] = make_uint2(o.z, o.w);
  }
}

// The groups [g0, end) of one request (the whole CTA works on them, so every
// branch below is uniform across it).  Group 0 starts head elements (pw =
// head es / 4 words) before the output.  When pw is a multiple of the unit
// size, group g is the 4 words from word off - pw + 4 g: exactly Philox block
// (off - pw)/4 + g when off - pw is a multiple of 4, else the tail of one
// block and the head of the next.  Otherwise (a Box-Muller pair split by the
// output's start) lanes transform pair-aligned virtual groups one element
// earlier.
template <int V>
__device__ __forceinline__ void batch_tile(const BatchReq& r, uint64_t off_lo, uint64_t off_hi,
                                           int64_t g0, int64_t end) {
  using I = VInfo<V>;
  constexpr int kEpg = 16 / I::es;
  const TransformParams& t = r.t;
  const uint32_t pw = (uint32_t)r.head * (uint32_t)(I::es / 4);
  const bool split = I::epu == 2 && (pw % (uint32_t)I::wpu) != 0;
  // word of (virtual) group 0, and the block of group g0's first word
  const uint32_t back = pw + (split ? (uint32_t)(I::es / 4) : 0u);
  const uint64_t a_lo = off_lo - back, a_hi = off_hi - ((off_lo < back) ? 1u : 0u);
  const uint32_t ph = (uint32_t)a_lo & 3u;
  uint64_t b_lo = (a_lo >> 2) | (a_hi << 62), b_hi = a_hi >> 2;
  add128(b_lo, b_hi, (uint64_t)g0);
  TileOut out;
  out.base = reinterpret_cast<char*>(r.out);
  out.n = r.n;
  out.count = (uint32_t)(end - g0);
  out.e0 = g0 * kEpg - r.head;
  out.dst = reinterpret_cast<uint4*>(out.base + out.e0 * I::es);
  out.wf = out.e0 < 0 ? 1u : 0u;
  out.wl = out.e0 + (end - g0) * kEpg <= r.n ? out.count : out.count - 1u;
  const bool cross = (uint64_t)(uint32_t)b_lo + out.count + 64u >= kPhiloxMaxBlocks;
  const TileBlocks q(r.key0, r.key1, b_lo, b_hi);
  if (I::epu == 2 && split) {
    if constexpr (I::epu == 2) {
      if (!cross) {
        tile_shift_loop<V, false, true>(t, q, ph, out);
      } else {
        tile_shift_loop<V, true, true>(t, q, ph, out);
      }
    }
  } else if (cross) {
    tile_shift_loop<V, true, false>(t, q, ph, out);
  } else if (ph == 0) {
    tile_blocks_loop<V>(t, q, out);
  } else if (I::es == 4 && I::epu == 2 && ph == 2) {
    if constexpr (I::es == 4 && I::epu == 2) tile_halves_loop<V>(t, q, out);
  } else if (I::wpu <= 2 && I::weight == 0 && ph == 2) {
    if constexpr (I::wpu <= 2 && I::weight == 0) tile_shift_loop<V, false, false, 2>(t, q, ph, out);
  } else if (I::wpu == 1 && I::weight == 0) {
    if constexpr (I::wpu == 1 && I::weight == 0) {
      if (ph == 1) {
        tile_shift_loop<V, false, false, 1>(t, q, ph, out);
      } else {
        tile_shift_loop<V, false, false, 3>(t, q, ph, out);
      }
    }
  } else {
    tile_shift_loop<V, false, false>(t, q, ph, out);
  }
}

// One kernel for all variants of a batch; kHeavy also those of the FP64
// fixed-point transforms, whose registers a batch without them need not carry.
// Bound by issue and the FMA-heavy pipe (bits: 59 instructions per group, 44 in
// the single-stream kernel; the rest is the set-up per run of tiles and
// fewer blocks in flight).  The table of 4096 requests at the built-in geometry:
// 858 -> 603 us a launch, 541 with the FP64 add for [-1, 1) and the phases as
// constants (at 603, five CTAs per SM, 48 registers and 376 bytes spilled:
// 5 % slower than four).
// With those transforms (a fifth each FP64 gaussians, lognormals, inverse CDFs, FP32
// uniforms and gaussians): 4096 requests 3.96 -> 2.90 ms (3.29 at the best geometry
// before), 1024 of up to 2^18 305 -> 225 us, 16 of up to 2^14 22.7 -> 19.3.  Both kernels
// stand at the cap of 64 registers.
template <bool kHeavy>
__global__ void __launch_bounds__(kThreads, 4) batch_fill_kernel(const BatchReq* __restrict__ reqs,
                                                              const uint64_t* __restrict__ off,
                                                              const int32_t* __restrict__ tile_req,
                                                              int64_t tiles, int ipt, int run,
                                                              uint64_t* arrivals, bool advance) {
  uint64_t launches = 0;
  if (arrivals != nullptr) {
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(launches) : "l"(arrivals) : "memory");
    launches >>= kArrivalBits;
  }
  // a CTA takes `run` consecutive tiles at a time; those of one request are
  // one longer tile, so that a request's set-up is shared
  for (int64_t t0 = (int64_t)blockIdx.x * run; t0 < tiles; t0 += (int64_t)gridDim.x * run) {
    const int64_t t1 = t0 + run < tiles ? t0 + run : tiles;
    for (int64_t t = t0; t < t1;) {
      const int32_t ri = tile_req[t];
      const BatchReq& r = reqs[ri];
      uint64_t off_lo = off[2 * ri], off_hi = off[2 * ri + 1];
      {
        const uint64_t add = r.adv_lo * launches;
        off_lo += add;
        off_hi += r.adv_hi * launches + __umul64hi(r.adv_lo, launches) + (off_lo < add ? 1u : 0u);
      }
      const int64_t tile = (int64_t)kThreads * ipt;
      const int64_t g0 = (t - r.first_tile) * tile;
      const int64_t left = (r.groups - g0 + tile - 1) / tile;
      const int64_t m = t1 - t < left ? t1 - t : left;
      const int64_t end = g0 + m * tile < r.groups ? g0 + m * tile : r.groups;
      t += m;
      switch (r.variant) {  // uniform per tile
        case V_BITS: batch_tile<V_BITS>(r, off_lo, off_hi, g0, end); break;
        case V_U01_F32: batch_tile<V_U01_F32>(r, off_lo, off_hi, g0, end); break;
        case V_UNI_F32: batch_tile<V_UNI_F32>(r, off_lo, off_hi, g0, end); break;
        case V_U01_F64: batch_tile<V_U01_F64>(r, off_lo, off_hi, g0, end); break;
        case V_AFF_F64: batch_tile<V_AFF_F64>(r, off_lo, off_hi, g0, end); break;
        case V_UNI_F64: batch_tile<V_UNI_F64>(r, off_lo, off_hi, g0, end); break;
        case V_GAUSS_F32: batch_tile<V_GAUSS_F32>(r, off_lo, off_hi, g0, end); break;
        case V_LOGN_F32: batch_tile<V_LOGN_F32>(r, off_lo, off_hi, g0, end); break;
        case V_ICDF_GAUSS_F32: batch_tile<V_ICDF_GAUSS_F32>(r, off_lo, off_hi, g0, end); break;
        case V_ICDF_LOGN_F32: batch_tile<V_ICDF_LOGN_F32>(r, off_lo, off_hi, g0, end); break;
        default:
          if constexpr (kHeavy) {
            switch (r.variant) {
              case V_GAUSS_F64: batch_tile<V_GAUSS_F64>(r, off_lo, off_hi, g0, end); break;
              case V_LOGN_F64: batch_tile<V_LOGN_F64>(r, off_lo, off_hi, g0, end); break;
              case V_ICDF_GAUSS_F64: batch_tile<V_ICDF_GAUSS_F64>(r, off_lo, off_hi, g0, end); break;
              case V_STDGAUSS_F64: batch_tile<V_STDGAUSS_F64>(r, off_lo, off_hi, g0, end); break;
              default: batch_tile<V_ICDF_LOGN_F64>(r, off_lo, off_hi, g0, end); break;
            }
          }
          break;
      }
    }
  }
  // every thread of this CTA has read the launch count: it arrives (a kernel of
  // its own for the offsets took 2.5 us a launch)
  if (arrivals != nullptr && advance) {
    __syncthreads();
    if (threadIdx.x == 0)
      atomicAdd((unsigned long long*)arrivals, (unsigned long long)batch_arrival(blockIdx.x, gridDim.x));
  }
}

}  // namespace

// Consecutive tiles a CTA takes at a time: up to eight, while that leaves 16
// such runs per SM (at 8 groups per thread, runs of at most 1, 4, 8: 4096
// requests 683, 610, 590 us; 1024 requests at most 4, 8: 151, 153).
static int run_of(int64_t tiles) {
  int dev = 0;
  const int64_t r = tiles / ((int64_t)current_device_sms(&dev) * 16);
  return (int)(r < 1 ? 1 : r < 8 ? r : 8);
}

static void launch_tiles(const BatchReq* reqs, const uint64_t* offs, const int32_t* tile_req,
                         int64_t tiles, int ipt, bool heavy, int64_t grid, uint64_t* arrivals,
                         bool advance, cudaStream_t stream) {
  const int run = run_of(tiles);
  if (grid > (tiles + run - 1) / run) grid = (tiles + run - 1) / run;
  if (grid < 1) grid = 1;
  if (grid > (int64_t(1) << kArrivalBits)) grid = int64_t(1) << kArrivalBits;
  (heavy ? batch_fill_kernel<true> : batch_fill_kernel<false>)<<<(unsigned)grid, kThreads, 0, stream>>>(
      reqs, offs, tile_req, tiles, ipt, run, arrivals, advance);
}

int64_t plan_parts(const PartDesc* parts, int32_t count, int ipt, BatchReq* reqs_out,
                   uint64_t* offs_out, int32_t* tiles_out, int64_t tile_cap) {
  const int64_t tile_groups = (int64_t)kThreads * ipt;
  int64_t t = 0;
  for (int32_t i = 0; i < count; ++i) {
    const PartDesc& q = parts[i];
    BatchReq& r = reqs_out[i];
    std::memset(&r, 0, sizeof(r));
    const int64_t epg = 16 / q.es;
    const int32_t head = (int32_t)((q.out & 15u) / (uint64_t)q.es);
    const int64_t groups = q.n == 0 ? 0 : (head + q.n + epg - 1) / epg;
    r.t = q.t;
    r.out = q.out;
    r.n = q.n;
    r.groups = groups;
    r.first_tile = t;
    r.variant = q.variant;
    r.head = head;
    r.key0 = q.key0;
    r.key1 = q.key1;
    offs_out[2 * i] = q.off_lo;
    offs_out[2 * i + 1] = q.off_hi;
    const int64_t nt = (groups + tile_groups - 1) / tile_groups;
    if (t + nt > tile_cap) return -1;
    for (int64_t k = 0; k < nt; ++k) tiles_out[t + k] = i;
    t += nt;
  }
  return t;
}

grng_status enqueue_fill(const BatchReq* d_reqs, const uint64_t* d_offs, const int32_t* d_tiles,
                         int64_t tiles, int ipt, bool heavy, int64_t grid, cudaStream_t stream) {
  if (tiles <= 0) return GRNG_OK;
  launch_tiles(d_reqs, d_offs, d_tiles, tiles, ipt, heavy, grid, nullptr, false, stream);
  const cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) {
    set_error("batch fill launch failed: %s", cudaGetErrorString(err));
    return GRNG_ERR_CUDA;
  }
  return GRNG_OK;
}

}  // namespace grng

struct grng_batch {
  int32_t count;
  int64_t tiles;
  int32_t ipt;           // groups per thread per tile
  int32_t ctas_per_sm;
  bool heavy;            // some request takes an FP64 fixed-point transform
  int32_t sms;
  int32_t device;
  void* workspace;
  size_t workspace_bytes;
  size_t reqs_off, offs_off, count_off, tiles_off;
  std::vector<grng::BatchReq> host_reqs;  // the request records as uploaded
  std::vector<int64_t> groups;            // per request
  int64_t groups_total;
  std::vector<grng_engine_t> engines;  // per request
  std::vector<int32_t> first_req_of_engine;  // per request: index of its engine's first request
  std::vector<uint64_t> start_lo, start_hi;  // per request: start offset at creation
};

using namespace grng;

namespace {

constexpr int32_t kMaxBatch = 1 << 20;

grng_status plan_sizes(const grng_request* reqs, int32_t count, int ipt, int64_t* tiles_out,
                       std::vector<int64_t>* groups, std::vector<int32_t>* heads,
                       std::vector<int>* variants, std::vector<TransformParams>* tps) {
  int64_t tiles = 0;
  const int64_t tile_groups = (int64_t)kThreads * ipt;
  for (int32_t i = 0; i < count; ++i) {
    const grng_request& q = reqs[i];
    uint64_t words = 0;
    grng_status st = grng_words_for(&q.dist, q.n, &words);
    if (st != GRNG_OK) return st;
    if (q.engine == nullptr) {
      set_error("request %d: engine is NULL", i);
      return GRNG_ERR_INVALID_ARG;
    }
    grng_engine_state es;
    grng_engine_get_state(q.engine, &es);
    if (es.kind != GRNG_PHILOX4X32X10) {
      set_error("request %d: batches take Philox4x32-10 engines", i);
      return GRNG_ERR_UNSUPPORTED;
    }
    const int esz = q.dist.dtype == GRNG_F64 ? 8 : 4;
    if ((q.n > 0 && q.out == nullptr) || ((uintptr_t)q.out % (uintptr_t)esz) != 0) {
      set_error("request %d: output pointer NULL or misaligned", i);
      return GRNG_ERR_INVALID_ARG;
    }
    TransformParams t;
    int v = 0;
    st = fill_transform_params(&q.dist, &t, &v);
    if (st != GRNG_OK) return st;
    const int32_t head = (int32_t)(((uintptr_t)q.out & 15u) / (uintptr_t)esz);
    const int64_t epg = 16 / esz;
    const int64_t g = q.n == 0 ? 0 : (head + q.n + epg - 1) / epg;
    groups->push_back(g);
    heads->push_back(head);
    variants->push_back(v);
    tps->push_back(t);
    tiles += (g + tile_groups - 1) / tile_groups;
  }
  *tiles_out = tiles;
  return GRNG_OK;
}

}  // namespace

extern "C" {

grng_status grng_batch_workspace_bytes(const grng_request* reqs, int32_t count, int32_t ipt,
                                       size_t* bytes) {
  if (reqs == nullptr || bytes == nullptr || count < 1 || count > kMaxBatch || ipt < 1 ||
      ipt > 64) {
    set_error("bad batch arguments (count in [1, 2^20], ipt in [1, 64])");
    return GRNG_ERR_INVALID_ARG;
  }
  std::vector<int64_t> groups;
  std::vector<int32_t> heads;
  std::vector<int> variants;
  std::vector<TransformParams> tps;
  int64_t tiles = 0;
  grng_status st = plan_sizes(reqs, count, ipt, &tiles, &groups, &heads, &variants, &tps);
  if (st != GRNG_OK) return st;
  *bytes = align256(sizeof(BatchReq) * (size_t)count) + align256(16u * (size_t)count) +
           align256(sizeof(uint64_t)) + align256(4u * (size_t)(tiles > 0 ? tiles : 1));
  return GRNG_OK;
}

grng_status grng_batch_create(grng_batch_t* out, const grng_request* reqs, int32_t count,
                              int32_t ipt, void* dev_workspace, size_t workspace_bytes,
                              grng_stream_t stream) {
  if (out == nullptr || dev_workspace == nullptr || ((uintptr_t)dev_workspace & 255u) != 0) {
    set_error("out NULL or workspace NULL / not 256-byte aligned");
    return GRNG_ERR_INVALID_ARG;
  }
  size_t need = 0;
  grng_status st = grng_batch_workspace_bytes(reqs, count, ipt, &need);
  if (st != GRNG_OK) return st;
  if (workspace_bytes < need) {
    set_error("workspace of %zu bytes is smaller than the %zu bytes needed", workspace_bytes, need);
    return GRNG_ERR_INVALID_ARG;
  }
  std::vector<int64_t> groups;
  std::vector<int32_t> heads;
  std::vector<int> variants;
  std::vector<TransformParams> tps;
  int64_t tiles = 0;
  st = plan_sizes(reqs, count, ipt, &tiles, &groups, &heads, &variants, &tps);
  if (st != GRNG_OK) return st;

  grng_batch* b = new (std::nothrow) grng_batch;
  if (b == nullptr) {
    set_error("batch allocation failed");
    return GRNG_ERR_OOM;
  }
  b->count = count;
  b->tiles = tiles;
  b->ipt = ipt;
  b->ctas_per_sm = 32;  // resident CTAs eight times over, so that the SMs refill
  b->heavy = false;
  for (int v : variants) b->heavy = b->heavy || variant_is_heavy(v);
  b->sms = current_device_sms(&b->device);
  b->workspace = dev_workspace;
  b->reqs_off = 0;
  b->offs_off = align256(sizeof(BatchReq) * (size_t)count);
  b->count_off = b->offs_off + align256(16u * (size_t)count);
  b->tiles_off = b->count_off + align256(sizeof(uint64_t));
  b->groups_total = 0;

  // Requests of one engine follow each other in its sequence, in table order.
  std::vector<BatchReq> h(count);
  std::vector<uint64_t> offs(2 * (size_t)count);
  std::vector<int32_t> tile_req((size_t)(tiles > 0 ? tiles : 1), 0);
  b->engines.resize(count);
  b->first_req_of_engine.resize(count);
  b->start_lo.resize(count);
  b->start_hi.resize(count);
  struct Acc {
    grng_engine_t e;
    uint64_t lo, hi;   // running offset
    int32_t first;
  };
  std::vector<Acc> acc;
  std::vector<int32_t> acc_of(count);
  std::unordered_map<grng_engine_t, int32_t> index_of;
  index_of.reserve((size_t)count * 2);
  for (int32_t i = 0; i < count; ++i) {
    int32_t a = -1;
    auto it = index_of.find(reqs[i].engine);
    if (it != index_of.end()) {
      a = it->second;
    } else {
      grng_engine_state es;
      grng_engine_get_state(reqs[i].engine, &es);
      acc.push_back({reqs[i].engine, es.offset_lo, es.offset_hi, i});
      a = (int32_t)acc.size() - 1;
      index_of.emplace(reqs[i].engine, a);
    }
    acc_of[i] = a;
    offs[2 * i] = acc[a].lo;
    offs[2 * i + 1] = acc[a].hi;
    b->start_lo[i] = acc[a].lo;
    b->start_hi[i] = acc[a].hi;
    uint64_t words = 0;
    grng_words_for(&reqs[i].dist, reqs[i].n, &words);
    const uint64_t lo = acc[a].lo + words;
    acc[a].hi += (lo < acc[a].lo) ? 1u : 0u;
    acc[a].lo = lo;
    b->engines[i] = reqs[i].engine;
    b->first_req_of_engine[i] = acc[a].first;
  }
  int64_t t = 0;
  const int64_t tile_groups = (int64_t)kThreads * ipt;
  for (int32_t i = 0; i < count; ++i) {
    BatchReq& r = h[i];
    std::memset(&r, 0, sizeof(r));
    r.t = tps[i];
    r.out = (uint64_t)(uintptr_t)reqs[i].out;
    r.n = reqs[i].n;
    r.groups = groups[i];
    r.first_tile = t;
    r.variant = variants[i];
    r.head = heads[i];
    grng_engine_state es;
    grng_engine_get_state(reqs[i].engine, &es);
    r.key0 = (uint32_t)es.seed;
    r.key1 = (uint32_t)(es.seed >> 32);
    // per launch the engine advances by all of its requests' words
    const Acc& A = acc[acc_of[i]];
    const uint64_t s_lo = b->start_lo[A.first], s_hi = b->start_hi[A.first];
    r.adv_lo = A.lo - s_lo;
    r.adv_hi = A.hi - s_hi - ((A.lo < s_lo) ? 1u : 0u);
    const int64_t nt = (groups[i] + tile_groups - 1) / tile_groups;
    for (int64_t k = 0; k < nt; ++k) tile_req[(size_t)(t + k)] = i;
    t += nt;
    b->groups_total += groups[i];
  }
  b->workspace_bytes = workspace_bytes;
  b->groups = groups;
  char* ws = reinterpret_cast<char*>(dev_workspace);
  cudaError_t err =
      cudaMemcpyAsync(ws + b->reqs_off, h.data(), sizeof(BatchReq) * (size_t)count,
                      cudaMemcpyHostToDevice, (cudaStream_t)stream);
  if (err == cudaSuccess)
    err = cudaMemcpyAsync(ws + b->offs_off, offs.data(), 16u * (size_t)count,
                          cudaMemcpyHostToDevice, (cudaStream_t)stream);
  if (err == cudaSuccess)
    err = cudaMemsetAsync(ws + b->count_off, 0, sizeof(uint64_t), (cudaStream_t)stream);
  if (err == cudaSuccess && tiles > 0)
    err = cudaMemcpyAsync(ws + b->tiles_off, tile_req.data(), 4u * (size_t)tiles,
                          cudaMemcpyHostToDevice, (cudaStream_t)stream);
  // the host vectors die here: wait for the copies
  if (err == cudaSuccess) err = cudaStreamSynchronize((cudaStream_t)stream);
  if (err != cudaSuccess) {
    set_error("batch upload failed: %s", cudaGetErrorString(err));
    cudaGetLastError();
    delete b;
    return GRNG_ERR_CUDA;
  }
  b->host_reqs = std::move(h);
  *out = b;
  return GRNG_OK;
}

}  // extern "C"

namespace {

// Tiles of the batch at ipt groups per thread, and whether their map fits the
// workspace given at creation.
int64_t tiles_at(const grng_batch* b, int ipt) {
  const int64_t tile_groups = (int64_t)kThreads * ipt;
  int64_t t = 0;
  for (int64_t g : b->groups) t += (g + tile_groups - 1) / tile_groups;
  return t;
}
bool fits(const grng_batch* b, int ipt) {
  const int64_t t = tiles_at(b, ipt);
  return b->tiles_off + 4u * (size_t)(t > 0 ? t : 1) <= b->workspace_bytes;
}

// Rebuilds the tile map and the requests' first tiles for ipt and uploads
// both (synchronises the stream: the host tables are temporaries).
grng_status replan(grng_batch* b, int ipt, cudaStream_t stream) {
  if (ipt == b->ipt) return GRNG_OK;
  const int64_t tile_groups = (int64_t)kThreads * ipt;
  const int64_t tiles = tiles_at(b, ipt);
  std::vector<int32_t> tile_req((size_t)(tiles > 0 ? tiles : 1), 0);
  std::vector<BatchReq> h = b->host_reqs;
  int64_t t = 0;
  for (int32_t i = 0; i < b->count; ++i) {
    h[i].first_tile = t;
    const int64_t nt = (b->groups[i] + tile_groups - 1) / tile_groups;
    for (int64_t k = 0; k < nt; ++k) tile_req[(size_t)(t + k)] = i;
    t += nt;
  }
  // the launch count is not touched: the device copy is the live one
  char* ws = reinterpret_cast<char*>(b->workspace);
  cudaError_t err = cudaMemcpyAsync(ws + b->reqs_off, h.data(), sizeof(BatchReq) * h.size(),
                                    cudaMemcpyHostToDevice, stream);
  if (err == cudaSuccess && tiles > 0)
    err = cudaMemcpyAsync(ws + b->tiles_off, tile_req.data(), 4u * (size_t)tiles,
                          cudaMemcpyHostToDevice, stream);
  if (err == cudaSuccess) err = cudaStreamSynchronize(stream);
  if (err != cudaSuccess) {
    set_error("batch re-plan upload failed: %s", cudaGetErrorString(err));
    cudaGetLastError();
    return GRNG_ERR_CUDA;
  }
  b->host_reqs = std::move(h);
  b->ipt = ipt;
  b->tiles = tiles;
  return GRNG_OK;
}

}  // namespace

extern "C" {

grng_status grng_batch_set_config(grng_batch_t b, int32_t ipt, int32_t ctas_per_sm,
                                  grng_stream_t stream) {
  if (b == nullptr || ctas_per_sm < 1 || ctas_per_sm > 32 || ipt < 1 || ipt > 64) {
    set_error("bad batch, ipt (1..64) or ctas_per_sm (1..32)");
    return GRNG_ERR_INVALID_ARG;
  }
  if (!fits(b, ipt)) {
    set_error("the tile map at %d groups per thread does not fit the batch's workspace", ipt);
    return GRNG_ERR_INVALID_ARG;
  }
  const grng_status st = replan(b, ipt, (cudaStream_t)stream);
  if (st != GRNG_OK) return st;
  b->ctas_per_sm = ctas_per_sm;
  return GRNG_OK;
}

static grng_status batch_enqueue(grng_batch_t b, cudaStream_t stream, bool advance) {
  char* ws = reinterpret_cast<char*>(b->workspace);
  const BatchReq* reqs = reinterpret_cast<const BatchReq*>(ws + b->reqs_off);
  const uint64_t* offs = reinterpret_cast<const uint64_t*>(ws + b->offs_off);
  const int32_t* tile_req = reinterpret_cast<const int32_t*>(ws + b->tiles_off);
  if (b->tiles > 0)
    launch_tiles(reqs, offs, tile_req, b->tiles, b->ipt, b->heavy, (int64_t)b->sms * b->ctas_per_sm,
                 reinterpret_cast<uint64_t*>(ws + b->count_off), advance, stream);
  const cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) {
    set_error("batch launch failed: %s", cudaGetErrorString(err));
    return GRNG_ERR_CUDA;
  }
  return GRNG_OK;
}

grng_status grng_batch_launch(grng_batch_t b, grng_stream_t stream) {
  if (b == nullptr) {
    set_error("batch is NULL");
    return GRNG_ERR_INVALID_ARG;
  }
  return batch_enqueue(b, (cudaStream_t)stream, true);
}

grng_status grng_batch_autotune(grng_batch_t b, grng_stream_t stream_in, int32_t* best_ipt,
                                int32_t* best_ctas, float* best_ms) {
  if (b == nullptr) {
    set_error("batch is NULL");
    return GRNG_ERR_INVALID_ARG;
  }
  cudaStream_t stream = (cudaStream_t)stream_in;
  const int32_t ipts[] = {1, 2, 4, 8, 16, 32};
  const int32_t ctas[] = {1, 2, 4, 6, 8, 12, 16, 24, 32};
  cudaEvent_t e0, e1;
  if (cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    set_error("event creation failed");
    cudaGetLastError();
    return GRNG_ERR_CUDA;
  }
  float best = 1e30f;
  int32_t arg_ipt = b->ipt, arg_ctas = b->ctas_per_sm;
  grng_status st = GRNG_OK;
  for (int32_t ipt : ipts) {
    if (!fits(b, ipt)) continue;  // a workspace sized for larger tiles
    if ((st = replan(b, ipt, stream)) != GRNG_OK) break;
    for (int32_t c : ctas) {
      b->ctas_per_sm = c;
      // tuning fills do not advance the offsets: they rewrite the same outputs
      if ((st = batch_enqueue(b, stream, false)) != GRNG_OK) break;
      cudaEventRecord(e0, stream);
      for (int k = 0; k < 3 && st == GRNG_OK; ++k) st = batch_enqueue(b, stream, false);
      cudaEventRecord(e1, stream);
      if (st != GRNG_OK) break;
      if (cudaEventSynchronize(e1) != cudaSuccess) {
        set_error("batch autotune: timing failed");
        cudaGetLastError();
        st = GRNG_ERR_CUDA;
        break;
      }
      float ms = 0.f;
      cudaEventElapsedTime(&ms, e0, e1);
      if (ms / 3 < best) {
        best = ms / 3;
        arg_ipt = ipt;
        arg_ctas = c;
      }
    }
    if (st != GRNG_OK) break;
  }
  cudaEventDestroy(e0);
  cudaEventDestroy(e1);
  if (st == GRNG_OK) st = replan(b, arg_ipt, stream);
  b->ctas_per_sm = arg_ctas;
  if (st != GRNG_OK) return st;
  if (best_ipt) *best_ipt = arg_ipt;
  if (best_ctas) *best_ctas = arg_ctas;
  if (best_ms) *best_ms = best;
  return GRNG_OK;
}

grng_status grng_batch_commit(grng_batch_t b, grng_stream_t stream) {
  if (b == nullptr) {
    set_error("batch is NULL");
    return GRNG_ERR_INVALID_ARG;
  }
  uint64_t arrivals = 0;
  const char* ws = reinterpret_cast<const char*>(b->workspace);
  cudaError_t err = cudaMemcpyAsync(&arrivals, ws + b->count_off, sizeof(arrivals), cudaMemcpyDeviceToHost,
                                    (cudaStream_t)stream);
  if (err == cudaSuccess) err = cudaStreamSynchronize((cudaStream_t)stream);
  if (err != cudaSuccess) {
    set_error("batch commit failed: %s", cudaGetErrorString(err));
    cudaGetLastError();
    return GRNG_ERR_CUDA;
  }
  // an engine continues at its first request's start plus the launches'
  // advances: skip it ahead to that offset
  for (int32_t i = 0; i < b->count; ++i) {
    if (b->first_req_of_engine[i] != i) continue;
    grng_engine_state es;
    grng_engine_get_state(b->engines[i], &es);
    const BatchReq& r = b->host_reqs[i];
    const unsigned __int128 at =
        (((unsigned __int128)b->start_hi[i] << 64) | b->start_lo[i]) +
        (((unsigned __int128)r.adv_hi << 64) | r.adv_lo) * (arrivals >> kArrivalBits);
    const unsigned __int128 skip = at - (((unsigned __int128)es.offset_hi << 64) | es.offset_lo);
    const uint64_t d_lo = (uint64_t)skip, d_hi = (uint64_t)(skip >> 64);
    grng_engine_skip_ahead(b->engines[i], d_lo, d_hi);
  }
  return GRNG_OK;
}

grng_status grng_batch_destroy(grng_batch_t b) {
  delete b;
  return GRNG_OK;
}

}  // extern "C"
