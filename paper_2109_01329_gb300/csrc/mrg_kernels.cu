// MRG32k3a fill kernels with the distribution transform fused in.
//
// MRG32k3a (L'Ecuyer 1999; the paper's "MRG-based generators", Sec. 4.1) is a
// sequential recursion, so the output is cut into per-thread chunks of
// consecutive units.  Each thread
//   1. jumps the call's starting state to its chunk, one matrix-vector product
//      per radix-32 digit of the distance, from a compile-time table of
//      A^(k 2^(5 d));
//   2. steps the two component recursions in registers, with products
//      reduced by folding 2^32 = c (mod 2^32 - c) instead of dividing;
//   3. transforms each 16 bytes of outputs and writes them to its row of a
//      per-warp shared-memory stage (swizzled: no bank conflicts);
//   4. with its warp, copies the 32 staged rows out with 16-byte stores, 8
//      lanes per 128-byte row.
// Chunks are placed so that every chunk starts on a 16-byte output boundary
// (the first chunk of a stream has virtual head units), hence aligned rows.
// When the output's start splits a Box-Muller pair (an odd element offset
// into a 16-byte group) each chunk starts one pair earlier, with the pair
// that straddles its first 16-byte boundary, and stages its outputs shifted
// by one element (a one-element carry from pair to pair), so the rows are
// again whole 16-byte groups; the straddling pair is computed by both
// neighbouring chunks.
#include <cuda_runtime.h>

#include <cstdint>

#include "device_common.cuh"
#include "grng_internal.h"
#include "mrg_tables.h"

namespace grng {

__device__ const mrg::DigitTable d_mrg_digits = mrg::make_digit_table();

namespace {

using namespace dev;

constexpr int kThreads = 256;
constexpr int kRowLg = 3;  // log2 of the 16-byte pieces of a staged row (128 bytes)

struct MrgParams {
  TransformParams t;
  void* out;
  int64_t n;                  // elements per stream
  int64_t units;              // units per stream
  int64_t out_words;          // output words per stream (n * es / 4)
  int64_t chunk_units;        // units per thread (multiple of 32 / wpu)
  int64_t chunks_per_stream;
  int64_t total_chunks;
  int64_t head_units;         // virtual units before `out` in the first chunk
  int32_t row_lg;             // log2 of a row's 16-byte pieces (mode 4; else kRowLg)
  uint64_t stride_lo, stride_hi;  // word stride between streams
  uint32_t m1, m2;            // the moduli, as operands the compiler does not know
  uint32_t x[6];              // state at the call's word offset
};

struct MrgRegs {
  uint32_t a0, a1, a2;  // x1_{n-3}, x1_{n-2}, x1_{n-1}
  uint32_t b0, b1, b2;  // x2_{n-3}, x2_{n-2}, x2_{n-1}
};

__device__ __forceinline__ uint64_t mul_wide(uint32_t a, uint32_t b) {
  uint64_t r;
  asm("mul.wide.u32 %0, %1, %2;" : "=l"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint64_t mad_wide(uint32_t a, uint32_t b, uint64_t c) {
  uint64_t r;
  asm("mad.wide.u32 %0, %1, %2, %3;" : "=l"(r) : "r"(a), "r"(b), "l"(c));
  return r;
}

// lo + 2^32 (h - 1) mod m = 2^32 - c, h c < 2^32: with L = lo + h c, the
// value is congruent to L - c.  Where the 32-bit sum carries, L - 2^32 is
// that value mod m and below m (h c < m); where it does not, L < 2^32 makes
// L - c < m.  So one comparison and one conditional subtraction give the
// canonical residue, where a fold of lo + 2^32 h needs one pair for the carry
// and one for the residue at or above m.
template <uint32_t kC>
__device__ __forceinline__ uint32_t fold_carry(uint32_t lo, uint32_t h) {
  uint32_t n = lo + h * kC;
  asm("{ .reg .pred p; setp.ge.u32 p, %0, %1; @p sub.u32 %0, %0, %2; }"
      : "+r"(n) : "r"(lo), "n"(kC));
  return n;
}

// One step of both components; returns z_n = (x1_n - x2_n) mod m1.
// -a13 x = a13 (m1 - x) (mod m1) keeps the sums non-negative and below 2^54;
// m1's sum folds at once (its high word times c1 fits 32 bits), m2's high
// word times c2 needs 37 bits, so one wide fold goes before.
//
// Bound by the FMA-heavy pipe, which takes every product (a wide one about
// 4.5 cycles per warp) and every add that the compiler issues as an IMAD; it
// splits the adds evenly between that pipe and the ALU, so fewer instructions
// of any kind relieve it.  Steps alone, per word and warp: 28.6 instructions
// and 44.4 cycles with two conditional corrections per component, 22.7 and
// 38.7 with fold_carry, 20.6 and 35.5 with the moduli read from the kernel's
// parameters (as immediates the two subtractions cost a further instruction
// each).  Wide products with a constant or (lo, 1) as the 64-bit addend in
// place of the two 32-bit adds cost two moves each (23.6 instructions).  In
// the fills: 10^9 bits 1.250 -> 0.976 ms, 16384 x 16384 FP64 gaussians
// 2.099 -> 1.986 ms.
__device__ __forceinline__ uint32_t mrg_next(MrgRegs& s, const MrgParams& p) {
  const uint64_t p1 = mad_wide(p.m1 - s.a0, mrg::A13, mul_wide(s.a1, mrg::A12));
  const uint64_t p2 = mad_wide(p.m2 - s.b0, mrg::A23, mul_wide(s.b2, mrg::A21));
  const uint32_t n1 = fold_carry<mrg::C1>((uint32_t)p1, (uint32_t)(p1 >> 32) + 1u);
  const uint64_t t = mul_wide((uint32_t)(p2 >> 32), mrg::C2);
  uint32_t tl, th;  // lo(p2) + t, its high word one up (below 2^6)
  asm("add.cc.u32 %0, %2, %3; addc.u32 %1, %4, 1;"
      : "=r"(tl), "=r"(th)
      : "r"((uint32_t)p2), "r"((uint32_t)t), "r"((uint32_t)(t >> 32)));
  const uint32_t n2 = fold_carry<mrg::C2>(tl, th);
  s.a0 = s.a1;
  s.a1 = s.a2;
  s.a2 = n1;
  s.b0 = s.b1;
  s.b1 = s.b2;
  s.b2 = n2;
  uint32_t z = n1 - n2;  // below 0: + m1, which is - c1 in 32 bits
  asm("{ .reg .pred p; setp.lt.u32 p, %1, %2; @p sub.u32 %0, %0, %3; }"
      : "+r"(z) : "r"(n1), "r"(n2), "n"(mrg::C1));
  return z;
}

// One row of y = M x mod m.  The three products' low and high words are summed
// apart (L < 3 2^32, H < 3 2^32), so one fold of L + 2^32 H serves all three:
// H c in one wide product (below 2^47) plus the carry of H times c^2, and the
// 48-bit sum folds as in a step.
template <uint32_t kC>
__device__ __forceinline__ uint32_t row_mod(uint32_t m0, uint32_t m1, uint32_t m2, uint32_t x0,
                                            uint32_t x1, uint32_t x2) {
  const uint64_t p0 = mul_wide(m0, x0), p1 = mul_wide(m1, x1), p2 = mul_wide(m2, x2);
  const uint64_t L = (uint64_t)(uint32_t)p0 + (uint32_t)p1 + (uint32_t)p2;
  const uint64_t H = (p0 >> 32) + (p1 >> 32) + (p2 >> 32);
  const uint64_t t = L + mul_wide((uint32_t)H, kC) + (uint32_t)(H >> 32) * (kC * kC);
  return fold_carry<kC>((uint32_t)t, (uint32_t)(t >> 32) + 1u);
}

// One component's three state words by the matrix at r (9 words).
template <uint32_t kC>
__device__ __forceinline__ void apply(const uint4* r, uint32_t& x0, uint32_t& x1, uint32_t& x2) {
  const uint4 q0 = __ldg(r), q1 = __ldg(r + 1);
  const uint32_t q2 = __ldg(&r[2].x);
  const uint32_t y0 = row_mod<kC>(q0.x, q0.y, q0.z, x0, x1, x2);
  const uint32_t y1 = row_mod<kC>(q0.w, q1.x, q1.y, x0, x1, x2);
  const uint32_t y2 = row_mod<kC>(q1.z, q1.w, q2, x0, x1, x2);
  x0 = y0;
  x1 = y1;
  x2 = y2;
}

// Jumps by e words: one matrix-vector product per radix-32 digit of e that is
// not zero in every lane (each lane its own digit; the identity where it is
// zero).  A thread's first word inside a fill of 2^20 words takes 3 or 4 of
// them, where one level per bit took 14 or more; the table serves every chunk
// length and stride, so a launch prepares nothing.
__device__ __forceinline__ void jump(MrgRegs& s, uint64_t e_lo, uint64_t e_hi) {
  const uint4* row = reinterpret_cast<const uint4*>(d_mrg_digits.row[0]);
  constexpr int kRow16 = mrg::kRowWords / 4;
  while (__any_sync(0xFFFFFFFFu, (e_lo | e_hi) != 0)) {
    const uint32_t k = (uint32_t)e_lo & 31u;
    if (__any_sync(0xFFFFFFFFu, k != 0)) {
      apply<mrg::C1>(row + k * kRow16, s.a0, s.a1, s.a2);
      apply<mrg::C2>(row + k * kRow16 + 3, s.b0, s.b1, s.b2);
    }
    e_lo = (e_lo >> 5) | (e_hi << 59);
    e_hi >>= 5;
    row += 32 * kRow16;
  }
}

// Generates one unit's words and writes its kWpu output words to o.
template <int V>
__device__ __forceinline__ void gen_unit(MrgRegs& st, uint32_t* o, const MrgParams& p,
                                         bool odd = false) {
  constexpr int kWpu = VInfo<V>::wpu;
  uint32_t w[kWpu];
#pragma unroll
  for (int i = 0; i < kWpu; ++i) w[i] = mrg_next(st, p);
  unit_outputs<V>(w, o, p.t, odd);
}

// The 16-byte stage chunk from 4 new output words: as they are, or (carry
// mode) shifted up by one element of kOwpe words behind the carried element,
// whose place the new last element takes.
template <bool kCarry, int kOwpe>
__device__ __forceinline__ uint4 shift_in(uint32_t* carry, const uint32_t* o4) {
  if constexpr (!kCarry) {
    return make_uint4(o4[0], o4[1], o4[2], o4[3]);
  } else if constexpr (kOwpe == 1) {
    const uint4 v = make_uint4(carry[0], o4[0], o4[1], o4[2]);
    carry[0] = o4[3];
    return v;
  } else {
    const uint4 v = make_uint4(carry[0], carry[1], o4[0], o4[1]);
    carry[0] = o4[2];
    carry[1] = o4[3];
    return v;
  }
}

// kMode: 1 chunks start on 16-byte boundaries at unit boundaries; 2 chunks start on
// 16-byte boundaries one element into a Box-Muller pair (carry mode);
// 3 substreams of unequal 16-byte phase: each stream has its own head, and
// its own carry mode when its start splits a pair (a warp's 32 chunks lie in
// one stream, so both are warp-uniform); 4 is 1 with rows shorter than 128
// bytes (a small fill; their length a run-time value costs a long fill 1 %).
template <int V, int kMode>
__global__ void __launch_bounds__(kThreads) mrg_fill_kernel(const __grid_constant__ MrgParams p) {
  constexpr bool kPerStream = kMode == 3;
  constexpr int kWpu = VInfo<V>::wpu;
  constexpr int kOwpe = VInfo<V>::ow_per_elem;
  // 16-byte pieces of a row, and its units (a sub-chunk of the chunk)
  const int lg = kMode == 4 ? p.row_lg : kRowLg;
  const int pieces = 1 << lg;
  const int su = 4 * pieces / kWpu;
  constexpr int kCopyUnroll = kMode == 4 ? 1 : 8;
  // per warp: 32 rows (one per lane) of 8 16-byte chunks; chunk q of row r is
  // kept at position q ^ (r & 7), so a lane's chunk stores and the copy-out's
  // row loads are both free of bank conflicts
  extern __shared__ uint4 stage[][32][8];
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int64_t cid = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const bool active = cid < p.total_chunks;
  int64_t s = 0, c = active ? cid : 0;
  if (p.total_chunks != p.chunks_per_stream && active) {  // several streams
    s = cid / p.chunks_per_stream;
    c = cid - s * p.chunks_per_stream;
  }
  // the stream's head (virtual units before its output's first 16-byte
  // group) and whether its start splits a pair
  int64_t hu = p.head_units;
  bool kCarry = kMode == 2;
  if constexpr (kPerStream) {
    const uint32_t he = (uint32_t)(((uintptr_t)p.out + (uintptr_t)(s * p.n * VInfo<V>::es)) &
                                   15u) /
                        (uint32_t)VInfo<V>::es;
    constexpr uint32_t kEpu = (uint32_t)VInfo<V>::epu;
    hu = (int64_t)((he + kEpu - 1) / kEpu);
    kCarry = kEpu == 2 && (he & 1u) != 0;
  }
  const int64_t u_first = c * p.chunk_units - hu;

  // words to skip: s * stride + max(u_first, 0) * wpu  (mod 2^128)
  MrgRegs st = {p.x[0], p.x[1], p.x[2], p.x[3], p.x[4], p.x[5]};
  uint64_t e_lo = 0, e_hi = 0;
  if (active) {
    const uint64_t us = (uint64_t)s;
    e_lo = us * p.stride_lo;
    e_hi = __umul64hi(us, p.stride_lo) + us * p.stride_hi;
    const uint64_t add = (uint64_t)((u_first > 0 ? u_first : 0) * kWpu);
    const uint64_t sum = e_lo + add;
    e_hi += (sum < e_lo) ? 1u : 0u;
    e_lo = sum;
  }
  jump(st, e_lo, e_hi);

  // carry mode: the chunk's first unit straddles its first 16-byte boundary;
  // only its second element is output here (the previous chunk outputs the
  // first), and every later element moves up one place
  uint32_t carry[kOwpe];
  if (kCarry) {
    uint32_t o[kWpu];
#pragma unroll
    for (int i = 0; i < kWpu; ++i) o[i] = 0u;
    if (active && u_first >= 0 && u_first < p.units) gen_unit<V>(st, o, p);
#pragma unroll
    for (int i = 0; i < kOwpe; ++i) carry[i] = o[kOwpe + i];
  }
  const int64_t nsub = p.chunk_units / su;
  uint32_t* out_words = reinterpret_cast<uint32_t*>(p.out);
  // Copy-out: of 8-piece rows a lane copies piece (lane & 7) of rows
  // it * 4 + (lane >> 3), it = 0..7, and likewise of shorter ones.  The host
  // makes chunks_per_stream a multiple of 32 when there are several streams,
  // so the 32 chunks of a warp lie in one stream and row r is chunk cw + r of
  // that stream.
  const int64_t cw = ((int64_t)blockIdx.x * blockDim.x + warp * 32);  // warp's first chunk id
  const int64_t sw = __shfl_sync(0xFFFFFFFFu, s, 0);
  const int64_t cw_in = cw - sw * p.chunks_per_stream;
  const int64_t lim_chunks = (sw + 1) * p.chunks_per_stream < p.total_chunks
                                 ? (sw + 1) * p.chunks_per_stream
                                 : p.total_chunks;
  const int rows_active = (int)((lim_chunks - cw) < 32 ? (lim_chunks - cw) : 32);
  const int piece = lane & (pieces - 1), row0 = lane >> lg, row_step = 32 >> lg;
  const int64_t row_stride = row_step * p.chunk_units * kWpu;  // words between rows it and it + 1
  const int64_t ow_lane = ((cw_in + row0) * p.chunk_units - hu) * kWpu +
                          (kCarry ? kOwpe : 0) + piece * 4;
  uint32_t* stream_out = out_words + sw * p.out_words;
  for (int64_t q = 0; q < nsub; ++q) {
    // first unit of this sub-chunk (in carry mode after the straddling one)
    const int64_t ub = u_first + (kCarry ? 1 : 0) + q * su;
    constexpr int kUpc = 4 / kWpu;          // units per 16-byte chunk
    if (active) {
      if (ub >= 0 && ub + su <= p.units) {
        constexpr int kChUnroll = VInfo<V>::weight == 0 ? 8 : VInfo<V>::weight == 1 ? 2 : 1;
#pragma unroll kChUnroll
        for (int ch = 0; ch < pieces; ++ch) {
          uint32_t w[4];
#pragma unroll
          for (int i = 0; i < 4; ++i) w[i] = mrg_next(st, p);
          const uint4 o = block_outputs<V>(make_uint4(w[0], w[1], w[2], w[3]), p.t);
          const uint32_t o4[4] = {o.x, o.y, o.z, o.w};
          stage[warp][lane][ch ^ (lane & 7)] = kCarry ? shift_in<true, kOwpe>(carry, o4)
                                                      : shift_in<false, kOwpe>(carry, o4);
        }
      } else {
        for (int ch = 0; ch < pieces; ++ch) {
          uint32_t o4[4] = {0u, 0u, 0u, 0u};
#pragma unroll
          for (int u = 0; u < kUpc; ++u) {
            const int64_t unit = ub + ch * kUpc + u;
            if (unit >= 0 && unit < p.units) gen_unit<V>(st, o4 + u * kWpu, p);
          }
          stage[warp][lane][ch ^ (lane & 7)] = kCarry ? shift_in<true, kOwpe>(carry, o4)
                                                      : shift_in<false, kOwpe>(carry, o4);
        }
      }
    }
    __syncwarp();
    // interior sub-chunks (every row present and inside the stream, the
    // common case) store without per-row checks
    const int64_t ow0 = ow_lane + q * (4 * pieces);
    const bool inside = ow0 >= 0 && ow0 + (pieces - 1) * row_stride + 4 <= p.out_words;
    if (__all_sync(0xFFFFFFFFu, inside && rows_active == 32)) {
      uint32_t* dst = stream_out + ow0;
      if (lg == kRowLg) {
#pragma unroll
        for (int it = 0; it < 8; ++it) {
          const int r = it * 4 + (lane >> 3);
          store16(dst + it * row_stride, stage[warp][r][(lane & 7) ^ (r & 7)]);
        }
      } else {
        for (int it = 0; it < pieces; ++it) {
          const int r = it * row_step + row0;
          store16(dst + it * row_stride, stage[warp][r][piece ^ (r & 7)]);
        }
      }
      __syncwarp();
      continue;
    }
#pragma unroll kCopyUnroll
    for (int it = 0; it < pieces; ++it) {
      const int r = it * row_step + row0;
      if (r >= rows_active) continue;
      const int64_t ow = ow_lane + it * row_stride + q * (4 * pieces);
      const uint4 v = stage[warp][r][piece ^ (r & 7)];
      if (ow >= 0 && ow + 4 <= p.out_words) {
        store16(stream_out + ow, v);
      } else {
        const uint32_t src[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int i = 0; i < 4; ++i)
          if (ow + i >= 0 && ow + i < p.out_words) stream_out[ow + i] = src[i];
      }
    }
    __syncwarp();
  }
}

template <int V>
grng_status launch_variant(const FillRequest& r, cudaStream_t stream) {
  using I = VInfo<V>;
  int dev = 0;
  const int sms = current_device_sms(&dev);
  MrgParams p;
  p.t = r.t;
  p.out = r.out;
  p.n = r.n;
  p.units = (r.n + I::epu - 1) / I::epu;
  p.out_words = r.n * (I::es / 4);
  p.stride_lo = r.stride_lo;
  p.stride_hi = r.stride_hi;
  p.m1 = mrg::M1;
  p.m2 = mrg::M2;
  for (int i = 0; i < 6; ++i) p.x[i] = r.mrg[i];

  const uintptr_t addr = (uintptr_t)r.out;
  const uint32_t phase_w = (uint32_t)((addr & 15u) / 4u);
  const uint64_t stream_bytes = (uint64_t)r.n * I::es;
  const bool uniform_streams = r.num_streams == 1 || (stream_bytes % 16u) == 0;
  const bool aligned = uniform_streams && (phase_w % (uint32_t)I::wpu) == 0;
  // a Box-Muller pair split by the output's start: head elements odd
  const int64_t head_e = (int64_t)(phase_w * 4u / I::es);
  const bool carry = uniform_streams && !aligned && I::epu == 2 && (head_e & 1) != 0;
  // substreams of unequal phase: per-stream heads up to the largest possible
  // one, ceil((16 / es - 1) / epu) units
  const bool per_stream = !uniform_streams;
  const int64_t hu_max = (16 / I::es - 1 + I::epu - 1) / I::epu;
  p.head_units = aligned ? (int64_t)(phase_w / I::wpu)
                 : carry ? (head_e + 1) / 2
                 : per_stream ? hu_max : 0;

  // Threads per SM of the chunk plan, one chunk each: 3072 (several waves,
  // so that an SM refills as its CTAs finish) while that leaves a thread 256
  // words or more, else 2048; or the tuned count.  10^9 bits 0.990 -> 0.958
  // ms, 10^9 FP64 uniforms 2.518 -> 2.410 ms with 3072; 10^8 bits 0.1125
  // with 2048, 0.1149 with 3072.
  const int32_t geom = fill_geometry(GRNG_MRG32K3A, V, r.n * r.num_streams);
  const int64_t span = p.units + p.head_units;
  const int64_t words = span * I::wpu * r.num_streams;
  const int64_t target_threads =
      (int64_t)sms * (geom > 0 ? 256 * (int64_t)geom : words >= (int64_t)sms * 3072 * 256 ? 3072 : 2048);
  int64_t per_stream_threads = target_threads / r.num_streams;
  if (per_stream_threads < 1) per_stream_threads = 1;
  // Rows of 128 bytes; in a small fill of the FP64 fixed-point transforms,
  // whose pair or inverse CDF is a long serial chain, shorter rows share that
  // chain among more threads, up to 256 per SM (FP64 gaussians: 10^3 13.4 ->
  // 3.7 us, 10^5 9.7 -> 5.3; with up to 512 per SM 3 10^5 take 9.6 us in place
  // of 7.0, the jumps outweighing the chain).
  int lg = kRowLg;
  if (I::weight == 2 && aligned)
    while (lg > 0 && words < ((int64_t)sms * 256 << (lg + 2))) --lg;
  p.row_lg = lg;
  const int64_t su = (4 << lg) / I::wpu;
  // At least two rows a thread where that leaves 4 warps per scheduler: the
  // jump costs a thread about 20 words' steps (10^7 FP32 uniforms 18.1 us
  // with 64 words a thread, 20.1 with 32; 10^6 4.9 with 32, 5.3 with 64).
  const int64_t min_cu = words >= (int64_t)sms * 512 * (8 << lg) ? 2 * su : su;
  int64_t cu = (span + per_stream_threads - 1) / per_stream_threads;
  if (cu < min_cu) cu = min_cu;
  cu = (cu + su - 1) / su * su;
  int64_t cps = (span + cu - 1) / cu;
  if (r.num_streams > 1) {
    // a multiple of 32 chunks per stream keeps each warp's 32 chunks inside
    // one stream; the units are spread over all of them
    cps = (cps + 31) / 32 * 32;
    cu = (span + cps - 1) / cps;
    cu = (cu + su - 1) / su * su;
  }
  p.chunk_units = cu;
  p.chunks_per_stream = cps;
  p.total_chunks = p.chunks_per_stream * r.num_streams;
  // Threads per CTA: 128 spreads a small fill's warps over more SMs and fits
  // the light kernels' registers better (10^8 FP32 uniforms 116.6 us against
  // 122.5 with 256, 10^5 3.7 against 4.5); the long chunks of the FP64
  // fixed-point transforms keep 256 (10^9 FP64 gaussians 6.99 ms against 7.09).
  const int threads = I::weight == 2 && cu * I::wpu >= 1024 ? 256 : 128;
  const int64_t grid = (p.total_chunks + threads - 1) / threads;
  const size_t smem = (size_t)(threads / 32) * 32 * 8 * sizeof(uint4);
  if (grid > 0x7FFFFFFF) {
    set_error("MRG32k3a fill: grid too large");
    return GRNG_ERR_UNSUPPORTED;
  }
  if (lg != kRowLg) {
    if constexpr (I::weight == 2) mrg_fill_kernel<V, 4><<<(unsigned)grid, threads, smem, stream>>>(p);
  } else if (aligned) {
    mrg_fill_kernel<V, 1><<<(unsigned)grid, threads, smem, stream>>>(p);
  } else if (carry) {
    if constexpr (I::epu == 2) mrg_fill_kernel<V, 2><<<(unsigned)grid, threads, smem, stream>>>(p);
  } else {
    mrg_fill_kernel<V, 3><<<(unsigned)grid, threads, smem, stream>>>(p);
  }
  const cudaError_t err = cudaGetLastError();
  if (err != cudaSuccess) {
    set_error("MRG32k3a fill launch failed: %s", cudaGetErrorString(err));
    return GRNG_ERR_CUDA;
  }
  return GRNG_OK;
}

}  // namespace

grng_status launch_mrg(const FillRequest& r, CUstream_st* stream) {
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

}  // namespace grng
