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
//   3. transforms each 16 bytes of outputs and stores them, 32 bytes at a time
//      where the output allows: a whole sector, so that the lanes' strided
//      stores move no more memory than coalesced ones.
// Chunks are placed so that every chunk starts on a 16-byte output boundary
// (the first chunk of a stream has virtual head units), hence aligned rows.
// When the output's start splits a Box-Muller pair (an odd element offset
// into a 16-byte group) each chunk starts one pair earlier, with the pair
// that straddles its first 16-byte boundary, and stores its outputs shifted
// by one element (a one-element carry from pair to pair), again in whole
// 16-byte groups; the straddling pair is computed by both neighbouring chunks.
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

struct MrgParams {
  TransformParams t;
  void* out;
  int64_t n;                  // elements per stream
  int64_t units;              // units per stream
  int64_t out_words;          // output words per stream (n * es / 4)
  int64_t chunk_units;        // units per thread (multiple of 8 / wpu: 32 bytes)
  int64_t chunks_per_stream;
  int64_t total_chunks;
  int64_t head_units;         // virtual units before `out` in the first chunk
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
  static_assert(alignof(mrg::DigitTable) >= 16 && mrg::kRowWords % 4 == 0);
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
__device__ __forceinline__ void gen_unit(MrgRegs& st, uint32_t* o, const MrgParams& p) {
  constexpr int kWpu = VInfo<V>::wpu;
  uint32_t w[kWpu];
#pragma unroll
  for (int i = 0; i < kWpu; ++i) w[i] = mrg_next(st, p);
  unit_outputs<V>(w, o, p.t);
}

// The 16-byte group from 4 new output words: as they are, or (carry
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

// A warp's lanes store 32 bytes each, a chunk apart.  Staging 32 rows per warp in
// shared memory to store them coalesced took 3 instructions per word more: 10^9
// bits 0.958 -> 0.840 ms, FP64 uniforms 2.41 -> 2.14, FP32 gaussians 1.575 ->
// 1.440, FP64 gaussians 7.06 -> 6.67.  With 16-byte stores, half a sector each, the
// FP64 gaussians took 8.08 ms.
__device__ __forceinline__ void store32(void* p, uint4 a, uint4 b) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y),
               "r"(a.z), "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}

// kMode: 1 chunks start on 16-byte boundaries at unit boundaries; 2 chunks start on
// 16-byte boundaries one element into a Box-Muller pair (carry mode);
// 3 substreams of unequal 16-byte phase: each stream has its own head, and
// its own carry mode when its start splits a pair.
template <int V, int kMode>
__global__ void __launch_bounds__(kThreads) mrg_fill_kernel(const __grid_constant__ MrgParams p) {
  constexpr bool kPerStream = kMode == 3;
  constexpr int kWpu = VInfo<V>::wpu;
  constexpr int kOwpe = VInfo<V>::ow_per_elem;
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
  if (!active) return;
  // the chunk's output words: its first 16-byte group starts at word w of the
  // stream, before word 0 in a first chunk with head units
  const int64_t w = u_first * kWpu + (kCarry ? kOwpe : 0);
  const int64_t left = p.out_words - w;
  const int64_t count = p.chunk_units * kWpu < left ? p.chunk_units * kWpu : left;  // words to write
  uint32_t* dst = reinterpret_cast<uint32_t*>(p.out) + s * p.out_words + w;
  // a group at either end of the stream: virtual units make no words, and each
  // output word is checked
  auto edge = [&](int64_t at) {
    uint32_t o4[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int u = 0; u < 4 / kWpu; ++u) {
      const int64_t unit = u_first + (kCarry ? 1 : 0) + at / kWpu + u;
      if (unit >= 0 && unit < p.units) gen_unit<V>(st, o4 + u * kWpu, p);
    }
    const uint4 v = kCarry ? shift_in<true, kOwpe>(carry, o4) : shift_in<false, kOwpe>(carry, o4);
    const uint32_t src[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (w + at + i >= 0 && at + i < count) dst[at + i] = src[i];
  };
  auto group = [&]() {
    uint32_t x[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) x[i] = mrg_next(st, p);
    const uint4 o = block_outputs<V>(make_uint4(x[0], x[1], x[2], x[3]), p.t);
    const uint32_t o4[4] = {o.x, o.y, o.z, o.w};
    return kCarry ? shift_in<true, kOwpe>(carry, o4) : shift_in<false, kOwpe>(carry, o4);
  };
  int64_t at = 0;
  if (w < 0 && count > 0) {
    edge(0);
    at = 4;
  }
  uint32_t* q = dst + at;
  uint32_t* const end = dst + (at < count ? at + (count - at) / 4 * 4 : at);  // whole groups
  if (q != end && ((uintptr_t)q & 31u) != 0) {
    store16(q, group());
    q += 4;
  }
  uint32_t* const end32 = end - ((end - q) & 4);
  // 48 or 24 words a turn: a multiple of three steps leaves the state where it
  // was without moves (10^9 bits at 24, 32, 48 words: 0.860, 0.852, 0.840 ms;
  // FP32 gaussians at 8, 24, 48: 1.476, 1.440, 1.420, lognormals 1.704, -,
  // 1.683); the FP64 fixed-point bodies would leave the instruction cache
  constexpr int kUnroll = VInfo<V>::weight == 0 ? 6 : VInfo<V>::weight == 1 ? 3 : 1;
#pragma unroll kUnroll
  for (; q != end32; q += 8) {
    const uint4 a = group();
    store32(q, a, group());
  }
  if (q != end) {
    store16(q, group());
    q += 4;
  }
  if (q - dst < count) edge(q - dst);
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

  // Threads per SM of the chunk plan, one chunk each, or the tuned count: 3072
  // for long fills (several waves, so that an SM refills as its CTAs finish:
  // 10^9 FP64 gaussians 6.67 ms, with 2048 6.78), 1536 for middling ones of the
  // shorter transforms (10^8 bits 96 us, with 2048 99), 2048 below.
  const int32_t geom = fill_geometry(GRNG_MRG32K3A, V, r.asked);
  const int64_t span = p.units + p.head_units;
  const int64_t words = span * I::wpu * r.num_streams;
  const int64_t per_sm = geom > 0                                              ? 256 * (int64_t)geom
                         : words >= (int64_t)sms * (I::weight == 2 ? 786432 : 2621440) ? 3072
                         : I::weight < 2 && words >= (int64_t)sms * 393216              ? 1536
                                                                                        : 2048;
  const int64_t target_threads = (int64_t)sms * per_sm;
  int64_t per_stream_threads = target_threads / r.num_streams;
  if (per_stream_threads < 1) per_stream_threads = 1;
  // Chunks of whole 32-byte pieces: at least 32 words a thread, since the jump
  // costs about 20 words' steps, and 64 where that leaves 4 warps per
  // scheduler (10^7 FP32 uniforms 18.1 us with 64 words a thread, 20.1 with 32;
  // 10^6 4.9 with 32, 5.3 with 64); the FP64 fixed-point transforms, whose pair
  // or inverse CDF is a long serial chain, down to 8 in small fills, up to 256
  // threads per SM (FP64 gaussians: 10^3 13.4 -> 3.7 us, 10^5 9.7 -> 5.3).
  const int64_t su = 8 / I::wpu;
  int64_t min_words = words >= (int64_t)sms * 512 * 64 ? 64 : 32;
  if (I::weight == 2)
    while (min_words > 8 && words < (int64_t)sms * 256 * min_words) min_words /= 2;
  const int64_t min_cu = min_words / I::wpu;
  int64_t cu = (span + per_stream_threads - 1) / per_stream_threads;
  if (cu < min_cu) cu = min_cu;
  cu = (cu + su - 1) / su * su;
  int64_t cps = (span + cu - 1) / cu;
  p.chunk_units = cu;
  p.chunks_per_stream = cps;
  p.total_chunks = p.chunks_per_stream * r.num_streams;
  // Threads per CTA: 128 spreads a small fill's warps over more SMs (10^5 FP32
  // uniforms 3.7 us against 4.5 with 256); the long chunks of the FP64
  // fixed-point transforms keep 256.
  const int threads = I::weight == 2 && cu * I::wpu >= 1024 ? 256 : 128;
  const int64_t grid = (p.total_chunks + threads - 1) / threads;
  if (grid > 0x7FFFFFFF) {
    set_error("MRG32k3a fill: grid too large");
    return GRNG_ERR_UNSUPPORTED;
  }
  if (aligned) {
    mrg_fill_kernel<V, 1><<<(unsigned)grid, threads, 0, stream>>>(p);
  } else if (carry) {
    if constexpr (I::epu == 2) mrg_fill_kernel<V, 2><<<(unsigned)grid, threads, 0, stream>>>(p);
  } else {
    mrg_fill_kernel<V, 3><<<(unsigned)grid, threads, 0, stream>>>(p);
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
