// Grain with one thread per instance, 16 clocks per step: the launches for
// handles with too few 32-lane groups to fill the chip with one thread per
// group (grain.cu).
//
// No tap of Grain reaches above s64 / b63, so the 16 next clocks depend on
// the present 80 + 80 bits only (b_{80+15} on b_{63+15}, z_{15} on s_{64+15}):
// a thread computes them at once, each tap a 16-bit window of the register,
// with the same logic as one bitsliced clock.  Five words w_k hold register
// bits 16k .. 16k + 31, bit 16k in bit 31 (each bit twice, w_4's low half
// unset), so the window from bit 16k + m is w_k << m in the top half: one
// multiply on the FMA pipe, while the logic pipe runs the 36 logic operations
// and the two byte permutes that append the new bits.  The words are renamed
// each step and are back in place after five.
//
// Measured (GB300, us): 4001 instances x 20,002 bits with the initialisation
// 1127 to 1488 -> 82; 155,648 x 8192 bits of bytes 1025 -> 204 (6.3 Tbit/s); rows off
// the 16-byte grid, 2^20 x 1001 bits 1196 -> 216.  A lone warp takes 4.7 ns
// per clock (9.7 cycles; its logic operations fill 4.9); at full occupancy
// 6.8 Tbit/s, 0.82 of what the logic pipe allows for 38 operations per 16
// clocks of 32 instances.
#include "../../include/mickey.h"
#include "grain_clock.cuh"
#include "internal.h"
#include "packed.cuh"

namespace mickey {
namespace {

using namespace grainc;

constexpr int kGpThreads = 32;    // one group per block: an even spread over the sub-partitions

struct GrainPacked {
  uint32_t s[5], b[5];
};

// The windows of 16 clocks at tap I (top half valid) when the words stand R
// steps rotated.
template <int R, int I>
__device__ __forceinline__ uint32_t win(const uint32_t (&w)[5]) {
  constexpr int k = I / 16, m = I % 16;
  const uint32_t x = w[(R + k) % 5];
  return m ? mad32(x, 1u << m, 0u) : x;
}

// Append the 16 new bits in n's top half: they complete w_4 and begin the next
// word, in the place of w_0.
template <int R>
__device__ __forceinline__ void append(uint32_t (&w)[5], uint32_t n) {
  w[(R + 4) % 5] = __byte_perm(n, w[(R + 4) % 5], 0x7632);
  w[R % 5] = n;
}

// 16 clocks; z of clock c in bit 31 - c (the low half undefined).
template <int R, bool INIT>
__device__ __forceinline__ uint32_t grain_step16(GrainPacked &q) {
#define S(i) win<R, i>(q.s)
#define B(i) win<R, i>(q.b)
  uint32_t h0, h1;
  grain_h01(S(3), S(25), S(46), S(64), h0, h1);
  const uint32_t b10 = B(10), b31 = B(31), b43 = B(43), b63 = B(63);
  const uint32_t z = xor3(xor3(B(1), B(2), B(4)), xor3(b10, b31, b43), B(56)) ^ xand(h0, b63, h1);
  const uint32_t s0 = S(0);
  const uint32_t la = xor3(S(62), S(51), S(38)), lb = xor3(S(23), S(13), s0);
  const uint32_t ns = INIT ? xor3(la, lb, z) : la ^ lb;
  const uint32_t nb = grain_feedback<INIT>(s0, z, B(0), B(9), B(14), B(15), B(21), B(28), B(33),
                                           B(37), B(45), B(52), B(60), B(62), b63);
#undef S
#undef B
  append<R>(q.s, ns);
  append<R>(q.b, nb);
  return z;
}

__device__ __forceinline__ void rotate(uint32_t (&w)[5]) {
  const uint32_t x = w[0];
#pragma unroll
  for (int k = 0; k < 4; ++k) w[k] = w[k + 1];
  w[4] = x;
}

// Up to 16 clocks, r of them kept (r <= 16), with the words moved in place.
__device__ __forceinline__ uint32_t grain_tail16(GrainPacked &q, int r) {
  if (r == 16) {
    const uint32_t z = grain_step16<0, false>(q);
    rotate(q.s);
    rotate(q.b);
    return z;
  }
  const uint32_t s0 = q.s[0], b0 = q.b[0];
  const uint32_t z = grain_step16<0, false>(q);
  auto shift = [r](uint32_t (&w)[5], uint32_t w0) {   // 96 bits w0 : w2 : w4 by r
    const uint32_t x0 = __funnelshift_l(w[2], w0, r), x1 = __funnelshift_l(w[4], w[2], r);
    const uint32_t x2 = w[4] << r;
    w[0] = x0;
    w[1] = __byte_perm(x1, x0, 0x5432);
    w[2] = x1;
    w[3] = __byte_perm(x2, x1, 0x5432);
    w[4] = x2;
  };
  shift(q.s, s0);
  shift(q.b, b0);
  return z;
}

// Group g's bitsliced state (rows s0..s79 then b0..b79 of P words) to the
// lanes' words and back.
__device__ __forceinline__ void gp_load(GrainPacked &q, const uint32_t *state, size_t P, uint32_t g,
                                        uint32_t lane) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t x[3];
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const int i = 32 * k + 31 - int(lane);          // register bit in bit `lane` of the word
      x[k] = i < kG ? state[size_t(h * kG + i) * P + g] : 0u;
    }
#pragma unroll
    for (int k = 0; k < 3; ++k) x[k] = warp_transpose(x[k], lane);
    uint32_t(&w)[5] = h ? q.b : q.s;
    w[0] = x[0];
    w[1] = __byte_perm(x[1], x[0], 0x5432);
    w[2] = x[1];
    w[3] = __byte_perm(x[2], x[1], 0x5432);
    w[4] = x[2];
  }
}

__device__ __forceinline__ void gp_store(const GrainPacked &q, uint32_t *state, size_t P,
                                         uint32_t g, uint32_t lane) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const uint32_t(&w)[5] = h ? q.b : q.s;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
      const uint32_t x = warp_transpose(w[2 * k], lane);
      const int i = 32 * k + 31 - int(lane);
      if (i < kG) state[size_t(h * kG + i) * P + g] = x;
    }
  }
}

// Tile t's z words of the lanes (first clock in bit 31) to the output.
template <int LAYOUT>
__device__ __forceinline__ void gp_emit(RowOut &row, uint32_t *gout, uint64_t t, uint32_t z,
                                        uint32_t lane, uint32_t lane_mask) {
  z = __brev(z);                                     // first clock in bit 0
  if constexpr (LAYOUT == MICKEY_LAYOUT_BITSLICED_U32)
    gout[32 * t + lane] = warp_transpose(z, lane) & lane_mask;
  else
    row.put(t, z);
}

template <int LAYOUT>
__global__ void __launch_bounds__(kGpThreads)
    grain_packed_kernel(KeystreamArgs a, uint32_t lane_mask) {
  const uint32_t lane = threadIdx.x, g = blockIdx.x;
  if (g != a.G - 1) lane_mask = ~0u;
  GrainPacked q;
  gp_load(q, a.state, a.Gpad, g, lane);
  const uint64_t pitch = (a.n_bits + 7) >> 3;
  RowOut row(static_cast<uint8_t *>(a.out) + (32ull * g + lane) * pitch,
             (reinterpret_cast<uintptr_t>(a.out) & 15u) == 0 && a.n_bits % 128 == 0,
             (lane_mask >> lane) & 1u);
  uint32_t *gout = static_cast<uint32_t *>(a.out) + size_t(g) * a.n_bits;
  uint64_t t = 0;                                    // tiles emitted
  const uint64_t full = a.n_bits / 160;
#pragma unroll 1
  for (uint64_t j = 0; j < full; ++j) {
    static_for<0, 5>([&](auto tc) {
      constexpr int i = decltype(tc)::value;
      const uint32_t z0 = grain_step16<(2 * i) % 5, false>(q);
      const uint32_t z1 = grain_step16<(2 * i + 1) % 5, false>(q);
      gp_emit<LAYOUT>(row, gout, t + i, __byte_perm(z1, z0, 0x7632), lane, lane_mask);
    });
    t += 5;
  }
  int rem = int(a.n_bits - full * 160);
#pragma unroll 1
  for (; rem >= 32; rem -= 32) {
    const uint32_t z0 = grain_tail16(q, 16), z1 = grain_tail16(q, 16);
    gp_emit<LAYOUT>(row, gout, t++, __byte_perm(z1, z0, 0x7632), lane, lane_mask);
  }
  uint32_t z = 0;
  if (rem) {
    z = grain_tail16(q, min(rem, 16)) & 0xffff0000u;
    if (rem > 16) z |= grain_tail16(q, rem - 16) >> 16;
    z = __brev(z & (~0u << (32 - rem)));
  }
  if constexpr (LAYOUT == MICKEY_LAYOUT_BITSLICED_U32) {
    z = warp_transpose(z, lane) & lane_mask;
    if (int(lane) < rem) gout[32 * t + lane] = z;
  } else {
    row.finish(t, (rem + 7) >> 3, z);
  }
  gp_store(q, a.state, a.Gpad, g, lane);
}

__device__ __forceinline__ uint32_t le32(const uint8_t *p) {
  return uint32_t(p[0]) | (uint32_t(p[1]) << 8) | (uint32_t(p[2]) << 16) | (uint32_t(p[3]) << 24);
}

// Loading (least significant bit of each byte first) and the 160 clocks with
// z fed back.
__global__ void __launch_bounds__(kGpThreads)
    grain_packed_init_kernel(const uint8_t *keys, const uint8_t *ivs, uint64_t n, size_t P,
                             uint32_t *state) {
  const uint32_t lane = threadIdx.x, g = blockIdx.x;
  const uint64_t i = 32ull * g + lane;
  uint32_t x[2][3] = {{0u, 0u, 0xffff0000u}, {0u, 0u, 0u}};
  if (i < n) {
    const uint8_t *k = keys + 10 * i, *v = ivs + 8 * i;
    x[0][0] = __brev(le32(v));
    x[0][1] = __brev(le32(v + 4));
    x[1][0] = __brev(le32(k));
    x[1][1] = __brev(le32(k + 4));
    x[1][2] = __brev(uint32_t(k[8]) | (uint32_t(k[9]) << 8));
  }
  GrainPacked q;
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t(&w)[5] = h ? q.b : q.s;
    w[0] = x[h][0];
    w[1] = __byte_perm(x[h][1], x[h][0], 0x5432);
    w[2] = x[h][1];
    w[3] = __byte_perm(x[h][2], x[h][1], 0x5432);
    w[4] = x[h][2];
  }
#pragma unroll 1
  for (int rep = 0; rep < 2; ++rep)
    static_for<0, 5>([&](auto rc) { grain_step16<decltype(rc)::value, true>(q); });
  gp_store(q, state, P, g, lane);
}

}  // namespace

cudaError_t launch_grain_packed(const KeystreamArgs &a, int layout, cudaStream_t st) {
  const uint32_t tail = uint32_t(a.n & 31u), mask = tail ? (1u << tail) - 1u : ~0u;
  if (layout == MICKEY_LAYOUT_BYTES)
    grain_packed_kernel<MICKEY_LAYOUT_BYTES><<<a.G, kGpThreads, 0, st>>>(a, mask);
  else
    grain_packed_kernel<MICKEY_LAYOUT_BITSLICED_U32><<<a.G, kGpThreads, 0, st>>>(a, mask);
  return cudaGetLastError();
}

cudaError_t launch_grain_packed_init(const uint8_t *keys, const uint8_t *ivs, uint64_t n,
                                     uint32_t G, uint32_t Gpad, uint32_t *state, cudaStream_t st) {
  grain_packed_init_kernel<<<G, kGpThreads, 0, st>>>(keys, ivs, n, Gpad, state);
  return cudaGetLastError();
}

}  // namespace mickey
