// Packed clock: one thread clocks one instance, its two 100-bit registers in
// eight 32-bit words, so that a warp clocks one 32-lane group (device code of
// the launches that are bound by the time per clock of one stream, not by the
// throughput of many).
//
// Layout.  R bit i is bit j of word w, i = 4j + w; S bit i is at position
// p = 99 - i = 4j + w.  With four words interleaved like this a shift of the
// register is a renaming of the words plus a one-bit shift of a single one,
// and with S reversed each control bit is one XOR of two bits at the same
// place: s34 ^ r67 at bit 16 of a[1] ^ r[3], s67 ^ r33 at bit 8 of
// a[0] ^ r[1].  Feedback bits: r99 is bit 24 of r[3], s99 bit 0 of a[0].
// The S words hold a_i = s_i ^ COMP0_i (i = 1..98), so that the AND term is
// a_i & (a_{i+1} ^ k_i) with k_i = COMP0_{i+1} ^ COMP1_i, and the constants
// COMP0_{i-1} ^ COMP0_i join the feedback word.  s0 (which is the last
// clock's feedback bit) is kept apart: its place in a[3] stays zero, so that
// the AND term of bit 0, which the cipher does not have, is zero without a
// mask; so does the one of bit 99, whose s_{i+1} is the zero shifted in.
// Bits 25..31 of the r words hold shifted-out garbage that only moves up.
//
// Pipes.  The half-rate logic pipe bounds a warp on its own, so everything
// that can be a multiply-add goes to the FMA pipe: left shifts, the feedback
// words k2 + fb (FB0 part) + fb cbs (FB1 part) (each bit a 0/1 times a
// constant, differences mod 2^32), fb_R x RTAPS and cb_R x r_i.  That leaves
// 22 logic and 21 multiply-add operations per clock of 32 instances.
// Measured (GB300, 2.07 GHz, with the row stores): 26.0 ns per clock for a lone
// warp, 27.6 with one warp per SM sub-partition; clocks alone 782 Gbit/s with
// eight (717 with the R update in logic operations).  The logic pipe would
// allow 21.3 ns; the rest is the schedule, which the compiler does best in a
// one-warp kernel whose loop holds the 32 clocks and a word store (control
// bits' words written first; other orders, register bounds or four words kept
// for a vector store: 28 to 44 ns).  The column form spread over a warp's
// lanes, which this one replaces, took 34.2 ns and at most 649 Gbit/s; one
// thread per 32-lane group takes 334 ns.
#pragma once

#include <cstdint>

#include "bitslice.cuh"

namespace mickey {

struct Packed {
  uint32_t r[4], a[4], s0;
};

__host__ __device__ constexpr bool packed_c0(int i) { return i >= 1 && i <= 98 && comp0(i); }

struct PackedMasks {
  uint32_t tap[4];   // RTAPS
  uint32_t c0[4];    // COMP0: a = s ^ c0
  uint32_t k[4];     // AND term a_i & (a_{i+1} ^ k_i)
  uint32_t k2[4];    // COMP0_{i-1} ^ COMP0_i
  uint32_t x[4];     // (k2 ^ FB0) - k2
  uint32_t y[4];     // (k2 ^ FB1) - (k2 ^ FB0)
};
constexpr PackedMasks make_packed_masks() {
  PackedMasks m{};
  for (int w = 0; w < 4; ++w) {
    uint32_t f0 = 0, f1 = 0;
    for (int j = 0; j < 25; ++j) {
      const uint32_t b = 1u << j;
      if (rtap(4 * j + w)) m.tap[w] |= b;
      const int i = 99 - (4 * j + w);
      if (i == 0) continue;                  // kept in Packed::s0
      if (packed_c0(i)) m.c0[w] |= b;
      if (fb0(i)) f0 |= b;
      if (fb1(i)) f1 |= b;
      if (packed_c0(i - 1) != packed_c0(i)) m.k2[w] |= b;
      if (i <= 98 && packed_c0(i + 1) != comp1(i)) m.k[w] |= b;
    }
    m.x[w] = (m.k2[w] ^ f0) - m.k2[w];
    m.y[w] = (m.k2[w] ^ f1) - (m.k2[w] ^ f0);
  }
  return m;
}
constexpr PackedMasks kPackedMasks = make_packed_masks();

// The control and feedback bits of a clock: CONTROL_BIT_R (0 / 1), FB_R (0 /
// ~0), FB_S and FB_S & CONTROL_BIT_S (0 / 1).
struct PackedCtl {
  uint32_t cbr, fbr, fbs, fc;
};

// MIX as in clock_kg, `in` 0 or 1.
template <bool MIX>
__device__ __forceinline__ PackedCtl packed_ctl(const Packed &q, uint32_t in) {
  static_assert(!packed_c0(34) && packed_c0(67) && !packed_c0(50), "control bits as held");
  PackedCtl c;
  c.fbs = MIX ? (q.a[0] ^ in) & 1u : q.a[0] & 1u;
  const uint32_t ncbs = (q.a[0] ^ q.r[1]) >> 8;            // bit 0: NOT CONTROL_BIT_S
  c.fc = lop3<0x20>(c.fbs, ncbs, 1u);                      // fbs & ~ncbs & 1
  c.cbr = ((q.a[1] ^ q.r[3]) >> 16) & 1u;
  c.fbr = MIX ? 0u - (((q.r[3] >> 24) ^ (q.a[1] >> 12) ^ in) & 1u)   // r99 ^ s50 ^ in
              : uint32_t(int32_t(q.r[3] << 7) >> 31);
  return c;
}

template <int W>
__device__ __forceinline__ uint32_t packed_r(const Packed &q, const PackedCtl &c) {
  constexpr uint32_t tap = 0u - kPackedMasks.tap[W];
  const uint32_t rm1 = W ? q.r[(W + 3) % 4] : q.r[3] << 1;                 // r_{i-1}
  return lop3<0x96>(rm1, mad32(q.r[W], c.cbr, 0u), mad32(c.fbr, tap, 0u));
}
template <int W>
__device__ __forceinline__ uint32_t packed_a(const Packed &q, const PackedCtl &c) {
  constexpr uint32_t k = kPackedMasks.k[W], k2 = kPackedMasks.k2[W], x = kPackedMasks.x[W],
                     y = kPackedMasks.y[W];
  const uint32_t sp1 = W ? q.a[(W + 3) % 4] : q.a[3] << 1;                 // a_{i+1}
  const uint32_t sm1 = W < 2    ? q.a[(W + 1) % 4]                         // a_{i-1}
                       : W == 2 ? mad32(q.s0, 1u << 24, q.a[3])
                                : q.a[0] >> 1;
  return lop3<0x96>(lop3<0x60>(q.a[W], sp1, k), sm1, mad32(c.fc, y, mad32(c.fbs, x, k2)));
}

// The registers one clock on.  The words that the next clock's control bits
// come from are written first.
__device__ __forceinline__ Packed packed_step(const Packed &q, const PackedCtl &c) {
  Packed n;
  n.a[0] = packed_a<0>(q, c);
  n.a[1] = packed_a<1>(q, c);
  n.r[1] = packed_r<1>(q, c);
  n.r[3] = packed_r<3>(q, c);
  n.a[2] = packed_a<2>(q, c);
  n.r[0] = packed_r<0>(q, c);
  n.s0 = c.fbs;
  n.a[3] = packed_a<3>(q, c);
  n.r[2] = packed_r<2>(q, c);
  return n;
}

// One CLOCK_KG of the thread's instance.
template <bool MIX>
__device__ __forceinline__ void clock_packed(Packed &q, uint32_t in) {
  q = packed_step(q, packed_ctl<MIX>(q, in));
}

// The zero state.
__device__ __forceinline__ void packed_zero(Packed &q) {
  static_for<0, 4>([&](auto wc) {
    constexpr int w = decltype(wc)::value;
    constexpr uint32_t c0 = kPackedMasks.c0[w];
    q.r[w] = 0u;
    q.a[w] = c0;
  });
  q.s0 = 0u;
}

// N clocks in non-mixing mode; z of clock c in bit N - 1 - c of the result
// (after N = 32: the first clock's in bit 31).
template <int N>
__device__ __forceinline__ uint32_t packed_clocks(Packed &q) {
  uint32_t z = 0;
#pragma unroll
  for (int c = 0; c < N; ++c) {
    z = mad32(z, 2u, lop3<0x28>(q.r[0], q.s0, 1u));   // (r0 ^ s0) & 1
    clock_packed<false>(q, 0u);
  }
  return z;
}

// The n < 32 clocks of a last partial tile, left-aligned as a whole tile.
__device__ __forceinline__ uint32_t packed_tail(Packed &q, int n) {
  uint32_t z = 0;
#pragma unroll 1
  for (int c = 0; c < n; ++c) {
    z = mad32(z, 2u, lop3<0x28>(q.r[0], q.s0, 1u));
    clock_packed<false>(q, 0u);
  }
  return z << (32 - n);
}

// 32 x 32 bit transpose across the warp: lane l's bit b <-> lane b's bit l.
__device__ __forceinline__ uint32_t warp_transpose(uint32_t x, uint32_t lane) {
  constexpr uint32_t kLow[5] = {0x0000ffffu, 0x00ff00ffu, 0x0f0f0f0fu, 0x33333333u, 0x55555555u};
#pragma unroll
  for (int st = 0; st < 5; ++st) {
    const uint32_t j = 16u >> st, m = kLow[st];
    const uint32_t y = __shfl_xor_sync(0xffffffffu, x, j);
    x = (lane & j) ? (x & ~m) | ((y >> j) & m) : (x & m) | ((y & m) << j);
  }
  return x;
}

// A lane's output row at o, written in whole words in memory order: four at a
// time (16-byte stores) where `vec` says that output and pitch allow it, else
// each word at the aligned addresses the row covers, put together from two
// words of a row that starts off a word boundary (its first and last bytes go
// singly).
struct RowOut {
  uint8_t *o;
  bool vec, valid;
  uint4 v;
  __device__ __forceinline__ RowOut(uint8_t *row, bool vec16, bool lane_valid)
      : o(row), vec(vec16), valid(lane_valid), v(make_uint4(0u, 0u, 0u, 0u)) {}
  __device__ __forceinline__ void put(uint64_t t, uint32_t w) {   // word t = 0, 1, 2, ...
    if (vec) {
      v = make_uint4(v.y, v.z, v.w, w);
      if ((t & 3) == 3 && valid) *reinterpret_cast<uint4 *>(o + 4 * (t - 3)) = v;
      return;
    }
    const uint32_t a = uint32_t(reinterpret_cast<uintptr_t>(o)) & 3u;
    const uint32_t x = __funnelshift_l(v.w, w, 8 * a);
    v.w = w;
    if (!valid) return;
    if (t > 0 || a == 0)
      *reinterpret_cast<uint32_t *>(o + 4 * t - a) = x;
    else
      for (uint32_t b = 0; b < 4 - a; ++b) o[b] = uint8_t(w >> (8 * b));
  }
  // After t whole words: the last one's bytes not yet written, then nbytes
  // more of w.
  __device__ __forceinline__ void finish(uint64_t t, int nbytes, uint32_t w) {
    if (!valid) return;
    const uint32_t a = uint32_t(reinterpret_cast<uintptr_t>(o)) & 3u;
    uint8_t *p = o + 4 * t;
    if (!vec && t > 0)
      for (uint32_t b = 0; b < a; ++b) p[int(b) - int(a)] = uint8_t(v.w >> (32 - 8 * (a - b)));
    for (int b = 0; b < nbytes; ++b) p[b] = uint8_t(w >> (8 * b));
  }
};

// Group g's bitsliced state (word-major rows of P words, r0..r99 then
// s0..s99) to the lanes' packed registers and back: lane j reads or writes
// the row of bit j of each word, and the transpose turns rows into lanes.
__device__ __forceinline__ void packed_load(Packed &q, const uint32_t *state, size_t P, uint32_t g,
                                            uint32_t lane) {
  uint32_t x[8];
#pragma unroll
  for (int w = 0; w < 4; ++w) {
    const int i = int(4 * lane) + w;
    x[w] = lane < 25 ? state[size_t(i) * P + g] : 0u;
    x[4 + w] = lane < 25 ? state[size_t(kReg + 99 - i) * P + g] : 0u;
  }
  static_for<0, 4>([&](auto wc) {
    constexpr int w = decltype(wc)::value;
    constexpr uint32_t c0 = kPackedMasks.c0[w];
    q.r[w] = warp_transpose(x[w], lane);
    q.a[w] = warp_transpose(x[4 + w], lane) ^ c0;
  });
  q.s0 = (q.a[3] >> 24) & 1u;
  q.a[3] &= 0x00ffffffu;
}

__device__ __forceinline__ void packed_store(const Packed &q, uint32_t *state, size_t P,
                                             uint32_t g, uint32_t lane) {
  static_for<0, 4>([&](auto wc) {
    constexpr int w = decltype(wc)::value;
    constexpr uint32_t c0 = kPackedMasks.c0[w];
    const uint32_t a = (w == 3 ? q.a[w] | (q.s0 << 24) : q.a[w]) ^ c0;
    const uint32_t xr = warp_transpose(q.r[w], lane), xs = warp_transpose(a, lane);
    const int i = int(4 * lane) + w;
    if (lane < 25) {
      state[size_t(i) * P + g] = xr;
      state[size_t(kReg + 99 - i) * P + g] = xs;
    }
  });
}

// A row of register bits in order, bit i at bit 31 - i % 32 of word i / 32
// (R in words 0..3, S in 4..7), to the packed registers and back.
__device__ __forceinline__ void packed_from_row(Packed &q, const uint32_t (&row)[8]) {
  static_for<0, 4>([&](auto wc) {
    constexpr int w = decltype(wc)::value;
    constexpr uint32_t c0 = kPackedMasks.c0[w];
    uint32_t r = 0u, s = 0u;
#pragma unroll
    for (int j = 0; j < 25; ++j) {
      const int i = 4 * j + w, k = 99 - i;
      r |= ((row[i >> 5] >> (31 - (i & 31))) & 1u) << j;
      s |= ((row[4 + (k >> 5)] >> (31 - (k & 31))) & 1u) << j;
    }
    q.r[w] = r;
    q.a[w] = s ^ c0;
  });
  q.s0 = (q.a[3] >> 24) & 1u;
  q.a[3] &= 0x00ffffffu;
}

__device__ __forceinline__ void packed_to_row(const Packed &q, uint32_t (&row)[8]) {
#pragma unroll
  for (int k = 0; k < 8; ++k) row[k] = 0u;
  static_for<0, 4>([&](auto wc) {
    constexpr int w = decltype(wc)::value;
    constexpr uint32_t c0 = kPackedMasks.c0[w];
    const uint32_t a = (w == 3 ? q.a[w] | (q.s0 << 24) : q.a[w]) ^ c0;
#pragma unroll
    for (int j = 0; j < 25; ++j) {
      const int i = 4 * j + w, k = 99 - i;
      row[i >> 5] |= ((q.r[w] >> j) & 1u) << (31 - (i & 31));
      row[4 + (k >> 5)] |= ((a >> j) & 1u) << (31 - (k & 31));
    }
  });
}

}  // namespace mickey
