// Initialisation and keystream of a streams handle with one thread per
// instance (packed.cuh): the launches for handles that are too small for one
// thread per 32-lane group to fill the chip.  A warp takes one group, so the
// state in HBM stays bitsliced and every other launch can go on from it.
#include "../../include/mickey.h"
#include "internal.h"
#include "packed.cuh"

namespace mickey {
namespace {

// One-warp blocks: a handle of a few hundred groups then spreads evenly over
// the SM sub-partitions.
constexpr int kPackedThreads = 32;

// Store word w (z_{t0} in bit 31) of tile t of the row at o.
template <int LAYOUT>
__device__ __forceinline__ void packed_store_word(uint8_t *o, uint64_t f32_off, uint64_t t,
                                                  int nb, uint32_t w) {
  o += 4 * t;
  if constexpr (LAYOUT == MICKEY_LAYOUT_BYTES) {
    const uint32_t v = __byte_perm(w, 0u, 0x0123);
    if (nb == 32 && (reinterpret_cast<uintptr_t>(o) & 3u) == 0) {
      *reinterpret_cast<uint32_t *>(o) = v;
    } else {
      const int nbytes = (nb + 7) >> 3;
      for (int b = 0; b < nbytes; ++b) o[b] = uint8_t(v >> (8 * b));
    }
  } else {
    *reinterpret_cast<uint32_t *>(o) = w;
    if constexpr (LAYOUT == MICKEY_LAYOUT_U32_F32)
      *reinterpret_cast<float *>(o + f32_off) = __uint2float_rn(w >> 8) * 0x1p-24f;
  }
}

// Keystream of group blockIdx.x, one instance per lane.  The row layouts
// store a word (or bytes, off the word grid) per tile; the bitsliced layout
// turns each tile round with a transpose across the warp.  The loop around
// packed_clocks holds nothing else: with four tiles' words kept for 16-byte
// stores the compiler's schedule of the clocks was 16 % slower.
template <int LAYOUT>
__global__ void __launch_bounds__(32)
    packed_keystream_kernel(KeystreamArgs a, uint32_t lane_mask) {
  const uint32_t lane = threadIdx.x, g = blockIdx.x;
  if (g != a.G - 1) lane_mask = ~0u;
  Packed q;
  packed_load(q, a.state, a.Gpad, g, lane);
  const uint64_t full = a.n_bits >> 5;
  const int rem = int(a.n_bits & 31);
  if constexpr (LAYOUT == MICKEY_LAYOUT_BITSLICED_U32) {
    uint32_t *o = static_cast<uint32_t *>(a.out) + size_t(g) * a.n_bits;
#pragma unroll 1
    for (uint64_t t = 0; t < full; ++t) {
      const uint32_t z = packed_clocks<32>(q);
      o[32 * t + lane] = warp_transpose(__brev(z), lane) & lane_mask;
    }
    if (rem) {
      const uint32_t z = warp_transpose(__brev(packed_tail(q, rem)), lane) & lane_mask;
      if (int(lane) < rem) o[32 * full + lane] = z;
    }
  } else {
    const bool valid = (lane_mask >> lane) & 1u;
    const uint64_t pitch = LAYOUT == MICKEY_LAYOUT_BYTES ? (a.n_bits + 7) >> 3 : a.n_bits >> 3;
    const uint64_t f32_off = pitch * a.n;
    uint8_t *o = static_cast<uint8_t *>(a.out) + (32ull * g + lane) * pitch;
#pragma unroll 1
    for (uint64_t t = 0; t < full; ++t) {
      const uint32_t z = packed_clocks<32>(q);
      if (valid) packed_store_word<LAYOUT>(o, f32_off, t, 32, z);
    }
    if (rem) {
      const uint32_t z = packed_tail(q, rem);
      if (valid) packed_store_word<LAYOUT>(o, f32_off, full, rem, z);
    }
  }
  packed_store(q, a.state, a.Gpad, g, lane);
}

__device__ __forceinline__ uint32_t be32(const uint8_t *p) {
  return (uint32_t(p[0]) << 24) | (uint32_t(p[1]) << 16) | (uint32_t(p[2]) << 8) | uint32_t(p[3]);
}

// Key/IV loading and the mixing clocks, one instance per lane: its IV bits,
// 80 key bits and 100 zero bits go in one per clock.  Lanes with shorter IVs
// wait at the end of the IV clocks (an instance's clocks are its own, so no
// alignment or masking is needed).  The seven pieces of the input (three
// words of IV, three of key, the zeros) share one copy of the clock's code.
__global__ void __launch_bounds__(kPackedThreads) packed_init_kernel(LoadArgs a, uint32_t *state) {
  const uint32_t lane = threadIdx.x, g = blockIdx.x;
  const uint64_t slot = 32ull * g + lane;
  const bool valid = slot < a.n;
  uint32_t word[6] = {0u, 0u, 0u, 0u, 0u, 0u};
  int len = 0;
  if (valid) {
    const uint64_t i = a.perm ? uint64_t(a.perm[slot]) : slot;
    const uint8_t *v = a.ivs + 10 * i, *k = a.keys + 10 * i;
    word[0] = be32(v);
    word[1] = be32(v + 4);
    word[2] = (uint32_t(v[8]) << 24) | (uint32_t(v[9]) << 16);
    word[3] = be32(k);
    word[4] = be32(k + 4);
    word[5] = (uint32_t(k[8]) << 24) | (uint32_t(k[9]) << 16);
    len = a.iv_lens ? int(min(a.iv_lens[i], 1000u)) : 80;
    if (len > 80) {
      atomicOr(a.err, kErrIvLen);
      len = 80;
    }
  }
  Packed q;
  packed_zero(q);
#pragma unroll 1
  for (int ph = 0; ph < 7; ++ph) {
    uint32_t w = word[0];
#pragma unroll
    for (int j = 0; j < 5; ++j) word[j] = word[j + 1];
    word[5] = 0u;
    // this lane's clocks of the phase
    const int lim = ph < 3 ? min(32, max(0, len - 32 * ph)) : ph < 5 ? 32 : ph == 5 ? 16 : 100;
    const int end = int(__reduce_max_sync(0xffffffffu, uint32_t(lim)));
#pragma unroll 1
    for (int c = 0; c < end; c += 4) {
      if (__all_sync(0xffffffffu, c + 4 <= lim)) {
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          clock_packed<true>(q, w >> 31);
          w <<= 1;
        }
      } else {
#pragma unroll 1
        for (int u = 0; u < 4; ++u) {
          if (c + u < lim) clock_packed<true>(q, w >> 31);
          w <<= 1;
        }
      }
    }
  }
  packed_store(q, state, a.Gpad, g, lane);
}

}  // namespace

cudaError_t launch_packed_keystream(const KeystreamArgs &a, int layout, cudaStream_t st) {
  const uint32_t tail = uint32_t(a.n & 31u), mask = tail ? (1u << tail) - 1u : ~0u;
  switch (layout) {
    case MICKEY_LAYOUT_BITSLICED_U32:
      packed_keystream_kernel<MICKEY_LAYOUT_BITSLICED_U32><<<a.G, kPackedThreads, 0, st>>>(a, mask);
      break;
    case MICKEY_LAYOUT_BYTES:
      packed_keystream_kernel<MICKEY_LAYOUT_BYTES><<<a.G, kPackedThreads, 0, st>>>(a, mask);
      break;
    case MICKEY_LAYOUT_U32:
      packed_keystream_kernel<MICKEY_LAYOUT_U32><<<a.G, kPackedThreads, 0, st>>>(a, mask);
      break;
    case MICKEY_LAYOUT_U32_F32:
      packed_keystream_kernel<MICKEY_LAYOUT_U32_F32><<<a.G, kPackedThreads, 0, st>>>(a, mask);
      break;
    default:
      return cudaErrorInvalidValue;
  }
  return cudaGetLastError();
}

cudaError_t launch_packed_init(const LoadArgs &a, uint32_t *state, cudaStream_t st) {
  packed_init_kernel<<<a.G, kPackedThreads, 0, st>>>(a, state);
  return cudaGetLastError();
}

}  // namespace mickey
