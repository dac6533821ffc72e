// Bitsliced Grain keystream: one thread clocks a 32-lane group, clock warps
// paired with emission warps and the work cut into equal segments, as in the
// MICKEY launch (keystream_persistent.cuh).
//
// State: s[0..79] (LFSR) and b[0..79] (NFSR), 160 words in registers; the
// shift is register renaming within a body of 32 clocks, one tile
// (grain_clock.cuh: 36 logic operations per clock).  The clock warp writes
// the tile's z words to shared memory, reversed for the bytes layout
// (kLayoutBytesLsb), and meets its emission warp once per tile; the emission
// warp transposes and stages rows while the next tile is clocked.
//
// What bounds it: the logic pipe of a sub-partition, on which one clock warp
// alone issues at 0.77 (94 cycles per clock for 72 of logic) when its body
// fits the instruction cache, and the emission's 0.2 of that.  2^20 x 2^14
// bits, a re-key and the call: bytes 2444 -> 1621 us, bitsliced 1750 -> 1310
// us against a warp per warp-group of 80-clock bodies with the emission in
// its own instruction stream (those bodies did not fit, and the busiest
// sub-partitions had two of 1024 chains where others had one; the segments
// give each the same).
#include "keystream_persistent.cuh"

#include "grain_clock.cuh"

namespace mickey {
namespace {

using namespace grainc;

template <int LAYOUT>
__device__ __forceinline__ void grain_clock_piece(const KeystreamArgs &a, uint32_t g, uint32_t *zb0,
                                                  uint32_t *zb1, uint32_t &par, uint32_t bar,
                                                  uint32_t tile_a, uint32_t tile_b) {
  const size_t P = a.Gpad;
  const bool valid = g < a.G;
  uint32_t s[kG], b[kG];
  const uint32_t *src = a.state + (valid ? g : 0);
#pragma unroll
  for (int i = 0; i < kG; ++i) {
    s[i] = src[size_t(i) * P];
    b[i] = src[size_t(kG + i) * P];
  }
  auto row = [](int c) { return (LAYOUT == kLayoutBytesLsb ? 31 - c : c) * kKsThreads; };
  // A last partial tile is clocked in full and its words past the call's end
  // are zeroed.  The state wanted is then `rem` clocks on, not 32: of the 112
  // words old state + new bits it takes words rem .. rem + 79, the first of
  // them stored before the tile's clocks replace them.
  const uint32_t full = uint32_t(a.n_bits >> 5);
  const int rem = tile_b > full ? int(a.n_bits & 31) : 0;
  uint32_t *dst = a.state + g;
#pragma unroll 1
  for (uint32_t tile = tile_a; tile < tile_b; ++tile) {
    uint32_t *cur = par ? zb1 : zb0;
    if (rem && tile == full && valid) {
#pragma unroll
      for (int i = 0; i < 32; ++i)
        if (i >= rem) {
          dst[size_t(i - rem) * P] = s[i];
          dst[size_t(kG + i - rem) * P] = b[i];
        }
    }
    grain_body<32, false>(s, b, [&](auto rc, uint32_t z) { cur[row(decltype(rc)::value)] = z; });
    if (rem && tile == full)
      for (int c = rem; c < 32; ++c) cur[row(c)] = 0u;
    pair_sync(bar);
    par ^= 1u;
  }
  if (valid) {
    const int back = rem ? 32 - rem : 0;
#pragma unroll
    for (int i = 0; i < kG; ++i)
      if (i + back < kG) {
        dst[size_t(i + back) * P] = s[i];
        dst[size_t(kG + i + back) * P] = b[i];
      }
  }
}

// Row emission, rows on the 16-byte grid (a last partial tile, whose words past
// the call's end are zero, then fills a row's last word).  Grain's clock is a
// ninth of MICKEY's, so here the emission warp's time per tile matters.
//   * A tile is transposed in registers: one read of its 32 words, no second
//     pass through shared memory.
//   * Its words are staged as [row][slot][thread], so that a warp's accesses
//     are consecutive words, in a ring of kRingSlots tiles, so that the rows
//     of a finished block of 8 tiles can go out a quarter per tile.  A row
//     store touches 32 lines and all four emission warps come to theirs at
//     the same time: 32 rows at once held the clock warps up for 9000 cycles
//     per block.
// 622,592 instances x 8192 bits (every sub-partition clocking one chain): the
// MICKEY emission 596 us, in registers 578 us, spread over the ring 521 us; the
// clocks alone 374 us.
constexpr int kRingSlots = 12;

// Rows r0 .. r1-1 of tiles ba .. bb (a whole block of 8, or the part of one
// that a piece has).
__device__ __forceinline__ void grain_flush(const uint32_t *rb, const KeystreamArgs &a, uint32_t g,
                                            uint32_t ba, uint32_t bb, int r0, int r1,
                                            uint32_t lane_mask) {
  const uint64_t pitch = (a.n_bits + 7) >> 3;
  uint8_t *o = static_cast<uint8_t *>(a.out) + (32ull * g + uint32_t(r0)) * pitch + uint64_t(ba) * 4;
  if (bb - ba == 7) {
    const uint32_t *h0 = rb + (ba % kRingSlots) * kKsThreads;         // slots 0, 4 or 8 on
    const uint32_t *h1 = rb + ((ba + 4) % kRingSlots) * kKsThreads;
#pragma unroll 4
    for (int l = r0; l < r1; ++l, o += pitch) {
      const int w = l * kRingSlots * kKsThreads;
      const uint4 v0 = make_uint4(h0[w], h0[w + kKsThreads], h0[w + 2 * kKsThreads],
                                  h0[w + 3 * kKsThreads]);
      const uint4 v1 = make_uint4(h1[w], h1[w + kKsThreads], h1[w + 2 * kKsThreads],
                                  h1[w + 3 * kKsThreads]);
      if ((lane_mask >> l) & 1u) {
        reinterpret_cast<uint4 *>(o)[0] = v0;
        reinterpret_cast<uint4 *>(o)[1] = v1;
      }
    }
  } else {
#pragma unroll 1
    for (int l = r0; l < r1; ++l, o += pitch)
      for (uint32_t t = ba; t <= bb; ++t)
        if ((lane_mask >> l) & 1u)
          reinterpret_cast<uint32_t *>(o)[t - ba] = rb[(l * kRingSlots + t % kRingSlots) * kKsThreads];
  }
}

__device__ __forceinline__ void grain_emit_rows(const KeystreamArgs &a, uint32_t g,
                                                const uint32_t *zb0, const uint32_t *zb1,
                                                uint32_t *rb, uint32_t &par, uint32_t bar,
                                                uint32_t tile_a, uint32_t tile_b,
                                                uint32_t lane_mask) {
  uint32_t ba = 0, bb = 0;   // the block going out
  int row = 32;              // its next row (32: none left)
#pragma unroll 1
  for (uint32_t tile = tile_a; tile < tile_b; ++tile) {
    pair_sync(bar);
    const uint32_t *z = par ? zb1 : zb0;
    par ^= 1u;
    if (g >= a.G) continue;
    uint32_t m[32];
#pragma unroll
    for (int i = 0; i < 32; ++i) m[i] = z[i * kKsThreads];
    transpose32_prmt(m);     // m[31 - l]: lane l's word, clock c in bit c
    const uint32_t slot = tile % kRingSlots;
#pragma unroll
    for (int l = 0; l < 32; ++l) rb[(l * kRingSlots + slot) * kKsThreads] = m[31 - l];
    const bool last = tile == tile_b - 1;
    if (last && row < 32) {
      grain_flush(rb, a, g, ba, bb, row, 32, lane_mask);
      row = 32;
    }
    if (last || (tile & 7) == 7) {
      ba = max(tile & ~7u, tile_a);
      bb = tile;
      row = 0;
    }
    if (row < 32) {
      const int end = last ? 32 : row + 8;
      grain_flush(rb, a, g, ba, bb, row, end, lane_mask);
      row = end;
    }
  }
}

// As keystream_ws_kernel, with Grain's clock.
template <int LAYOUT>
__global__ void __launch_bounds__(2 * kKsThreads, 1)
    grain_ws_kernel(KeystreamArgs a, EmitCtx e, PersistArgs p) {
  extern __shared__ uint32_t zs[];
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t t = threadIdx.x & (kKsThreads - 1);   // thread of the clock side
  const uint32_t pair = t >> 5;
  const uint32_t slot = blockIdx.x * (kKsThreads / 32) + pair;
  const uint64_t NT = (a.n_bits + 31) >> 5;
  uint32_t *zb0 = zs + t, *zb1 = zs + 32 * kKsThreads + t;
  uint32_t par = 0;
#pragma unroll 1
  for (uint32_t k = 0;; ++k) {
    uint32_t w, ta, tb;
    if (!segment_piece(p, NT, slot, k, w, ta, tb)) break;
    const uint32_t g = w * 32 + lane;
    if (threadIdx.x < kKsThreads) {
      if (ta > 0) await_head(p, w, lane);
      grain_clock_piece<LAYOUT>(a, g, zb0, zb1, par, 1 + pair, ta, tb);
      if (ta > 0) take_back(p, w, lane);
      if (ta == 0 && tb < NT) publish_head(p, w, lane);
    } else if (LAYOUT == kLayoutBytesLsb && e.stage) {
      grain_emit_rows(a, g, zb0, zb1, zs + kTileBufWords + t, par, 1 + pair, ta, tb,
                      g == a.G - 1 ? e.lane_mask : ~0u);
    } else {
      emit_piece<LAYOUT, 8>(a, e, g, zb0, zb1, nullptr, par, 1 + pair, ta, tb);   // no staging
    }
  }
}

template <int LAYOUT>
cudaError_t launch_layout(const KeystreamArgs &a, const EmitCtx &e, const PersistArgs &p,
                          cudaStream_t st) {
  const cudaError_t err = allow_smem(grain_ws_kernel<LAYOUT>, kRingSlots);
  if (err != cudaSuccess) return err;
  cudaLaunchConfig_t cfg = {};
  cfg.dynamicSmemBytes = smem_bytes(e, kRingSlots);
  cfg.gridDim = dim3(p.blocks);
  cfg.blockDim = dim3(2 * kKsThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = p.cooperative ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, grain_ws_kernel<LAYOUT>, a, e, p);
}

}  // namespace

cudaError_t launch_grain_ws(const KeystreamArgs &a, int layout, const PersistArgs &p,
                            cudaStream_t st) {
  EmitCtx e;
  const uint32_t tail = uint32_t(a.n & 31u);
  const uintptr_t addr = reinterpret_cast<uintptr_t>(a.out);
  e.lane_mask = tail ? (1u << tail) - 1u : ~0u;
  e.vec_ok = addr % 16 == 0 && a.n_bits % 4 == 0;
  e.word_ok = addr % 4 == 0 && ((a.n_bits + 7) / 8) % 4 == 0;
  // a last block of fewer tiles than eight goes out word by word.  2^20 instances
  // x 16,380 bits: 1632 us, unstaged 8415
  e.stage = layout == MICKEY_LAYOUT_BYTES && grain_rows16(a.n_bits, a.out);
  return layout == MICKEY_LAYOUT_BYTES ? launch_layout<kLayoutBytesLsb>(a, e, p, st)
                                       : launch_layout<MICKEY_LAYOUT_BITSLICED_U32>(a, e, p, st);
}

}  // namespace mickey
