// Ragged keystream generation on a streams handle: every stream continues by
// its own number of bits in one call (the instance-per-lane design of
// Sec. IV-D with uneven lengths).
//
// Few groups (ragged_packed_kernel): one thread per instance (packed.cuh).  A
// thread clocks its own stream as often as it needs and is done.
//
// Many groups (ragged_ws_kernel): one thread per 32-lane group, clock warps
// paired with emission warps as in the keystream launch
// (keystream_persistent.cuh); a group is clocked as often as its longest lane
// needs.  What differs from equal lengths:
//   * A warp-group has as many blocks of 128 clocks as its longest lane needs,
//     and the work line is cut on their prefix sums (ragged_cuts.h).
//   * A lane's state must be the one after exactly its own number of clocks.
//     The clock loop has no test per clock: before every block the lanes that
//     end within its 128 clocks are merged into the state in HBM
//     (their bits were cleared there when the piece started, so one
//     fire-and-forget OR per word sets them), and ragged_rest_kernel runs
//     each lane's remaining 0 .. 127 clocks with a thread per instance.
//   * The emission warp knows where each row ends: whole words go out at the
//     aligned addresses a row covers (rows start at any byte), the last ones
//     byte by byte.
// Bound by the logic pipe: the clocks of the longest lanes (0.76 of the clocked
// bits are output below), then the emission warp's share of it.  Measured, 2^20
// streams, lengths uniform in [2^13, 2^14], bytes at the packed offsets, call
// by call: 21.9 -> 11.3 ms (1145 Gbit/s); before, one warp clocked, tested each
// clock for ends and emitted with byte stores.
#include "keystream_persistent.cuh"
#include "packed.cuh"

namespace mickey {
namespace {

// Tiles per block.  States are handed on at block boundaries only: a lane that
// has been merged then has no output left in the next segment.
constexpr uint32_t kSnapTiles = kRaggedBlockBits / 32;

// ------------------------------------------------------- one thread per group

// Shared memory of a block after the two tile buffers, all [lane][thread]:
// a row's address, the previous tile's word, the tiles that hold the lane's
// bits, and the tile before which its state is merged (~0: no bits asked for).
struct LaneTab {
  uint64_t *row;
  uint32_t *carry, *tiles, *snap;
};
constexpr size_t kRaggedSmem = 4 * kTileBufWords + size_t(32) * kKsThreads * (8 + 4 + 4 + 4);

__device__ __forceinline__ LaneTab lane_tab(uint32_t *zs, uint32_t t) {
  uint64_t *row = reinterpret_cast<uint64_t *>(zs + kTileBufWords);
  uint32_t *w = reinterpret_cast<uint32_t *>(row + 32 * kKsThreads);
  return LaneTab{row + t, w + t, w + 32 * kKsThreads + t, w + 64 * kKsThreads + t};
}

// The lanes for which f(snap tile) holds.
template <class F>
__device__ __forceinline__ uint32_t lanes_where(const uint32_t *snap, F f) {
  uint32_t m = 0;
#pragma unroll 8
  for (int l = 0; l < 32; ++l) m |= (f(snap[l * kKsThreads]) ? 1u : 0u) << l;
  return m;
}

// The address of the group's state and the row pitch through an opaque move,
// so that the 200 word addresses are formed where they are used and are not
// held live across the clock loop (which spilled).
__device__ __forceinline__ uint32_t *opaque(uint32_t *st0, size_t P0, size_t &P) {
  uint32_t *st;
  asm volatile("mov.b64 %0, %1;" : "=l"(st) : "l"(st0));
  asm volatile("mov.b64 %0, %1;" : "=l"(P) : "l"(P0));
  return st;
}

// OR the lanes in `m` of the current state into the state in HBM.
__device__ __forceinline__ void merge_lanes(uint32_t *st0, size_t P0, const uint32_t (&r)[kReg],
                                            const uint32_t (&s)[kReg], uint32_t m) {
  size_t P;
  uint32_t *st = opaque(st0, P0, P);
#pragma unroll
  for (int i = 0; i < kReg; ++i) {
    atomicOr(st + size_t(i) * P, r[i] & m);
    atomicOr(st + size_t(kReg + i) * P, s[i] & m);
  }
}

// Row of the tile buffer that takes clock c's word, such that the transposed
// word of a lane is in memory order (bytes) or big-endian (u32).
template <int LAYOUT>
__device__ __forceinline__ int clock_row(int c) {
  return LAYOUT == MICKEY_LAYOUT_BYTES ? 24 - (c & ~7) + (c & 7) : c;
}

template <int LAYOUT>
__device__ __forceinline__ void ragged_clock_piece(const RaggedArgs &a, const LaneTab &lt,
                                                   uint32_t g, uint32_t *zb0, uint32_t *zb1,
                                                   uint32_t &par, uint32_t bar, uint32_t ta,
                                                   uint32_t tb, bool ends) {
  const size_t P = a.Gpad;
  const bool valid = g < a.G;
  uint32_t r[kReg], s[kReg];
  uint32_t *st = a.state + (valid ? g : 0);
  // lanes whose state this piece carries on: their bits leave HBM
  const uint32_t live = valid ? lanes_where(lt.snap, [ta](uint32_t x) { return x != ~0u && x >= ta; })
                              : 0u;
#pragma unroll
  for (int i = 0; i < kReg; ++i) {
    r[i] = st[size_t(i) * P];
    s[i] = st[size_t(kReg + i) * P];
  }
  if (live) {
    size_t Q;
    uint32_t *wr = opaque(st, P, Q);
#pragma unroll
    for (int i = 0; i < kReg; ++i) {
      wr[size_t(i) * Q] = r[i] & ~live;
      wr[size_t(kReg + i) * Q] = s[i] & ~live;
    }
  }
#pragma unroll 1
  for (uint32_t T = ta;; ++T) {
    // lanes that end before the next look; after the last tile those that end
    // there, or, where the next segment goes on, all that run on
    if (valid && T % kSnapTiles == 0) {      // tb too is a multiple
      const bool hand_on = T == tb && !ends;
      const uint32_t m = lanes_where(
          lt.snap, [=](uint32_t x) { return x == T || (hand_on && x > T && x != ~0u); });
      if (m) merge_lanes(st, P, r, s, m);
    }
    if (T == tb) break;
    uint32_t *cur = par ? zb1 : zb0;
#pragma unroll 1
    for (int c = 0; c < 32; c += 4) {
      uint32_t *row = cur + clock_row<LAYOUT>(c) * kKsThreads;
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        row[u * kKsThreads] = r[0] ^ s[0];
        clock_kg<false, false>(r, s, 0u, 0u);
      }
    }
    pair_sync(bar);
    par ^= 1u;
  }
}

// Store the tile's words of the group's rows.  `first`: the piece's first tile;
// `final`: the last tile of a piece that the next segment continues.  The rows
// that go on past the tile take the loop; its code and the one copy of the
// byte-wise cases stay small beside the clock loop in the instruction cache
// (all 32 rows unrolled with their cases: 34.6 ms where the clocks take 10).
template <int LAYOUT>
__device__ __forceinline__ void ragged_rows(const RaggedArgs &a, const LaneTab &lt, uint32_t g,
                                            uint32_t *z, uint32_t T, bool first, bool final) {
  uint32_t m[32];
#pragma unroll
  for (int i = 0; i < 32; ++i) m[i] = z[i * kKsThreads];
  transpose32_prmt(m);                       // m[31 - l]: lane l's word
#pragma unroll
  for (int l = 0; l < 32; ++l) z[l * kKsThreads] = m[31 - l];
  uint32_t whole = 0, ending = 0;
#pragma unroll 4
  for (int l = 0; l < 32; ++l) {
    const uint32_t n_tiles = lt.tiles[l * kKsThreads];
    ending |= (T + 1 == n_tiles ? 1u : 0u) << l;
    if (T + 1 >= n_tiles) continue;
    whole |= 1u << l;
    const uint64_t base = lt.row[l * kKsThreads];
    const uint32_t al = uint32_t(base) & 3u; // the row starts `al` bytes into its first word
    const uint32_t w = z[l * kKsThreads], prev = lt.carry[l * kKsThreads];
    lt.carry[l * kKsThreads] = w;
    if (!first)
      *reinterpret_cast<uint32_t *>(base - al + 4ull * T) = __funnelshift_l(prev, w, 8 * al);
  }
  // rows byte by byte: the part of the first word that is theirs, and what is
  // left of the last one
  for (uint32_t todo = ending | (first || final ? whole : 0u); todo; todo &= todo - 1) {
    const int l = __ffs(int(todo)) - 1;
    const uint64_t base = lt.row[l * kKsThreads];
    const uint32_t al = uint32_t(base) & 3u;
    uint8_t *o = reinterpret_cast<uint8_t *>(base - al) + 4ull * T;
    uint32_t w = z[l * kKsThreads];
    if ((whole >> l) & 1u) {
      for (uint32_t b = al; first && b < 4; ++b) o[b] = uint8_t(w >> (8 * (b - al)));
      for (uint32_t b = 0; final && b < al; ++b) o[4 + b] = uint8_t(w >> (8 * (4 - al + b)));
    } else {
      const int nb = int((a.n_bits[32ull * g + l] - 1) & 31u) + 1;
      if (LAYOUT == MICKEY_LAYOUT_BYTES) w &= __byte_perm(~0u << (32 - nb), 0u, 0x0123);
      const uint32_t prev = lt.carry[l * kKsThreads];
      for (uint32_t b = 0; !first && b < al; ++b) o[b] = uint8_t(prev >> (8 * (4 - al + b)));
      for (int b = 0; b < (nb + 7) >> 3; ++b) o[al + b] = uint8_t(w >> (8 * b));
    }
  }
}

// The tile's words of a bitsliced row (T in words of the group's longest lane).
__device__ __forceinline__ void ragged_words(const RaggedArgs &a, const LaneTab &lt, uint32_t g,
                                             uint32_t *z, uint32_t T, uint64_t words) {
  uint32_t alive = 0;
  for (int l = 0; l < 32; ++l) {
    const uint32_t n_tiles = lt.tiles[l * kKsThreads];
    if (T >= n_tiles) continue;
    alive |= 1u << l;
    if (T + 1 == n_tiles)                           // ends inside: its later clocks' bits go
      for (int c = int((a.n_bits[32ull * g + l] - 1) & 31u) + 1; c < 32; ++c)
        z[c * kKsThreads] &= ~(1u << l);
  }
  if (!alive) return;
  uint32_t *o = reinterpret_cast<uint32_t *>(a.out + a.offsets[g]) + 32ull * T;
  const uint64_t left = words - 32ull * T;
  const int n = left < 32 ? int(left) : 32;
  // vectors from the first 16-byte boundary on
  int c = 0;
  for (; c < n && (reinterpret_cast<uintptr_t>(o + c) & 15u); ++c) o[c] = z[c * kKsThreads] & alive;
#pragma unroll 2
  for (; c + 4 <= n; c += 4)
    *reinterpret_cast<uint4 *>(o + c) =
        make_uint4(z[c * kKsThreads] & alive, z[(c + 1) * kKsThreads] & alive,
                   z[(c + 2) * kKsThreads] & alive, z[(c + 3) * kKsThreads] & alive);
  for (; c < n; ++c) o[c] = z[c * kKsThreads] & alive;
}

template <int LAYOUT>
__global__ void __launch_bounds__(2 * kKsThreads, 1)
    ragged_ws_kernel(RaggedArgs a, PersistArgs p) {
  extern __shared__ __align__(16) uint32_t zs[];
  const uint32_t lane = threadIdx.x & 31u;
  const uint32_t t = threadIdx.x & (kKsThreads - 1);
  const uint32_t pair = t >> 5;
  const bool clocker = threadIdx.x < kKsThreads;
  const uint32_t slot = blockIdx.x * (kKsThreads / 32) + pair;
  uint32_t *zb0 = zs + t, *zb1 = zs + 32 * kKsThreads + t;
  const LaneTab lt = lane_tab(zs, t);
  uint32_t par = 0;
#pragma unroll 1
  for (uint32_t k = 0;; ++k) {
    uint32_t pos;
    uint64_t ba, bb;
    if (!ragged_piece(a.line, p.tails_first, slot, k, pos, ba, bb)) break;
    if (ba == bb) continue;                  // a warp-group that asks for no bits
    const uint32_t w = uint32_t(a.line.order[pos]), g = w * 32 + lane;
    const uint32_t ta = kSnapTiles * uint32_t(ba), tb = kSnapTiles * uint32_t(bb);
    const bool ends = a.line.blocks[pos] + bb == a.line.blocks[pos + 1];
    if (clocker && ta > 0) await_head(p, w, lane);
    // The lane table: the clock side fills what it reads itself (snap), the
    // emission side the rest.  Every thread uses its own columns only.
    uint64_t words = 0;
    for (int l = 0; l < 32; ++l) {
      const uint64_t i = 32ull * g + l;
      const uint64_t n = g < a.G && i < a.n ? a.n_bits[i] : 0;
      if (clocker) {
        lt.snap[l * kKsThreads] = n ? uint32_t(n / kRaggedBlockBits) * kSnapTiles : ~0u;
      } else {
        lt.tiles[l * kKsThreads] = uint32_t((n + 31) >> 5);
        if (LAYOUT != MICKEY_LAYOUT_BITSLICED_U32)
          lt.row[l * kKsThreads] = n ? reinterpret_cast<uint64_t>(a.out + a.offsets[i]) : 0ull;
        words = max(words, n);
      }
    }
    if (clocker) {
      ragged_clock_piece<LAYOUT>(a, lt, g, zb0, zb1, par, 1 + pair, ta, tb, ends);
      if (ta > 0) take_back(p, w, lane);
      if (!ends) publish_head(p, w, lane);
    } else {
#pragma unroll 1
      for (uint32_t T = ta; T < tb; ++T) {
        pair_sync(1 + pair);
        uint32_t *z = par ? zb1 : zb0;
        par ^= 1u;
        if (32ull * T >= words) continue;    // the group's lanes have all ended
        if constexpr (LAYOUT == MICKEY_LAYOUT_BITSLICED_U32)
          ragged_words(a, lt, g, z, T, words);
        else
          ragged_rows<LAYOUT>(a, lt, g, z, T, T == ta, T == tb - 1 && !ends);
      }
    }
  }
}

// The clocks that ragged_ws_kernel left: each lane's own 0 .. kRaggedBlockBits - 1,
// a thread per instance.
__global__ void __launch_bounds__(32) ragged_rest_kernel(RaggedArgs a) {
  const uint32_t lane = threadIdx.x, g = blockIdx.x;
  const uint64_t i = 32ull * g + lane;
  const uint32_t rest = i < a.n ? uint32_t(a.n_bits[i] % kRaggedBlockBits) : 0u;
  const uint32_t most = __reduce_max_sync(0xffffffffu, rest);
  if (most == 0) return;
  Packed q;
  packed_load(q, a.state, a.Gpad, g, lane);
#pragma unroll 1
  for (uint32_t c = 0; c < most; c += 8) {
    if (__all_sync(0xffffffffu, c + 8 <= rest)) {
#pragma unroll
      for (int u = 0; u < 8; ++u) clock_packed<false>(q, 0u);
    } else {
#pragma unroll 1
      for (uint32_t u = c; u < c + 8; ++u)
        if (u < rest) clock_packed<false>(q, 0u);
    }
  }
  packed_store(q, a.state, a.Gpad, g, lane);
}

// ---------------------------------------------------- one thread per instance

template <int LAYOUT>
__global__ void __launch_bounds__(32) ragged_packed_kernel(RaggedArgs a) {
  const uint32_t lane = threadIdx.x, g = blockIdx.x;
  const uint64_t i = 32ull * g + lane;
  const uint64_t n = i < a.n ? a.n_bits[i] : 0;
  if (__all_sync(0xffffffffu, n == 0)) return;
  const uint64_t full = n >> 5;
  const int rem = int(n & 31);
  Packed q;
  packed_load(q, a.state, a.Gpad, g, lane);
  if constexpr (LAYOUT == MICKEY_LAYOUT_BITSLICED_U32) {
    uint32_t *o = reinterpret_cast<uint32_t *>(a.out + a.offsets[g]);
    const uint32_t tiles = __reduce_max_sync(0xffffffffu, uint32_t((n + 31) >> 5));
    const uint32_t ends = __reduce_max_sync(0xffffffffu, (n + 31) >> 5 == tiles ? uint32_t((n - 1) & 31) + 1 : 0u);
#pragma unroll 1
    for (uint32_t t = 0; t < tiles; ++t) {
      uint32_t z = 0;
      if (t < full) z = packed_clocks<32>(q);
      else if (t == full && rem) z = packed_tail(q, rem);
      __syncwarp();
      z = warp_transpose(__brev(z), lane);
      if (t + 1 < tiles || lane < ends) o[32ull * t + lane] = z;
    }
  } else {
    uint8_t *o = n ? a.out + a.offsets[i] : nullptr;
    const bool words = (reinterpret_cast<uintptr_t>(o) & 3u) == 0;
#pragma unroll 1
    for (uint64_t t = 0; t < full; ++t, o += 4) {
      const uint32_t z = packed_clocks<32>(q);
      const uint32_t w = LAYOUT == MICKEY_LAYOUT_BYTES ? __byte_perm(z, 0u, 0x0123) : z;
      if (words) {
        *reinterpret_cast<uint32_t *>(o) = w;
      } else {
        for (int b = 0; b < 4; ++b) o[b] = uint8_t(w >> (8 * b));
      }
    }
    if (rem) {
      const uint32_t w = __byte_perm(packed_tail(q, rem), 0u, 0x0123);
      for (int b = 0; b < (rem + 7) >> 3; ++b) o[b] = uint8_t(w >> (8 * b));
    }
    __syncwarp();
  }
  packed_store(q, a.state, a.Gpad, g, lane);
}

template <int LAYOUT>
cudaError_t launch_layout(const RaggedArgs &a, const PersistArgs *p, cudaStream_t st) {
  if (!p) {
    ragged_packed_kernel<LAYOUT><<<a.G, 32, 0, st>>>(a);
    return cudaGetLastError();
  }
  cudaError_t e = cudaFuncSetAttribute(
      ragged_ws_kernel<LAYOUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(kRaggedSmem));
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.dynamicSmemBytes = kRaggedSmem;
  cfg.gridDim = dim3(p->blocks);
  cfg.blockDim = dim3(2 * kKsThreads);
  cfg.stream = st;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeCooperative;
  attr[0].val.cooperative = p->cooperative ? 1 : 0;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  e = cudaLaunchKernelEx(&cfg, ragged_ws_kernel<LAYOUT>, a, *p);
  if (e != cudaSuccess) return e;
  ragged_rest_kernel<<<a.G, 32, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_ragged(const RaggedArgs &a, int layout, const PersistArgs *p, cudaStream_t st) {
  switch (layout) {
    case MICKEY_LAYOUT_BITSLICED_U32: return launch_layout<MICKEY_LAYOUT_BITSLICED_U32>(a, p, st);
    case MICKEY_LAYOUT_BYTES: return launch_layout<MICKEY_LAYOUT_BYTES>(a, p, st);
    case MICKEY_LAYOUT_U32: return launch_layout<MICKEY_LAYOUT_U32>(a, p, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mickey
