// Keystream of handles with fewer warp-groups than SM sub-partitions: four
// warps clock one warp-group (32 groups of 32 instances), a quarter of the
// state each, one on every sub-partition of an SM.
//
// Warp 0 holds R bits 0..49 of every group, warp 1 R 50..99, warp 2 S 0..49,
// warp 3 S 50..99 (a thread its group's words, as in the other launches: one
// logic instruction per bit, compile-time tables).  What a quarter needs of
// the others per clock are the boundary words and the control and feedback
// bits: r33, r49, r67, r99, s34, s49, s50, s67, s99.  Each warp computes its
// own of these first in a clock and publishes them in shared memory (two
// parities); the four meet at a named barrier once per clock, read the words
// of the next one, and the rest of their bits hide that.  A fifth warp XORs
// the r0 and s0 words of a finished tile, transposes and stores it, as the
// emission warp of the paired launch does.
//
// A block has room for three warp-groups (slots); warp-group w is slot w /
// blocks of block w % blocks.  The parts of a slot are turned by its number,
// so that an SM with several has a mix of R and S work on each sub-partition.
//
// Bound by the exchange's latency with one warp-group per SM and by the logic
// pipe with more (654 cycles of it per warp-group and clock on four
// sub-partitions).  Measured, ns per clock with 1 / 2 / 3 warp-groups per SM:
// bytes 117 / 187 / 269, bitsliced 110 / 181 / 256; one thread per group on
// one warp 334 with any number up to four.  With an mbarrier per slot (arrive
// early, wait in mid-clock) in place of the barrier: 162 / 230 / 295.
#include "keystream_device.cuh"

namespace mickey {
namespace {

constexpr int kSlots = 3;
constexpr int kQuarterThreads = kSlots * 32 * 5;

// Words published per clock: per slot and clock parity, 9 rows of 32 lanes.
enum { kR33, kR49, kR67, kR99, kS34, kS49, kS50, kS67, kS99, kWords };
constexpr int kParWords = kWords * 32;

struct Exchange {
  uint32_t *w;        // this lane's column of the slot's words: [parity][word][lane]
  uint32_t bar;       // named barrier of the slot's four quarters
  __device__ __forceinline__ uint32_t get(uint32_t par, int k) const {
    return *reinterpret_cast<volatile uint32_t *>(w + par * kParWords + k * 32);
  }
  __device__ __forceinline__ void put(uint32_t par, int k, uint32_t x) const {
    *reinterpret_cast<volatile uint32_t *>(w + par * kParWords + k * 32) = x;
  }
  // every quarter's words of the next clock are there (and those of the clock
  // before have been read, so that their place is free)
  __device__ __forceinline__ void wait() const {
    asm volatile("bar.sync %0, 128;" ::"r"(bar) : "memory");
  }
};

__device__ __forceinline__ void tile_sync(uint32_t id) {   // parts 0 and 2 and the emission warp
  asm volatile("barrier.sync %0, 96;" ::"r"(id) : "memory");
}

template <int I>
__device__ __forceinline__ uint32_t next_r(uint32_t rm1, uint32_t r, uint32_t cbr, uint32_t fbr) {
  if constexpr (I == 0) return lop3<0x6A>(cbr, r, fbr);
  uint32_t v = lop3<0x78>(rm1, cbr, r);
  if constexpr (rtap(I)) v ^= fbr;
  return v;
}
template <int I>
__device__ __forceinline__ uint32_t next_s(uint32_t sm1, uint32_t s, uint32_t sp1, uint32_t fbs,
                                           uint32_t f0, uint32_t f1) {
  if constexpr (I == 0) return fbs;
  uint32_t v = sm1;
  if constexpr (I < kReg - 1) v = lop3<s_lut(comp0(I), comp1(I))>(sm1, s, sp1);
  if constexpr (fb0(I) || fb1(I)) v ^= s_feedback<I>(fbs, f0, f1);
  return v;
}

// One quarter: x[j] is bit 50 (PART % 2) + j of R (PART 0, 1) or S (2, 3).
template <int PART>
struct Quarter {
  static constexpr bool kIsR = PART < 2;
  static constexpr int kBase = PART % 2 ? 50 : 0;
  uint32_t x[50];
  uint32_t in[4];   // of the coming clock, as read() orders them

  __device__ __forceinline__ void publish(const Exchange &e, uint32_t par, const uint32_t (&y)[3]) {
    if constexpr (PART == 0) { e.put(par, kR33, y[0]); e.put(par, kR49, y[1]); }
    if constexpr (PART == 1) { e.put(par, kR67, y[0]); e.put(par, kR99, y[1]); }
    if constexpr (PART == 2) { e.put(par, kS34, y[0]); e.put(par, kS49, y[1]); }
    if constexpr (PART == 3) { e.put(par, kS50, y[0]); e.put(par, kS67, y[1]); e.put(par, kS99, y[2]); }
  }
  __device__ __forceinline__ void read(const Exchange &e, uint32_t par) {
    if constexpr (PART == 0) { in[0] = e.get(par, kS34); in[1] = e.get(par, kR67); in[2] = e.get(par, kR99); }
    if constexpr (PART == 1) { in[0] = e.get(par, kS34); in[1] = e.get(par, kR49); }
    if constexpr (PART == 2) {
      in[0] = e.get(par, kS67); in[1] = e.get(par, kR33); in[2] = e.get(par, kS99); in[3] = e.get(par, kS50);
    }
    if constexpr (PART == 3) { in[0] = e.get(par, kS49); in[1] = e.get(par, kR33); }
  }
  // Bit kBase + J of the next state.
  template <int J>
  __device__ __forceinline__ uint32_t next(uint32_t c, uint32_t fb, uint32_t f0, uint32_t f1) const {
    constexpr int I = kBase + J;
    const uint32_t m1 = J ? x[J ? J - 1 : 0] : PART == 1 ? in[1] : PART == 3 ? in[0] : 0u;
    if constexpr (kIsR) return next_r<I>(m1, x[J], c, fb);
    const uint32_t p1 = J < 49 ? x[J < 49 ? J + 1 : 0] : PART == 2 ? in[3] : 0u;
    return next_s<I>(m1, x[J], p1, fb, f0, f1);
  }
  // One clock; publishes into the words of parity `par` and ends with the
  // inputs of the clock after it.
  __device__ __forceinline__ void clock(const Exchange &e, uint32_t par) {
    uint32_t c = 0, fb, f0 = 0, f1 = 0;
    if constexpr (kIsR) {
      c = in[0] ^ (PART == 0 ? in[1] : x[67 - 50]);          // CONTROL_BIT_R
      fb = PART == 0 ? in[2] : x[49];
    } else {
      const uint32_t s67 = PART == 2 ? in[0] : x[67 - 50], r33 = in[1];
      fb = PART == 2 ? in[2] : x[49];
      f0 = lop3<0x90>(fb, s67, r33);
      f1 = lop3<0x60>(fb, s67, r33);
    }
    uint32_t y[3] = {0u, 0u, 0u};
    if constexpr (PART == 0) { y[0] = next<33>(c, fb, f0, f1); y[1] = next<49>(c, fb, f0, f1); }
    if constexpr (PART == 1) { y[0] = next<17>(c, fb, f0, f1); y[1] = next<49>(c, fb, f0, f1); }
    if constexpr (PART == 2) { y[0] = next<34>(c, fb, f0, f1); y[1] = next<49>(c, fb, f0, f1); }
    if constexpr (PART == 3) {
      y[0] = next<0>(c, fb, f0, f1);
      y[1] = next<17>(c, fb, f0, f1);
      y[2] = next<49>(c, fb, f0, f1);
    }
    publish(e, par, y);
    // from the top down: a word's last use is the bit above or below it, so
    // the new words can take the places of the old ones
    uint32_t n[50];
    n[0] = next<0>(c, fb, f0, f1);             // the one that reads `in` besides bit 49
    e.wait();
    read(e, par);
    static_for<0, 48>([&](auto jc) {
      constexpr int j = 48 - decltype(jc)::value;
      n[j] = next<j>(c, fb, f0, f1);
    });
    if constexpr (PART == 0) { n[33] = y[0]; n[49] = y[1]; }
    if constexpr (PART == 1) { n[17] = y[0]; n[49] = y[1]; }
    if constexpr (PART == 2) { n[34] = y[0]; n[49] = y[1]; }
    if constexpr (PART == 3) { n[0] = y[0]; n[17] = y[1]; n[49] = y[2]; }
#pragma unroll
    for (int j = 0; j < 50; ++j) x[j] = n[j];
  }
};

template <int PART>
__device__ __forceinline__ void run_quarter(const KeystreamArgs &a, Exchange e, uint32_t g,
                                            uint32_t *z0, uint32_t *z1, uint32_t bar) {
  constexpr bool kLow = PART % 2 == 0;    // holds r0 or s0, the output's words
  const bool valid = g < a.G;
  const size_t P = a.Gpad;
  Quarter<PART> q;
  uint32_t *st = a.state + size_t(50 * PART) * P + (valid ? g : 0);
#pragma unroll
  for (int j = 0; j < 50; ++j) q.x[j] = valid ? st[size_t(j) * P] : 0u;
  uint32_t y[3] = {0u, 0u, 0u};
  if constexpr (PART == 0) { y[0] = q.x[33]; y[1] = q.x[49]; }
  if constexpr (PART == 1) { y[0] = q.x[17]; y[1] = q.x[49]; }
  if constexpr (PART == 2) { y[0] = q.x[34]; y[1] = q.x[49]; }
  if constexpr (PART == 3) { y[0] = q.x[0]; y[1] = q.x[17]; y[2] = q.x[49]; }
  uint32_t par = 0;
  q.publish(e, par, y);
  e.wait();
  q.read(e, par);
  const uint32_t full = uint32_t(a.n_bits >> 5);
  const int rem = int(a.n_bits & 31);
  uint32_t *cur = z0, *other = z1;
#pragma unroll 1
  for (uint32_t t = 0; t < full; ++t) {
#pragma unroll 1
    for (int c = 0; c < 32; c += 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        if constexpr (kLow) cur[(c + u) * kKsThreads] = q.x[0];
        par ^= 1u;
        q.clock(e, par);
      }
    }
    if constexpr (kLow) {
      tile_sync(bar);
      uint32_t *s = cur;
      cur = other;
      other = s;
    }
  }
  if (rem) {
#pragma unroll 1
    for (int c = 0; c < rem; ++c) {
      if constexpr (kLow) cur[c * kKsThreads] = q.x[0];
      par ^= 1u;
      q.clock(e, par);
    }
    if constexpr (kLow) {
      for (int c = rem; c < 32; ++c) cur[c * kKsThreads] = 0u;
      tile_sync(bar);
    }
  }
  if (valid) {
#pragma unroll
    for (int j = 0; j < 50; ++j) st[size_t(j) * P] = q.x[j];
  }
}

constexpr int kQStage = 8;   // tiles per staged row
// Shared memory: r0 and s0 words of two tiles (four 32-row buffers of kKsThreads
// columns), the published words, the row staging.
constexpr size_t kQWords = 4 * 32 * kKsThreads, kQExchange = size_t(kSlots) * 2 * kParWords;

template <int LAYOUT>
__global__ void __launch_bounds__(kQuarterThreads, 1)
    quarters_kernel(KeystreamArgs a, EmitCtx e, uint32_t W) {
  extern __shared__ __align__(16) uint32_t zs[];
  const uint32_t lane = threadIdx.x & 31u, warp = threadIdx.x >> 5;
  const bool clocker = warp < 4 * kSlots;
  const uint32_t slot = clocker ? warp >> 2 : warp - 4 * kSlots;
  const uint32_t w = blockIdx.x + slot * gridDim.x;
  if (w >= W) return;
  const uint32_t g = w * 32 + lane, col = slot * 32 + lane, bar = 1 + slot;
  uint32_t *zr0 = zs + col, *zr1 = zr0 + 32 * kKsThreads, *zs0 = zr1 + 32 * kKsThreads,
           *zs1 = zs0 + 32 * kKsThreads;
  const Exchange x{zs + kQWords + slot * 2 * kParWords + lane, 1 + kSlots + slot};
  if (clocker) {
    switch ((warp - slot) & 3u) {
      case 0: run_quarter<0>(a, x, g, zr0, zr1, bar); break;
      case 1: run_quarter<1>(a, x, g, zr0, zr1, bar); break;
      case 2: run_quarter<2>(a, x, g, zs0, zs1, bar); break;
      default: run_quarter<3>(a, x, g, zs0, zs1, bar); break;
    }
    return;
  }
  uint32_t *rb = zs + kQWords + kQExchange + kQStage * col;
  if (g != a.G - 1) e.lane_mask = ~0u;
  const uint32_t full = uint32_t(a.n_bits >> 5), tiles = uint32_t((a.n_bits + 31) >> 5);
#pragma unroll 1
  for (uint32_t t = 0; t < tiles; ++t) {
    tile_sync(bar);
    if (g >= a.G) continue;
    uint32_t *zr = t & 1 ? zr1 : zr0, *zo = t & 1 ? zs1 : zs0;
#pragma unroll 8
    for (int c = 0; c < 32; ++c) zr[c * kKsThreads] ^= zo[c * kKsThreads];
    emit_tile<LAYOUT, kQStage>(zr, rb, a, g, uint64_t(t) << 5, t < full ? 32 : int(a.n_bits & 31), e);
    if (LAYOUT != MICKEY_LAYOUT_BITSLICED_U32 && e.stage &&
        ((t & (kQStage - 1)) == kQStage - 1 || t == tiles - 1))
      flush_rows<LAYOUT, kQStage>(rb, a, g, t & ~uint32_t(kQStage - 1), t, e);
  }
}

template <int LAYOUT>
cudaError_t launch_layout(const KeystreamArgs &a, const EmitCtx &e, uint32_t W, uint32_t blocks,
                          cudaStream_t st) {
  const size_t smem = 4 * (kQWords + kQExchange + row_stage_words(kQStage));
  const cudaError_t c = cudaFuncSetAttribute(
      quarters_kernel<LAYOUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(smem));
  if (c != cudaSuccess) return c;
  quarters_kernel<LAYOUT><<<blocks, kQuarterThreads, smem, st>>>(a, e, W);
  return cudaGetLastError();
}

}  // namespace

cudaError_t launch_quarters(const KeystreamArgs &a, int layout, int sm_count, cudaStream_t st) {
  const uint32_t W = (a.G + 31) / 32;
  static_assert(kSlots == kQuartersPerSm, "room for the dispatch's limit");
  if (W > uint32_t(kSlots * sm_count)) return cudaErrorInvalidValue;
  const uint32_t blocks = W < uint32_t(sm_count) ? W : uint32_t(sm_count);
  EmitCtx e;
  const uint32_t tail = uint32_t(a.n & 31u);
  const uintptr_t addr = reinterpret_cast<uintptr_t>(a.out);
  e.lane_mask = tail ? (1u << tail) - 1u : ~0u;
  e.vec_ok = addr % 16 == 0 && a.n_bits % 4 == 0;
  e.word_ok = addr % 4 == 0 && ((a.n_bits + 7) / 8) % 4 == 0;
  e.stage = layout != MICKEY_LAYOUT_BITSLICED_U32 && addr % 16 == 0 && a.n_bits % (32 * kQStage) == 0;
  switch (layout) {
    case MICKEY_LAYOUT_BITSLICED_U32: return launch_layout<MICKEY_LAYOUT_BITSLICED_U32>(a, e, W, blocks, st);
    case MICKEY_LAYOUT_BYTES: return launch_layout<MICKEY_LAYOUT_BYTES>(a, e, W, blocks, st);
    case MICKEY_LAYOUT_U32: return launch_layout<MICKEY_LAYOUT_U32>(a, e, W, blocks, st);
    case MICKEY_LAYOUT_U32_F32: return launch_layout<MICKEY_LAYOUT_U32_F32>(a, e, W, blocks, st);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace mickey
