// Internal interfaces between the C ABI (capi.cu) and the kernel
// translation units.  Plain pointers and sizes only.
#pragma once

#include <cuda_runtime.h>

#include <cstddef>
#include <cstdint>

#include "ragged_cuts.h"

namespace mickey {

// Device-side error bits, OR-ed into a per-handle flag word.
constexpr int kErrIvLen = 1;
constexpr int kErrTimeout = 2;

// Rows of the bitsliced input scratch, each Gpad words long:
//   [0, 80)    key words K[j], bit l = key bit j of lane l
//   [80, 160)  IV-phase input words, right-aligned per lane
//   [160, 240) IV-phase activity masks (only read for mixed-length groups)
// followed by one info word per group: max IV length | (mixed << 8).
constexpr int kKeyRow = 0;
constexpr int kIvRow = 80;
constexpr int kActRow = 160;
constexpr int kScratchRows = 240;

// Bitsliced state: 200 rows of Gpad words, r0..r99 then s0..s99.
constexpr int kStateRows = 200;

constexpr int kInitThreads = 128;

struct LoadArgs {
  const uint8_t *keys;      // n x 10, device
  const uint8_t *ivs;       // n x 10, device
  const uint32_t *iv_lens;  // n, device, or nullptr (= 80)
  uint64_t n;
  const uint32_t *perm;     // lane slot -> instance, or nullptr (identity)
  uint32_t G, Gpad;
  uint32_t *scratch;        // kScratchRows * Gpad + Gpad words
  int *err;
};

// Key/IV loading and preclocking of every group (init_kernels.cu): the
// scratch rows of `a`, then the 200-word state into `state` (kStateRows *
// Gpad words).
cudaError_t launch_init(const LoadArgs &a, uint32_t *state, cudaStream_t st);

// The same with one thread per instance (packed.cu); the scratch of `a` is
// not used.
cudaError_t launch_packed_init(const LoadArgs &a, uint32_t *state, cudaStream_t st);

// Launches of a handle whose mode is left to the library take one thread per
// instance up to this many groups per SM.  Measured (152 SMs, us; 2048 bits of
// bytes: packed, four warps per warp-group, thread per group; re-key: packed,
// thread per group):
//   groups    608       2432           4864           7296           9728
//   2048 bits 69, -, 712 212, 240, 711 407, 240, 713  604, 385, 713  -, 385, 713
//   re-key    27, 118   49, 119        77, 119        108, 119       136, 120
// The packed times grow with the groups once every SM sub-partition has a
// warp; four warps take a warp-group's clock in 117 ns with one per SM, 187
// with two, 270 with three; a thread per group takes 334 ns until all 608
// sub-partitions have a warp of 32 groups.  Rows of bytes that are not whole
// words cost the emission warps byte stores: there the packed launch goes as
// far as it beats a thread per group.  A call of up to 8 clocks mostly moves
// states, which costs the packed launch its transposes (1 bit, bitsliced: 2719
// groups 15 against 11 us, 7813 groups 24 against 11).
constexpr uint32_t kPackedShortPerSm = 13;
constexpr uint32_t kPackedKeystreamPerSm = 18;
constexpr uint32_t kPackedPerSm = 52;

struct KeystreamArgs {
  uint32_t *state;          // kStateRows * Gpad words, read and written back
  uint32_t G, Gpad;
  uint64_t n;               // instances
  uint64_t n_bits;          // keystream bits per instance in this call
  void *out;                // device output, layout-dependent
};

// Record the thread-local error reported by mickey_last_error (code 0
// clears it); returns `code`.
int set_error(int code, const char *msg);

}  // namespace mickey
struct mickey_streams;
namespace mickey {
// Device state words of a handle (kStateRows x Gpad, word-major).
const uint32_t *handle_state(const mickey_streams *s, uint32_t *G, uint32_t *Gpad);

// Unroll factors compiled for the keystream kernel.
constexpr int kUnrolls[] = {2, 4};
// Largest n_bits of one keystream launch: a row of the row-major layouts
// must stay below 4 GiB.
constexpr uint64_t kMaxBitsPerCall = 1ull << 34;
constexpr int kKsThreads = 128;

// Persistent mode (see keystream_persistent_kernel): W warp-groups, L tiles
// per warp, one flag word per warp-group: zero before a cooperative launch, 1
// from the end of a head piece until its tail piece has seen it, zero after it.
struct PersistArgs {
  uint32_t blocks;      // grid: 1 or 2 blocks per SM (cooperative), or one block per
                        // 4 warp-groups (paired launch with L = NT, not cooperative)
  uint32_t cooperative; // 1: all blocks resident (needed when segments hand off)
  uint32_t stage_tiles; // row staging depth in tiles: 2, 4 or 8 (paired kernel), 4 (two-block)
  uint32_t paired;      // 1: clock warps paired with emission warps; 0: two-block kernel
  uint32_t W;           // warp-groups = ceil(G / 32)
  uint64_t L;           // tiles of the work line per warp
  uint32_t *flags;      // W words
  uint32_t wait_flag;   // value a tail piece waits for (1; differs only under the
                        // MICKEY_TEST_UNPUBLISHED test hook, to make the wait run out)
  uint32_t spin_limit;  // bounded wait of a tail piece (iterations of ~256 ns)
  int *err;
  uint32_t tails_first; // 1: each segment runs its tail piece first, so that every hand-off
                        // is waited for (a test's order; 0: heads first, hardly any wait)
};

// Ragged generation on a handle (ragged.cu): stream i continues by
// n_bits[i] bits; its output starts at byte offsets[i] of out (row layouts)
// or, for the bitsliced layout, group g's words start at offsets[g].
struct RaggedArgs {
  uint32_t *state;          // kStateRows * Gpad words, read and written back
  uint32_t G, Gpad;
  uint64_t n;
  const uint64_t *n_bits;   // n values, device
  const uint64_t *offsets;  // n (row layouts) or G (bitsliced) byte offsets, device
  uint8_t *out;
  RaggedLine line;          // the warp-groups in blocks of kRaggedBlockBits clocks (their
                            // longest lane's), arrays on the device; only with `p`
};
constexpr uint32_t kRaggedBlockBits = 128;
// p == nullptr: one thread per instance; else clock and emission warps on the
// pieces of `line` (cooperative where it may be cut).
cudaError_t launch_ragged(const RaggedArgs &a, int layout, const PersistArgs *p, cudaStream_t st);

// One thread per instance (packed.cu), any n_bits, layout and alignment that
// launch_keystream takes.
cudaError_t launch_packed_keystream(const KeystreamArgs &a, int layout, cudaStream_t st);

// Four warps per warp-group (keystream_quarters.cu), at most kQuartersPerSm
// warp-groups per SM; any n_bits, layout and alignment that launch_keystream
// takes.
constexpr uint32_t kQuartersPerSm = 3;
cudaError_t launch_quarters(const KeystreamArgs &a, int layout, int sm_count, cudaStream_t st);

// Grain with one thread per instance (grain_packed.cu): the bitsliced or the
// bytes layout, any n_bits and alignment that grain_generate takes; loading and
// the 160 initialisation clocks.  State: s0..s79 then b0..b79, rows of Gpad words.
cudaError_t launch_grain_packed(const KeystreamArgs &a, int layout, cudaStream_t st);
// Whether Grain's byte rows lie on the 16-byte grid: the paired launch stages
// them then, whatever the last tile holds (a row is a whole number of words).
inline bool grain_rows16(uint64_t n_bits, const void *out) {
  return ((n_bits + 7) / 8) % 16 == 0 && (reinterpret_cast<uintptr_t>(out) & 15u) == 0;
}
// Grain with clock warps paired with emission warps (grain_ws.cu), any
// n_bits and alignment; `p` as for the paired keystream launch.
cudaError_t launch_grain_ws(const KeystreamArgs &a, int layout, const PersistArgs &p,
                            cudaStream_t st);
cudaError_t launch_grain_packed_init(const uint8_t *keys, const uint8_t *ivs, uint64_t n,
                                     uint32_t G, uint32_t Gpad, uint32_t *state, cudaStream_t st);

// p == nullptr: grid mode (one thread per group); else persistent mode.
// stage: row layouts stage this many tiles per row (grid: 2 or 4; persistent:
// p->stage_tiles) and write whole chunks of 4 x stage bytes per row, used when
// n_bits is a multiple of 32 x stage and `out` is 16-byte aligned; 0: direct
// 4-byte row stores.
cudaError_t launch_keystream(const KeystreamArgs &a, int layout, int unroll, int stage,
                             const PersistArgs *p, cudaStream_t st);

}  // namespace mickey
