// Bitsliced Grain (version 1) keystream generation: the paper's second
// stream cipher (Sec. II-C-3: an 80-bit LFSR and an 80-bit NFSR shifted
// together each clock, 80-bit key, 64-bit IV, 160 initialisation clocks),
// in the column-major representation of Sec. IV-A: a 32-bit word holds the
// same register bit of 32 instances, one thread clocks a 32-lane group.
//
// State: s[0..79] (LFSR) and b[0..79] (NFSR), 160 words in registers.  The
// shift of both registers is never executed: slot (R + i) % 80 holds s_{i}
// when R clocks have passed (mod 80), and a clock overwrites slot R (the
// oldest bit) with the new bit s_{i+80} (register renaming, Sec. IV-C).
//
// Per clock, with 3-input logic instructions (lop3.b32):
//   LFSR   s_{i+80} = s62+s51+s38+s23+s13+s0                        3 ops
//   NFSR   b_{i+80} = s0 + g(b): 12 linear terms and 11 products of 2 to 6
//          taps, with the partial products b63b60, b37b33, b15b9, b60b52,
//          b52b45, b33b28b21 and b63b45b28 shared                   23 ops
//   output z = b1+b2+b4+b10+b31+b43+b56 + h(s3,s25,s46,s64,b63), h written
//          as H0 + b63 H1, H0 and H1 of LFSR bits only             10 ops
//   init   z is added into both new bits (into the LFSR's last XOR)  +1
// This file: initialisation with a thread per group, the handle and the C ABI;
// the keystream kernels are in grain_ws.cu (a thread per group) and
// grain_packed.cu (a thread per instance).
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <new>
#include <vector>

#include "../../include/grain.h"
#include "../../include/mickey.h"
#include "bitslice.cuh"
#include "grain_clock.cuh"
#include "internal.h"

namespace mickey {
namespace {

using namespace grainc;

// ---------------------------------------------------------------- init

struct GrainInitArgs {
  const uint8_t *keys;  // n x 10
  const uint8_t *ivs;   // n x 8
  uint64_t n;
  uint32_t G, Gpad;
  uint32_t *state;
};

constexpr int kInitT = 64;                   // groups per block
constexpr int kKeyWords = 81;                // 80 words of 32 keys + a spare (odd stride)
constexpr int kIvWords = 65;                 // 64 words of 32 IVs + a spare

// Copy `bytes` bytes of src into rows of row_bytes bytes, stride_words apart:
// 4-byte cp.async copies (all in flight at once; the caller waits) when src
// is 4-byte aligned, byte loads otherwise and for a last partial word.
__device__ __forceinline__ void stage(const uint8_t *src, uint64_t bytes, uint32_t *dst,
                                      int row_bytes, int stride_words) {
  const int row_words = row_bytes / 4;
  const bool aligned = (reinterpret_cast<uintptr_t>(src) & 3u) == 0;
  for (uint64_t w = threadIdx.x; w * 4 < bytes; w += kInitT) {
    uint32_t *d = dst + (w / row_words) * stride_words + w % row_words;
    if (aligned && w * 4 + 4 <= bytes) {
      const uint32_t da = uint32_t(__cvta_generic_to_shared(d));
      asm volatile("cp.async.ca.shared.global [%0], [%1], 4;" ::"r"(da),
                   "l"(reinterpret_cast<const uint32_t *>(src) + w) : "memory");
    } else {
      uint32_t v = 0;
      for (int k = 0; k < 4 && w * 4 + k < bytes; ++k) v |= uint32_t(src[w * 4 + k]) << (8 * k);
      *d = v;
    }
  }
}

// Little-endian 32 bits at byte offset o of a staged row, bit-reversed: bit
// (31 - j) of the result is bit j of the byte string from o on (least
// significant bit of each byte first), i.e. the row of a 32x32 transpose.
__device__ __forceinline__ uint32_t lsb_chunk(const uint32_t *row, int o) {
  const uint32_t w0 = row[o >> 2], w1 = row[(o >> 2) + 1];
  return __brev(__funnelshift_r(w0, w1, 8 * (o & 3)));
}

__global__ void __launch_bounds__(kInitT) grain_init_kernel(GrainInitArgs a) {
  __shared__ uint32_t ks[kInitT * kKeyWords], vs[kInitT * kIvWords];
  const uint64_t first = 32ull * blockIdx.x * kInitT;
  const uint64_t count = min(uint64_t(32) * kInitT, a.n - first);
  stage(a.keys + first * 10, count * 10, ks, 320, kKeyWords);
  stage(a.ivs + first * 8, count * 8, vs, 256, kIvWords);
  asm volatile("cp.async.wait_all;" ::: "memory");
  __syncthreads();
  const uint32_t g = blockIdx.x * blockDim.x + threadIdx.x;
  if (g >= a.G) return;
  const uint64_t left = a.n - 32ull * g;
  const int nv = left >= 32 ? 32 : int(left);
  const uint32_t *krow = ks + threadIdx.x * kKeyWords, *vrow = vs + threadIdx.x * kIvWords;
  uint32_t s[kG], b[kG];
  // key bits 32q .. 32q+31 of the 32 lanes: row r of the matrix is lane
  // 31 - r, so that after the transpose word j has bit l = that bit of lane l
  static_for<0, 3>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    uint32_t m[32];
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      const int l = 31 - r;
      uint32_t v = l < nv ? lsb_chunk(krow, 10 * l + 4 * q) : 0u;
      if (q == 2) v &= 0xFFFF0000u;           // bits 64..79 only
      m[r] = v;
    }
    transpose32(m);
    static_for<0, 32>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      if constexpr (32 * q + j < kG) b[32 * q + j] = m[j];
    });
  });
  static_for<0, 2>([&](auto qc) {
    constexpr int q = decltype(qc)::value;
    uint32_t m[32];
#pragma unroll
    for (int r = 0; r < 32; ++r) {
      const int l = 31 - r;
      m[r] = l < nv ? lsb_chunk(vrow, 8 * l + 4 * q) : 0u;
    }
    transpose32(m);
    static_for<0, 32>([&](auto jc) {
      constexpr int j = decltype(jc)::value;
      s[32 * q + j] = m[j];
    });
  });
#pragma unroll
  for (int i = 64; i < kG; ++i) s[i] = ~0u;    // s64..s79 = 1
#pragma unroll 1
  for (int rep = 0; rep < 4; ++rep) grain_body<40, true>(s, b, [](auto, uint32_t) {});
  const size_t P = a.Gpad;
#pragma unroll
  for (int i = 0; i < kG; ++i) {
    a.state[size_t(i) * P + g] = s[i];
    a.state[size_t(kG + i) * P + g] = b[i];
  }
}

// A few clocks of the bitsliced layout, a thread per group: no more than moving
// the states.  The paired launch clocks a whole tile for them, and with more
// warp-groups than clock warps one behind the other.
__global__ void __launch_bounds__(kInitT) grain_short_kernel(KeystreamArgs a, uint32_t lane_mask) {
  const uint32_t g = blockIdx.x * kInitT + threadIdx.x;
  if (g >= a.G) return;
  if (g != a.G - 1) lane_mask = ~0u;
  const size_t P = a.Gpad;
  uint32_t s[kG], b[kG];
#pragma unroll
  for (int i = 0; i < kG; ++i) {
    s[i] = a.state[size_t(i) * P + g];
    b[i] = a.state[size_t(kG + i) * P + g];
  }
  uint32_t *o = static_cast<uint32_t *>(a.out) + size_t(g) * a.n_bits;
#pragma unroll 1
  for (uint32_t c = 0; c < a.n_bits; ++c) o[c] = grain_clock_shift(s, b) & lane_mask;
#pragma unroll
  for (int i = 0; i < kG; ++i) {
    a.state[size_t(i) * P + g] = s[i];
    a.state[size_t(kG + i) * P + g] = b[i];
  }
}

// Logic ops per clock per 32-lane group, as written above (keystream clock
// including z, or an initialisation clock).
constexpr int kGrainOps = 10 + 3 + 23;
constexpr int kGrainInitOps = kGrainOps + 1;

}  // namespace
}  // namespace mickey

using namespace mickey;

struct grain_streams {
  size_t n = 0;
  uint32_t G = 0, Gpad = 0;
  uint32_t *d_state = nullptr;
  uint8_t *d_inputs = nullptr;   // host inputs staged: keys (10n), ivs (8n)
  uint32_t *d_flags = nullptr;   // one word per warp-group (hand-off between segments)
  int *d_err = nullptr;
  cudaStream_t stream = nullptr;
  uint64_t pos = 0;
  int sm_count = 0;
  uint32_t spin_limit = 1u << 24;
  int force = -1;                // MICKEY_GRAIN_QUEUE=1: paired launch with hand-offs at any
                                 // size, =0: paired launch; neither: one thread per instance
                                 // for few groups, else as 0
};

namespace {

int grain_fail(int code, const char *msg) { return set_error(code, msg); }

void grain_release(grain_streams *s) {
  if (!s) return;
  if (s->stream) cudaStreamSynchronize(s->stream);
  cudaFree(s->d_state);
  cudaFree(s->d_inputs);
  cudaFree(s->d_flags);
  cudaFree(s->d_err);
  delete s;
}

// Up to how many groups per SM a launch left to the library takes one thread
// per instance.  Measured (152 SMs; us; packed, thread per group):
//   groups                       126      7296      9728      14592      32768
//   bitsliced, 8192 bits      40, 388   343, 390  454, 390  672, 389   -, 661
//   bytes, 8192 bits          41, 506   290, 514  380, 509  561, 517  1265, 818
//   initialisation            11, 28    18, 27    21, 27     25, 27     44, 35
//   (the initialisation is level at 15,625: 26, 26; at 19,456: 30, 27)
// The packed launches' work grows with the groups from one warp per SM
// sub-partition on; a thread per group takes one warp-group's chain until
// every sub-partition has one (19456 groups; the initialisation: two).
constexpr uint32_t kGrainPackedInitPerSm = 102;
constexpr uint32_t kGrainPackedBitslicedPerSm = 54, kGrainPackedBytesPerSm = 86;
// Short calls are moving states, which costs a thread per instance its
// transposes, 1.6 us per 1000 groups (us; packed, thread per group):
//   groups                       2719      4844      7813      12500     19456     32768
//   bitsliced, 8 bits          13, 13    15, 13    21, 14    28, 15    40, 15    58, 20
//   bitsliced, 256 bits        17, 23    21, 23    29, 24    -
//   rows of one byte           14, 17    16, 17    21, 17    29, 18    40, 19    58, 25
//   rows of 24 bits            13, 24    17, 24    21, 25    29, 26    40, 30    58, 50
//   rows of one word           12, 14    16, 15    21, 16    28, 16    39, 15    57, 24
// Longer rows off the 16-byte grid cost the thread-per-group launch byte
// stores (1001 bits, 2^20 instances: 1196 against 216): packed at any size.
// Bitsliced calls of up to this many clocks that are not packed take
// grain_short_kernel (us; paired launch, this kernel: 500,000 instances x 8 bits
// 14.6, 11.5; x 16 15.3, 13.2; 2^21 x 8 32.3, 20.2; x 16 34.4, 24.7).
constexpr uint64_t kGrainShortBits = 16;
constexpr uint32_t kGrainPackedShortRowsPerSm = 32, kGrainPackedThreeBytesPerSm = 64;

bool grain_use_packed(const grain_streams *s, uint32_t per_sm) {
  return s->force < 0 && s->G <= per_sm * uint32_t(s->sm_count);
}

bool grain_generate_packed(const grain_streams *s, uint64_t n_bits, const void *out, int layout) {
  if (layout == MICKEY_LAYOUT_BITSLICED_U32) {
    // the two estimates behind the table's bitsliced lines:
    //   packed 8.4 + (0.243 + 0.00076 n_bits) per_sm,  thread per group 12.6 + 0.0445 n_bits
    const double per_sm = double(s->G) / s->sm_count;
    return grain_use_packed(s, kGrainPackedBitslicedPerSm) &&
           double(n_bits) * (0.0445 - 0.00076 * per_sm) >= 0.243 * per_sm - 4.2;
  }
  const uint64_t row = (n_bits + 7) / 8;
  const uint32_t per_sm = grain_rows16(n_bits, out) ? kGrainPackedBytesPerSm
                          : row == 1 || (row == 4 && reinterpret_cast<uintptr_t>(out) % 4 == 0)
                              ? kGrainPackedShortRowsPerSm
                          : row <= 3 ? kGrainPackedThreeBytesPerSm
                                     : ~0u / uint32_t(s->sm_count);
  return grain_use_packed(s, per_sm);
}

// Loading and initialisation clocks from device inputs.
cudaError_t grain_init(const grain_streams *s, const uint8_t *dk, const uint8_t *dv) {
  if (grain_use_packed(s, kGrainPackedInitPerSm))
    return launch_grain_packed_init(dk, dv, s->n, s->G, s->Gpad, s->d_state, s->stream);
  GrainInitArgs ia{dk, dv, s->n, s->G, s->Gpad, s->d_state};
  grain_init_kernel<<<(s->G + kInitT - 1) / kInitT, kInitT, 0, s->stream>>>(ia);
  return cudaGetLastError();
}

size_t grain_out_bytes(size_t n, uint64_t n_bits, int layout) {
  if (layout == MICKEY_LAYOUT_BITSLICED_U32) return size_t((n + 31) / 32 * n_bits * 4);
  if (layout == MICKEY_LAYOUT_BYTES) return size_t(n * ((n_bits + 7) / 8));
  return 0;
}

}  // namespace

extern "C" {

MICKEY_API grain_streams *grain_init_streams(const void *keys, const void *ivs, size_t n, int mem,
                                             void *cuda_stream) {
  if (!keys || !ivs || n == 0 || n > (size_t(1) << 36) ||
      (mem != MICKEY_MEM_HOST && mem != MICKEY_MEM_DEVICE)) {
    grain_fail(MICKEY_E_ARG, "keys/ivs must not be NULL, 0 < n <= 2^36, mem host or device");
    return nullptr;
  }
  grain_streams *s = new (std::nothrow) grain_streams;
  if (!s) {
    grain_fail(MICKEY_E_OOM, "host allocation failed");
    return nullptr;
  }
  s->n = n;
  s->G = uint32_t((n + 31) / 32);
  s->Gpad = (s->G + 31u) & ~31u;
  s->stream = static_cast<cudaStream_t>(cuda_stream);
  const uint8_t *dk = static_cast<const uint8_t *>(keys), *dv = static_cast<const uint8_t *>(ivs);
  int dev = 0;
  bool ok = cudaGetDevice(&dev) == cudaSuccess &&
            cudaDeviceGetAttribute(&s->sm_count, cudaDevAttrMultiProcessorCount, dev) ==
                cudaSuccess &&
            cudaMalloc(&s->d_state, size_t(2 * kG) * s->Gpad * 4) == cudaSuccess &&
            cudaMalloc(&s->d_flags, size_t(s->Gpad / 32) * 4) == cudaSuccess &&
            cudaMalloc(&s->d_err, sizeof(int)) == cudaSuccess &&
            cudaMemsetAsync(s->d_flags, 0, size_t(s->Gpad / 32) * 4, s->stream) == cudaSuccess &&
            cudaMemsetAsync(s->d_err, 0, sizeof(int), s->stream) == cudaSuccess;
  if (const char *v = getenv("MICKEY_SPIN_LIMIT")) {
    const long long l = atoll(v);
    if (l > 0 && l < (1ll << 31)) s->spin_limit = uint32_t(l);
  }
  if (const char *v = getenv("MICKEY_GRAIN_QUEUE")) s->force = atoi(v) != 0 ? 1 : 0;
  if (ok && mem == MICKEY_MEM_HOST) {
    ok = cudaMalloc(&s->d_inputs, n * 18) == cudaSuccess &&
         cudaMemcpyAsync(s->d_inputs, keys, n * 10, cudaMemcpyHostToDevice, s->stream) ==
             cudaSuccess &&
         cudaMemcpyAsync(s->d_inputs + n * 10, ivs, n * 8, cudaMemcpyHostToDevice, s->stream) ==
             cudaSuccess;
    dk = s->d_inputs;
    dv = s->d_inputs + n * 10;
  }
  if (ok) {
    ok = grain_init(s, dk, dv) == cudaSuccess;
  }
  if (!ok) {
    grain_release(s);
    grain_fail(MICKEY_E_CUDA, "device allocation, copy or launch failed");
    return nullptr;
  }
  set_error(MICKEY_OK, "");
  return s;
}

MICKEY_API int grain_reset_streams(grain_streams *s, const void *keys, const void *ivs, int mem) {
  if (!s || !keys || !ivs || (mem != MICKEY_MEM_HOST && mem != MICKEY_MEM_DEVICE))
    return grain_fail(MICKEY_E_ARG, "NULL argument or bad memory kind");
  const size_t n = s->n;
  const uint8_t *dk = static_cast<const uint8_t *>(keys), *dv = static_cast<const uint8_t *>(ivs);
  if (mem == MICKEY_MEM_HOST) {
    if (!s->d_inputs && cudaMalloc(&s->d_inputs, n * 18) != cudaSuccess)
      return grain_fail(MICKEY_E_OOM, "input staging");
    if (cudaMemcpyAsync(s->d_inputs, keys, n * 10, cudaMemcpyHostToDevice, s->stream) !=
            cudaSuccess ||
        cudaMemcpyAsync(s->d_inputs + n * 10, ivs, n * 8, cudaMemcpyHostToDevice, s->stream) !=
            cudaSuccess)
      return grain_fail(MICKEY_E_CUDA, "key/IV upload");
    dk = s->d_inputs;
    dv = s->d_inputs + n * 10;
  }
  if (grain_init(s, dk, dv) != cudaSuccess) return grain_fail(MICKEY_E_CUDA, "grain init launch");
  s->pos = 0;
  return set_error(MICKEY_OK, "");
}

MICKEY_API int grain_generate(grain_streams *s, uint64_t n_bits, void *out, int layout) {
  if (!s || !out || n_bits == 0) return grain_fail(MICKEY_E_ARG, "NULL argument or n_bits == 0");
  if (n_bits > kMaxBitsPerCall) return grain_fail(MICKEY_E_ARG, "n_bits per call is limited to 2^34");
  if (layout != MICKEY_LAYOUT_BITSLICED_U32 && layout != MICKEY_LAYOUT_BYTES)
    return grain_fail(MICKEY_E_LAYOUT, "Grain takes the bitsliced or the bytes layout");
  if (layout == MICKEY_LAYOUT_BITSLICED_U32 && (reinterpret_cast<uintptr_t>(out) & 3u))
    return grain_fail(MICKEY_E_ARG, "bitsliced output must be 4-byte aligned");
  const KeystreamArgs ka{s->d_state, s->G, s->Gpad, s->n, n_bits, out};
  if (grain_generate_packed(s, n_bits, out, layout)) {
    if (launch_grain_packed(ka, layout, s->stream) != cudaSuccess)
      return grain_fail(MICKEY_E_CUDA, "grain keystream launch");
    s->pos += n_bits;
    return set_error(MICKEY_OK, "");
  }
  if (layout == MICKEY_LAYOUT_BITSLICED_U32 && n_bits <= kGrainShortBits && s->force < 0) {
    const uint32_t tail = uint32_t(s->n & 31u);
    grain_short_kernel<<<(s->G + kInitT - 1) / kInitT, kInitT, 0, s->stream>>>(
        ka, tail ? (1u << tail) - 1u : ~0u);
    if (cudaGetLastError() != cudaSuccess)
      return grain_fail(MICKEY_E_CUDA, "grain keystream launch");
    s->pos += n_bits;
    return set_error(MICKEY_OK, "");
  }
  // Equal segments of the groups x tiles work line, one per clock warp, once
  // there is a warp-group for each; with fewer, a warp-group per pair.  Rows
  // that are staged in blocks of eight tiles are cut between blocks (a block in
  // two segments goes out word by word: 800,000 instances x 256 bits 72 us, 50 when not cut).
  // Forced hand-offs: one segment fewer than warp-groups, tails first.
  const uint64_t W = (s->G + 31) / 32, NT = (n_bits + 31) / 32;
  const bool hand_off = s->force == 1;
  const uint64_t slots = std::min<uint64_t>(4ull * uint32_t(s->sm_count),
                                            hand_off ? std::max<uint64_t>(W - 1, 1) : W);
  PersistArgs pa{};
  pa.blocks = uint32_t((slots + 3) / 4);
  pa.W = uint32_t(W);
  pa.L = (W * NT + slots - 1) / slots;
  if (layout == MICKEY_LAYOUT_BYTES && NT % 8 == 0 && grain_rows16(n_bits, out) && !hand_off)
    pa.L = (pa.L + 7) / 8 * 8;
  pa.cooperative = pa.L % NT != 0;        // else no warp-group is cut
  pa.flags = s->d_flags;
  pa.wait_flag = 1;
  pa.spin_limit = s->spin_limit;
  pa.err = s->d_err;
  pa.tails_first = hand_off;
  if (launch_grain_ws(ka, layout, pa, s->stream) != cudaSuccess)
    return grain_fail(MICKEY_E_CUDA, "grain keystream launch");
  s->pos += n_bits;
  return set_error(MICKEY_OK, "");
}

MICKEY_API size_t grain_output_bytes(size_t n, uint64_t n_bits, int layout) {
  return grain_out_bytes(n, n_bits, layout);
}

MICKEY_API int grain_set_stream(grain_streams *s, void *cuda_stream) {
  if (!s) return grain_fail(MICKEY_E_ARG, "NULL handle");
  s->stream = static_cast<cudaStream_t>(cuda_stream);
  return set_error(MICKEY_OK, "");
}

MICKEY_API int grain_sync(grain_streams *s) {
  if (!s) return grain_fail(MICKEY_E_ARG, "NULL handle");
  if (cudaStreamSynchronize(s->stream) != cudaSuccess)
    return grain_fail(MICKEY_E_CUDA, "cudaStreamSynchronize");
  int flag = 0;
  if (cudaMemcpy(&flag, s->d_err, sizeof flag, cudaMemcpyDeviceToHost) != cudaSuccess)
    return grain_fail(MICKEY_E_CUDA, "error flag copy");
  if (flag) {
    cudaMemset(s->d_err, 0, sizeof(int));
    // the hand-offs that nobody waited for any more
    cudaMemsetAsync(s->d_flags, 0, size_t(s->Gpad / 32) * 4, s->stream);
    return grain_fail(MICKEY_E_TIMEOUT, "a device-side wait timed out");
  }
  return set_error(MICKEY_OK, "");
}

MICKEY_API uint64_t grain_position(const grain_streams *s) { return s ? s->pos : UINT64_MAX; }

MICKEY_API int grain_export_state(grain_streams *s, uint8_t *states) {
  if (!s || !states) return grain_fail(MICKEY_E_ARG, "NULL argument");
  std::vector<uint32_t> w(size_t(2 * kG) * s->Gpad);
  if (cudaStreamSynchronize(s->stream) != cudaSuccess ||
      cudaMemcpy(w.data(), s->d_state, w.size() * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
    return grain_fail(MICKEY_E_CUDA, "state copy");
  for (size_t i = 0; i < s->n; ++i) {
    const size_t g = i / 32, l = i % 32;
    uint8_t *rec = states + 20 * i;
    std::memset(rec, 0, 20);
    for (int k = 0; k < 2 * kG; ++k)
      if ((w[size_t(k) * s->Gpad + g] >> l) & 1u) rec[k / 8] |= uint8_t(1u << (k % 8));
  }
  return set_error(MICKEY_OK, "");
}

MICKEY_API int grain_ops_per_clock(int init) { return init ? kGrainInitOps : kGrainOps; }

MICKEY_API void grain_free(grain_streams *s) { grain_release(s); }

}  // extern "C"
