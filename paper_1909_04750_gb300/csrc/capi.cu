// Host side of the C ABI declared in include/mickey.h: argument checking,
// device memory of a handle, kernel launches, chunked device-to-host
// generation, checkpoint export/import and error reporting.
#include <cuda_runtime.h>

#include <algorithm>
#include <cstdarg>
#include <cstdio>
#include <cstring>
#include <new>
#include <utility>
#include <vector>

#include "../../include/mickey.h"
#include "internal.h"
#include "tables.cuh"

using namespace mickey;

struct mickey_streams {
  size_t n = 0;
  uint32_t G = 0, Gpad = 0;
  uint32_t *d_state = nullptr;    // kStateRows x Gpad
  uint32_t *d_scratch = nullptr;  // (kScratchRows + 1) x Gpad
  uint8_t *d_inputs = nullptr;    // staging for host inputs: keys, ivs, lens
  int *d_err = nullptr;
  cudaStream_t stream = nullptr;
  int unroll = 4;
  int mode = 0;                   // 0 auto, 1 grid, 2 persistent
  int stage = 1;                  // row layouts: 0 direct stores, 1 the mode's default
                                  // staging depth, 2 / 4 / 8 that many tiles
  struct LayoutCfg {
    bool set = false;
    int mode = 0, unroll = 4;
    int stage = 1;
  } cfg[4];                       // per-layout settings (mickey_set_config / tune)
  int sm_count = 0;
  int persist_blocks = 0;         // blocks of the persistent kernel (<= SMs)
  uint32_t *d_flags = nullptr;    // one word per warp-group (hand-off between segments)
  uint32_t spin_limit = 1u << 24;   // polls of ~256 ns before a tail piece gives up
  bool test_unpublished = false;    // test hook: tails wait for a value no head writes
  bool test_tails_first = false;    // test hook: every hand-off is waited for
  // Keystream position of stream i = pos_base + pos[i]: a call that
  // continues every stream by the same count moves pos_base only (O(1) host
  // work, whatever n is); ragged calls and imports set pos[i]; pos_max is
  // the largest pos[i], so that the 2^40 limit check of a uniform call is
  // O(1) as well.
  uint64_t pos_base = 0, pos_max = 0;
  std::vector<uint64_t> pos;
  // device staging for mickey_generate_host
  void *d_stage[2] = {nullptr, nullptr};
  size_t stage_bytes = 0;
  cudaStream_t copy_stream = nullptr;
  cudaEvent_t ev_gen[2] = {nullptr, nullptr}, ev_copy[2] = {nullptr, nullptr};
  // mickey_generate_ragged: device copies of the per-stream lengths and
  // output offsets, and the event after the last launch that reads them;
  // two pinned host buffers they are copied from, each with the event after
  // its last copy
  uint64_t *d_ragged = nullptr;
  size_t ragged_words = 0;
  cudaEvent_t ev_ragged = nullptr;
  uint64_t *h_ragged[2] = {nullptr, nullptr};
  cudaEvent_t ev_h2d[2] = {nullptr, nullptr};
  int ragged_flip = 0;
};

namespace {

thread_local int t_err = MICKEY_OK;
thread_local char t_msg[512] = "";

int fail(int code, const char *fmt, ...) {
  t_err = code;
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(t_msg, sizeof t_msg, fmt, ap);
  va_end(ap);
  return code;
}

int ok() {
  t_err = MICKEY_OK;
  t_msg[0] = '\0';
  return MICKEY_OK;
}

int cuda_fail(cudaError_t e, const char *what) {
  return fail(e == cudaErrorMemoryAllocation ? MICKEY_E_OOM : MICKEY_E_CUDA,
              "%s: %s", what, cudaGetErrorString(e));
}

#define CUDA_TRY(call, what)                     \
  do {                                           \
    cudaError_t e_ = (call);                     \
    if (e_ != cudaSuccess) return cuda_fail(e_, what); \
  } while (0)

// Index of the first IV length above 80 bits in host memory, or n.  The
// maximum of each block is taken by a loop without an early exit (so the
// compiler vectorises it); only a block that holds an offender is scanned.
size_t first_long_iv(const uint32_t *lens, size_t n) {
  constexpr size_t kBlock = 4096;
  for (size_t b = 0; b < n; b += kBlock) {
    const size_t e = std::min(n, b + kBlock);
    uint32_t mx = 0;
    for (size_t i = b; i < e; ++i) mx = std::max(mx, lens[i]);
    if (mx > MICKEY_MAX_IV_BITS)
      for (size_t i = b; i < e; ++i)
        if (lens[i] > MICKEY_MAX_IV_BITS) return i;
  }
  return n;
}

int default_mode() {
  const char *v = getenv("MICKEY_MODE");
  if (v && !strcmp(v, "grid")) return MICKEY_MODE_GRID;
  if (v && !strcmp(v, "persistent")) return MICKEY_MODE_PERSISTENT;
  if (v && !strcmp(v, "persistent2")) return MICKEY_MODE_PERSISTENT2;
  return MICKEY_MODE_AUTO;
}

int default_unroll() {
  const char *v = getenv("MICKEY_UNROLL");
  if (v) {
    const int u = atoi(v);
    for (int k : kUnrolls)
      if (k == u) return u;
  }
  return 4;
}

bool layout_ok(int layout) {
  return layout >= MICKEY_LAYOUT_BITSLICED_U32 && layout <= MICKEY_LAYOUT_U32_F32;
}

// Output bytes of one call; 0 if the layout cannot hold n_bits.
size_t out_bytes(size_t n, uint64_t n_bits, int layout) {
  const uint64_t G = (n + 31) / 32;
  switch (layout) {
    case MICKEY_LAYOUT_BITSLICED_U32: return size_t(G * n_bits * 4);
    case MICKEY_LAYOUT_BYTES: return size_t(n * ((n_bits + 7) / 8));
    case MICKEY_LAYOUT_U32: return n_bits % 32 ? 0 : size_t(n * (n_bits / 8));
    case MICKEY_LAYOUT_U32_F32: return n_bits % 32 ? 0 : size_t(2 * n * (n_bits / 8));
    default: return 0;
  }
}

void release(mickey_streams *s) {
  if (!s) return;
  if (s->stream) cudaStreamSynchronize(s->stream);
  if (s->copy_stream) {
    cudaStreamSynchronize(s->copy_stream);
    cudaStreamDestroy(s->copy_stream);
  }
  for (int k = 0; k < 2; ++k) {
    if (s->ev_gen[k]) cudaEventDestroy(s->ev_gen[k]);
    if (s->ev_copy[k]) cudaEventDestroy(s->ev_copy[k]);
    if (s->d_stage[k]) cudaFree(s->d_stage[k]);
  }
  cudaFree(s->d_state);
  cudaFree(s->d_scratch);
  cudaFree(s->d_inputs);
  cudaFree(s->d_err);
  cudaFree(s->d_flags);
  cudaFree(s->d_ragged);
  if (s->ev_ragged) cudaEventDestroy(s->ev_ragged);
  for (int k = 0; k < 2; ++k) {
    if (s->h_ragged[k]) cudaFreeHost(s->h_ragged[k]);
    if (s->ev_h2d[k]) cudaEventDestroy(s->ev_h2d[k]);
  }
  delete s;
}

int allocate(mickey_streams *s, size_t n) {
  s->n = n;
  s->G = uint32_t((n + 31) / 32);
  s->Gpad = (s->G + 31u) & ~31u;
  s->pos.assign(n, 0);
  s->unroll = default_unroll();
  s->mode = default_mode();
  if (const char *v = getenv("MICKEY_STAGE")) {
    const int d = atoi(v);
    s->stage = (d == 0 || d == 1 || d == 2 || d == 4 || d == 8) ? d : 1;
  }
  if (const char *v = getenv("MICKEY_SPIN_LIMIT")) {
    const long long l = atoll(v);
    if (l > 0 && l < (1ll << 31)) s->spin_limit = uint32_t(l);
  }
  if (const char *v = getenv("MICKEY_TEST_UNPUBLISHED")) s->test_unpublished = atoi(v) != 0;
  if (const char *v = getenv("MICKEY_TEST_TAILS_FIRST")) s->test_tails_first = atoi(v) != 0;
  int dev = 0;
  CUDA_TRY(cudaGetDevice(&dev), "cudaGetDevice");
  CUDA_TRY(cudaDeviceGetAttribute(&s->sm_count, cudaDevAttrMultiProcessorCount, dev),
           "cudaDeviceGetAttribute");
  s->persist_blocks = s->sm_count;
  if (const char *v = getenv("MICKEY_PERSIST_BLOCKS")) {
    const int b = atoi(v);
    if (b > 0 && b < s->sm_count) s->persist_blocks = b;
  }
  CUDA_TRY(cudaMalloc(&s->d_flags, size_t((s->G + 31) / 32) * 4), "cudaMalloc(flags)");
  CUDA_TRY(cudaMemsetAsync(s->d_flags, 0, size_t((s->G + 31) / 32) * 4, s->stream),
           "cudaMemset(flags)");
  CUDA_TRY(cudaMalloc(&s->d_state, size_t(kStateRows) * s->Gpad * 4), "cudaMalloc(state)");
  CUDA_TRY(cudaMalloc(&s->d_scratch, size_t(kScratchRows + 1) * s->Gpad * 4),
           "cudaMalloc(scratch)");
  CUDA_TRY(cudaMalloc(&s->d_err, sizeof(int)), "cudaMalloc(err)");
  CUDA_TRY(cudaMemsetAsync(s->d_err, 0, sizeof(int), s->stream), "cudaMemset(err)");
  return ok();
}

// Whether initialisations and ragged calls left to the library clock one
// instance per thread.
bool use_packed(const mickey_streams *s) {
  return s->G <= kPackedPerSm * uint32_t(s->sm_count);
}

// Whether launches left to the library take four warps per warp-group when
// they do not clock one instance per thread.
bool use_quarters(const mickey_streams *s) {
  return (s->G + 31) / 32 <= kQuartersPerSm * uint32_t(s->sm_count);
}

// Key/IV loading + preclock for all instances of s.
int run_init(mickey_streams *s, const void *keys, const void *ivs,
             const uint32_t *iv_lens, int mem) {
  if (!keys || !ivs) return fail(MICKEY_E_ARG, "keys and ivs must not be NULL");
  if (mem != MICKEY_MEM_HOST && mem != MICKEY_MEM_DEVICE)
    return fail(MICKEY_E_ARG, "mem must be MICKEY_MEM_HOST or MICKEY_MEM_DEVICE");
  const size_t n = s->n;
  const uint8_t *dk, *di;
  const uint32_t *dl = nullptr;
  if (mem == MICKEY_MEM_HOST) {
    if (iv_lens) {
      const size_t i = first_long_iv(iv_lens, n);
      if (i < n) return fail(MICKEY_E_IVLEN, "iv_lens[%zu] = %u exceeds 80 bits", i, iv_lens[i]);
    }
    // keys, IVs and lengths each at a 16-byte aligned offset (the init
    // kernel then reads them with 16-byte loads)
    const size_t rec = (n * 10 + 15) & ~size_t(15);
    if (!s->d_inputs)
      CUDA_TRY(cudaMalloc(&s->d_inputs, 2 * rec + n * 4), "cudaMalloc(inputs)");
    uint8_t *p = s->d_inputs;
    CUDA_TRY(cudaMemcpyAsync(p, keys, n * 10, cudaMemcpyHostToDevice, s->stream), "H2D keys");
    CUDA_TRY(cudaMemcpyAsync(p + rec, ivs, n * 10, cudaMemcpyHostToDevice, s->stream),
             "H2D ivs");
    dk = p;
    di = p + rec;
    if (iv_lens) {
      uint32_t *lens = reinterpret_cast<uint32_t *>(p + 2 * rec);
      CUDA_TRY(cudaMemcpyAsync(lens, iv_lens, n * 4, cudaMemcpyHostToDevice, s->stream),
               "H2D iv_lens");
      dl = lens;
    }
  } else {
    dk = static_cast<const uint8_t *>(keys);
    di = static_cast<const uint8_t *>(ivs);
    dl = iv_lens;
  }
  LoadArgs la{dk, di, dl, n, nullptr, s->G, s->Gpad, s->d_scratch, s->d_err};
  if (s->mode == MICKEY_MODE_AUTO && use_packed(s))
    CUDA_TRY(launch_packed_init(la, s->d_state, s->stream), "packed_init_kernel launch");
  else
    CUDA_TRY(launch_init(la, s->d_state, s->stream), "init_kernel launch");
  if (s->pos_max) std::fill(s->pos.begin(), s->pos.end(), 0);
  s->pos_base = s->pos_max = 0;
  return ok();
}

int check_limit(const mickey_streams *s, uint64_t n_bits) {
  // positions stay at or below 2^40, so these sums cannot wrap
  const uint64_t room = n_bits <= MICKEY_MAX_STREAM_BITS ? MICKEY_MAX_STREAM_BITS - n_bits : 0;
  if (n_bits <= MICKEY_MAX_STREAM_BITS && s->pos_base + s->pos_max <= room) return MICKEY_OK;
  for (size_t i = 0; i < s->n; ++i)   // name the first stream that would pass it
    if (n_bits > MICKEY_MAX_STREAM_BITS || s->pos_base + s->pos[i] > room)
      return fail(MICKEY_E_LIMIT,
                  "stream %zu would pass 2^40 keystream bits (at %llu, +%llu)", i,
                  (unsigned long long)(s->pos_base + s->pos[i]), (unsigned long long)n_bits);
  return MICKEY_OK;
}

int check_generate(const mickey_streams *s, uint64_t n_bits, const void *out, int layout) {
  if (!s || !out) return fail(MICKEY_E_ARG, "handle and output must not be NULL");
  if (n_bits == 0) return fail(MICKEY_E_ARG, "n_bits must be > 0");
  if (!layout_ok(layout)) return fail(MICKEY_E_LAYOUT, "unknown layout %d", layout);
  if ((layout == MICKEY_LAYOUT_U32 || layout == MICKEY_LAYOUT_U32_F32) && n_bits % 32)
    return fail(MICKEY_E_LAYOUT, "u32 layouts need n_bits %% 32 == 0 (got %llu)",
                (unsigned long long)n_bits);
  if (layout != MICKEY_LAYOUT_BYTES && reinterpret_cast<uintptr_t>(out) % 4)
    return fail(MICKEY_E_ARG, "output of a 32-bit layout must be 4-byte aligned");
  return check_limit(s, n_bits);
}

// Blocks per SM of a persistent launch in `mode`.
uint32_t persist_per_sm(int mode) { return mode == MICKEY_MODE_PERSISTENT2 ? 2u : 1u; }

// Whether a launch can use a persistent kernel of `mode`: there must be at
// least as many warp-groups as warps that clock.
bool use_persistent(const mickey_streams *s, int mode) {
  const uint64_t W = (s->G + 31) / 32;
  const uint64_t slots = uint64_t(s->persist_blocks) * persist_per_sm(mode) * 4;
  return mode != MICKEY_MODE_GRID && W >= slots;
}

// What the segments of one launch hand states on with.
void set_hand_off(const mickey_streams *s, PersistArgs &pa) {
  pa.flags = s->d_flags;
  pa.wait_flag = s->test_unpublished ? 2 : 1;
  pa.spin_limit = s->spin_limit;
  pa.err = s->d_err;
  pa.tails_first = s->test_tails_first;
}

// One keystream launch of `bits` clocks into a device buffer.
//   AUTO, few groups          one thread per instance, or four warps per warp-group
//                             (calls of a few clocks go over to the latter earlier:
//                             250,000 x 1 bit of bytes 24 against 15 us)
//   GRID                      one thread per group, clocking and emitting
//   PERSISTENT2, enough groups two clocking warps per SM sub-partition
//   otherwise (AUTO, PERSISTENT) the paired kernel: clock warps beside emission
//                             warps; with enough warp-groups the cooperative
//                             launch with equal segments, else one warp-group
//                             per pair.  It outruns the others at every size
//                             measured above the first line's, so AUTO takes it.
int launch_generate(mickey_streams *s, uint64_t bits, void *out, int layout) {
  KeystreamArgs ka{s->d_state, s->G, s->Gpad, s->n, bits, out};
  const auto &c = s->cfg[layout];
  int mode = c.set ? c.mode : s->mode;
  const int unroll = c.set ? c.unroll : s->unroll;
  const int stage = c.set ? c.stage : s->stage;
  if (mode == MICKEY_MODE_AUTO) {
    const uint32_t sms = uint32_t(s->sm_count);
    const bool words = layout != MICKEY_LAYOUT_BYTES ||
                       ((bits + 7) / 8 % 4 == 0 && reinterpret_cast<uintptr_t>(out) % 4 == 0);
    const uint32_t per_sm = bits <= 8 ? kPackedShortPerSm : words ? kPackedKeystreamPerSm : kPackedPerSm;
    if (s->G <= per_sm * sms) {
      CUDA_TRY(launch_packed_keystream(ka, layout, s->stream), "packed_keystream_kernel launch");
      return MICKEY_OK;
    }
    if (use_quarters(s)) {
      CUDA_TRY(launch_quarters(ka, layout, s->sm_count, s->stream), "quarters_kernel launch");
      return MICKEY_OK;
    }
  }
  if (mode == MICKEY_MODE_GRID) {
    CUDA_TRY(launch_keystream(ka, layout, unroll, stage, nullptr, s->stream),
             "keystream_kernel launch");
    return MICKEY_OK;
  }
  if (mode == MICKEY_MODE_PERSISTENT2 && !use_persistent(s, mode)) mode = MICKEY_MODE_PERSISTENT;
  const uint32_t per_sm = persist_per_sm(mode);
  const uint64_t W = (s->G + 31) / 32, NT = (bits + 31) / 32;
  PersistArgs pa;
  // the two-block kernel stages 4 tiles; the paired kernel 8 unless told otherwise
  pa.paired = per_sm == 2 ? 0u : 1u;
  pa.stage_tiles = per_sm == 2 ? 4u : (stage == 2 || stage == 4 ? uint32_t(stage) : 8u);
  pa.W = uint32_t(W);
  if (use_persistent(s, mode)) {
    const uint64_t slots = uint64_t(s->persist_blocks) * per_sm * 4;
    pa.blocks = uint32_t(s->persist_blocks) * per_sm;
    pa.L = (W * NT + slots - 1) / slots;
    pa.cooperative = pa.L % NT != 0;     // else no warp-group is cut
  } else {  // one warp-group per clock/emission pair, four pairs per block
    pa.blocks = uint32_t((W + 3) / 4);
    pa.cooperative = 0;
    pa.L = NT;
  }
  set_hand_off(s, pa);
  CUDA_TRY(launch_keystream(ka, layout, unroll, stage, &pa, s->stream),
           "keystream persistent launch");
  return MICKEY_OK;
}

// Byte offsets of the packed ragged output (rows, or for the bitsliced layout
// the groups' word arrays, back to back) into offs; returns the total size.
uint64_t ragged_packed(size_t n, const uint64_t *n_bits, int layout, uint64_t *offs) {
  uint64_t off = 0;
  if (layout == MICKEY_LAYOUT_BITSLICED_U32) {
    for (size_t g = 0; g * 32 < n; ++g) {
      uint64_t c = 0;
      for (size_t i = 32 * g; i < n && i < 32 * g + 32; ++i) c = std::max(c, n_bits[i]);
      if (offs) offs[g] = off;
      off += 4 * c;
    }
    return off;
  }
  for (size_t i = 0; i < n; ++i) {
    if (offs) offs[i] = off;
    off += layout == MICKEY_LAYOUT_U32 ? n_bits[i] / 8 : (n_bits[i] + 7) / 8;
  }
  return off;
}

// Copy m lengths and return the longest, in one pass (a pass of its own over
// 2^20 lengths cost the call 0.7 ms): four maxima, so that they do not wait for
// one another.
uint64_t copy_longest(const uint64_t *src, size_t m, uint64_t *dst) {
  uint64_t top[4] = {0, 0, 0, 0};
  size_t i = 0;
  for (; i + 4 <= m; i += 4)
    for (int k = 0; k < 4; ++k) {
      const uint64_t v = src[i + k];
      dst[i + k] = v;
      top[k] = v > top[k] ? v : top[k];
    }
  for (; i < m; ++i) top[0] = std::max(top[0], dst[i] = src[i]);
  return std::max(std::max(top[0], top[1]), std::max(top[2], top[3]));
}

// True when every stream asks for the same number of bits and the offsets
// (NULL = packed) are the packed ones: row i at i * row bytes, group g's
// words at g * 4 * n_bits.
bool equal_packed(size_t n, const uint64_t *n_bits, const uint64_t *offs, int layout) {
  const uint64_t b = n_bits[0];
  for (size_t i = 1; i < n; ++i)
    if (n_bits[i] != b) return false;
  if (b == 0 || !offs) return b != 0;
  const size_t n_off = layout == MICKEY_LAYOUT_BITSLICED_U32 ? (n + 31) / 32 : n;
  const uint64_t step = layout == MICKEY_LAYOUT_BITSLICED_U32 ? 4 * b
                        : layout == MICKEY_LAYOUT_U32         ? b / 8
                                                              : (b + 7) / 8;
  for (size_t k = 0; k < n_off; ++k)
    if (offs[k] != k * step) return false;
  return true;
}

}  // namespace

namespace mickey {
int set_error(int code, const char *msg) { return code ? fail(code, "%s", msg) : ok(); }

const uint32_t *handle_state(const mickey_streams *s, uint32_t *G, uint32_t *Gpad) {
  *G = s->G;
  *Gpad = s->Gpad;
  return s->d_state;
}
}  // namespace mickey

extern "C" {

mickey_streams *mickey_init_streams(const uint8_t *keys, const uint8_t *ivs,
                                    const uint32_t *iv_lens, size_t n) {
  return mickey_init_streams_ex(keys, ivs, iv_lens, n, MICKEY_MEM_HOST, nullptr);
}

mickey_streams *mickey_init_streams_ex(const void *keys, const void *ivs,
                                       const uint32_t *iv_lens, size_t n, int mem,
                                       void *cuda_stream) {
  if (!keys || !ivs || n == 0) {
    fail(MICKEY_E_ARG, "keys/ivs must not be NULL and n must be > 0");
    return nullptr;
  }
  if (n > (size_t(1) << 36)) {
    fail(MICKEY_E_ARG, "n = %zu instances is above the supported 2^36", n);
    return nullptr;
  }
  if (mem == MICKEY_MEM_HOST && iv_lens) {
    const size_t i = first_long_iv(iv_lens, n);
    if (i < n) {
      fail(MICKEY_E_IVLEN, "iv_lens[%zu] = %u exceeds 80 bits", i, iv_lens[i]);
      return nullptr;
    }
  }
  mickey_streams *s = new (std::nothrow) mickey_streams;
  if (!s) {
    fail(MICKEY_E_OOM, "host allocation failed");
    return nullptr;
  }
  s->stream = static_cast<cudaStream_t>(cuda_stream);
  if (allocate(s, n) != MICKEY_OK || run_init(s, keys, ivs, iv_lens, mem) != MICKEY_OK) {
    const int code = t_err;
    char msg[512];
    memcpy(msg, t_msg, sizeof msg);
    release(s);
    fail(code, "%s", msg);
    return nullptr;
  }
  ok();
  return s;
}

int mickey_reset_streams(mickey_streams *s, const void *keys, const void *ivs,
                         const uint32_t *iv_lens, int mem) {
  if (!s) return fail(MICKEY_E_ARG, "handle must not be NULL");
  return run_init(s, keys, ivs, iv_lens, mem);
}

int mickey_set_stream(mickey_streams *s, void *cuda_stream) {
  if (!s) return fail(MICKEY_E_ARG, "handle must not be NULL");
  s->stream = static_cast<cudaStream_t>(cuda_stream);
  return ok();
}

int mickey_generate(mickey_streams *s, uint64_t n_bits, void *out, int layout) {
  int rc = check_generate(s, n_bits, out, layout);
  if (rc) return rc;
  if (n_bits > kMaxBitsPerCall)
    return fail(MICKEY_E_ARG, "n_bits per call is limited to 2^34 (got %llu)",
                (unsigned long long)n_bits);
  rc = launch_generate(s, n_bits, out, layout);
  if (rc) return rc;
  s->pos_base += n_bits;
  return ok();
}

size_t mickey_output_bytes(size_t n, uint64_t n_bits, int layout) {
  return out_bytes(n, n_bits, layout);
}

int mickey_generate_ragged(mickey_streams *s, const uint64_t *n_bits, void *out,
                           const uint64_t *out_offsets, int layout) {
  if (!s || !n_bits || !out) return fail(MICKEY_E_ARG, "handle, n_bits and out must not be NULL");
  if (layout != MICKEY_LAYOUT_BITSLICED_U32 && layout != MICKEY_LAYOUT_BYTES &&
      layout != MICKEY_LAYOUT_U32)
    return fail(MICKEY_E_LAYOUT, "ragged generation takes the bitsliced, bytes or u32 layout "
                "(got %d)", layout);
  const size_t n = s->n, G = s->G;
  const size_t n_off = layout == MICKEY_LAYOUT_BITSLICED_U32 ? G : n;
  uint64_t any = 0;
  for (size_t i = 0; i < n; ++i) {
    if (n_bits[i] > kMaxBitsPerCall)
      return fail(MICKEY_E_ARG, "n_bits[%zu] = %llu is above 2^34 per call", i,
                  (unsigned long long)n_bits[i]);
    if (s->pos_base + s->pos[i] + n_bits[i] > MICKEY_MAX_STREAM_BITS)
      return fail(MICKEY_E_LIMIT, "stream %zu would pass 2^40 keystream bits", i);
    if (layout == MICKEY_LAYOUT_U32 && n_bits[i] % 32)
      return fail(MICKEY_E_LAYOUT, "the u32 layout needs n_bits[%zu] %% 32 == 0", i);
    any |= n_bits[i];
  }
  // 32-bit layouts: every output that receives words starts 4-byte aligned.
  // Packed offsets are multiples of 4 there, so only the base can be off.
  const uintptr_t base = reinterpret_cast<uintptr_t>(out);
  if (layout != MICKEY_LAYOUT_BYTES && any) {
    for (size_t k = 0; k < (out_offsets ? n_off : 1); ++k) {
      if ((base + (out_offsets ? out_offsets[k] : 0)) % 4 == 0) continue;
      uint64_t c = 0;   // the words this output receives (none: no constraint)
      if (!out_offsets) c = any;
      else if (layout == MICKEY_LAYOUT_U32) c = n_bits[k];
      else
        for (size_t i = 32 * k; i < n && i < 32 * k + 32; ++i) c = std::max(c, n_bits[i]);
      if (c)
        return fail(MICKEY_E_ARG, "output %zu of a 32-bit layout is not 4-byte aligned", k);
    }
  }
  if (!any) return ok();                              // nothing to generate
  // Equal lengths at the packed offsets are exactly mickey_generate's
  // layout ([n][row] or [G][n_bits]): take the keystream launch.
  if (equal_packed(n, n_bits, out_offsets, layout)) {
    const int rc = launch_generate(s, n_bits[0], out, layout);
    if (rc) return rc;
    s->pos_base += n_bits[0];
    return ok();
  }
  // The lengths and offsets reach the kernel through one of two pinned
  // buffers (so that the copy is a DMA and the next call can fill the other
  // buffer while this one is in flight) and one device buffer.
  // ... then, for the launch with a thread per group, its work line
  const size_t W = (G + 31) / 32, words = n + n_off + 2 * W + 1;
  if (s->ragged_words < words) {
    if (s->ev_ragged) CUDA_TRY(cudaEventSynchronize(s->ev_ragged), "sync");
    for (int k = 0; k < 2; ++k) {
      if (s->ev_h2d[k]) CUDA_TRY(cudaEventSynchronize(s->ev_h2d[k]), "sync");
      if (s->h_ragged[k]) cudaFreeHost(s->h_ragged[k]);
      s->h_ragged[k] = nullptr;
    }
    cudaFree(s->d_ragged);
    s->d_ragged = nullptr;
    s->ragged_words = 0;
    CUDA_TRY(cudaMalloc(&s->d_ragged, words * 8), "cudaMalloc(ragged lengths)");
    for (int k = 0; k < 2; ++k)
      CUDA_TRY(cudaMallocHost(&s->h_ragged[k], words * 8), "cudaMallocHost(ragged lengths)");
    s->ragged_words = words;
  }
  for (int k = 0; k < 2; ++k)
    if (!s->ev_h2d[k])
      CUDA_TRY(cudaEventCreateWithFlags(&s->ev_h2d[k], cudaEventDisableTiming), "event");
  if (!s->ev_ragged)
    CUDA_TRY(cudaEventCreateWithFlags(&s->ev_ragged, cudaEventDisableTiming), "event");
  const int kb = s->ragged_flip;
  CUDA_TRY(cudaEventSynchronize(s->ev_h2d[kb]), "staging buffer");  // its last copy is done
  uint64_t *h = s->h_ragged[kb];
  if (out_offsets)
    std::copy(out_offsets, out_offsets + n_off, h + n);
  else
    ragged_packed(n, n_bits, layout, h + n);
  const auto &c = s->cfg[layout];
  const bool packed = (c.set ? c.mode : s->mode) == MICKEY_MODE_AUTO && use_packed(s);
  const uint64_t slots = std::min<uint64_t>(W, 4ull * uint32_t(s->persist_blocks));
  RaggedLine line{};
  if (packed) {
    std::copy(n_bits, n_bits + n, h);
  } else {
    std::vector<uint64_t> blocks(W);
    for (size_t w = 0; w < W; ++w)
      blocks[w] = (copy_longest(n_bits + 1024 * w, std::min<size_t>(n - 1024 * w, 1024),
                                h + 1024 * w) + kRaggedBlockBits - 1) / kRaggedBlockBits;
    uint64_t *order = h + n + n_off;
    line = ragged_cuts(blocks.data(), uint32_t(W), slots, order, order + W);
    line.order = s->d_ragged + n + n_off;    // where the copy below puts them
    line.blocks = line.order + W;
  }
  // the previous ragged launch (perhaps on another stream) has read d_ragged
  CUDA_TRY(cudaStreamWaitEvent(s->stream, s->ev_ragged, 0), "wait");
  CUDA_TRY(cudaMemcpyAsync(s->d_ragged, h, (packed ? n + n_off : words) * 8,
                           cudaMemcpyHostToDevice, s->stream),
           "H2D ragged lengths");
  CUDA_TRY(cudaEventRecord(s->ev_h2d[kb], s->stream), "record");
  s->ragged_flip = kb ^ 1;
  RaggedArgs ra{s->d_state, s->G, s->Gpad, n, s->d_ragged, s->d_ragged + n,
                static_cast<uint8_t *>(out), line};
  PersistArgs pa{};
  pa.blocks = uint32_t((slots + 3) / 4);
  pa.cooperative = line.alone < W;
  pa.W = uint32_t(W);
  if (!packed) {
    set_hand_off(s, pa);
    // By the cuts a tail hardly waits.  The limit grows with the segments all
    // the same: a warp whose rows cost it more stores may come to the hand-off
    // a part of its segment later than the next one.
    const uint64_t clocks = std::min<uint64_t>(line.L, ~0u / kRaggedBlockBits) * kRaggedBlockBits;
    pa.spin_limit = uint32_t(std::min<uint64_t>(pa.spin_limit + clocks, ~0u));
  }
  CUDA_TRY(launch_ragged(ra, layout, packed ? nullptr : &pa, s->stream), "ragged launch");
  CUDA_TRY(cudaEventRecord(s->ev_ragged, s->stream), "record");
  for (size_t i = 0; i < n; ++i) {
    s->pos[i] += n_bits[i];
    s->pos_max = std::max(s->pos_max, s->pos[i]);
  }
  return ok();
}

size_t mickey_ragged_output_bytes(size_t n, const uint64_t *n_bits, int layout) {
  if (!n_bits) return 0;
  if (layout != MICKEY_LAYOUT_BITSLICED_U32 && layout != MICKEY_LAYOUT_BYTES &&
      layout != MICKEY_LAYOUT_U32)
    return 0;
  for (size_t i = 0; i < n; ++i)   // above the per-call limit, or the sum could wrap
    if (n_bits[i] > kMaxBitsPerCall || (layout == MICKEY_LAYOUT_U32 && n_bits[i] % 32))
      return 0;
  return size_t(ragged_packed(n, n_bits, layout, nullptr));
}

int mickey_generate_host(mickey_streams *s, uint64_t n_bits, void *host_out, int layout) {
  int rc = check_generate(s, n_bits, host_out, layout);
  if (rc) return rc;
  // Chunk of keystream bits per launch: a multiple of 32 giving about
  // 256 MiB of output, so that two staging buffers stay small and copies
  // overlap with generation.
  const size_t per_bit = std::max<size_t>(1, out_bytes(s->n, 32, layout) / 32);
  uint64_t chunk = (uint64_t(256) << 20) / per_bit;
  chunk = std::max<uint64_t>(32, chunk & ~uint64_t(31));
  chunk = std::min<uint64_t>(chunk, (n_bits + 31) & ~uint64_t(31));
  const size_t need = out_bytes(s->n, chunk, layout);
  if (s->stage_bytes < need) {
    for (int k = 0; k < 2; ++k) {
      if (s->d_stage[k]) cudaFree(s->d_stage[k]);
      s->d_stage[k] = nullptr;
    }
    s->stage_bytes = 0;
    for (int k = 0; k < 2; ++k) CUDA_TRY(cudaMalloc(&s->d_stage[k], need), "cudaMalloc(stage)");
    s->stage_bytes = need;
  }
  if (!s->copy_stream) {
    CUDA_TRY(cudaStreamCreateWithFlags(&s->copy_stream, cudaStreamNonBlocking),
             "cudaStreamCreate");
    for (int k = 0; k < 2; ++k) {
      CUDA_TRY(cudaEventCreateWithFlags(&s->ev_gen[k], cudaEventDisableTiming), "event");
      CUDA_TRY(cudaEventCreateWithFlags(&s->ev_copy[k], cudaEventDisableTiming), "event");
    }
  }
  uint8_t *host = static_cast<uint8_t *>(host_out);
  const uint64_t G = s->G;
  uint64_t done = 0;
  int k = 0;
  while (done < n_bits) {
    const uint64_t bits = std::min<uint64_t>(chunk, n_bits - done);
    void *buf = s->d_stage[k];
    CUDA_TRY(cudaStreamWaitEvent(s->stream, s->ev_copy[k], 0), "wait copy");
    rc = launch_generate(s, bits, buf, layout);
    if (rc) return rc;
    CUDA_TRY(cudaEventRecord(s->ev_gen[k], s->stream), "record");
    CUDA_TRY(cudaStreamWaitEvent(s->copy_stream, s->ev_gen[k], 0), "wait gen");
    // copy the chunk's rows into their columns of the full host array
    switch (layout) {
      case MICKEY_LAYOUT_BITSLICED_U32:
        CUDA_TRY(cudaMemcpy2DAsync(host + done * 4, n_bits * 4, buf, bits * 4, bits * 4, G,
                                   cudaMemcpyDeviceToHost, s->copy_stream), "D2H");
        break;
      case MICKEY_LAYOUT_BYTES:
        CUDA_TRY(cudaMemcpy2DAsync(host + done / 8, (n_bits + 7) / 8, buf, (bits + 7) / 8,
                                   (bits + 7) / 8, s->n, cudaMemcpyDeviceToHost,
                                   s->copy_stream), "D2H");
        break;
      default: {
        const size_t w = bits / 8, W = n_bits / 8;  // bytes per row
        CUDA_TRY(cudaMemcpy2DAsync(host + done / 8, W, buf, w, w, s->n,
                                   cudaMemcpyDeviceToHost, s->copy_stream), "D2H");
        if (layout == MICKEY_LAYOUT_U32_F32)
          CUDA_TRY(cudaMemcpy2DAsync(host + s->n * W + done / 8, W,
                                     static_cast<uint8_t *>(buf) + s->n * w, w, w, s->n,
                                     cudaMemcpyDeviceToHost, s->copy_stream), "D2H");
      }
    }
    CUDA_TRY(cudaEventRecord(s->ev_copy[k], s->copy_stream), "record");
    s->pos_base += bits;
    done += bits;
    k ^= 1;
  }
  CUDA_TRY(cudaStreamSynchronize(s->copy_stream), "sync copy");
  return ok();
}

int mickey_sync(mickey_streams *s) {
  if (!s) return fail(MICKEY_E_ARG, "handle must not be NULL");
  CUDA_TRY(cudaStreamSynchronize(s->stream), "cudaStreamSynchronize");
  int flag = 0;
  CUDA_TRY(cudaMemcpy(&flag, s->d_err, sizeof flag, cudaMemcpyDeviceToHost), "D2H err");
  if (flag) {
    CUDA_TRY(cudaMemset(s->d_err, 0, sizeof(int)), "clear err");
    if (flag & kErrTimeout)   // the hand-offs that nobody waited for any more
      CUDA_TRY(cudaMemsetAsync(s->d_flags, 0, size_t((s->G + 31) / 32) * 4, s->stream),
               "clear flags");
    if (flag & kErrIvLen) return fail(MICKEY_E_IVLEN, "an IV length above 80 bits was given");
    if (flag & kErrTimeout) return fail(MICKEY_E_TIMEOUT, "a device-side wait timed out");
  }
  return ok();
}

size_t mickey_num_streams(const mickey_streams *s) { return s ? s->n : 0; }

uint64_t mickey_position(const mickey_streams *s, size_t i) {
  if (!s || i >= s->n) return UINT64_MAX;
  return s->pos_base + s->pos[i];
}

int mickey_export_state(mickey_streams *s, uint8_t *states, uint64_t *positions) {
  if (!s || !states) return fail(MICKEY_E_ARG, "handle and states must not be NULL");
  std::vector<uint32_t> words(size_t(kStateRows) * s->Gpad);
  CUDA_TRY(cudaStreamSynchronize(s->stream), "sync");
  CUDA_TRY(cudaMemcpy(words.data(), s->d_state, words.size() * 4, cudaMemcpyDeviceToHost),
           "D2H state");
  for (size_t i = 0; i < s->n; ++i) {
    const size_t g = i / 32, l = i % 32;
    uint8_t *rec = states + 26 * i;
    memset(rec, 0, 26);
    for (int half = 0; half < 2; ++half)
      for (int b = 0; b < kReg; ++b) {
        const uint32_t w = words[size_t(half * kReg + b) * s->Gpad + g];
        if ((w >> l) & 1u) rec[13 * half + b / 8] |= uint8_t(0x80u >> (b % 8));
      }
    if (positions) positions[i] = s->pos_base + s->pos[i];
  }
  return ok();
}

mickey_streams *mickey_import_state(const uint8_t *states, const uint64_t *positions,
                                    size_t n, void *cuda_stream) {
  if (!states || n == 0) {
    fail(MICKEY_E_ARG, "states must not be NULL and n must be > 0");
    return nullptr;
  }
  mickey_streams *s = new (std::nothrow) mickey_streams;
  if (!s) {
    fail(MICKEY_E_OOM, "host allocation failed");
    return nullptr;
  }
  s->stream = static_cast<cudaStream_t>(cuda_stream);
  if (allocate(s, n) != MICKEY_OK) {
    const int code = t_err;
    release(s);
    t_err = code;
    return nullptr;
  }
  std::vector<uint32_t> words(size_t(kStateRows) * s->Gpad, 0u);
  for (size_t i = 0; i < n; ++i) {
    const size_t g = i / 32, l = i % 32;
    const uint8_t *rec = states + 26 * i;
    for (int half = 0; half < 2; ++half)
      for (int b = 0; b < kReg; ++b)
        if ((rec[13 * half + b / 8] >> (7 - b % 8)) & 1u)
          words[size_t(half * kReg + b) * s->Gpad + g] |= 1u << l;
    if (positions) {
      if (positions[i] > MICKEY_MAX_STREAM_BITS) {
        release(s);
        fail(MICKEY_E_LIMIT, "position of stream %zu is beyond 2^40", i);
        return nullptr;
      }
      s->pos[i] = positions[i];
      s->pos_max = std::max(s->pos_max, positions[i]);
    }
  }
  cudaError_t e = cudaMemcpy(s->d_state, words.data(), words.size() * 4, cudaMemcpyHostToDevice);
  if (e != cudaSuccess) {
    release(s);
    cuda_fail(e, "H2D state");
    return nullptr;
  }
  ok();
  return s;
}

int mickey_set_config(mickey_streams *s, int layout, int mode, int unroll, int stage) {
  if (!s) return fail(MICKEY_E_ARG, "handle must not be NULL");
  if (!layout_ok(layout)) return fail(MICKEY_E_LAYOUT, "unknown layout %d", layout);
  if (mode < MICKEY_MODE_AUTO || mode > MICKEY_MODE_PERSISTENT2)
    return fail(MICKEY_E_ARG, "unknown mode %d", mode);
  bool known = false;
  for (int k : kUnrolls) known |= (k == unroll);
  if (!known) return fail(MICKEY_E_ARG, "unroll %d is not compiled (2 or 4)", unroll);
  if (stage != 0 && stage != 1 && stage != 2 && stage != 4 && stage != 8)
    return fail(MICKEY_E_ARG, "stage must be 0, 1, 2, 4 or 8 (got %d)", stage);
  auto &c = s->cfg[layout];
  c.set = true;
  c.mode = mode;
  c.unroll = unroll;
  c.stage = stage;
  return ok();
}

int mickey_get_config(const mickey_streams *s, int layout, int *mode, int *unroll, int *stage) {
  if (!s || !mode || !unroll || !stage) return fail(MICKEY_E_ARG, "NULL argument");
  if (!layout_ok(layout)) return fail(MICKEY_E_LAYOUT, "unknown layout %d", layout);
  const auto &c = s->cfg[layout];
  *mode = c.set ? c.mode : s->mode;
  *unroll = c.set ? c.unroll : s->unroll;
  *stage = c.set ? c.stage : s->stage;
  return ok();
}

int mickey_tune(mickey_streams *s, uint64_t n_bits, int layout, mickey_tune_result *results,
                int max_results, int *n_results) {
  if (!s || n_bits == 0) return fail(MICKEY_E_ARG, "handle must not be NULL, n_bits > 0");
  if (!layout_ok(layout)) return fail(MICKEY_E_LAYOUT, "unknown layout %d", layout);
  if ((layout == MICKEY_LAYOUT_U32 || layout == MICKEY_LAYOUT_U32_F32) && n_bits % 32)
    return fail(MICKEY_E_LAYOUT, "u32 layouts need n_bits %% 32 == 0");
  int rc = MICKEY_OK;
  if (n_bits > kMaxBitsPerCall) return fail(MICKEY_E_ARG, "n_bits per call is limited to 2^34");
  const size_t out_sz = out_bytes(s->n, n_bits, layout);
  const size_t st_sz = size_t(kStateRows) * s->Gpad * 4;
  void *out = nullptr, *saved = nullptr;
  cudaEvent_t e0 = nullptr, e1 = nullptr;
  auto cleanup = [&]() {
    if (out) cudaFree(out);
    if (saved) cudaFree(saved);
    if (e0) cudaEventDestroy(e0);
    if (e1) cudaEventDestroy(e1);
  };
  if (cudaMalloc(&out, out_sz) != cudaSuccess || cudaMalloc(&saved, st_sz) != cudaSuccess ||
      cudaEventCreate(&e0) != cudaSuccess || cudaEventCreate(&e1) != cudaSuccess) {
    cleanup();
    return fail(MICKEY_E_OOM, "tuning buffers (%zu + %zu bytes)", out_sz, st_sz);
  }
  cudaMemcpyAsync(saved, s->d_state, st_sz, cudaMemcpyDeviceToDevice, s->stream);
  const auto keep = s->cfg[layout];
  const bool row = layout != MICKEY_LAYOUT_BITSLICED_U32;
  const uint64_t W = (s->G + 31) / 32;
  int count = 0;
  // every candidate timed: (configuration, best of two)
  std::vector<std::pair<mickey_streams::LayoutCfg, float>> timed;
  for (int mode : {MICKEY_MODE_AUTO, MICKEY_MODE_GRID, MICKEY_MODE_PERSISTENT,
                   MICKEY_MODE_PERSISTENT2}) {
    if (mode == MICKEY_MODE_PERSISTENT2 && !use_persistent(s, mode)) continue;
    if (mode == MICKEY_MODE_AUTO && !use_quarters(s)) continue;   // the same as PERSISTENT
    // output tile: direct row stores, or rows staged this many tiles deep
    // (the depths the mode's kernels are compiled for)
    std::vector<int> stages{mode == MICKEY_MODE_AUTO ? 1 : 0};
    if (row && mode != MICKEY_MODE_AUTO) {
      const std::vector<int> depths = mode == MICKEY_MODE_GRID      ? std::vector<int>{2, 4}
                                      : mode == MICKEY_MODE_PERSISTENT ? std::vector<int>{2, 4, 8}
                                                                    : std::vector<int>{4};
      for (int d : depths)
        if (n_bits % (32 * uint64_t(d)) == 0) stages.push_back(d);
    }
    for (int unroll : kUnrolls) {
      if (mode == MICKEY_MODE_AUTO && unroll != 4) continue;      // its own launches have no choice
      for (int stage : stages) {
        auto &c = s->cfg[layout];
        c.set = true;
        c.mode = mode;
        c.unroll = unroll;
        c.stage = stage;
        float ms = 1e30f;
        for (int rep = 0; rep < 2 && rc == MICKEY_OK; ++rep) {
          cudaMemcpyAsync(s->d_state, saved, st_sz, cudaMemcpyDeviceToDevice, s->stream);
          cudaEventRecord(e0, s->stream);
          rc = launch_generate(s, n_bits, out, layout);
          cudaEventRecord(e1, s->stream);
          if (rc == MICKEY_OK && cudaEventSynchronize(e1) == cudaSuccess) {
            float t = 0.f;
            cudaEventElapsedTime(&t, e0, e1);
            ms = t < ms ? t : ms;
          }
        }
        if (rc != MICKEY_OK) break;
        if (results && count < max_results) results[count] = {mode, unroll, stage, ms};
        ++count;
        timed.push_back({c, ms});
      }
    }
  }
  // The fastest, except that among candidates within 1 % of it (timing
  // noise: the launch is logic-bound, not memory-bound) the deepest row
  // staging wins: rows written as whole 32-byte sectors need no partial
  // sector merges (with 16-byte chunks DRAM moved 6.1 GB per 2 GiB launch
  // of the plain workload, against 2.3 GB with 32-byte chunks, at the same
  // speed).
  float best_ms = 1e30f;
  for (const auto &t : timed) best_ms = std::min(best_ms, t.second);
  auto depth = [](const mickey_streams::LayoutCfg &c) {
    return c.stage == 1 ? (c.mode == MICKEY_MODE_GRID || c.mode == MICKEY_MODE_PERSISTENT2 ? 4 : 8)
                        : c.stage;
  };
  mickey_streams::LayoutCfg best = keep;
  float chosen = 1e30f;
  for (const auto &t : timed) {
    if (t.second > best_ms * 1.01f) continue;
    if (chosen == 1e30f || depth(t.first) > depth(best) ||
        (depth(t.first) == depth(best) && t.second < chosen)) {
      best = t.first;
      chosen = t.second;
    }
  }
  cudaMemcpyAsync(s->d_state, saved, st_sz, cudaMemcpyDeviceToDevice, s->stream);
  cudaError_t e = cudaStreamSynchronize(s->stream);
  cleanup();
  if (rc != MICKEY_OK) {
    s->cfg[layout] = keep;
    return rc;
  }
  if (e != cudaSuccess) return cuda_fail(e, "tune sync");
  s->cfg[layout] = best;
  s->cfg[layout].set = true;
  if (n_results) *n_results = count;
  return ok();
}

void mickey_free(mickey_streams *s) { release(s); }

int mickey_last_error(void) { return t_err; }
const char *mickey_last_error_message(void) { return t_msg; }

const char *mickey_error_string(int code) {
  switch (code) {
    case MICKEY_OK: return "ok";
    case MICKEY_E_ARG: return "invalid argument";
    case MICKEY_E_IVLEN: return "IV length above 80 bits";
    case MICKEY_E_LIMIT: return "more than 2^40 keystream bits for one key/IV";
    case MICKEY_E_LAYOUT: return "invalid layout for this request";
    case MICKEY_E_OOM: return "out of memory";
    case MICKEY_E_CUDA: return "CUDA error";
    case MICKEY_E_TIMEOUT: return "device-side wait timed out";
    case MICKEY_E_STATE: return "handle not usable for this call";
    default: return "unknown error";
  }
}

void mickey_tables(uint32_t masks[5][4]) {
  memset(masks, 0, sizeof(uint32_t) * 20);
  static_for<0, kReg>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    constexpr uint32_t bit = 1u << (i % 32);
    if constexpr (rtap(i)) masks[0][i / 32] |= bit;
    if constexpr (comp0(i)) masks[1][i / 32] |= bit;
    if constexpr (comp1(i)) masks[2][i / 32] |= bit;
    if constexpr (fb0(i)) masks[3][i / 32] |= bit;
    if constexpr (fb1(i)) masks[4][i / 32] |= bit;
  });
}

int mickey_ops_per_clock(int mixing) {
  constexpr int keystream = ops_per_clock(false), init = ops_per_clock(true);
  return mixing ? init : keystream;
}

const char *mickey_version(void) { return "mickey-gb300 0.1 (sm_103a)"; }

}  // extern "C"
