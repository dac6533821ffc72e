"""The performance cases: the calls a user of this framework makes, with the
sizes they are made at.

A case is a dict of plain values.  `listed()` gives the fixed ones, `draw(rng)`
one more of the same ranges, `prepare(case, seed)` what a program has in hand
before the call (inputs on the device, the handle or plan it keeps),
`run(state)` one pass through the public entry points and its outputs,
`work(case)` the bytes and 32-bit logic operations of a pass, and
`exact(case, seed)` the outputs computed with plain torch where that is quick.

Every output is whole numbers or bytes (the u32_f32 layout returns the float
words as their bits), so outputs are compared for equality.
"""
import numpy as np
import torch

from paper_1909_04750_gb300.batch import Batch
from paper_1909_04750_gb300.grain import GrainStreams
from paper_1909_04750_gb300.lfsr import crc8, lfsr_generate
from paper_1909_04750_gb300.streams import Streams, output_shape

# Logic operations (three-input) per clock of a 32-instance group, as the
# library's mickey_ops_per_clock / grain_ops_per_clock count them.
MICKEY_OPS, MICKEY_INIT_OPS, MICKEY_INIT_CLOCKS = 327, 329, 180
GRAIN_OPS, GRAIN_INIT_OPS, GRAIN_INIT_CLOCKS = 36, 37, 160

CRC_POLYS = (0x07, 0x1D, 0x2F, 0x31, 0x9B, 0xD5)


def listed():
    return [
        # One group of keystreams for a short message each: the smallest call,
        # all latency (the smoke test's shape).
        dict(name="streams_32x2048", kind="streams", n=32, bits=2048, layout="bytes", iv=80),
        # A thousand sessions with IVs of mixed length and a length that is no
        # whole number of bytes, words or tiles.
        dict(name="streams_1000x10001_iv", kind="streams", n=1000, bits=10001, layout="bytes",
             iv=0),
        # A medium set of generators drawing 32-bit words (2^16 instances).
        dict(name="streams_64k_u32", kind="streams", n=1 << 16, bits=1 << 14, layout="u32", iv=80),
        # A quarter of a million generators whose bits stay bitsliced; the last
        # group is not full.
        dict(name="streams_250k_bitsliced", kind="streams", n=250_001, bits=4096,
             layout="bitsliced", iv=80),
        # The plain workload at scale: 2^20 instances, 2 KiB each, row-major bytes.
        dict(name="streams_1m_bytes", kind="streams", n=1 << 20, bits=1 << 14, layout="bytes",
             iv=80),
        # Random numbers as u32 and FP32 at once, many instances, short rows.
        dict(name="streams_4m_u32_f32", kind="streams", n=1 << 22, bits=1 << 12,
             layout="u32_f32", iv=80),
        # A million resident streams each continued by its own length.
        dict(name="ragged_1m", kind="ragged", n=1 << 20, lo=1 << 13, hi=1 << 14, layout="bytes"),
        # A batch of independent streams of very uneven length, each with its own
        # IV length, as the plan is made (no tuning run).
        dict(name="batch_20k", kind="batch", n=20_000, lo_log2=10, hi_log2=18),
        # Grain at the plain workload's size, row-major bytes.
        dict(name="grain_1m_bytes", kind="grain", n=1 << 20, bits=1 << 14, layout="bytes"),
        # A few thousand Grain streams, bitsliced, an odd count and length.
        dict(name="grain_4k_bitsliced", kind="grain", n=4_001, bits=20_002, layout="bitsliced"),
        # CRC-8 of a million 1 KiB messages (preset and final XOR of SAE J1850).
        dict(name="crc8_1m_1k", kind="crc8", n=1 << 20, len=1024, poly=0x1D, init=0xFF,
             xorout=0xFF),
        # A million degree-64 LFSRs with four taps, 4096 bits each.
        dict(name="lfsr_1m_d64", kind="lfsr", n=1 << 20, degree=64, taps=0b11011, bits=4096),
    ]


def _log(rng, lo, hi):
    return int(round(2.0 ** rng.uniform(np.log2(lo), np.log2(hi))))


def draw(rng):
    kind = rng.choice(["streams", "streams", "streams", "streams", "ragged", "batch", "grain",
                       "grain", "crc8", "lfsr"])
    if kind == "streams":
        layout = rng.choice(["bytes", "bytes", "bitsliced", "u32", "u32_f32"])
        n = _log(rng, 32, 1 << 20)
        bits = _log(rng, 256, min(1 << 16, (1 << 33) // n))
        if layout in ("u32", "u32_f32"):
            bits = max(256, bits // 32 * 32)
        return dict(kind=kind, n=n, bits=bits, layout=layout, iv=rng.choice([80, 80, 64, 0]))
    if kind == "ragged":
        n = _log(rng, 1000, 1 << 20)
        hi = _log(rng, 1 << 10, min(1 << 15, (1 << 34) // n))
        layout = rng.choice(["bytes", "bytes", "u32", "bitsliced"])
        return dict(kind=kind, n=n, lo=rng.choice([hi // 2, hi // 8, 0]), hi=hi, layout=layout)
    if kind == "batch":
        return dict(kind=kind, n=_log(rng, 1000, 40_000), lo_log2=10,
                    hi_log2=rng.choice([14, 15, 16, 17]))
    if kind == "grain":
        n = _log(rng, 32, 1 << 20)
        bits = _log(rng, 256, min(1 << 16, (1 << 34) // n))
        return dict(kind=kind, n=n, bits=bits, layout=rng.choice(["bytes", "bitsliced"]))
    if kind == "crc8":
        n = _log(rng, 1000, 1 << 20)
        length = _log(rng, 8, min(4096, (1 << 30) // n))
        if rng.random() < 0.5:
            length = max(16, length // 16 * 16)
        poly = rng.choice(CRC_POLYS) if rng.random() < 0.7 else rng.randrange(1, 256)
        return dict(kind=kind, n=n, len=length, poly=poly, init=rng.choice([0, 0xFF]),
                    xorout=rng.choice([0, 0xFF]))
    degree = rng.choice([16, 24, 31, 32, 48, 63, 64])
    taps = 1
    for _ in range(rng.choice([1, 3, 3, 5, 24])):
        taps |= 1 << rng.randrange(1, degree)
    n = _log(rng, 1000, 1 << 20)
    return dict(kind="lfsr", n=n, degree=degree, taps=taps,
                bits=_log(rng, 128, min(1 << 15, (1 << 32) // n)))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) * 1_000_003 + 17)


def _bytes(gen, n, width):
    return torch.randint(0, 256, (n, width), dtype=torch.uint8, device="cuda", generator=gen)


def _seeds(case, gen):
    """Seeds in [1, 2^degree)."""
    top = (1 << min(case["degree"], 62)) - 1
    return torch.randint(1, top, (case["n"],), dtype=torch.int64, device="cuda", generator=gen)


def prepare(case, seed):
    gen, kind, n = _gen(seed), case["kind"], case["n"]
    if kind == "crc8":
        return dict(case=case, data=_bytes(gen, n, case["len"]),
                    out=torch.empty(n, dtype=torch.uint8, device="cuda"))
    if kind == "lfsr":
        return dict(case=case, seeds=_seeds(case, gen),
                    out=torch.empty((case["bits"], (n + 31) // 32), dtype=torch.int32,
                                    device="cuda"))
    if kind == "grain":
        keys, ivs = _bytes(gen, n, 10), _bytes(gen, n, 8)
        shape, dtype = output_shape(n, case["bits"], case["layout"])
        return dict(case=case, keys=keys, ivs=ivs, handle=GrainStreams(keys, ivs),
                    out=torch.empty(shape, dtype=dtype, device="cuda"))
    keys, ivs = _bytes(gen, n, 10), _bytes(gen, n, 10)
    if kind == "streams":
        lens = None
        if case["iv"] == 0:      # mixed: 0, 16, ..., 80 bits
            lens = 16 * torch.randint(0, 6, (n,), dtype=torch.int32, device="cuda", generator=gen)
        elif case["iv"] != 80:
            lens = torch.full((n,), case["iv"], dtype=torch.int32, device="cuda")
        shape, dtype = output_shape(n, case["bits"], case["layout"])
        return dict(case=case, keys=keys, ivs=ivs, lens=lens, handle=Streams(keys, ivs, lens),
                    out=torch.empty(shape, dtype=dtype, device="cuda"))
    # the lengths of a ragged or batch case are the same set for every seed, in
    # another order, so that the outputs have one size
    base, order = np.random.default_rng(n), np.random.default_rng(int(seed))
    if kind == "ragged":
        step = 32 if case["layout"] == "u32" else 1
        lengths = base.integers(case["lo"] // step, case["hi"] // step + 1, n).astype(np.uint64)
        lengths = order.permutation(lengths * np.uint64(step))
        if case["layout"] == "bitsliced":     # at most the longest length for every group
            total = 4 * ((n + 31) // 32) * case["hi"]
        else:
            total = int(((lengths + np.uint64(7)) // np.uint64(8)).sum())
        return dict(case=case, keys=keys, ivs=ivs, lengths=lengths, handle=Streams(keys, ivs),
                    out=torch.zeros(max(total, 16), dtype=torch.uint8, device="cuda"))
    # batch: lengths log-uniform, whole bytes; IVs of 0, 16, ..., 80 bits
    bits = 2.0 ** order.permutation(base.uniform(case["lo_log2"], case["hi_log2"], n))
    plan = Batch(bits.astype(np.uint64) // np.uint64(8) * np.uint64(8),
                 (16 * order.integers(0, 6, n)).astype(np.uint32))
    return dict(case=case, keys=keys, ivs=ivs, plan=plan,
                out=torch.zeros(plan.output_bytes, dtype=torch.uint8, device="cuda"))


def run(state):
    case, kind = state["case"], state["case"]["kind"]
    if kind == "crc8":
        return crc8(state["data"], case["poly"], case["init"], case["xorout"], out=state["out"])
    if kind == "lfsr":
        return lfsr_generate(state["seeds"], case["degree"], case["taps"], case["bits"],
                             out=state["out"])
    if kind == "batch":
        return state["plan"].run(state["keys"], state["ivs"], out=state["out"])
    h = state["handle"]
    if kind == "grain":
        h.reset(state["keys"], state["ivs"])
        return h.generate(case["bits"], case["layout"], out=state["out"])
    if kind == "ragged":
        h.reset(state["keys"], state["ivs"])
        return h.generate_ragged(state["lengths"], case["layout"], out=state["out"])[0]
    h.reset(state["keys"], state["ivs"], state["lens"])
    return h.generate(case["bits"], case["layout"], out=state["out"])


def work(case):
    kind, n = case["kind"], case["n"]
    G = (n + 31) // 32
    if kind == "crc8":
        return dict(bytes=n * (case["len"] + 1), flops=0)
    if kind == "lfsr":
        ops = (bin(case["taps"]).count("1") // 2) * G * case["bits"]
        return dict(bytes=8 * n + 4 * G * case["bits"], flops=ops)
    if kind == "grain":
        per = 4 * G * case["bits"] if case["layout"] == "bitsliced" else n * ((case["bits"] + 7) // 8)
        ops = G * (GRAIN_OPS * case["bits"] + GRAIN_INIT_OPS * GRAIN_INIT_CLOCKS)
        return dict(bytes=18 * n + per, flops=ops)
    if kind == "streams":
        iv = 40 if case["iv"] == 0 else case["iv"]
        per = {"bitsliced": 4 * G * case["bits"], "u32_f32": n * (case["bits"] // 4)}.get(
            case["layout"], n * ((case["bits"] + 7) // 8))
        bits = case["bits"]
    elif kind == "ragged":
        iv, bits = 80, (case["lo"] + case["hi"]) // 2
        per = n * ((bits + 7) // 8)
    else:
        lo, hi = case["lo_log2"], case["hi_log2"]
        iv, bits = 40, int((2.0 ** hi - 2.0 ** lo) / ((hi - lo) * np.log(2.0)))
        per = n * (bits // 8)
    ops = G * (MICKEY_OPS * bits + MICKEY_INIT_OPS * (MICKEY_INIT_CLOCKS + iv))
    return dict(bytes=20 * n + per, flops=ops)


def exact(case, seed):
    gen, n = _gen(seed), case["n"]
    if case["kind"] == "crc8":
        # most significant bit first, a table step per byte
        table = []
        for b in range(256):
            for _ in range(8):
                b = ((b << 1) ^ (case["poly"] if b & 0x80 else 0)) & 0xFF
            table.append(b)
        table = torch.tensor(table, dtype=torch.int64, device="cuda")
        data = _bytes(gen, n, case["len"])
        c = torch.full((n,), case["init"], dtype=torch.int64, device="cuda")
        for k in range(case["len"]):
            c = table[c ^ data[:, k].long()]
        return (c ^ case["xorout"]).to(torch.uint8)
    if case["kind"] == "lfsr":
        # s_{t+d} = XOR of s_{t+j} over the taps j, on 32-instance words
        seeds = _seeds(case, gen)
        G, d = (n + 31) // 32, case["degree"]
        x = torch.zeros(G * 32, dtype=torch.int64, device="cuda")
        x[:n] = seeds
        x = x.view(G, 32)
        lane = torch.arange(32, device="cuda")
        w = torch.zeros((case["bits"], G), dtype=torch.int32, device="cuda")
        js = [j for j in range(d) if case["taps"] >> j & 1]
        for t in range(case["bits"]):
            if t < d:
                v = (((x >> t) & 1) << lane).sum(1)
                w[t] = torch.where(v >= 1 << 31, v - (1 << 32), v).to(torch.int32)
            else:
                v = w[t - d + js[0]]
                for j in js[1:]:
                    v = v ^ w[t - d + j]
                w[t] = v
        return w
    return None   # the ciphers bit by bit in torch would take minutes
