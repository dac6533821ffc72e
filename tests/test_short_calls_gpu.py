"""Calls of a few clocks, which move states more than they clock, on both sides of
the lines between the launches, and rows staged in blocks that a segment of the
work line could cut."""
import os

import numpy as np
import pytest

import oracle
from paper_1909_04750_gb300 import _native as N
from paper_1909_04750_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

THREADS = os.cpu_count() or 4


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1909_04750_gb300 import build as B
    B.build()
    N.lib()


def _sms():
    return torch.cuda.get_device_properties(0).multi_processor_count


def _sample(n, k=600):
    return np.unique(np.concatenate([np.random.default_rng(n).integers(0, n, k), np.arange(40),
                                     np.arange(max(0, n - 40), n)]))


# Grain: groups per SM at the lines of short rows (32, 64), of bitsliced calls
# whose line moves with the clocks (30, 50), of the loading (102), and above all;
# every kind of row on and off the grid, at an aligned output and an odd one
@pytest.mark.parametrize("per_sm,extra", [(30, 0), (32, 0), (32, 1), (50, 0), (64, 0), (64, 1),
                                          (102, 0), (102, 1), (140, 3)])
def test_grain_short_calls(per_sm, extra):
    from oracle import grain as og
    from paper_1909_04750_gb300.grain import GrainStreams
    n = (per_sm * _sms() + extra) * 32 - 5
    s = workloads.grain_streams(n, seed=41)
    idx = _sample(n)
    calls = [1, 8, 9, 16, 24, 32, 33, 64, 128, 256]
    bits = np.unpackbits(og.batch_bytes(s.keys[idx], s.ivs[idx], 2 * sum(calls), threads=THREADS),
                         axis=1, bitorder="little")
    dev = torch.from_numpy(idx).cuda()
    for layout in ("bytes", "bitsliced"):
        st = GrainStreams(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda())
        at = 0
        for odd in (0, 1):
            for b in calls:
                want = bits[:, at:at + b]
                at += b
                if layout == "bytes":
                    row = (b + 7) // 8
                    buf = torch.full((n * row + 16,), 0xA5, dtype=torch.uint8, device="cuda")
                    st.generate(b, layout, out=buf[odd:])
                    got = buf[odd:odd + n * row].view(n, row)[dev].cpu().numpy()
                    assert np.array_equal(got, np.packbits(want, axis=1, bitorder="little")), b
                    assert (buf[odd + n * row:] == 0xA5).all() and (buf[:odd] == 0xA5).all()
                else:
                    words = st.generate(b, layout).view((n + 31) // 32, b)
                    got = words[(dev // 32)].cpu().numpy().view(np.uint32)
                    got = (got >> (idx % 32).astype(np.uint32)[:, None]) & 1
                    assert np.array_equal(got, want), b
        st.sync()


# more warp-groups than clock warps, by one and by a part: blocks of eight tiles
# whole in a segment, and rows of other numbers of tiles
@pytest.mark.parametrize("groups", [1, 300])
@pytest.mark.parametrize("n_bits", [128, 250, 256, 384, 512, 768, 1024, 2304])
def test_grain_segments_end_between_blocks(groups, n_bits):
    from oracle import grain as og
    from paper_1909_04750_gb300.grain import GrainStreams
    n = (4 * _sms() * 32 + groups) * 32 - 7
    s = workloads.grain_streams(n, seed=42)
    idx = _sample(n)
    st = GrainStreams(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda())
    got = [st.generate(n_bits, "bytes")[torch.from_numpy(idx).cuda()].cpu().numpy() for _ in range(2)]
    st.sync()
    bits = np.unpackbits(og.batch_bytes(s.keys[idx], s.ivs[idx], 2 * n_bits, threads=THREADS), axis=1,
                         bitorder="little")
    for k in range(2):
        want = np.packbits(bits[:, k * n_bits:(k + 1) * n_bits], axis=1, bitorder="little")
        assert np.array_equal(got[k], want)


@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("per_sm", [13, 52])
def test_mickey_short_calls_agree_with_a_thread_per_group(monkeypatch, per_sm, extra):
    from paper_1909_04750_gb300.streams import Streams
    n = (per_sm * _sms() + extra) * 32 - 5
    s = workloads.plain_scale(n)
    keys, ivs = torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda()
    auto = Streams(keys, ivs)
    monkeypatch.setenv("MICKEY_MODE", "grid")
    grid = Streams(keys, ivs)
    for b in (1, 8, 9, 3):
        for layout in ("bytes", "bitsliced"):
            assert torch.equal(auto.generate(b, layout), grid.generate(b, layout))
    idx = _sample(n)
    want = oracle.batch_bytes(s.keys[idx], s.ivs[idx], s.iv_lens[idx], 42 + 8, threads=THREADS)
    got = auto.generate(8, "bytes")[torch.from_numpy(idx).cuda()].cpu().numpy()
    assert np.array_equal(np.packbits(np.unpackbits(want, axis=1)[:, 42:50], axis=1), got)


def test_grain_one_byte_costs_about_what_the_paired_launch_costs():
    # 2^21 instances x 24 bits bitsliced take 36 us, rows of a byte 40; 105 when
    # those took the launch of a thread per instance
    from paper_1909_04750_gb300.grain import GrainStreams
    n = 1 << 21
    k, v = (torch.randint(0, 256, (n, w), dtype=torch.uint8, device="cuda") for w in (10, 8))
    st = GrainStreams(k, v)
    us = {}
    for n_bits, layout in ((8, "bytes"), (24, "bitsliced")):
        out, best = st.generate(n_bits, layout), 1e9
        for _ in range(6):
            e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            e0.record()
            st.generate(n_bits, layout, out=out)
            e1.record()
            e1.synchronize()
            best = min(best, 1e3 * e0.elapsed_time(e1))
        us[layout] = best
    assert us["bytes"] < 2 * us["bitsliced"], us


# above the packed launch's line: up to 16 clocks in a kernel of their own, the
# paired launch from 17; the lanes past the last instance stay zero
@pytest.mark.parametrize("n", [60 * 152 * 32 + 11, 700_003])
def test_grain_few_bitsliced_clocks(n):
    from oracle import grain as og
    from paper_1909_04750_gb300.grain import GrainStreams
    s = workloads.grain_streams(n, seed=43)
    idx = _sample(n)
    st = GrainStreams(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda())
    calls = [16, 1, 17, 15, 2, 32, 7]
    bits = np.unpackbits(og.batch_bytes(s.keys[idx], s.ivs[idx], sum(calls), threads=THREADS), axis=1,
                         bitorder="little")
    at = 0
    for b in calls:
        words = st.generate(b, "bitsliced").view((n + 31) // 32, b).cpu().numpy().view(np.uint32)
        got = (words[idx // 32] >> (idx % 32).astype(np.uint32)[:, None]) & 1
        assert np.array_equal(got, bits[:, at:at + b])
        assert not (words[-1] >> np.uint32(n % 32)).any()
        at += b
    st.sync()
