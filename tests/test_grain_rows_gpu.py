"""Grain's byte rows on the 16-byte grid whose last tile is partial: staged as
whole rows are, in the paired launch of many groups."""
import os

import numpy as np
import pytest

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


def _grain(s):
    from paper_1909_04750_gb300.grain import GrainStreams
    return GrainStreams(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda())


# every last tile that fills a row of whole 16 bytes; fewer than eight tiles,
# whole blocks of eight, and a part of one behind them
@pytest.mark.parametrize("queue", ["0", "1"])
@pytest.mark.parametrize("n_bits", [121, 124, 127, 249, 250, 1020, 1021, 1407, 2046, 4092])
def test_partial_last_tile_against_the_oracle(monkeypatch, n_bits, queue):
    from oracle import grain as og
    monkeypatch.setenv("MICKEY_GRAIN_QUEUE", queue)
    s = workloads.grain_streams(2 * 1024 + 70, seed=31)
    st = _grain(s)
    got = [st.generate(n_bits, "bytes").cpu().numpy() for _ in range(2)]
    st.sync()
    bits = np.unpackbits(og.batch_bytes(s.keys, s.ivs, 2 * n_bits, threads=THREADS), axis=1,
                         bitorder="little")
    for k in range(2):
        want = np.packbits(bits[:, k * n_bits:(k + 1) * n_bits], axis=1, bitorder="little")
        assert np.array_equal(got[k], want)


def test_partial_last_tile_costs_no_more_stores():
    # 2^19 instances of 4092 and of 4096 bits write the same rows; stored word
    # by word the former took 4.4 times as long
    k, v = (torch.randint(0, 256, (1 << 19, w), dtype=torch.uint8, device="cuda") for w in (10, 8))
    from paper_1909_04750_gb300.grain import GrainStreams
    st = GrainStreams(k, v)
    out = torch.empty((1 << 19, 512), dtype=torch.uint8, device="cuda")
    ms = {}
    for n_bits in (4096, 4092, 4096, 4092):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        for _ in range(5):
            st.generate(n_bits, "bytes", out=out)
        e1.record()
        e1.synchronize()
        ms[n_bits] = e0.elapsed_time(e1)            # of the second turn
    assert ms[4092] < 2 * ms[4096], ms
