"""The arrangement a new batch plan takes, and a batch large enough to load its
keys through the permutation with a thread per group."""
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


def test_thread_items_where_equal_lengths_fill_every_warp():
    # 1024 streams for each of the 8 warps per SM: 12.8 ms, all split 13.2
    from paper_1909_04750_gb300.batch import Batch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    full = 8 * sms * 1024
    assert Batch(np.full(full, 2048, np.uint64)).get_config()["split_groups"] == 0
    for n, lo in ((full // 2, 2048), (full * 5 // 4, 2048), (full, 256)):
        nb = np.linspace(lo, 2048, n).astype(np.uint64)
        cfg = Batch(nb).get_config()
        assert cfg["split_groups"] == (n + 31) // 32 and cfg["split_clocks"] == 1


@pytest.mark.parametrize("split", [True, False])
def test_batch_above_the_packed_loading_sampled(split):
    # IV lengths 0..80 mixed, lengths that sort into another order than the
    # caller's; 300,000 streams are 62 groups per SM
    from paper_1909_04750_gb300.batch import Batch
    n = 300_000
    s = workloads.plain_scale(n)
    rng = np.random.default_rng(6)
    s.iv_lens[:] = rng.integers(0, 81, n)
    nb = rng.integers(0, 1500, n).astype(np.uint64)
    b = Batch(nb, s.iv_lens)
    assert b.get_config()["split_groups"] == (n + 31) // 32
    if not split:
        b.set_config(4, 2, 0)
    out = b.run(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda())
    b.sync()
    idx = np.unique(np.concatenate([rng.integers(0, n, 4000), np.argsort(nb)[:64],
                                    np.argsort(nb)[-64:], np.arange(64), np.arange(n - 64, n)]))
    sub = s.subset(idx)
    want = oracle.batch_bytes(sub.keys, sub.ivs, sub.iv_lens, nb[idx], threads=THREADS)
    host = out.cpu().numpy()
    for k, i in enumerate(idx):
        o, c = int(b.offsets[i]), (int(nb[i]) + 7) // 8
        assert np.array_equal(host[o:o + c], np.asarray(want[k])[:c]), i


def test_a_reported_configuration_can_be_set_again():
    # 40 of 80 streams empty: a whole group has nothing to clock
    from paper_1909_04750_gb300.batch import Batch
    s = workloads.plain_scale(80)
    nb = np.where(np.arange(80) % 2, 4096, 0).astype(np.uint64)
    b = Batch(nb, s.iv_lens)
    cfg = b.get_config()
    assert cfg["split_groups"] == 3
    b.set_config(cfg["unroll"], cfg["blocks_per_sm"], cfg["split_clocks"], cfg["split_mode"])
    assert b.get_config() == cfg
    out = b.run(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda())
    b.sync()
    want = oracle.batch_bytes(s.keys, s.ivs, s.iv_lens, nb, threads=THREADS)
    for got, row in zip(b.rows(out), want):
        assert np.array_equal(got, np.asarray(row)[:got.size])


def test_streams_past_the_thread_items_tile_count():
    # 2^37 bits are 2^32 tiles; planned only, such a stream runs for an hour
    from paper_1909_04750_gb300.batch import Batch
    nb = np.full(2000, 100, np.uint64)
    nb[7] = 1 << 37
    b = Batch(nb)
    for cfg, split in (((4, 2, 0), 1), ((4, 2, 1 << 39), 1), ((4, 1, 64), 63), ((4, 1, 1), 63)):
        b.set_config(*cfg)
        assert b.get_config()["split_groups"] == split
    nb[7] -= 1
    b = Batch(nb)
    b.set_config(4, 2, 0)
    assert b.get_config()["split_groups"] == 0
