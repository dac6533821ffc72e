"""Launches whose segments hand states on: a captured call that is replayed,
and waits that run out."""
import numpy as np
import pytest

import oracle
from paper_1909_04750_gb300 import _native as N
from paper_1909_04750_gb300 import workloads

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1909_04750_gb300 import build as B
    B.build()
    N.lib()


def _streams(s):
    from paper_1909_04750_gb300.streams import Streams
    return Streams(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda(),
                   torch.from_numpy(s.iv_lens.astype(np.int32)).cuda())


# tails first: every segment waits for the one before it, so a flag left by the
# replay before would be taken for the hand-off of this one
@pytest.mark.parametrize("tails_first", ["0", "1"])
@pytest.mark.parametrize("mode", ["persistent", "persistent2"])
@pytest.mark.parametrize("layout,n_bits", [("bytes", 512), ("bitsliced", 333)])
def test_keystream_hand_offs_in_a_replayed_graph(monkeypatch, layout, n_bits, mode, tails_first):
    s = workloads.plain_scale(9 * 1024 + 70)
    plain = _streams(s)
    monkeypatch.setenv("MICKEY_MODE", mode)
    monkeypatch.setenv("MICKEY_PERSIST_BLOCKS", "1")
    monkeypatch.setenv("MICKEY_TEST_TAILS_FIRST", tails_first)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        st = _streams(s)
        out = st.generate(n_bits, layout)
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            st.generate(n_bits, layout, out=out)
    plain.generate(n_bits, layout)
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, plain.generate(n_bits, layout))
    st.sync()


# a stream of 2^17 bits among short ones, in the first warp-group, between
# others and in the last: 44 ms of clocks, where a tail may wait for about 1 ms
@pytest.mark.parametrize("layout", ["bytes", "bitsliced"])
@pytest.mark.parametrize("long", [[5], [2500], [6 * 1024 - 10], [1030, 3077, 5200]])
def test_ragged_hand_offs_beside_a_long_stream(monkeypatch, layout, long):
    n = 6 * 1024 - 9
    s = workloads.plain_scale(n)
    nb = np.random.default_rng(8).integers(0, 400, n).astype(np.uint64)
    nb[long] = 1 << 17
    plain = _streams(s)                              # few groups: a thread per instance
    monkeypatch.setenv("MICKEY_MODE", "persistent")
    monkeypatch.setenv("MICKEY_PERSIST_BLOCKS", "1")
    monkeypatch.setenv("MICKEY_SPIN_LIMIT", "2000")
    st = _streams(s)
    for _ in range(2):
        got, want = (h.generate_ragged(nb, layout)[0] for h in (st, plain))
        st.sync()
        assert torch.equal(got, want)
    assert all(np.array_equal(a, b) for a, b in zip(st.export_state(), plain.export_state()))


@pytest.mark.parametrize("tails_first", ["0", "1"])
def test_ragged_hand_offs_waited_for(monkeypatch, tails_first):
    # 7 warp-groups on 4 clock warps, each tail waiting for its head
    n = 7 * 1024 - 100
    s = workloads.plain_scale(n)
    nb = np.random.default_rng(9).integers(0, 3000, n).astype(np.uint64)
    plain = _streams(s)
    monkeypatch.setenv("MICKEY_MODE", "persistent")
    monkeypatch.setenv("MICKEY_PERSIST_BLOCKS", "1")
    monkeypatch.setenv("MICKEY_TEST_TAILS_FIRST", tails_first)
    st = _streams(s)
    for _ in range(2):
        got, want = (h.generate_ragged(nb, "bytes")[0] for h in (st, plain))
        st.sync()
        assert torch.equal(got, want)


def test_ragged_wait_runs_out_without_a_fault(monkeypatch):
    # no head publishes the value the tails wait for: the call returns, the sync
    # reports it, and the context goes on working
    n = 7 * 1024 - 100
    s = workloads.plain_scale(n)
    nb = np.random.default_rng(10).integers(0, 3000, n).astype(np.uint64)
    want = _streams(s).generate_ragged(nb, "bytes")[0]
    monkeypatch.setenv("MICKEY_MODE", "persistent")
    monkeypatch.setenv("MICKEY_PERSIST_BLOCKS", "1")
    monkeypatch.setenv("MICKEY_SPIN_LIMIT", "2000")
    monkeypatch.setenv("MICKEY_TEST_UNPUBLISHED", "1")
    st = _streams(s)
    st.generate_ragged(nb, "bytes")
    with pytest.raises(N.MickeyError) as e:
        st.sync()
    assert e.value.code == N.E_TIMEOUT
    monkeypatch.delenv("MICKEY_TEST_UNPUBLISHED")
    ok = _streams(s)
    got = ok.generate_ragged(nb, "bytes")[0]
    ok.sync()
    assert torch.equal(got, want)
