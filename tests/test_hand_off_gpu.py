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
