"""Loading with a thread per group on small handles, which load with a thread per
instance unless their mode is set, and the rows that four warps per warp-group
stage over several blocks."""
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


def _at(arr, offset, dtype=torch.uint8):
    """arr's bytes on the device, `offset` bytes behind a 16-byte boundary."""
    raw = np.frombuffer(np.ascontiguousarray(arr).tobytes(), np.uint8)
    buf = torch.zeros(raw.size + 64, dtype=torch.uint8, device="cuda")
    buf[offset:offset + raw.size] = torch.from_numpy(raw.copy()).cuda()
    return buf[offset:offset + raw.size].view(dtype)


# 16-byte loads and through shared memory, with the IV clocks uniform (whole and
# not a multiple of four, none), absent lengths, and mixed inside groups
@pytest.mark.parametrize("mode", ["grid", "persistent"])
@pytest.mark.parametrize("kind", ["none", "0", "37", "48", "80", "mixed"])
@pytest.mark.parametrize("n", [32 * 300, 32 * 300 + 7])
def test_thread_per_group_loading(monkeypatch, n, kind, mode):
    from paper_1909_04750_gb300.streams import Streams
    monkeypatch.setenv("MICKEY_MODE", mode)
    s = workloads.plain_scale(n)
    if kind == "mixed":
        s.iv_lens[:] = np.random.default_rng(n).integers(0, 81, n)
    elif kind != "none":
        s.iv_lens[:] = int(kind)
    want = oracle.batch_bytes(s.keys, s.ivs, s.iv_lens, 96, threads=THREADS)
    for key_off, iv_off, len_off in ((0, 0, 0), (1, 0, 0), (0, 6, 4), (3, 5, 8)):
        lens = None if kind == "none" else _at(s.iv_lens.astype(np.int32), len_off, torch.int32)
        st = Streams(_at(s.keys, key_off).view(n, 10), _at(s.ivs, iv_off).view(n, 10), lens)
        assert np.array_equal(st.generate(96, "bytes").cpu().numpy(), want)
        st.sync()


# one, two and three warp-groups per SM, the last one not full; two, three, four
# and eight blocks of eight tiles per row, and rows that are not staged between them
@pytest.mark.parametrize("groups_per_sm", [20, 40, 90])
def test_staged_rows_of_several_blocks(monkeypatch, groups_per_sm):
    from paper_1909_04750_gb300.streams import Streams
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = workloads.plain_scale(groups_per_sm * sms * 32 - 5)
    keys, ivs = torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda()
    auto = Streams(keys, ivs)
    monkeypatch.setenv("MICKEY_MODE", "grid")
    grid = Streams(keys, ivs)
    for n_bits, layout in ((512, "bytes"), (768, "u32"), (1024, "u32_f32"), (288, "bytes"),
                           (2048, "bytes"), (512, "u32_f32")):
        assert torch.equal(auto.generate(n_bits, layout), grid.generate(n_bits, layout))
