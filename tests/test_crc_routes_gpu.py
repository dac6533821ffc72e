"""CRC-8 on each side of the lines between its kernels (a table step per byte, tiles
of 2048 messages, a warp per 32 messages), at sizes where each loops over
its grid, and the choice between them."""
import numpy as np
import pytest

from paper_1909_04750_gb300 import _native as N

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1909_04750_gb300 import build as B
    B.build()
    N.lib()


def _check(n, length, poly, init, xorout, offset=0, seed=1):
    """Every 64th message, the first and last 64 and those around the tiles' and
    the grids' ends against the oracle."""
    from oracle import lfsr as ol
    from paper_1909_04750_gb300.lfsr import crc8
    gen = torch.Generator(device="cuda").manual_seed(seed)
    buf = torch.randint(0, 256, (n * length + 16,), dtype=torch.uint8, device="cuda", generator=gen)
    data = buf[offset:offset + n * length].view(n, length)
    got = crc8(data, poly, init, xorout)
    tiles = np.arange(2048, n, 2048)
    idx = np.unique(np.concatenate([np.arange(0, n, 64), np.arange(min(n, 64)),
                                    np.arange(max(0, n - 64), n), tiles - 1, tiles]))
    dev = torch.from_numpy(idx).cuda()
    rows = data[dev].cpu().numpy()
    assert np.array_equal(got[dev].cpu().numpy(), ol.crc8_batch(rows, poly, init, xorout))


POLYS = [(0x1D, 0xFF, 0xFF), (0x8D, 0xA5, 0x3C)]     # with a kernel of its own, and without


# aligned lengths of the tiles, a whole and a half last pass, a last tile that is
# not full; one wave and more
@pytest.mark.parametrize("poly,init,xorout", POLYS)
@pytest.mark.parametrize("length", [32, 48, 64, 80, 96, 112, 128, 144, 160, 176, 192])
@pytest.mark.parametrize("n", [(1 << 19) + 37, (1 << 20) + 2049])
def test_tiles(n, length, poly, init, xorout):
    _check(n, length, poly, init, xorout)


# tiles for a polynomial without a kernel only
@pytest.mark.parametrize("length", [208, 256, 272, 320])
def test_longer_tiles(length):
    _check((1 << 20) + 5, length, 0x8D, 0, 0)


# the table and the units looping over their grids
@pytest.mark.parametrize("poly,init,xorout", POLYS)
@pytest.mark.parametrize("length,offset", [(60, 0), (16, 0), (112, 1), (113, 0), (127, 3), (500, 0),
                                           (1000, 8)])
def test_grid_loops(length, offset, poly, init, xorout):
    _check((1 << 20) + 33, length, poly, init, xorout, offset)


# the lines between the kernels, few messages and the numbers from which tiles win
@pytest.mark.parametrize("n", [1, 2049, 114_687, 114_688, 179_999, 180_000, 229_999, 230_000])
@pytest.mark.parametrize("length", [48, 64, 96, 111, 112, 113, 128, 144, 160, 176])
def test_lines(n, length):
    for poly, init, xorout in POLYS:
        _check(n, length, poly, init, xorout)


def _us(n, length, poly):
    from paper_1909_04750_gb300.lfsr import crc8
    data = torch.zeros((n, length), dtype=torch.uint8, device="cuda")
    out = torch.empty(n, dtype=torch.uint8, device="cuda")
    best = 1e9
    for _ in range(6):
        e0, e1 = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        e0.record()
        crc8(data, poly, 0, 0, out=out)
        e1.record()
        e1.synchronize()
        best = min(best, e0.elapsed_time(e1))
    return 1e3 * best


# a little longer messages do not cost half as much again: lengths next to a line
# that lay wrong for a polynomial without a kernel of its own, or for the number
# of messages (229 us against 118, 58 against 29)
@pytest.mark.parametrize("n,short,long,poly", [(1 << 20, 160, 192, 0x8D), (1 << 19, 160, 176, 0x8D),
                                               (350_000, 56, 64, 0x1D)])
def test_no_step_in_time_at_a_line(n, short, long, poly):
    a, b = _us(n, short, poly), _us(n, long, poly)
    assert b < 1.5 * a, (a, b)
