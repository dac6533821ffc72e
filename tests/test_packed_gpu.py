"""The one-thread-per-instance launches of a streams handle (keystream and
initialisation) against the oracle and against the one-thread-per-group
launches, on whose state in HBM they go on and the other way round."""
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


def _streams(s):
    from paper_1909_04750_gb300.streams import Streams
    return Streams(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda(),
                   torch.from_numpy(s.iv_lens.astype(np.int32)).cuda())


def _mixed(n):
    s = workloads.plain_scale(n)
    s.iv_lens[:] = np.random.default_rng(n).integers(0, 81, n)
    return s


# one tile less or more a bit, the 16-byte row stores (multiples of 128) and what is left of them
@pytest.mark.parametrize("n_bits", [1, 31, 32, 33, 96, 124, 128, 160, 256, 1001])
@pytest.mark.parametrize("n", [1, 31, 33, 1000])
def test_every_layout_two_calls_against_the_oracle(n, n_bits):
    s = _mixed(n)
    ref = oracle.batch_bytes(s.keys, s.ivs, s.iv_lens, n_bits + 64, threads=THREADS)
    bits = np.unpackbits(ref, axis=1)
    for layout in ("bytes", "bitsliced", "u32", "u32_f32"):
        if layout.startswith("u32") and n_bits % 32:
            continue
        st = _streams(s)
        first, second = st.generate(n_bits, layout), st.generate(64, layout)
        st.sync()
        for got, lo, hi in ((first, 0, n_bits), (second, n_bits, n_bits + 64)):
            want = np.packbits(bits[:, lo:hi], axis=1)
            a = got.cpu().numpy()
            if layout == "bytes":
                assert np.array_equal(a, want)
            elif layout == "bitsliced":
                assert np.array_equal(a.view(np.uint32), oracle.to_bitsliced(want, hi - lo))
            else:
                u = oracle.to_u32(want, hi - lo)
                assert np.array_equal((a if layout == "u32" else a[0]).view(np.uint32), u)
                if layout == "u32_f32":
                    assert np.array_equal(a[1].view(np.float32), oracle.to_f32(u))


@pytest.mark.parametrize("offset", [1, 2, 4, 8, 12])
@pytest.mark.parametrize("n_bits", [96, 256, 1001])
def test_output_at_any_alignment(n_bits, offset):
    s = _mixed(70)
    want = oracle.batch_bytes(s.keys, s.ivs, s.iv_lens, n_bits, threads=THREADS)
    st = _streams(s)
    buf = torch.full((70 * want.shape[1] + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    st.generate(n_bits, "bytes", out=buf[offset:])
    st.sync()
    got = buf.cpu().numpy()
    assert np.array_equal(got[offset:offset + want.size].reshape(want.shape), want)
    assert (got[:offset] == 0xA5).all() and (got[offset + want.size:] == 0xA5).all()


# the last groups per SM of the packed launch, of one and two warp-groups per
# SM, of the packed initialisation, of three warp-groups, and one group more
@pytest.mark.parametrize("extra", [0, 1])
@pytest.mark.parametrize("per_sm", [18, 32, 52, 64, 96])
def test_last_size_and_the_next_agree_with_a_thread_per_group(monkeypatch, per_sm, extra):
    # against an explicit grid launch: output, calls that go on, the state
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = _mixed((per_sm * sms + extra) * 32 - 5)
    auto = _streams(s)
    monkeypatch.setenv("MICKEY_MODE", "grid")
    grid = _streams(s)
    for n_bits, layout in ((64, "bytes"), (96, "u32"), (33, "bitsliced"), (544, "bytes"),
                           (1, "bytes"), (256, "u32_f32"), (45, "bytes"), (100, "bitsliced")):
        assert torch.equal(auto.generate(n_bits, layout), grid.generate(n_bits, layout))
    out = torch.zeros(s.n * 8 + 3, dtype=torch.uint8, device="cuda")   # off the word grid
    got = auto.generate(64, "bytes", out=out[3:])
    assert torch.equal(got.view(s.n, 8), grid.generate(64, "bytes"))
    assert torch.equal(auto.generate(96, "bytes"), grid.generate(96, "bytes"))
    k = 20_000
    if extra == 0 and per_sm in (18, 32):
        states = [h.export_state()[0][:k] for h in (auto, grid)]
        assert np.array_equal(*states)


@pytest.mark.parametrize("n", [32 * 300 + 7, 5 * 1024 + 1])
def test_thread_per_group_loading_paths_small(monkeypatch, n):
    # small handles of an explicit mode load with a thread per group: 16-byte
    # loads, and through shared memory when unaligned
    from paper_1909_04750_gb300.streams import Streams
    monkeypatch.setenv("MICKEY_MODE", "grid")
    s = _mixed(n)
    want = oracle.batch_bytes(s.keys, s.ivs, s.iv_lens, 96, threads=THREADS)
    lens = torch.from_numpy(s.iv_lens.astype(np.int32)).cuda()
    for off in (0, 1, 6):
        keys, ivs = (torch.zeros(n * 10 + 16, dtype=torch.uint8, device="cuda")[off:off + n * 10]
                     for _ in range(2))
        keys.copy_(torch.from_numpy(s.keys.reshape(-1)))
        ivs.copy_(torch.from_numpy(s.ivs.reshape(-1)))
        st = Streams(keys.view(n, 10), ivs.view(n, 10), lens)
        assert np.array_equal(st.generate(96, "bytes").cpu().numpy(), want)
        st.sync()


def test_a_long_iv_is_reported():
    s = _mixed(100)
    lens = torch.from_numpy(s.iv_lens.astype(np.int32)).cuda()
    lens[77] = 81
    from paper_1909_04750_gb300.streams import Streams
    st = Streams(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda(), lens)
    with pytest.raises(N.MickeyError) as e:
        st.sync()
    assert e.value.code == N.E_IVLEN


@pytest.mark.parametrize("offset", [0, 4])
def test_new_batch_plan_row_ends_at_any_tile(offset):
    # every group split; rows of one group end inside and at the ends of tiles
    # and of the four-tile row stores, with 16- and 4-byte aligned rows
    from paper_1909_04750_gb300.batch import Batch
    s = _mixed(200)
    nb = np.arange(200, dtype=np.uint64) * 3
    nb[:10] = [0, 1, 31, 32, 33, 127, 128, 129, 256, 4096]
    b = Batch(nb, s.iv_lens)
    assert b.get_config()["split_groups"] == 7
    buf = torch.full((b.output_bytes + 16,), 0xA5, dtype=torch.uint8, device="cuda")
    out = b.run(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda(), buf[offset:])
    b.sync()
    want = oracle.batch_bytes(s.keys, s.ivs, s.iv_lens, nb, threads=THREADS)
    for got, row in zip(b.rows(out), want):
        assert np.array_equal(got, np.asarray(row)[:got.size])
    host = out.cpu().numpy()
    used = np.zeros(host.size, bool)
    for o, n in zip(b.offsets, nb):
        used[int(o):int(o) + (int(n) + 7) // 8] = True
    assert (host[~used] == 0xA5).all()


def _grain(s):
    from paper_1909_04750_gb300.grain import GrainStreams
    return GrainStreams(torch.from_numpy(s.keys).cuda(), torch.from_numpy(s.ivs).cuda())


# the 16-clock steps, the 160-clock body, tiles and 16-byte row stores, and what is left of each
@pytest.mark.parametrize("n_bits", [1, 15, 16, 17, 31, 32, 33, 48, 128, 159, 160, 161, 176, 325,
                                    1281])
@pytest.mark.parametrize("n", [1, 33, 1000])
def test_grain_two_calls_against_the_oracle(n, n_bits):
    from oracle import grain as og
    s = workloads.grain_streams(n, seed=21)
    bits = np.unpackbits(og.batch_bytes(s.keys, s.ivs, n_bits + 67, threads=THREADS), axis=1,
                         bitorder="little")
    for layout in ("bytes", "bitsliced"):
        st = _grain(s)
        first, second = st.generate(n_bits, layout), st.generate(67, layout)
        st.sync()
        for got, lo, hi in ((first, 0, n_bits), (second, n_bits, n_bits + 67)):
            want = np.packbits(bits[:, lo:hi], axis=1, bitorder="little")
            a = got.cpu().numpy()
            if layout == "bytes":
                assert np.array_equal(a, want)
            else:
                assert np.array_equal(a.view(np.uint32), og.to_bitsliced(want, hi - lo))


@pytest.mark.parametrize("offset", [1, 2, 3, 4, 8])
@pytest.mark.parametrize("n_bits", [5, 96, 256, 1001])
def test_grain_output_at_any_alignment(n_bits, offset):
    from oracle import grain as og
    s = workloads.grain_streams(70, seed=22)
    want = og.batch_bytes(s.keys, s.ivs, n_bits, threads=THREADS)
    buf = torch.full((want.size + 64,), 0xA5, dtype=torch.uint8, device="cuda")
    st = _grain(s)
    st.generate(n_bits, "bytes", out=buf[offset:])
    st.sync()
    got = buf.cpu().numpy()
    assert np.array_equal(got[offset:offset + want.size].reshape(want.shape), want)
    assert (got[:offset] == 0xA5).all() and (got[offset + want.size:] == 0xA5).all()


@pytest.mark.parametrize("per_sm,layout", [(54, "bitsliced"), (86, "bytes"), (128, "bytes")])
@pytest.mark.parametrize("extra", [0, 1])
def test_grain_last_size_and_the_next_agree_with_a_thread_per_group(monkeypatch, per_sm, layout,
                                                                    extra):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    s = workloads.grain_streams((per_sm * sms + extra) * 32 - 5, seed=23)
    auto = _grain(s)
    monkeypatch.setenv("MICKEY_GRAIN_QUEUE", "0")
    grid = _grain(s)
    for n_bits in (256, 333):
        assert torch.equal(auto.generate(n_bits, layout), grid.generate(n_bits, layout))
    k = 50_000
    assert np.array_equal(auto.export_state()[:k], grid.export_state()[:k])


@pytest.mark.parametrize("queue", ["0", "1"])
@pytest.mark.parametrize("n_bits", [32, 33, 128, 384, 256 * 3, 640, 2048 + 128, 1000])
def test_grain_paired_launch_tiles_and_blocks(monkeypatch, n_bits, queue):
    # row blocks of 8 tiles that end early, the ring of 12, segments that start
    # and end inside a block (queue 1: three warp-groups on two chains), twice
    from oracle import grain as og
    monkeypatch.setenv("MICKEY_GRAIN_QUEUE", queue)
    s = workloads.grain_streams(2 * 1024 + 70, seed=24)
    bits = np.unpackbits(og.batch_bytes(s.keys, s.ivs, 2 * n_bits, threads=THREADS), axis=1,
                         bitorder="little")
    for layout in ("bytes", "bitsliced"):
        st = _grain(s)
        for k in range(2):
            a = st.generate(n_bits, layout).cpu().numpy()
            st.sync()
            want = np.packbits(bits[:, k * n_bits:(k + 1) * n_bits], axis=1, bitorder="little")
            if layout == "bytes":
                assert np.array_equal(a, want)
            else:
                assert np.array_equal(a.view(np.uint32), og.to_bitsliced(want, n_bits))


@pytest.mark.parametrize("n_bits", [1001, 1002, 67])
def test_bitsliced_rows_off_the_16_byte_grid(monkeypatch, n_bits):
    # the paired MICKEY launch stores a tile's words in vectors from the first
    # 16-byte boundary on
    monkeypatch.setenv("MICKEY_MODE", "persistent")
    s = _mixed(300)
    want = oracle.batch_bytes(s.keys, s.ivs, s.iv_lens, n_bits, threads=THREADS)
    got = _streams(s).generate(n_bits, "bitsliced").cpu().numpy().view(np.uint32)
    assert np.array_equal(got, oracle.to_bitsliced(want, n_bits))


def _ragged_lengths(n, layout, seed):
    rng = np.random.default_rng(seed)
    nb = rng.integers(0, 700, n).astype(np.uint64)
    nb[:24] = [0, 1, 7, 31, 32, 33, 64, 95, 96, 97, 127, 128, 129, 159, 160, 161, 255, 256, 257, 384,
               512, 639, 640, 641]
    nb[1024:2048] = rng.integers(0, 40, 1024)      # a warp-group of short lanes
    if n > 3072:
        nb[2048:3072] = 0                          # one that asks for nothing
    return nb // 32 * 32 if layout == "u32" else nb


# 3 warp-groups on pairs of their own; 6 on 4 clock warps, which hand states on
@pytest.mark.parametrize("n", [2 * 1024 + 70, 6 * 1024 - 9])
@pytest.mark.parametrize("layout", ["bytes", "u32", "bitsliced"])
def test_ragged_thread_per_group_and_per_instance_agree(monkeypatch, n, layout):
    s = _mixed(n)
    handles = [_streams(s)]                        # few groups: a thread per instance
    monkeypatch.setenv("MICKEY_MODE", "persistent")
    monkeypatch.setenv("MICKEY_PERSIST_BLOCKS", "1")
    handles.append(_streams(s))                    # a thread per group
    for call in range(3):
        nb = _ragged_lengths(n, layout, 10 * n + call)
        if layout == "bytes" and call == 2:        # rows at any byte, gaps between them
            gaps = np.random.default_rng(1).integers(0, 6, n).astype(np.uint64)
            offs = np.cumsum((nb + np.uint64(7)) // np.uint64(8) + gaps) - (
                (nb + np.uint64(7)) // np.uint64(8))
            size = int(offs[-1]) + 200
        else:
            offs, size = None, int(nb.sum()) // 8 + n + 64
            if layout == "bitsliced":
                size = 4 * 700 * ((n + 31) // 32)
        outs = []
        for h in handles:
            out = torch.full((size,), 0x5A, dtype=torch.uint8, device="cuda")
            h.generate_ragged(nb, layout, out=out, offsets=offs)
            h.sync()
            outs.append(out)
        assert torch.equal(*outs)
    states, positions = zip(*(h.export_state() for h in handles))
    assert np.array_equal(*states) and np.array_equal(*positions)
    # and the oracle, over the state both ended in: the next bits of some streams
    idx = np.arange(0, n, 37)
    nxt = [h.generate(64, "bytes").cpu().numpy()[idx] for h in handles]
    want = oracle.batch_bytes(s.keys[idx], s.ivs[idx], s.iv_lens[idx],
                              positions[0][idx] + np.uint64(64), threads=THREADS)
    for k, i in enumerate(idx):
        lo = int(positions[0][i])
        bits = np.unpackbits(np.asarray(want[k]))[lo:lo + 64]
        assert np.array_equal(np.packbits(bits), nxt[0][k])
        assert np.array_equal(nxt[0][k], nxt[1][k])


# the covering units: first and last unit in one, one chunk to several, every
# alignment of data and length, the edges of the buffer, presets of 0 and not
@pytest.mark.parametrize("length", [25, 26, 31, 33, 47, 161, 176, 481, 482, 497, 498, 511, 513, 528,
                                    1000, 1009, 1536 + 7])
@pytest.mark.parametrize("poly,init,xorout", [(0x1D, 0xFF, 0xFF), (0x07, 0, 0), (0x55, 0xA5, 0x3C),
                                              (0x32, 0xFF, 0)])
def test_crc8_any_length_and_alignment(length, poly, init, xorout):
    from oracle import lfsr as ol
    from paper_1909_04750_gb300.lfsr import crc8
    for n in (1, 31, 33, 150):
        raw = np.random.default_rng(length + n).integers(0, 256, n * length).astype(np.uint8)
        want = ol.crc8_batch(raw.reshape(n, length), poly, init, xorout)
        for offset in (0, 1, 8, 15):
            buf = torch.zeros(n * length + 16, dtype=torch.uint8, device="cuda")
            buf[offset:offset + n * length] = torch.from_numpy(raw).cuda()
            buf[:offset] = 0xC3
            buf[offset + n * length:] = 0xC3
            data = buf[offset:offset + n * length].view(n, length)
            got = crc8(data, poly, init, xorout).cpu().numpy()
            assert np.array_equal(got, want), (n, offset)


def test_grain_hand_offs_in_a_replayed_graph(monkeypatch):
    # a captured call whose segments hand states on, replayed three times,
    # continues the streams as three calls do
    monkeypatch.setenv("MICKEY_GRAIN_QUEUE", "1")
    s = workloads.grain_streams(3 * 1024 + 17, seed=25)
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        st = _grain(s)
        out = torch.zeros((s.n, 64), dtype=torch.uint8, device="cuda")
        st.generate(512, "bytes", out=out)
        side.synchronize()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=side):
            st.generate(512, "bytes", out=out)
    plain = _grain(s)
    plain.generate(512, "bytes")
    for _ in range(3):
        graph.replay()
        torch.cuda.synchronize()
        assert torch.equal(out, plain.generate(512, "bytes"))
