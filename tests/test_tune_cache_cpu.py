"""The tuning cache holds for the sources it was measured on."""
import types

import numpy as np

from paper_1909_04750_gb300 import autotune, batch, build


def _keys(monkeypatch):
    torch = __import__("torch")
    gpu = types.SimpleNamespace(name="GPU", multi_processor_count=152)
    monkeypatch.setattr(torch.cuda, "get_device_properties", lambda d: gpu)
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    plan = types.SimpleNamespace(n=3, n_bits=np.arange(3, dtype=np.uint64), max_clocks=2,
                                 total_clocks=2)
    return autotune.shape_key(1024, 256, 1), batch.shape_key(plan)


def test_another_build_is_another_key(monkeypatch):
    first = _keys(monkeypatch)
    assert first == _keys(monkeypatch)
    monkeypatch.setattr(build, "library_digest", lambda: "another")
    assert all(a != b for a, b in zip(first, _keys(monkeypatch)))


def test_the_digest_covers_every_source(tmp_path, monkeypatch):
    import os
    import shutil
    shutil.copytree(build.CSRC, tmp_path / "csrc")
    monkeypatch.setattr(build, "CSRC", str(tmp_path / "csrc"))
    seen = set()
    for name in sorted(os.listdir(tmp_path / "csrc")):
        build.library_digest.cache_clear()
        seen.add(build.library_digest())
        with open(tmp_path / "csrc" / name, "a") as f:
            f.write("\nint %s;\n" % name.replace(".", "_"))
    build.library_digest.cache_clear()
    seen.add(build.library_digest())
    assert len(seen) == len(os.listdir(tmp_path / "csrc")) + 1
    build.library_digest.cache_clear()


def test_the_librarys_own_launch_is_described_as_what_it_is():
    from paper_1909_04750_gb300 import _native as N
    own = autotune.describe({"mode": N.MODE_AUTO, "unroll": 4, "stage": 1})
    assert "clocks/step" not in own and "staged" not in own and own.startswith("auto")
    paired = autotune.describe({"mode": N.MODE_PERSISTENT, "unroll": 4, "stage": 1})
    assert paired == "persistent, 4 clocks/step, staged rows"
