"""The tuner's cache key names the library that was timed (no GPU): a choice cached with
other kernels is not applied."""
import os

import pytest


def test_key_changes_with_the_library(tmp_path, monkeypatch):
    pytest.importorskip("torch")
    from paper_1603_04100_gb300 import build, tune
    lib = tmp_path / "libmvgd.so"
    monkeypatch.setattr(build, "LIB", lib)
    keys = [tune.shape_key(1 << 20, 20, 1, 2)]  # not built yet
    lib.write_bytes(b"one")
    keys.append(tune.shape_key(1 << 20, 20, 1, 2))
    assert tune.shape_key(1 << 20, 20, 1, 2) == keys[-1]
    lib.write_bytes(b"two")
    os.utime(lib, ns=(1, 1))
    keys.append(tune.shape_key(1 << 20, 20, 1, 2))
    assert len(set(keys)) == 3
    lib.write_bytes(b"one")  # the same bytes, built again: the same key
    os.utime(lib, ns=(2, 2))
    assert tune.shape_key(1 << 20, 20, 1, 2) == keys[1]
