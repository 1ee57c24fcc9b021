"""The autotuner's cache: a choice measured with other kernels is not used (no GPU)."""
import json

import pytest
import torch

from paper_2011_05755_gb300 import MRA_BF16_RESCORE, MRA_KERNEL_MMA_SYNC, autotune

ARGS = (76, 1, 35, 1, 4.0, 1.0, 1, MRA_BF16_RESCORE, 100)


class _Measured(Exception):
    pass


@pytest.fixture
def cache(monkeypatch, tmp_path):
    def measure(*a, **kw):
        raise _Measured
    monkeypatch.setattr(torch.cuda, "current_device", lambda: 0)
    monkeypatch.setattr(torch.cuda, "get_device_name", lambda dev=None: "NVIDIA GB300")
    monkeypatch.setattr(torch, "Generator", measure)  # the first step of a measurement
    return tmp_path / "tune.json"


def _tune(path):
    return autotune.tune(*ARGS, cache=str(path))


def test_entries_of_other_kernels_are_measured_again(cache, monkeypatch):
    entry = {"kernel": MRA_KERNEL_MMA_SYNC, "chunk_images": 1024, "ms_per_image": 0.01}
    # as written before the key named the library
    cache.write_text(json.dumps({"NVIDIA_GB300|L76|r1-35-1|s4/1|m1|p1|K100": entry}))
    with pytest.raises(_Measured):
        _tune(cache)
    key = autotune._key(torch.device("cuda", 0), *ARGS)
    cache.write_text(json.dumps({key: entry}))
    assert _tune(cache) == entry
    monkeypatch.setattr(autotune, "library_id", lambda: "0" * 12)
    with pytest.raises(_Measured):
        _tune(cache)


def test_the_library_id_follows_the_sources(monkeypatch, tmp_path):
    csrc = tmp_path / "csrc"
    csrc.mkdir()
    (csrc / "k.cu").write_text("a")
    monkeypatch.setattr(autotune, "__file__", str(tmp_path / "autotune.py"))
    ids = []
    for text in ("a", "b"):
        (csrc / "k.cu").write_text(text)
        autotune.library_id.cache_clear()
        ids.append(autotune.library_id())
    autotune.library_id.cache_clear()
    assert ids[0] != ids[1] and all(len(i) == 12 for i in ids)
