"""Tuning of few samples of a large grid, which untuned calls give a cluster of
CTAs each, and of entries that other kernels were measured for (no GPU)."""
import json

import pytest

torch = pytest.importorskip("torch")

import paper_1903_08741_gb300 as R  # noqa: E402
from paper_1903_08741_gb300 import autotune  # noqa: E402

GRID = dict(nx=256, nz=256, precision=R.MIXED)


def test_candidates_hold_the_automatic_shape_for_few_samples():
    few, many = R.Problem(**GRID), R.Problem(nx=32, nz=64, precision=R.MIXED)
    assert autotune.candidates(few, 76, 152) == (0,) + autotune.shapes(few)
    assert autotune.candidates(few, 77, 152) == autotune.shapes(few)
    assert autotune.candidates(many, 2, 152) == autotune.shapes(many)
    assert autotune.candidates(R.Problem(**GRID, cycle=2), 2, 152) == autotune.shapes(few)


def test_few_samples_have_their_own_entries():
    pb = R.Problem(**GRID)
    assert autotune._bucket(70) == autotune._bucket(80)
    assert autotune._key(pb, 70, "GPU", 152) != autotune._key(pb, 80, "GPU", 152)
    assert autotune._key(pb, 80, "GPU", 152) == autotune._key(pb, 80, "GPU")


@pytest.fixture
def gpu(monkeypatch, tmp_path):
    """A GB300 as far as the choice of an entry goes; the calls of set_tuning."""
    calls = []
    monkeypatch.setenv("RICH_TUNE_CACHE", str(tmp_path / "t.json"))
    monkeypatch.setattr(autotune, "_device", lambda d: (torch.device("cpu"), "NVIDIA GB300", 152))
    monkeypatch.setattr(R, "set_tuning", lambda *a: calls.append(a))
    return tmp_path / "t.json", calls


def test_shipped_entries_are_for_the_present_kernels_and_not_for_few_samples(gpu):
    path, calls = gpu
    assert autotune._load(autotune.SHIPPED).keys() == autotune._read(autotune.SHIPPED).keys()
    pb = R.Problem(**GRID)
    assert autotune.source(pb, 80) == "shipped"
    assert autotune.source(pb, 70) == "measure"
    bt, mi = autotune.tune(pb, 80)
    assert bt in autotune.shapes(pb) and calls == [(bt, mi, 0)]


def test_entries_of_other_kernels_are_not_used(gpu):
    path, calls = gpu
    pb = R.Problem(**GRID)
    key = autotune._key(pb, 70, "NVIDIA GB300", 152)
    entry = {"block_threads": 1024, "mixed_inner": 3}
    for kernels in (None, autotune.KERNELS - 1):
        path.write_text(json.dumps({key: dict(entry, kernels=kernels) if kernels else entry}))
        assert autotune.source(pb, 70) == "measure"
    path.write_text(json.dumps({key: dict(entry, kernels=autotune.KERNELS)}))
    assert autotune.source(pb, 70) == "cache"
    assert autotune.tune(pb, 70) == (1024, 3) and calls == [(1024, 3, 0)]
