"""The tuner does not make few samples of a large grid slower than no tuning."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_tuning_keeps_the_clusters(tmp_path, monkeypatch):
    """24 samples of 256^2 on six SMs each take about a third of the time of one
    CTA a sample, so the library's own shape wins by far."""
    import paper_1903_08741_gb300 as R
    from paper_1903_08741_gb300 import autotune, build
    build.build()
    monkeypatch.setenv("RICH_TUNE_CACHE", str(tmp_path / "t.json"))
    pb = R.Problem(nx=256, nz=256, nsteps=2, dt=0.1 / 80)
    try:
        assert autotune.tune(pb, 24)[0] == 0
        assert autotune.source(pb, 24) == "cache" and autotune.tune(pb, 24)[0] == 0
    finally:
        R.set_tuning(0, 0)
