"""A batch whose launch shape would hold more slots than the device has memory for
runs with fewer CTAs, to the same bits."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_fewer_slots_where_memory_is_short(monkeypatch):
    """4864 samples of 32^2 take eight CTAs an SM, 1216 slots of 0.19 MiB (240 MB);
    512-thread CTAs, two an SM, would take 60 MB.  150 MB are left."""
    import paper_1903_08741_gb300 as R
    from paper_1903_08741_gb300 import build
    build.build()
    n, S = 32, 4864
    lk, al = R.sample_fields(n, n, S, R.FieldModel(seed=1))
    pb = R.Problem(nx=n, nz=n, nsteps=1, dt=0.01)
    want = R.solve_batch(pb, lk, al)               # (outputs and local memory are allocated now)
    h = C.c_void_p()
    assert R.lib().rich_create(C.byref(h), 0) == 0
    monkeypatch.setattr(R, "_ctx", {0: h})
    fill = None
    try:
        torch.cuda.synchronize()
        fill = torch.empty(torch.cuda.mem_get_info()[0] - (150 << 20), dtype=torch.uint8, device="cuda")
        got = R.solve_batch(pb, lk, al)
    finally:
        del fill
        torch.cuda.empty_cache()
        R.lib().rich_destroy(h)
    assert torch.equal(got[0].nan_to_num(7.0), want[0].nan_to_num(7.0)) and torch.equal(got[2], want[2])
