"""Memory of the adjoint's states: kept or recomputed from checkpoints to the same
bits, within the caller's limit, and given back."""
import ctypes as C

import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1903_08741_gb300 as R
    from paper_1903_08741_gb300 import build
    build.build()
    return R


def inputs(nx, nz, S):
    g = torch.Generator(device="cuda").manual_seed(nx + S)
    basis = torch.randn((4, nz, nx), dtype=torch.float64, device="cuda", generator=g) * 0.05
    xi = torch.randn((S, 4), dtype=torch.float64, device="cuda", generator=g)
    return basis, xi, torch.full((S, nz, nx), 0.7, dtype=torch.float64, device="cuda")


# one CTA a sample (16^2, 64^2 with GMRES or W-cycles) and a cluster (64^2 FP64,
# 128^2 mixed); intervals of one step, with a short last segment, of all steps and
# beyond them
@pytest.mark.parametrize("n,S,kw,method", [(16, 3, dict(), 1), (16, 3, dict(precision=1), 0), (64, 2, dict(), 1),
                                           (128, 2, dict(precision=1), 1), (64, 2, dict(), 2),
                                           (64, 2, dict(cycle=2), 1)])
def test_recomputed_states_give_the_kept_ones_bits(R, n, S, kw, method):
    basis, xi, al = inputs(n, n, S)
    pb = R.Problem(nx=n, nz=n, nsteps=7, dt=0.005, **kw)
    try:
        R.set_adjoint_method(method)
        kept = R.solve_batch_adjoint(pb, basis, xi, al, ckpt_every=3, want_dlnks=True)
        R.set_adjoint_memory(0)
        for ck in (1, 3, 7, 10):
            got = R.solve_batch_adjoint(pb, basis, xi, al, ckpt_every=ck, want_dlnks=True)
            for a, b in zip(kept[:4], got[:4]):
                assert torch.equal(a, b)
            assert (kept[4].picard_iters, kept[4].mg_cycles) == (got[4].picard_iters, got[4].mg_cycles)
    finally:
        R.set_adjoint_memory()
        R.set_adjoint_method(R.BICGSTAB)
    assert torch.isfinite(kept[1]).all()


@pytest.fixture
def fresh(R, monkeypatch):
    """fresh(limit): a new library context for the calls that follow."""
    made = []

    def make(limit):
        h = C.c_void_p()
        assert R.lib().rich_create(C.byref(h), 0) == 0
        made.append(h)
        monkeypatch.setattr(R, "_ctx", {0: h})
        if limit is not None:
            R.set_adjoint_memory(limit)
    yield make
    for h in made:
        R.lib().rich_destroy(h)


@pytest.mark.parametrize("steps,limit,kept_mib", [(40, None, 46), (40, 0, 1), (40, 46 << 20, 25), (140, None, 0)])
def test_states_stay_within_the_limit_and_are_given_back(R, fresh, steps, limit, kept_mib):
    """What a context holds after a call beyond that after a call of one step.  A
    state of the 152 samples on 32^2 is 1.19 MiB.  40 steps kept: 47.5 MiB.  Never
    kept: a second checkpoint.  40 steps above the limit (one step below it): two
    checkpoints and a segment of 20.  140 steps kept, 166 MiB, above the pool's 64:
    nothing."""
    basis, xi, al = inputs(32, 32, 152)
    ck = 20

    def held(n):
        fresh(limit)
        pb = R.Problem(nx=32, nz=32, nsteps=n, dt=0.001, precision=R.MIXED, picard_tol=1e-4, mg_tol=1e-3)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        R.solve_batch_adjoint(pb, basis, xi, al, ckpt_every=ck)
        return (before - torch.cuda.mem_get_info()[0]) / 2 ** 20

    few = held(1)
    more = held(steps) - few
    assert kept_mib - 6 <= more <= kept_mib + 6
