"""Level loops of the fused solver: the 16-byte (two FP64 or four FP32 cells a
thread) and the one-cell loops of a level give the same bits, whichever launch
shape picks them, and solves that need no cycle leave the head alone."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1903_08741_gb300 as R
    from paper_1903_08741_gb300 import build
    build.build()
    return R


def fields(nx, nz, S, seed):
    from tests.inputs import smooth_random_fields
    lk, al = smooth_random_fields(nx, nz, S, seed)
    return torch.from_numpy(lk).cuda(), torch.from_numpy(al).cuda()


# half rows of 18 and 14 (even, no multiple of 4), 20, 10 and 13 (odd: never wide),
# the smallest split grid, and one level only
@pytest.mark.parametrize("nx,nz", [(36, 20), (40, 24), (28, 36), (20, 36), (26, 8), (6, 6), (5, 7)])
@pytest.mark.parametrize("kw", [dict(precision=0), dict(precision=1), dict(precision=0, cycle=2),
                                dict(precision=0, nu1=0), dict(precision=0, nu2=0), dict(precision=1, nu1=1)])
def test_wide_and_narrow_loops_agree(R, nx, nz, kw):
    """One-warp CTAs take every aligned level of at least 64 cells of a colour
    through the wide loops, 1024-thread CTAs none of these levels."""
    lk, al = fields(nx, nz, 3, nx + nz)
    pb = R.Problem(nx=nx, nz=nz, nsteps=2, dt=0.01, **kw)
    out = {}
    try:
        for nt in (32, 256, 1024):
            R.set_tuning(nt, 0)
            out[nt] = R.solve_batch(pb, lk, al, 0.6, want_p=True)
    finally:
        R.set_tuning(0, 0)
    for nt in (32, 256):
        assert torch.equal(out[nt][2], out[1024][2])
        assert torch.equal(out[nt][1], out[1024][1])
        assert (out[nt][3].picard_iters, out[nt][3].mg_cycles) == (out[1024][3].picard_iters, out[1024][3].mg_cycles)


@pytest.mark.parametrize("n", [3, 16, 64])
@pytest.mark.parametrize("precision", [0, 1])
def test_solve_without_a_cycle_changes_nothing(R, n, precision):
    """A right-hand side already below the multigrid target has the zero
    correction (the red cells' seed is not one): one Picard iteration a step,
    no cycle, the head stays at its initial value."""
    lk, al = fields(n, n, 2, n)
    pb = R.Problem(nx=n, nz=n, nsteps=2, dt=0.01, mg_tol=2.0, precision=precision)
    _, p, s, st, rc = R.solve_batch(pb, lk, al, want_p=True)
    assert rc == 0 and st.mg_cycles == 0 and st.picard_iters == 4
    assert torch.equal(p, torch.full_like(p, pb.p_init))


def test_adjoint_checkpoints_match_kept_states(R):
    """Beyond the memory for kept states (4 GiB over the resident samples) the
    adjoint recomputes its segments from checkpoints: same bits as the kept
    states that a smaller batch of the same samples uses."""
    n, S, steps = 64, 152, 900
    g = torch.Generator(device="cuda").manual_seed(3)
    basis = torch.randn((4, n, n), dtype=torch.float64, device="cuda", generator=g) * 0.05
    xi = torch.randn((S, 4), dtype=torch.float64, device="cuda", generator=g)
    al = torch.full((S, n, n), 0.5, dtype=torch.float64, device="cuda")
    pb = R.Problem(nx=n, nz=n, nsteps=steps, dt=0.02, precision=R.MIXED, picard_tol=1e-6)
    assert min(S, torch.cuda.get_device_properties(0).multi_processor_count) * steps * n * n * 8 > 4 << 30
    big = R.solve_batch_adjoint(pb, basis, xi, al, ckpt_every=30)
    few = R.solve_batch_adjoint(pb, basis, xi[:3].contiguous(), al[:3].contiguous(), ckpt_every=30)
    assert torch.equal(big[0][:3], few[0]) and torch.equal(big[1][:3], few[1])
    assert torch.isfinite(big[1]).all()
