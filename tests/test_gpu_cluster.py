"""A cluster of CTAs per sample (small batches of large grids) gives the bits of
one CTA per sample."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1903_08741_gb300 as R
    from paper_1903_08741_gb300 import build
    build.build()
    return R


# clusters of 8 (one sample), 4, 2 (the last size that fits) and none; rows that
# are no multiple of the wide loops' width; a coarsest level of several cells
@pytest.mark.parametrize("nx,nz,S", [(64, 64, 1), (64, 64, 70), (80, 96, 5), (112, 80, 3), (128, 128, 24),
                                     (256, 256, 2), (128, 128, 77)])
@pytest.mark.parametrize("kw", [dict(), dict(precision=1), dict(nu1=0), dict(nu2=0), dict(precision=1, nu2=1)])
def test_cluster_matches_one_cta(R, nx, nz, S, kw):
    from tests.inputs import smooth_random_fields
    lk, al = (torch.from_numpy(v).cuda() for v in smooth_random_fields(nx, nz, S, nx + S))
    pb = R.Problem(nx=nx, nz=nz, nsteps=2, dt=0.01, picard_maxit=30, mg_maxit=12, **kw)
    a = R.solve_batch(pb, lk, al, 0.6, want_p=True)
    try:
        R.set_tuning(512, 0)
        b = R.solve_batch(pb, lk, al, 0.6, want_p=True)
    finally:
        R.set_tuning(0, 0)
    assert torch.equal(a[2], b[2]) and torch.equal(a[1].nan_to_num(7.0), b[1].nan_to_num(7.0))
    assert torch.equal(a[0].nan_to_num(7.0), b[0].nan_to_num(7.0))
    assert (a[3].picard_iters, a[3].mg_cycles, a[3].max_picard) == (b[3].picard_iters, b[3].mg_cycles, b[3].max_picard)
    assert 0 < a[3].sm_seconds <= a[3].seconds * torch.cuda.get_device_properties(0).multi_processor_count


@pytest.mark.parametrize("precision", [0, 1])
def test_cluster_matches_one_cta_van_genuchten(R, precision):
    from tests.inputs import smooth_random_fields
    lk, al = (torch.from_numpy(v).cuda() for v in smooth_random_fields(128, 128, 3, 1))
    n = torch.full_like(al, 1.6)
    pb = R.Problem.infiltration(nx=128, nz=128, nsteps=2, dt=1.0 / 64, precision=precision, cycle=1)
    a = R.solve_soil(pb, lk - 1.6, al, n, want_p=True)
    try:
        R.set_tuning(512, 0)
        b = R.solve_soil(pb, lk - 1.6, al, n, want_p=True)
    finally:
        R.set_tuning(0, 0)
    assert torch.equal(a[2], b[2]) and torch.equal(a[1].nan_to_num(7.0), b[1].nan_to_num(7.0))


@pytest.mark.parametrize("method,n,S,precision", [(0, 64, 2, 0), (1, 64, 50, 0), (1, 128, 3, 1), (2, 64, 3, 0)])
def test_adjoint_cluster_matches_one_cta(R, method, n, S, precision):
    """Same forward bits; the J^T solves differ by the order of their sums, within
    their 1e-11 residual target times the operators' condition: 1e-8."""
    g = torch.Generator(device="cuda").manual_seed(5)
    basis = torch.randn((4, n, n), dtype=torch.float64, device="cuda", generator=g) * 0.05
    xi = torch.randn((S, 4), dtype=torch.float64, device="cuda", generator=g)
    al = torch.full((S, n, n), 0.7, dtype=torch.float64, device="cuda")
    pb = R.Problem(nx=n, nz=n, nsteps=3, dt=0.01, precision=precision)
    out = []
    try:
        assert R.lib().rich_set_adjoint_method(R.context(0), method) == 0
        for nt in (0, 512):
            R.set_tuning(nt, 0)
            out.append(R.solve_batch_adjoint(pb, basis, xi, al))
    finally:
        R.set_tuning(0, 0)
        R.lib().rich_set_adjoint_method(R.context(0), 1)
    a, b = out
    assert torch.equal(a[0], b[0]) and torch.isfinite(a[1]).all()
    assert (a[1] - b[1]).abs().max() <= 1e-8 * b[1].abs().max()
    if method == 2:
        assert torch.equal(a[1], b[1])


def test_cluster_launch_is_captured(R):
    """A cluster launch inside a CUDA graph replays to the direct call's bits."""
    from tests.inputs import smooth_random_fields
    n, S = 64, 3
    lk, al = (torch.from_numpy(v).cuda() for v in smooth_random_fields(n, n, S, 2))
    pb = R.Problem(nx=n, nz=n, nsteps=2, dt=0.01)
    q, st = torch.empty(S, dtype=torch.float64, device="cuda"), torch.empty(S, dtype=torch.int32, device="cuda")
    side = torch.cuda.Stream()
    with torch.cuda.stream(side):
        R.solve_batch_async(pb, lk, al, q, st)                      # set-up outside the capture
        torch.cuda.synchronize()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=side):
            R.solve_batch_async(pb, lk, al, q, st)
    q.zero_()
    g.replay()
    torch.cuda.synchronize()
    want = R.solve_batch(pb, lk, al)
    assert torch.equal(q.nan_to_num(7.0), want[0].nan_to_num(7.0)) and torch.equal(st, want[2])
