"""A sample's gradient is its own: the number of samples in the call, and with it
the number of CTAs that share a sample, does not change its bits."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1903_08741_gb300 as R
    from paper_1903_08741_gb300 import build
    build.build()
    return R


# clusters of 8, 3 and 2 CTAs a sample, and one CTA a sample (100); 112 x 80 has
# rows that are no multiple of a warp, and cells that fill the last chains partly
@pytest.mark.parametrize("nx,nz,precision", [(64, 64, 0), (112, 80, 0), (128, 128, 1)])
@pytest.mark.parametrize("method", [0, 1])
def test_gradient_does_not_depend_on_the_batch(R, nx, nz, precision, method):
    g = torch.Generator(device="cuda").manual_seed(11)
    basis = torch.randn((4, nz, nx), dtype=torch.float64, device="cuda", generator=g) * 0.05
    xi = torch.randn((100, 4), dtype=torch.float64, device="cuda", generator=g)
    al = torch.full((100, nz, nx), 0.7, dtype=torch.float64, device="cuda")
    pb = R.Problem(nx=nx, nz=nz, nsteps=2, dt=0.01, precision=precision)
    out = {}
    try:
        R.set_adjoint_method(method)
        for S in (100, 70, 48, 1):
            out[S] = R.solve_batch_adjoint(pb, basis, xi[:S].contiguous(), al[:S].contiguous(), want_dlnks=True)
    finally:
        R.set_adjoint_method(R.BICGSTAB)
    q, dq, gr = out[100][:3]
    assert torch.isfinite(dq).all()
    for S in (70, 48, 1):
        assert torch.equal(out[S][0], q[:S])
        assert torch.equal(out[S][1], dq[:S]) and torch.equal(out[S][2], gr[:S])
