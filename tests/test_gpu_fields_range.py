"""Variances over the whole FP64 range: a power of four times the variance is
exactly the power of two times the field and leaves the uniform field alone."""
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def R():
    import paper_1903_08741_gb300 as R
    from paper_1903_08741_gb300 import build
    build.build()
    return R


# (1024 eigenvalues of 2^1016 add up to more than the largest FP64 number; with
# the correlated field's variance of 2^1000 none of them does)
@pytest.mark.parametrize("corr,log_sd", [(1e-7, 508), (1e-7, -500), (0.3, 500), (0.3, -500), (0.3, -20)])
def test_the_variance_scales_the_field(R, corr, log_sd):
    ref = R.sample_fields(16, 16, 5, R.FieldModel(seed=3, corr_len=corr))
    got = R.sample_fields(16, 16, 5, R.FieldModel(seed=3, corr_len=corr, sigma2=2.0 ** (2 * log_sd)))
    assert torch.isfinite(ref[0]).all()
    assert torch.equal(got[0], ref[0] * 2.0 ** log_sd)
    assert torch.equal(got[1], ref[1])
