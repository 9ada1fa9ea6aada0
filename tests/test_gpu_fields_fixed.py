"""Fixed-point field transforms: every pass plan (radices 8, 4, 2) and ragged
line blocks, against the oracle's FP64 generator."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

import oracle as O  # noqa: E402


@pytest.fixture(scope="module")
def R():
    import paper_1903_08741_gb300 as R
    from paper_1903_08741_gb300 import build
    build.build()
    O.build()
    return R


# torus sides 2 ... 4096: one pass of 2, 4, 8; fours at the end; blocks of many
# short lines and of one long line, the last block partly filled
SIZES = [(1, 1, 3), (2, 1, 5), (1, 4, 2), (4, 2, 37), (8, 16, 7), (64, 4, 3), (4, 64, 3), (256, 8, 5), (8, 256, 5),
         (128, 32, 2), (2048, 2, 1), (2, 1024, 3)]


@pytest.mark.parametrize("nx,nz,S", SIZES)
def test_white_field_is_the_noise(R, nx, nz, S):
    """With a covariance of one cell the filter is one and the field is the
    noise.  FP64 normals are off by up to 4e-15 (the rounding of the angle times
    the largest radius 8.6) and their transforms by about 2e-15 of 5 deviations;
    the bar is 2e-14."""
    kw = dict(corr_len=1e-7, corr_len_z=1e-7)
    lo, ao = O.sample_fields(nx, nz, S, seed=5, level=1, first_sample=2, **kw)
    lk, al = R.sample_fields(nx, nz, S, R.FieldModel(seed=5, **kw), level=1, first_sample=2)
    assert np.abs(lk.cpu().numpy() - lo).max() < 2e-14
    assert np.abs(al.cpu().numpy() - ao).max() < 2e-14


# (the 2 x 1024 grid's covariance needs a torus above the largest side)
@pytest.mark.parametrize("nx,nz,S", [s for s in SIZES if min(s[:2]) > 1 and s != (2, 1024, 3)] + [(2, 64, 3)])
def test_pair_fields_match_oracle(R, nx, nz, S):
    """The bar of the other field tests (rounding of the spectrum amplified by
    its small eigenvalues): 1e-12."""
    o = O.sample_fields_pair(nx, nz, S, seed=9, level=2, first_sample=1)
    g = R.sample_fields_pair(nx, nz, S, R.FieldModel(seed=9), level=2, first_sample=1)
    for a, b in zip(g, o):
        assert np.abs(a.cpu().numpy() - b).max() < 1e-12


def test_infinite_variance_gives_no_finite_field(R):
    lk, _ = R.sample_fields(8, 8, 2, R.FieldModel(sigma2=float("inf")))
    assert not torch.isfinite(lk).any()
