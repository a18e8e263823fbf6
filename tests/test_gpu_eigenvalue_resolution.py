"""Singular values beyond the resolution of the eigenvalue search.  The search
stops at an interval of 2^8 eps of the norm, so its midpoint is off by up to 128 eps;
what the Rayleigh quotient leaves is the backward error of the Gram and the
tridiagonalisation, a few eps of the norm (32 allowed).  Oracle: numpy's SVD."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def C():
    from paper_1512_04205_gb300 import build, cdmd
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    build.build()
    return cdmd


@pytest.mark.parametrize("n,r", [(7, 5), (40, 10), (130, 12), (300, 32), (512, 20)])
def test_singular_values_past_the_search(C, n, r):
    ctx = C.Context(0)
    rng = np.random.default_rng(n + r)
    k = 530
    U = np.linalg.qr(rng.standard_normal((k, n)))[0]
    V = np.linalg.qr(rng.standard_normal((n, n)))[0]
    DY = (U * (10.0 * 0.8 ** np.minimum(np.arange(n), 40))) @ V.T
    out = C.cdmd_decompose(ctx, torch.from_numpy(np.ascontiguousarray(DY.T)).cuda(), r, min(r, 4))
    C.cdmd_status_sync(ctx)
    s = np.linalg.svd(DY[:, :-1], compute_uv=False)[:r]
    eps = np.finfo(np.float64).eps
    assert np.max(np.abs(out["sigma"].cpu().numpy() ** 2 - s ** 2)) <= 32 * eps * s[0] ** 2
