"""Singular values of wanted pairs that lie within some 30 to 10,000 eps of the norm of
each other, so near that one shift of the eigenvalue search cannot tell them
apart: each is still off by no more than the backward error of the
tridiagonalisation and of numpy's symmetric eigen-solver on the same matrix, a few
eps of the norm each (32 allowed together), and they come in order."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

EPS = np.finfo(np.float64).eps


@pytest.fixture(scope="module")
def C():
    from paper_1512_04205_gb300 import build, cdmd
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    build.build()
    return cdmd


@pytest.mark.parametrize("p", [12, 63, 199, 300])
@pytest.mark.parametrize("gap", [3, 30, 100, 250, 1000, 4000, 10000])
def test_close_singular_values(C, p, gap):
    ctx = C.Context(0)
    r = 10
    worst = 0.0
    for seed in range(4):
        rng = np.random.default_rng(100 * p + seed)
        # two leading values, a cluster of two or three, more wanted ones, a tail
        q = 2 + seed % 2
        lam = np.concatenate([[1.0, 0.8], 0.5 + gap * EPS * np.arange(q)[::-1] * rng.uniform(0.5, 1.0),
                              0.3 * 0.7 ** np.arange(p - 2 - q)])
        Q = np.linalg.qr(rng.standard_normal((p, p)))[0]
        S = (Q * lam) @ Q.T
        S = 0.5 * (S + S.T)
        w = rng.standard_normal(p) / np.sqrt(p)
        R = np.empty((p + 1, p + 1))
        R[:p, :p] = S
        R[:p, p] = R[p, :p] = S @ w
        R[p, p] = w @ S @ w + 1.0
        out = C.cdmd_decompose_gram(ctx, torch.from_numpy(R).cuda(), r, 4)
        C.cdmd_status_sync(ctx)
        sigma = out["sigma"].cpu().numpy()
        ref = np.linalg.eigvalsh(S)[::-1][:r]
        assert np.all(np.diff(sigma) <= 0.0)
        worst = max(worst, np.max(np.abs(sigma ** 2 - ref)) / (EPS * ref[0]))
    assert worst <= 32.0, worst
