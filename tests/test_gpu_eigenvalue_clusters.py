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


@pytest.mark.parametrize("n,k,ratio,q", [(40, 200, 1e-1, 4), (40, 200, 1e-3, 4), (200, 400, 1e-3, 6), (300, 400, 1e-3, 6),
                                         (100, 300, 1e-4, 6)])
def test_repeated_values_below_larger_ones(C, n, k, ratio, q):
    # Three large singular values, one repeated q times, a tail.  The Gram and its
    # tridiagonal form are off by some eps of the largest eigenvalue, l1, so a vector of
    # the repeated one, lc, is off by eps l1 / lc: the compressed modes by some of
    # that, the eigenvalues by that times the condition of their vectors (Bauer and Fike).
    ctx = C.Context(0)
    r, p = 3 + q, n - 1
    for seed in range(3):
        rng = np.random.default_rng(seed)
        U = np.linalg.qr(rng.standard_normal((k, p)))[0]
        V = np.linalg.qr(rng.standard_normal((p, p)))[0]
        s = np.concatenate([[1.0, 0.7, 0.4], np.full(q, ratio), ratio * 0.02 * 0.9 ** np.arange(p - r)])
        Y = (U * s) @ V.T
        A = 0.9 * np.linalg.qr(rng.standard_normal((r, r)))[0]
        DY = np.concatenate([Y, (U[:, :r] @ (A @ (U[:, :r].T @ Y[:, -1])))[:, None]], 1)
        out = C.cdmd_decompose(ctx, torch.from_numpy(np.ascontiguousarray(DY.T)).cuda(), r, 3, with_phiy=True)
        C.cdmd_status_sync(ctx)
        Y, Y1 = DY[:, :-1], DY[:, 1:]
        U, s, Vh = np.linalg.svd(Y, full_matrices=False)
        U, s, V = U[:, :r], s[:r], Vh[:r].T
        lam, W = np.linalg.eig((U.T @ Y1 @ V) / s)
        W = W / np.linalg.norm(W, axis=0)
        P = Y1 @ ((V / s) @ W)
        unit = EPS * (s[0] / s[-1]) ** 2
        assert np.max(np.abs(out["sigma"].cpu().numpy() ** 2 - s ** 2)) <= 32 * EPS * s[0] ** 2
        got, gotP = (torch.view_as_complex(out[x]).cpu().numpy() for x in ("lam", "PhiY"))
        for c in range(r):
            j = int(np.argmin(np.abs(lam - got[c])))
            assert abs(got[c] - lam[j]) <= np.linalg.cond(W) * unit
            # up to the phase, which the basis of the repeated value's vectors decides
            phase = np.vdot(P[:, j], gotP[c])
            assert np.linalg.norm(gotP[c] - P[:, j] * phase / abs(phase)) <= 64 * unit * np.linalg.norm(P[:, j])
