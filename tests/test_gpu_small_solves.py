"""The small solves on sketches that reach the rare branches of their kernels:
repeated singular values (the inverse iteration's vectors are then not
orthogonal and the Gram-Schmidt branch runs), every block edge of the
reflectors, clustered eigenvalues of A~.

Oracle: numpy's SVD and eigenvalues of the same sketch."""
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


@pytest.fixture(scope="module")
def ctx(C):
    return C.Context(0)


def _solve(C, ctx, DY, r, K, **kw):
    out = C.cdmd_decompose(ctx, torch.from_numpy(np.ascontiguousarray(DY.T)).cuda(), r, K, with_phiy=True, **kw)
    C.cdmd_status_sync(ctx)
    d = {q: v.cpu().numpy() for q, v in out.items()}
    return d, d["lam"][:, 0] + 1j * d["lam"][:, 1]


def _reference(DY, r):
    Y, Y1 = DY[:, :-1], DY[:, 1:]
    U, s, Vh = np.linalg.svd(Y, full_matrices=False)
    At = (U[:, :r].T @ Y1 @ Vh[:r].T) / s[:r]
    return s[:r], np.linalg.eigvals(At), At


def _match(a, b):
    """Largest distance of two spectra, paired greedily."""
    b = list(b)
    worst = 0.0
    for x in a:
        i = int(np.argmin([abs(x - y) for y in b]))
        worst = max(worst, abs(x - b.pop(i)))
    return worst


@pytest.mark.parametrize("n,r", [(12, 5), (40, 6), (40, 32), (258, 7), (300, 20)])
def test_repeated_singular_values(C, ctx, n, r):
    # r equal singular values, the rest 1e-4 of them: every orthonormal basis
    # of the leading subspace gives the same A~ up to similarity
    rng = np.random.default_rng(n + r)
    p, k = n - 1, 600
    V = np.linalg.qr(rng.standard_normal((p, p)))[0]
    U = np.linalg.qr(rng.standard_normal((k, p)))[0]
    s = np.full(p, 5e-4)
    s[:r] = 5.0
    Y = (U * s) @ V.T
    DY = np.concatenate([Y, Y[:, :1] + 0.1 * rng.standard_normal((k, 1))], axis=1)
    d, lam = _solve(C, ctx, DY, r, min(r, 4))
    s_ref, lam_ref, At = _reference(DY, r)
    assert np.max(np.abs(d["sigma"] - s_ref)) < 1e-11 * s_ref[0]
    # the subspace errs by about eps (sigma_1 / gap)^2 p, an eigenvalue by that
    # times its condition number
    _, W = np.linalg.eig(At)
    cond = np.linalg.cond(W)
    assert _match(lam, lam_ref) < 1e-12 * n * max(1.0, cond) * np.linalg.norm(At, 2)


@pytest.mark.parametrize("n", [3, 4, 5, 18, 19, 33, 34, 35, 36, 66, 129, 255, 256, 257, 258, 259, 274, 275, 400, 512])
def test_reflector_block_edges(C, ctx, n):
    # p - 2 reflectors around multiples of the block sizes 16 and 32, and the
    # cluster's row splits; a decaying spectrum with random dynamics
    rng = np.random.default_rng(n)
    p, k = n - 1, 530
    r = min(8, p)
    U = np.linalg.qr(rng.standard_normal((k, n)))[0]
    V = np.linalg.qr(rng.standard_normal((n, n)))[0]
    DY = (U * (10.0 * 0.7 ** np.minimum(np.arange(n), 30))) @ V.T
    d, lam = _solve(C, ctx, DY, r, min(r, 4))
    s_ref, lam_ref, At = _reference(DY, r)
    assert np.max(np.abs(d["sigma"] - s_ref)) < 1e-11 * s_ref[0]
    _, W = np.linalg.eig(At)
    # the Gram form squares the spread: eps (sigma_1 / sigma_r)^2 over a relative gap of about 1/2
    assert _match(lam, lam_ref) < 1e-14 * n * (s_ref[0] / s_ref[-1]) ** 2 * max(1.0, np.linalg.cond(W)) * max(
        1.0, np.linalg.norm(At, 2))
    # Phi_Y = Y' G
    G = (d["G"][..., 0] + 1j * d["G"][..., 1]).T
    P = (d["PhiY"][..., 0] + 1j * d["PhiY"][..., 1]).T
    assert np.linalg.norm(P - DY[:, 1:] @ G) < 1e-10 * np.linalg.norm(P)
