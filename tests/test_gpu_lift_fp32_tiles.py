"""The FP32 lift over its mode tiles (1 to 8 modes, one tile and several) and its
batches of eight frames (shorter clips, remainders), ragged and unaligned
frames.  Bound per entry: p products added in FP32, each with G rounded to
FP32: (p + 2) 2^-24 times the sum of their magnitudes."""
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


@pytest.mark.parametrize("m,n,ncols,pad", [(1, 2, 1, 1), (3, 3, 2, 4), (511, 8, 3, 1), (512, 9, 4, 4), (513, 10, 5, 4),
                                           (1030, 17, 6, 1), (700, 18, 7, 4), (515, 25, 8, 4), (900, 30, 9, 1),
                                           (640, 33, 17, 4), (519, 40, 33, 4), (800, 12, 64, 4)])
def test_mode_tiles_and_frame_batches(C, m, n, ncols, pad):
    ctx = C.Context(0)
    rng = np.random.default_rng(m + n + ncols)
    buf = rng.integers(0, 256, size=(n, -(-m // pad) * pad), dtype=np.uint8)
    G = rng.standard_normal((ncols, n - 1)) + 1j * rng.standard_normal((ncols, n - 1))
    Gt = torch.from_numpy(np.stack([G.real, G.imag], axis=-1)).cuda()
    Phi = C.cdmd_lift(ctx, torch.from_numpy(buf).cuda()[:, :m], Gt, prec="fp32").cpu().numpy()
    Phi = (Phi[..., 0] + 1j * Phi[..., 1]) if Phi.shape[-1] == 2 and Phi.ndim == 3 else Phi
    X = buf[1:, :m].astype(np.float64)
    want = X.T @ G.T
    for part in (np.real, np.imag):
        bound = (n + 1) * 2.0 ** -24 * (X.T @ np.abs(part(G)).T)
        assert np.all(np.abs(part(Phi) - part(want)) <= bound + 1e-30)
