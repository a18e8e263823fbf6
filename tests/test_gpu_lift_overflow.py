"""The tensor-core lift with entries of G that its FP16 parts cannot hold: the
part (Re or Im) of a mode with such an entry comes back non-finite, never as a
finite number; the rest of the result does not see it.  Each mode is scaled by a
power of two clamped to 2^-100 .. 2^100 (2^15 past 1e300), so an entry overflows
FP16 from 2^116 on."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

INF, NAN = float("inf"), float("nan")


@pytest.fixture(scope="module")
def C():
    from paper_1512_04205_gb300 import build, cdmd
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    build.build()
    return cdmd


@pytest.mark.parametrize("part", [0, 1])
@pytest.mark.parametrize("v", [2.0 ** 116, 2.0 ** 227, -2.0 ** 228, 2.0 ** 229, 1e200, -1e300, 1e301, -1.7e308, INF,
                               -INF, NAN])
def test_overflowing_entry(C, v, part):
    ctx = C.Context(0)
    rng = np.random.default_rng(7)
    n, m, r = 40, 1000, 4
    D = torch.zeros((n, 1008), dtype=torch.uint8, device="cuda")[:, :m]
    D.copy_(torch.from_numpy(rng.integers(0, 256, (n, m), dtype=np.uint8)))
    G = rng.standard_normal((r, n - 1, 2)) * 1e-8      # far below 1: the scale matters
    clean = G.copy()
    clean[1, 17, part] = 0.0
    G[1, 17, part] = v
    ref = C.cdmd_lift(ctx, D, torch.from_numpy(clean).cuda(), prec="bf16x2")
    got = C.cdmd_lift(ctx, D, torch.from_numpy(G).cuda(), prec="bf16x2")
    assert not torch.isfinite(got[:, 1, part]).any()
    for c in (0, 2, 3):
        assert torch.equal(got[:, c], ref[:, c])
    if np.isnan(v):        # NaN has no part in the mode's scale
        assert torch.equal(got[:, 1, 1 - part], ref[:, 1, 1 - part])
    else:
        assert torch.isfinite(got[:, 1, 1 - part]).all()
