"""One clip under a Rademacher C on the tensor cores: more frames than one
launch packs (512), and C words drawn for 16 K steps at a time over several such batches
of one split, the last of them partial.  Exact integers against the oracle."""
import numpy as np
import pytest

from oracle import cdmd as O
from oracle import measurement as M

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def C():
    from paper_1512_04205_gb300 import build, cdmd
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    build.build()
    return cdmd


# k = 19400: 152 row blocks, so one split walks all 51 K steps; k = 1: one row
@pytest.mark.parametrize("m,n,k", [(700, 600, 40), (3205, 9, 19400), (64 * 48, 17, 19456), (1, 2, 1), (65, 513, 129)])
def test_single_clip_is_exact(C, m, n, k):
    ctx = C.Context(0)
    frames = np.random.default_rng(m + n).integers(0, 256, size=(n, m), dtype=np.uint8)
    padded = np.full((n, (m + 15) // 16 * 16), 255, dtype=np.uint8)
    padded[:, :m] = frames
    D = torch.from_numpy(padded).cuda()[:, :m]
    DY = C.cdmd_sketch(ctx, D, k, 5 + k, ctype="rademacher", prec="bf16x2")
    C.cdmd_status_sync(ctx)
    Cm = M.measurement_matrix("rademacher", 5 + k, k, m)
    assert np.array_equal(DY.cpu().numpy(), O.sketch(Cm, frames.T.astype(np.float64)).T)
