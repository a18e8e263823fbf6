"""The FP32 sketch at the edges of its 32-pixel chunks: one chunk in a split, two, a
ragged last one, splits of several, frames that are not 4-byte aligned, slabs of 1
to 8 groups of 32 frames and a second slab.  A Rademacher C gives exact
integers (255 m < 2^24), compared with the oracle's."""
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


@pytest.mark.parametrize("m,n,k,pad", [(1, 2, 1, 1), (31, 33, 65, 4), (32, 64, 64, 1), (33, 96, 63, 4), (64, 128, 5, 1),
                                       (1541, 160, 100, 1), (12321, 192, 130, 4), (9999, 224, 70, 1),
                                       (20000, 256, 66, 4), (4097, 257, 64, 1)])
def test_chunk_edges_are_exact(C, m, n, k, pad):
    ctx = C.Context(0)
    buf = np.random.default_rng(m + n).integers(0, 256, size=(n, -(-m // pad) * pad), dtype=np.uint8)
    D = torch.from_numpy(buf).cuda()[:, :m]
    DY = C.cdmd_sketch(ctx, D, k, 3 + k, ctype="rademacher", prec="fp32")
    C.cdmd_status_sync(ctx)
    Cm = M.measurement_matrix("rademacher", 3 + k, k, m)
    assert np.array_equal(DY.cpu().numpy(), O.sketch(Cm, buf[:, :m].T.astype(np.float64)).T)
