"""The median of masks whose rows are whole words, on clips long enough that a
thread walks a strip of more than four rows: strips that divide the height and
not, a last strip of one row, heights below the strip.  Bit for bit against the
oracle, first, middle and last frame."""
import numpy as np
import pytest

from oracle import cdmd as O

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def C():
    from paper_1512_04205_gb300 import build, cdmd
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    build.build()
    return cdmd


@pytest.mark.parametrize("W,H,n", [(64, 333, 900), (32, 2051, 1000), (1920, 46, 1500), (96, 33, 38000), (32, 17, 220000)])
def test_long_strips_match_oracle(C, W, H, n):
    ctx = C.Context(0)
    m = W * H
    g = torch.Generator(device="cuda").manual_seed(W + H)
    words = torch.randint(-2 ** 31, 2 ** 31 - 1, (n, m // 32), dtype=torch.int32, device="cuda", generator=g)
    out = C.cdmd_median3x3(ctx, words, W, H)
    pick = [0, 1, n // 2, n - 1]
    mask = C.unpack_mask(words[pick], m)
    got = out[pick].cpu().numpy().view(np.uint32)
    assert np.array_equal(got, O.pack_mask(O.median3x3_mask(mask, W, H)))
