"""A context whose workspace the largest decomposition has sized serves smaller
ones under stream capture, where nothing can be allocated: the room of the small
solves does not grow when n or k falls."""
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


def _sketch(n, k):
    rng = np.random.default_rng(n + k)
    return torch.from_numpy(rng.standard_normal((n, k)) * np.linspace(1.0, 2.0, n)[:, None]).cuda()


@pytest.mark.parametrize("largest,smaller", [((256, 1000), [(224, 1000), (200, 900), (256, 700), (33, 1000)]),
                                             ((512, 800), [(512, 680), (480, 800), (100, 500)]),
                                             ((300, 5000), [(290, 5000), (300, 1000), (64, 4000)])])
def test_smaller_problems_capture_after_the_largest(C, largest, smaller):
    ctx = C.Context(0)
    r, K = 6, 3
    C.cdmd_decompose(ctx, _sketch(*largest), r, K)
    C.cdmd_status_sync(ctx)
    for n, k in smaller:
        DY = _sketch(n, k)
        out = C.decompose_outputs(n, k, r, K, "cuda")
        g = torch.cuda.CUDAGraph()
        torch.cuda.synchronize()
        with torch.cuda.graph(g):
            C.cdmd_decompose(ctx, DY, r, K, out=out)
        g.replay()
        torch.cuda.synchronize()
        C.cdmd_status_sync(ctx)
        s = np.linalg.svd(DY.cpu().numpy()[:-1], compute_uv=False)[:r]
        assert np.allclose(out["sigma"].cpu().numpy(), s, rtol=1e-12, atol=0.0)


@pytest.mark.parametrize("n,k", [(33, 3000), (60, 250000), (512, 20000)])
def test_long_sketches(C, n, k):
    # chunks past 256 rows (n = 60, k = 250000; n = 512, k = 20000): the Gram's rounding
    # is that of its blocks of 256, far below sqrt(k) eps
    ctx = C.Context(0)
    DY = _sketch(n, k)
    out = C.cdmd_decompose(ctx, DY, 5, 2)
    C.cdmd_status_sync(ctx)
    s = np.linalg.svd(DY.cpu().numpy()[:-1], compute_uv=False)[:5]
    assert np.allclose(out["sigma"].cpu().numpy(), s, rtol=1e-12, atol=0.0)
