"""A batch of more clips than a grid has rows (65,535): tiny clips of one video, so
that every one of them has the mask of the first."""
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

import videogen  # noqa: E402


@pytest.fixture(scope="module")
def C():
    from paper_1512_04205_gb300 import build, cdmd
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    build.build()
    return cdmd


def test_more_clips_than_grid_rows(C):
    # waves get equal work, so three larger clips (each the work of all the tiny ones)
    # leave the fourth wave to those
    clips, n, m = 65600, 3, 64
    small = dict(D=torch.from_numpy(videogen.make_clip(8, 8, n, seed=3).frames).cuda(), k=4, r=1, K=1, seed=5)
    large = dict(D=torch.from_numpy(videogen.make_clip(64, 64, 200, seed=4).frames).cuda(), k=64, r=4, K=2, seed=5)
    args = dict(prec="fp32", selector="omp", graph=False, grouped=True)
    one = C.Batch([small], 2.0, **args)
    one.run()
    one.status_sync()
    want = one.masks[0].clone()
    one.close()
    assert small["D"].shape == (n, m)
    b = C.Batch([large] * 3 + [small] * clips, 2.0, **args)
    b.status_sync()
    assert b.tuning()["waves"] == 4
    looked_at = (3, 4, 65535, 65536, 65537, 65538, clips + 2)
    for i in looked_at:
        b.masks[i].fill_(-1)
    b.run()
    b.status_sync()
    for i in looked_at:
        assert torch.equal(b.masks[i], want), i
    b.close()
