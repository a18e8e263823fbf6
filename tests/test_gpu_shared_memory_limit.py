"""A shared run whose clips' small solves do not fit into the device's free memory side
by side solves them one after another: the results are those of the clips' own runs."""
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


def test_solves_one_after_another_when_memory_is_short(C):
    # eight clips of 512 frames, k = 1000: about 40 MB of workspace for the solves of each
    w, h, n, k, r, K, clips = 32, 24, 512, 1000, 8, 4, 8
    Ds = [torch.from_numpy(videogen.make_clip(w, h, n, seed=70 + i).frames).cuda() for i in range(clips)]
    p = C.make_params(k, r, K, 25.0, seed=2, prec="fp32", selector="omp")
    ctx = C.Context(0)                                # with a single clip's workspace
    want = [C.cdmd_run(ctx, D, p) for D in Ds]
    modes = C.workspace_tensors(ctx, w * h, n, k, r, K)
    masks = [torch.empty_like(m) for m in want]
    C.cdmd_status_sync(ctx)
    torch.cuda.empty_cache()
    leave = 112 << 20                                 # for the eight sketches and one clip's solves
    ballast = torch.empty(torch.cuda.mem_get_info()[0] - leave, dtype=torch.uint8, device="cuda")
    try:
        C.cdmd_run_shared(ctx, Ds, p, masks=masks)
        C.cdmd_status_sync(ctx)
    finally:
        del ballast
        torch.cuda.empty_cache()
    for a, b in zip(masks, want):
        assert torch.equal(a, b)
    got = C.workspace_tensors(ctx, w * h, n, k, r, K)
    for q in ("sigma", "lam", "G", "beta", "sel"):
        assert torch.equal(got[q], modes[q]), q
    ctx.close()
