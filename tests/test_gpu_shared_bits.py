"""A clip's small solves give the same bits whichever clips share the launches
(FP32 sketches are per clip, so every stage sees the same inputs).  Unlike a k of
one Gram block, these k are summed in several, whose size must not follow the
companions' lengths, and clips on both sides of 257 frames apply their reflectors
in blocks of 32 and of 16; each clip takes its turn as the last, whose results the
context shows."""
import numpy as np
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


@pytest.mark.parametrize("ns,k", [((200, 200, 200), 1000), ((200, 61, 130), 1000), ((40, 256, 33, 90, 100), 333),
                                  ((100,) * 8, 700), ((120, 120), 4099),
                                  ((30, 260), 300), ((257, 130, 258), 200)])
def test_solves_keep_their_bits_in_company(C, ns, k):
    w, h, r, K = 64, 48, 8, 4
    ctx = C.Context(0)
    clips = [torch.from_numpy(videogen.make_clip(w, h, n, seed=50 + i).frames).cuda() for i, n in enumerate(ns)]
    p = C.make_params(k, r, K, 25.0, seed=9, prec="fp32", selector="omp")
    for last in range(len(ns) if len(set(ns)) > 1 else 1):
        order = [i for i in range(len(ns)) if i != last] + [last]
        masks = C.cdmd_run_shared(ctx, [clips[i] for i in order], p)
        got = C.workspace_tensors(ctx, w * h, ns[last], k, r, K)
        for i, mk in zip(order, masks):
            assert torch.equal(mk, C.cdmd_run(ctx, clips[i], p)), i
        want = C.workspace_tensors(ctx, w * h, ns[last], k, r, K)
        C.cdmd_status_sync(ctx)
        for q in ("DY", "sigma", "lam", "G", "beta", "sel", "nsel", "Phi"):
            assert torch.equal(got[q], want[q]), (q, ns[last])
