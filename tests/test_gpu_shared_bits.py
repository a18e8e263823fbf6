"""A clip's small solves in company (FP32 sketches are per clip, so every stage sees
the inputs of the clip's own run).  The sums over the sketch rows are split by the
tiles of all clips of a call: with rows for one split only, every bit is that of the
clip's own run, also where clips on both sides of 257 frames share the launches, whose
reflectors go in blocks of 32 and of 16; with several splits the results agree to
the rounding of the sums.  Each clip takes its turn as the last, whose results the
context shows."""
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


@pytest.mark.parametrize("ns,k", [((30, 260), 64), ((257, 130, 258), 50), ((40, 256, 33, 90, 100), 64),
                                  ((100,) * 8, 60),
                                  ((200, 200, 200, 200, 200), 1000), ((200, 61, 130), 1000), ((257, 130, 258), 333),
                                  ((120, 120), 4099)])
def test_solves_in_company(C, ns, k):
    w, h, r, K = 64, 48, 8, 4
    ctx = C.Context(0)
    clips = [torch.from_numpy(videogen.make_clip(w, h, n, seed=50 + i).frames).cuda() for i, n in enumerate(ns)]
    p = C.make_params(k, r, K, 25.0, seed=9, prec="fp32", selector="omp")
    for last in range(len(ns) if len(set(ns)) > 1 else 1):
        order = [i for i in range(len(ns)) if i != last] + [last]
        masks = C.cdmd_run_shared(ctx, [clips[i] for i in order], p)
        got = C.workspace_tensors(ctx, w * h, ns[last], k, r, K)
        solo = [C.cdmd_run(ctx, clips[i], p) for i in order]
        want = C.workspace_tensors(ctx, w * h, ns[last], k, r, K)
        C.cdmd_status_sync(ctx)
        assert torch.equal(got["DY"], want["DY"])
        if k <= 64:
            for a, b in zip(masks, solo):
                assert torch.equal(a, b)
            for q in ("sigma", "lam", "G", "beta", "sel", "nsel", "Phi"):
                assert torch.equal(got[q], want[q]), (q, ns[last])
        else:
            # the Gram rounds by some eps of the largest eigenvalue, sigma_1^2
            s2 = got["sigma"] ** 2
            assert ((s2 - want["sigma"] ** 2).abs() <= 32 * 2.0 ** -52 * s2[0]).all()
            assert torch.equal(got["sel"][:1], want["sel"][:1])
