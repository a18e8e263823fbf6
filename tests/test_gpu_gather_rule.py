"""Which of its two kernels the sparse gather takes.  The packed one is exact at the
sizes it is taken at (row counts on both sides of its two layouts, reached on few
SMs, where one CTA has many pixels, and the ends of the rule's ranges), and a call
whose frames are 4-byte aligned takes no longer than the same call on frames that
are not, which only the plain one serves."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

from test_gpu_gather_packed import C, _check, _draw  # noqa: E402,F401


@pytest.mark.parametrize("m,n,k,density,sms", [
    (12289, 64, 2048, 0.0015, 1), (12290, 17, 2049, 0.0015, 1), (30003, 40, 3400, 0.001, 1),   # 18 warps; 16 frames
    (3071, 33, 16, 0.004, 0), (3073, 33, 16, 0.004, 0), (6145, 31, 16, 0.004, 0),              # a round and past it
    (20001, 40, 1000, 1e-6, 0), (20001, 24, 1000, 0.0099, 2), (20001, 23, 1000, 0.0099, 2)])   # ends of the ranges
def test_both_kernels_are_exact(C, m, n, k, density, sms):  # noqa: F811
    ctx = C.Context(0)
    C.cdmd_set_sm_limit(ctx, sms)
    rng = np.random.default_rng(m + n + k)
    col_ptr, row_idx = _draw(rng, m, k, density)
    _check(C, ctx, m, n, k, col_ptr, row_idx, density, seed=m)


def _median_us(call, reps=25):
    for _ in range(3):
        call()
    times = []
    for _ in range(reps):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        a.record()
        call()
        b.record()
        b.synchronize()
        times.append(a.elapsed_time(b) * 1e3)
    return sorted(times)[reps // 2]


@pytest.mark.parametrize("m,n,k,density", [(57600, 8, 1000, 9e-3), (76800, 64, 2048, 2e-3), (345600, 300, 2100, 9e-3),
                                           (2073600, 2, 1000, 9e-3)])
def test_aligned_frames_are_no_slower(C, m, n, k, density):  # noqa: F811
    ctx = C.Context(0)
    meas = C.Measure(ctx, "sparse", m, k, 3, density=density)
    buf = torch.randint(0, 256, (n * (m + 4) + 1,), dtype=torch.uint8, device="cuda")
    DY = torch.empty((n, k), dtype=torch.float64, device="cuda")
    aligned, odd = (buf[o:o + n * (m + 4)].view(n, m + 4)[:, :m] for o in (0, 1))
    fast = _median_us(lambda: C.cdmd_sketch_gather(ctx, aligned, meas, DY=DY))
    general = _median_us(lambda: C.cdmd_sketch_gather(ctx, odd, meas, DY=DY))
    assert fast <= 1.2 * general + 5.0, (fast, general)      # the same kernel twice at these sizes
