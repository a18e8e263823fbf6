"""Two host threads with a context each, whose calls need different amounts of
shared memory of the same kernels: no call of either is refused, whatever the
other sets between its preparation and its launch."""
import threading

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

ROUNDS = 6000


@pytest.fixture(scope="module")
def C():
    from paper_1512_04205_gb300 import build, cdmd
    if not torch.cuda.is_available():
        pytest.fail("CUDA device required for -m gpu tests")
    build.build()
    return cdmd


def _video(n, m, ldd):
    return torch.randint(0, 256, (n, ldd), dtype=torch.uint8, device="cuda")[:, :m]


def _subtract(C, ctx, n, m, ldd, ncols):
    D = _video(n, m, ldd)
    Phi = torch.randn((m, ncols, 2), device="cuda")
    lam = torch.tensor([[0.9, 0.0]] * ncols, dtype=torch.float64, device="cuda")
    mask = torch.empty((n, (m + 31) // 32), dtype=torch.int32, device="cuda")
    bg = torch.empty((n, m), dtype=torch.float32, device="cuda")
    return lambda: C.cdmd_subtract(ctx, D, Phi, lam, lam, 25.0, want_bg=True, mask=mask, bg=bg)


def _sketch(C, ctx, n):
    D = _video(n, 640, 640)
    DY = torch.empty((n, 64), dtype=torch.float64, device="cuda")
    return lambda: C.cdmd_sketch(ctx, D, 64, 3, prec="bf16x2", DY=DY)


@pytest.mark.parametrize("what", ["staged subtract", "plain subtract", "sketch"])
def test_calls_of_two_threads(C, what):
    ctxs = [C.Context(0), C.Context(0)]
    if what == "staged subtract":
        calls = [_subtract(C, ctxs[0], 512, 64, 64, 12), _subtract(C, ctxs[1], 2, 64, 64, 12)]
    elif what == "plain subtract":
        calls = [_subtract(C, ctxs[0], 512, 63, 63, 30), _subtract(C, ctxs[1], 2, 63, 63, 30)]
    else:
        calls = [_sketch(C, ctxs[0], 256), _sketch(C, ctxs[1], 16)]
    for call in calls:
        call()
    torch.cuda.synchronize()
    errors, start = [], threading.Barrier(2)

    def work(call):
        torch.zeros(1, device="cuda")      # the thread's CUDA context
        start.wait()
        for _ in range(ROUNDS):
            try:
                call()
            except C.CdmdError as e:
                errors.append(str(e))

    threads = [threading.Thread(target=work, args=(c,)) for c in calls]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    torch.cuda.synchronize()
    for ctx in ctxs:
        C.cdmd_status_sync(ctx)
    assert not errors, (len(errors), errors[0])


@pytest.mark.parametrize("prec", ["fp32", "bf16x2"])
def test_first_call_of_a_thread(C, prec):
    # a thread's first CUDA call may be the library's: a sketch whose workspace exists
    # starts with the tensor map of the video
    ctx = C.Context(0)
    D = _video(40, 640, 640)
    DY = torch.empty((40, 64), dtype=torch.float64, device="cuda")
    stream = torch.cuda.current_stream()
    C.cdmd_sketch(ctx, D, 64, 3, prec=prec, DY=DY, stream=stream)
    torch.cuda.synchronize()
    want, errors = DY.clone(), []
    DY.zero_()

    def work():
        try:
            C.cdmd_sketch(ctx, D, 64, 3, prec=prec, DY=DY, stream=stream)
        except C.CdmdError as e:
            errors.append(str(e))

    torch.cuda.synchronize()
    t = threading.Thread(target=work)
    t.start()
    t.join()
    torch.cuda.synchronize()
    assert not errors, errors
    assert torch.equal(DY, want)
