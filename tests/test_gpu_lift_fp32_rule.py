"""Tile width and frame batches of the FP32 lift: results where the rule takes tiles
of eight (few frames, a large output) are those of the equal tiles, bit for bit
(a sum runs over the frames in order whatever the tile), aligned or not, and
neither few frames with many modes nor unaligned frames cost what they do not have to."""
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


def _inputs(m, n, ncols, pad, seed=0):
    gen = torch.Generator(device="cuda")
    gen.manual_seed(seed + m + n)
    ldd = -(-m // pad) * pad
    D = torch.randint(0, 256, (n, ldd), dtype=torch.uint8, device="cuda", generator=gen)[:, :m]
    G = torch.randn((ncols, n - 1, 2), dtype=torch.float64, device="cuda", generator=gen)
    return D, G


@pytest.mark.parametrize("pad", [1, 4])
@pytest.mark.parametrize("m,n,ncols", [(87383, 24, 13), (87383, 25, 13), (80661, 40, 28), (80661, 41, 28),
                                       (116511, 12, 9), (116511, 13, 9), (52430, 5, 20)])
def test_tiles_agree(C, m, n, ncols, pad):
    ctx = C.Context(0)
    D, G = _inputs(m, n, ncols, pad)
    got = C.cdmd_lift(ctx, D, G, prec="fp32")
    for c in range(ncols):      # one mode at a time: a tile of one
        assert torch.equal(got[:, c], C.cdmd_lift(ctx, D, G[c:c + 1].contiguous(), prec="fp32")[:, 0]), c
    want = D[1:].double().T @ G.permute(1, 0, 2).reshape(n - 1, -1)
    bound = (n + 1) * 2.0 ** -24 * (D[1:].double().T @ G.abs().permute(1, 0, 2).reshape(n - 1, -1))
    assert ((got.reshape(m, -1).double() - want).abs() <= bound + 1e-30).all()


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


@pytest.mark.parametrize("n,few,many", [(5, 24, 28), (5, 16, 20)])
def test_a_few_more_modes_cost_a_little_more(C, n, few, many):
    # 10^6 pixels, bound by the stores: time follows the number of modes
    ctx = C.Context(0)
    us = []
    for ncols in (few, many):
        D, G = _inputs(1000000, n, ncols, 4)
        Phi = torch.empty((1000000, ncols, 2), device="cuda")
        us.append(_median_us(lambda: C.cdmd_lift(ctx, D, G, prec="fp32", Phi=Phi)))
    assert us[1] <= 1.4 * us[0] * many / few, us


def test_unaligned_frames(C):
    ctx = C.Context(0)
    us = []
    for pad in (4, 1):
        D, G = _inputs(230401, 200, 13, pad)
        Phi = torch.empty((230401, 13, 2), device="cuda")
        us.append(_median_us(lambda: C.cdmd_lift(ctx, D, G, prec="fp32", Phi=Phi)))
    assert us[1] <= 1.15 * us[0], us
