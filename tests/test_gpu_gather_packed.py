"""The packed gather sketch (sparse C, 4-byte aligned frames) at the edges of
its tiles: frames per slab, 128-pixel tiles, ragged last pixels, both row
layouts, and rows that collect more entries than a 16-bit sum holds, spread
over the clip (accumulators emptied in between) or packed into one round (added
to the partials directly).  Exact integers, against numpy."""
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


@pytest.fixture(scope="module")
def ctx(C):
    return C.Context(0)


class _Given:
    """A SPARSE measurement matrix from given CSC arrays."""

    def __init__(self, C, m, k, col_ptr, row_idx, density):
        self.col_ptr = torch.from_numpy(col_ptr.astype(np.int64)).cuda()
        self.row_idx = torch.from_numpy(row_idx.astype(np.uint32).view(np.int32)).cuda()
        self.struct = C.cdmd_measure(C.CTYPES["sparse"], k, m, 0, density, self.col_ptr.data_ptr(),
                                     self.row_idx.data_ptr(), self.row_idx.numel(), None)


def _check(C, ctx, m, n, k, col_ptr, row_idx, density, seed, pad=4, high=False):
    rng = np.random.default_rng(seed)
    ldd = -(-m // pad) * pad
    buf = rng.integers(200 if high else 0, 256, size=(n, ldd), dtype=np.uint8)
    D = torch.from_numpy(buf).cuda()[:, :m]
    DY = C.cdmd_sketch_gather(ctx, D, _Given(C, m, k, col_ptr, row_idx, density))
    C.cdmd_status_sync(ctx)
    rows = (row_idx & 0x7FFFFFFF).astype(np.int64)
    sign = np.where(row_idx >> 31, -1, 1)
    pix = np.repeat(np.arange(m), np.diff(col_ptr))
    want = np.zeros((n, k), dtype=np.int64)
    vals = buf[:, :m].astype(np.int64)
    for t in range(n):
        np.add.at(want[t], rows, sign * vals[t, pix])
    assert np.array_equal(DY.cpu().numpy(), want.astype(np.float64))


def _draw(rng, m, k, density):
    cnt = rng.binomial(k, density, size=m)
    cnt[m // 2] = max(cnt[m // 2], 1)          # an empty C is refused
    col_ptr = np.concatenate([[0], np.cumsum(cnt)])
    row_idx = np.concatenate([np.sort(rng.choice(k, c, replace=False)) for c in cnt if c] or [np.zeros(0, int)])
    return col_ptr, (row_idx | (rng.integers(0, 2, row_idx.size) << 31)).astype(np.uint32)


@pytest.mark.parametrize("m,n,k", [(1, 2, 1), (127, 31, 5), (128, 32, 7), (129, 33, 1023), (5000, 65, 100),
                                   (12289, 64, 2048), (12290, 17, 2049), (30003, 40, 3400), (70001, 100, 33)])
def test_packed_gather_is_exact(C, ctx, m, n, k):
    rng = np.random.default_rng(m + n + k)
    col_ptr, row_idx = _draw(rng, m, k, min(0.008, 40.0 / k))
    _check(C, ctx, m, n, k, col_ptr, row_idx, 0.008, seed=m)


def test_row_sums_past_sixteen_bits(C, ctx):
    # every pixel adds to row 3 with one sign: far past 128 entries per round
    # and per CTA, the case a random C of this density never brings
    m, n, k = 40000, 35, 9
    _check(C, ctx, m, n, k, np.arange(m + 1), np.full(m, 3, np.uint32), 0.001, seed=1, high=True)
    _check(C, ctx, m, n, k, np.arange(m + 1), np.full(m, 3 | 0x80000000, np.uint32), 0.001, seed=2, high=True)
    # one pixel in twelve: below the limit within a round, past it over several
    col_ptr = np.concatenate([[0], np.cumsum(np.arange(m) % 40 == 0)])
    _check(C, ctx, m, n, k, col_ptr, np.full(int(col_ptr[-1]), 5, np.uint32), 0.001, seed=3, high=True)


@pytest.mark.parametrize("pad", [1, 2])
def test_unaligned_frames_take_the_plain_kernel(C, ctx, pad):
    rng = np.random.default_rng(9)
    m, n, k = 1001, 37, 50
    col_ptr, row_idx = _draw(rng, m, k, 0.02)
    _check(C, ctx, m, n, k, col_ptr, row_idx, 0.005, seed=4, pad=pad)
