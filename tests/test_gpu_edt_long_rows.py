"""The EDT of images with long rows and few of them.

Rows of 2048 pixels and more that are no more than the SMs take sixteen warps
each instead of four.  On both sides of that rule, with and without edge pixels,
with a scratch of its own and in a result, and inside a window of either
storage, the squared distances are the exact ones; and four rows of 16384
pixels, which have the chip to themselves, take at most a fifth of the time of
1024 (with four warps a row it was three tenths).
"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def eb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2112_10591_gb300 as m
    m.load()
    return m


def _exact(E):
    ndimage = pytest.importorskip("scipy.ndimage")
    if not E.any():
        return np.full(E.shape, 2147483647, np.int64)
    i = ndimage.distance_transform_edt(E == 0, return_distances=False, return_indices=True)
    y, x = np.indices(E.shape)
    return (i[0] - y) ** 2 + (i[1] - x) ** 2


def _images(W, H):
    rng = np.random.default_rng(W + H)
    E = np.zeros((H, W), np.uint8)
    yield E
    for x in (0, W - 1, W // 3):
        F = E.copy()
        F[H // 2, x] = 1
        yield F
    for share in (0.0005, 0.05):
        yield (rng.random((H, W)) < share).astype(np.uint8)


@pytest.mark.parametrize("W,H", [(2047, 9), (2048, 1), (2048, 152), (2048, 153), (2049, 33),
                                 (4100, 7), (8191, 2), (16384, 1), (16384, 40)])
def test_long_rows_are_exact(eb, W, H):
    for E in _images(W, H):
        D = _exact(E)
        e = torch.from_numpy(np.ascontiguousarray(E)).cuda()
        scratch = torch.empty((H, W), dtype=torch.int32, device="cuda")
        edt = torch.empty_like(scratch)
        eb.check(eb.ebof_edt(e, W, H, scratch, edt, None))
        assert np.array_equal(edt.cpu().numpy(), D)
        eb.check(eb.ebof_edt(e, W, H, scratch, scratch, None))
        assert np.array_equal(scratch.cpu().numpy(), D)


@pytest.mark.parametrize("storage", [0, 1])
def test_long_rows_of_a_window_are_exact(eb, storage):
    W, H = 2100, 21
    rng = np.random.default_rng(7)
    E = (rng.random((H, W)) < 0.01).astype(np.uint8)
    p = eb.ebof_default_params(W, H)
    p.n_d, p.storage = 0, storage
    st, s = eb.ebof_stream_create(p, 0)
    eb.check(st)
    y, x = np.argwhere(E).T
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
           for a in (x.astype(np.uint16), y.astype(np.uint16), np.zeros(len(x), np.int64))]
    flow = torch.empty((2, H, W), dtype=torch.float32, device="cuda")
    edt = torch.empty((H, W), dtype=torch.int32, device="cuda")
    assert eb.ebof_process_window(s, *dev, None, 0, 10000, flow, edt=edt) == eb.EBOF_NO_PREVIOUS
    eb.check(eb.ebof_stream_sync(s, 1)[0])
    assert np.array_equal(edt.cpu().numpy(), _exact(E))
    s.close()


def test_a_few_long_rows_have_the_chip_to_themselves(eb):
    W = 16384

    def us(H):
        e = torch.from_numpy((np.random.default_rng(H).random((H, W)) < 0.03).astype(np.uint8))
        e = e.cuda()
        scratch = torch.empty((H, W), dtype=torch.int32, device="cuda")
        edt = torch.empty_like(scratch)
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(200000)
            a.record()
            for _ in range(10):
                eb.check(eb.ebof_edt(e, W, H, scratch, edt, None))
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 1000 / 10)
        return best

    assert us(4) <= 0.2 * us(1024)
