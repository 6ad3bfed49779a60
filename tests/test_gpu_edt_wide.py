"""The stand-alone EDT of low and wide images.

Its rows start while its columns end where the column blocks leave SMs enough
for them.  On both sides of that rule the squared distances are the exact ones;
and where they leave few, as at 4096 columns, 300 rows must not take longer than
700 (rows that start early crowd the few SMs left: 82 us for 300 of them).
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


def _call(eb, E):
    H, W = E.shape
    e = torch.from_numpy(E).cuda()
    scratch = torch.empty((H, W), dtype=torch.int32, device="cuda")
    edt = torch.empty_like(scratch)
    return edt, lambda: eb.check(eb.ebof_edt(e, W, H, scratch, edt, None))


@pytest.mark.parametrize("W,H", [(1000, 200), (2048, 300), (4096, 27), (4096, 300), (4800, 2),
                                 (4864, 9), (4900, 40), (8192, 200)])
def test_wide_images_are_exact(eb, W, H):
    ndimage = pytest.importorskip("scipy.ndimage")
    E = (np.random.default_rng(W + H).random((H, W)) < 0.01).astype(np.uint8)
    i = ndimage.distance_transform_edt(E == 0, return_distances=False, return_indices=True)
    y, x = np.indices(E.shape)
    edt, run = _call(eb, E)
    for _ in range(3):  # a call's columns behind the rows of the one before
        run()
    assert np.array_equal(edt.cpu().numpy(), (i[0] - y) ** 2 + (i[1] - x) ** 2)


def test_fewer_rows_do_not_take_longer(eb):
    def us(H):
        _, run = _call(eb, (np.random.default_rng(H).random((H, 4096)) < 0.03).astype(np.uint8))
        best = float("inf")
        for _ in range(6):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            torch.cuda._sleep(200000)
            a.record()
            for _ in range(20):
                run()
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b) * 1000 / 20)
        return best

    assert us(300) <= 1.1 * us(700)
