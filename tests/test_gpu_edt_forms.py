"""The EDT's two passes at the sizes where their tiles and words end.

Column pass: 32-row words (heights around 32, one word, several), 32-column
blocks.  Row pass: 32-pixel bands, quads of columns, the levels of the owner
search (widths around 32, 128, 256, 1024), single frames (four warps a row) and
batches (one warp a row), rows whose only edge pixel lies at one end, columns
without edge pixels, images without any.  Squared distances are integers and
must equal scipy's exact transform; the surface is Eq. 1 of them within 1e-6.
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
    d = ndimage.distance_transform_edt(E == 0, return_distances=False, return_indices=True)
    y, x = np.indices(E.shape)
    return (d[0] - y) ** 2 + (d[1] - x) ** 2


def _images(rng, W, H):
    E = np.zeros((H, W), np.uint8)
    yield E
    for y, x in ((0, 0), (H - 1, W - 1), (H // 2, 0), (0, W - 1)):
        F = E.copy()
        F[y, x] = 1
        yield F
    for share in (0.001, 0.02, 0.3):
        yield (rng.random((H, W)) < share).astype(np.uint8)
    F = E.copy()
    F[:, W // 3] = 1  # one full column: the others have none
    yield F
    F = E.copy()
    F[H // 3] = 1
    yield F


@pytest.mark.parametrize("W,H", [(1, 1), (1, 40), (40, 1), (31, 31), (32, 32), (33, 33), (64, 65),
                                 (97, 31), (128, 64), (129, 96), (257, 33), (300, 257),
                                 (1023, 70), (1025, 97), (2049, 34), (35, 1030)])
def test_edt_is_exact(eb, W, H):
    rng = np.random.default_rng(W * 5000 + H)
    for E in _images(rng, W, H):
        D = _exact(E)
        e = torch.from_numpy(np.ascontiguousarray(E)).cuda()
        scratch = torch.empty((H, W), dtype=torch.int32, device="cuda")
        edt = torch.empty((H, W), dtype=torch.int32, device="cuda")
        surf = torch.empty((H, W), dtype=torch.float32, device="cuda")
        eb.check(eb.ebof_edt(e, W, H, scratch, edt, surf))
        assert np.array_equal(edt.cpu().numpy(), D)
        S = np.where(D == 2147483647, 1.0, 1.0 - np.exp(-np.sqrt(D.astype(np.float64)) / 1.08))
        assert np.abs(surf.cpu().numpy() - S).max() <= 1e-6
        # the scratch given as the result: read off the edge image
        eb.check(eb.ebof_edt(e, W, H, scratch, scratch, None))
        assert np.array_equal(scratch.cpu().numpy(), D)


@pytest.mark.parametrize("W,H", [(33, 31), (129, 65), (346, 260), (1025, 40)])
def test_batched_rows_are_exact(eb, W, H):
    """Three windows a call take one warp a row: the same distances."""
    n = 3
    rng = np.random.default_rng(W + H)
    p = eb.ebof_default_params(W, H)
    p.max_batch, p.n_d = n, 0
    st, s = eb.ebof_stream_create(p, 0)
    eb.check(st)
    E = [(rng.random((H, W)) < share).astype(np.uint8) for share in (0.0, 0.004, 0.2)]
    y, x = np.concatenate([np.argwhere(f) for f in E]).T
    t = np.concatenate([np.full(int(f.sum()), 10000 * k) for k, f in enumerate(E)])
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda()
           for a in (x.astype(np.uint16), y.astype(np.uint16), t.astype(np.int64))]
    flow = torch.empty((n, 2, H, W), dtype=torch.float32, device="cuda")
    edt = torch.empty((n, H, W), dtype=torch.int32, device="cuda")
    eb.check(eb.ebof_process_windows(s, n, *dev, None, 0, 10000, flow, edt=edt))
    eb.check(eb.ebof_stream_sync(s, 1)[0])
    for k in range(n):
        assert np.array_equal(edt[k].cpu().numpy(), _exact(E[k])), k
    s.close()
