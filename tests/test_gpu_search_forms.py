"""The patch search where its warps' tiles end and its early stop acts.

A warp serves a tile of patches (4 x 2, 2 x 2, one) and stops once none of them
moves any more, so patch grids that do not fill the tiles, images whose patches
are all flat (guarded), flat on one side or all textured, and iteration counts
from none to the default are each compared with the oracle: 0.05 px mean
endpoint error; a flat image's flow is exactly zero.
"""
import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def eb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2112_10591_gb300 as m
    m.load()
    return m


def _surface(W, H, kind, shift):
    y, x = np.mgrid[0:H, 0:W].astype(np.float64)
    s = 0.5 + 0.25 * np.sin(0.31 * (x - shift)) * np.cos(0.27 * y) + 0.2 * np.sin(0.11 * x + 0.4 * y)
    if kind == "flat":
        s[:] = 0.5
    elif kind == "left":
        s[:, W // 2:] = 0.5
    return s.astype(np.float32)


def _flow(eb, W, H, kind, iters, patch, stride, storage):
    p = eb.ebof_default_params(W, H)
    p.levels, p.patch, p.stride, p.gn_iters, p.storage = 1, patch, stride, iters, storage
    p.var_outer = 0
    st, s = eb.ebof_stream_create(p, 0)
    eb.check(st)
    flow = torch.empty((2, H, W), dtype=torch.float32, device="cuda")
    for shift in (0.0, 0.8):
        eb.check(eb.ebof_process_surface(s, torch.from_numpy(_surface(W, H, kind, shift)).cuda(),
                                         flow))
    eb.check(eb.ebof_stream_sync(s, 1)[0])
    s.close()
    return flow.cpu().numpy()


@pytest.mark.parametrize("W,H,patch,stride", [
    (12, 12, 12, 4), (17, 13, 12, 4), (45, 29, 12, 4), (61, 53, 12, 5), (33, 41, 8, 4),
    (30, 27, 8, 3), (64, 48, 16, 6),
    (370, 365, 12, 4)])  # 91 x 90 patches: the first grid of the wide layout
@pytest.mark.parametrize("kind", ["flat", "left", "full"])
@pytest.mark.parametrize("storage", [0, 1])
def test_search_matches_the_oracle(eb, W, H, patch, stride, kind, storage):
    s0, s1 = (_surface(W, H, kind, k).astype(np.float64) * 255.0 for k in (0.0, 0.8))
    for iters in (0, 1, 12):
        f = _flow(eb, W, H, kind, iters, patch, stride, storage)
        U = oracle.flow(s0, s1, levels=1, patch=patch, stride=stride, gn_iters=iters,
                        var_outer=0)
        assert np.hypot(f[0] - U[0], f[1] - U[1]).mean() <= 0.05
    if kind == "flat":
        assert not f.any()
