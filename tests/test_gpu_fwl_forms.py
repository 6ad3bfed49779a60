"""The Flow Warping Loss at the sizes where its sums' passes end.

Images below one quad, below one block's pixels, of a pixel count that is no
multiple of four, and of more than one pass of the grid; scratch that is and is
not aligned to 16 bytes (quads and single loads); votes at odd and even columns
and across the borders.  The same gate as the other FWL tests: 1e-5 relative to
the FP64 oracle on the same flow (the votes' weights are FP32).
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


@pytest.mark.parametrize("W,H,n", [(2, 1, 5), (3, 1, 7), (5, 3, 40), (33, 31, 2000),
                                   (346, 260, 20000), (1601, 901, 60000)])
@pytest.mark.parametrize("offset", [0, 8])
def test_fwl_matches_oracle(eb, W, H, n, offset):
    rng = np.random.default_rng(W * H + n)
    x = rng.integers(0, W, n).astype(np.uint16)
    y = rng.integers(0, H, n).astype(np.uint16)
    t = np.sort(rng.integers(0, 10000, n)).astype(np.int64)
    p = np.where(rng.random(n) < 0.7, 1, -1).astype(np.int8)
    U = rng.uniform(-3.0, 3.0, (2, H, W)).astype(np.float32)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, y, t, p, U)]
    raw = torch.empty(eb.ebof_fwl_scratch_bytes(W, H) + 256, dtype=torch.uint8, device="cuda")
    st, out = eb.ebof_fwl(*dev[:4], 0, 10000, dev[4], W, H, raw[offset:])
    eb.check(st)
    o = oracle.fwl(W, H, x, y, t, p, 0, 10000, U.astype(np.float64))
    assert np.allclose(out.cpu().numpy(), o, rtol=1e-5, atol=0.0)
