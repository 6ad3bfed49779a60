"""The Flow Warping Loss's variances against exact sums of its own images.

The call leaves I_comp and I_uncomp at the start of its scratch.  Their moments
are summed here in rational arithmetic; with u = 2^-53 the call, whose sums are
those of doubles or better, rounds each moment at most 3 times up to four blocks'
sums, the mean and the square once more each, and the difference once:
|var - exact| <= 4 u E[I^2] + 9 u E[I]^2 + u var <= 10 u (E[I^2] + E[I]^2).
"""
from fractions import Fraction

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


@pytest.mark.parametrize("W,H,n", [(3, 1, 9), (32, 32, 3000), (31, 33, 400), (64, 64, 20000)])
@pytest.mark.parametrize("seed", range(6))
def test_variances_are_as_exact_as_sums_in_double(eb, W, H, n, seed):
    rng = np.random.default_rng(seed)
    x = rng.integers(0, W, n).astype(np.uint16)
    y = rng.integers(0, H, n).astype(np.uint16)
    t = np.sort(rng.integers(0, 10000, n)).astype(np.int64)
    p = np.where(rng.random(n) < 0.8, 1, -1).astype(np.int8)
    U = rng.uniform(-3.0, 3.0, (2, H, W)).astype(np.float32)
    dev = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (x, y, t, p, U)]
    scratch = torch.empty(eb.ebof_fwl_scratch_bytes(W, H), dtype=torch.uint8, device="cuda")
    st, out = eb.ebof_fwl(*dev[:4], 0, 10000, dev[4], W, H, scratch)
    eb.check(st)
    out = out.cpu().numpy()
    P, plane = W * H, (4 * W * H + 255) // 256 * 256
    for k in range(2):
        img = scratch[k * plane:k * plane + 4 * P].cpu().numpy().view(np.float32)
        v = [Fraction(float(a)) for a in img]
        m1, m2 = sum(v) / P, sum(a * a for a in v) / P
        var = m2 - m1 * m1
        assert abs(Fraction(float(out[1 + k])) - var) <= Fraction(10, 2 ** 53) * (m2 + m1 * m1)
