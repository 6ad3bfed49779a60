"""The stand-alone EDT with a scratch that is one of its results, or lies across them.

Column distances are then kept in a result, in place.  The squared distances and
the surface equal, bit for bit, those of a call with a buffer of its own, at the
sizes where the column words and the rows' bands end; the edge image may lie in
the result that holds no distances.  An image without edge pixels costs a pass
over the image, not one over a column for every pixel: 4096 x 4096 within ten
times the call with a separate buffer (a column walk a pixel: several hundred).
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


def _ints(n):
    return torch.empty(n, dtype=torch.int32, device="cuda")


@pytest.mark.parametrize("W,H", [(1, 1), (40, 1), (1, 40), (31, 32), (33, 33), (97, 31), (64, 65),
                                 (129, 96), (1025, 97), (35, 1030), (16384, 3), (2, 16384)])
def test_scratch_in_a_result(eb, W, H):
    rng = np.random.default_rng(W + 3 * H)
    n = W * H
    for share in (0.0, 0.002, 0.05, 0.6):
        e = torch.from_numpy((rng.random((H, W)) < share).astype(np.uint8)).cuda()
        D, S = _ints(n), _ints(n).view(torch.float32)
        eb.check(eb.ebof_edt(e, W, H, _ints(n), D, S))

        def same(edge, scratch, d, s):
            eb.check(eb.ebof_edt(edge, W, H, scratch, d, s))
            return torch.equal(d, D) and (s is None or torch.equal(s, S))

        a, b = _ints(n), _ints(n)
        assert same(e, a, a, None)
        assert same(e, a, a, b.view(torch.float32))
        assert same(e, b, a, b.view(torch.float32))
        # across both results, half a plane off
        c = _ints(2 * n)
        assert same(e, c[n // 2:n // 2 + n], c[:n], c[n:].view(torch.float32))
        # the edge image in the result that is not the scratch
        a.view(torch.uint8)[:n] = e.flatten()
        assert same(a.view(torch.uint8)[:n], b, a, b.view(torch.float32))
        b.view(torch.uint8)[-n:] = e.flatten()
        assert same(b.view(torch.uint8)[-n:], a, a, b.view(torch.float32))
        if n > 1:
            # ... and the scratch half in the other one
            c[:n].view(torch.uint8)[:n] = e.flatten()
            if n // 2 * 4 >= n:
                assert same(c[:n].view(torch.uint8)[:n], c[n // 2:n // 2 + n], c[:n],
                            c[n:].view(torch.float32))


def test_an_empty_image_costs_a_pass(eb):
    W = H = 4096
    e = torch.zeros((H, W), dtype=torch.uint8, device="cuda")
    scratch, d = _ints(W * H), _ints(W * H)

    def ms(buf):
        a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
        best = float("inf")
        for _ in range(4):
            a.record()
            eb.check(eb.ebof_edt(e, W, H, buf, d, None))
            b.record()
            torch.cuda.synchronize()
            best = min(best, a.elapsed_time(b))
        return best

    assert ms(d) <= 10.0 * ms(scratch)
    assert int(d.min()) == 2147483647
