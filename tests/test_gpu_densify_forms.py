"""Densification with one pixel a thread and with two.

Grids of many blocks (a call of many windows) take two pixels a thread where the
stride is even and divides the patch; a window alone takes one.  The arithmetic
is the same, so the flows are equal bit for bit: with two, three and four
patches a pixel and axis, at widths and heights around the tiles of 32 x 16 and
at odd ones, where the flush patches cover part of a tile, and in both storages.
"""
import numpy as np
import pytest

from paper_2112_10591_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


@pytest.mark.parametrize("storage", [0, 1])
@pytest.mark.parametrize("W,H,patch,stride,n", [
    (199, 131, 12, 4, 21), (192, 128, 8, 4, 26), (225, 145, 16, 4, 18), (161, 97, 12, 6, 35),
    (130, 127, 4, 2, 34), (199, 131, 12, 5, 21)])
def test_two_pixels_a_thread_are_one(W, H, patch, stride, n, storage):
    import paper_2112_10591_gb300 as eb
    assert -(-W // 32) * -(-H // 8) * n >= 2432
    ev = synth.translating_segments(width=W, height=H, n_windows=n + 1, n_segments=12,
                                    events_per_window=W * H // 8, seed=W + patch)
    flows = []
    for batch in (1, n):
        p = eb.ebof_default_params(W, H)
        p.patch, p.stride, p.storage, p.max_batch = patch, stride, storage, batch
        st, s = eb.ebof_stream_create(p, 0)
        eb.check(st)
        flow = torch.zeros((n + 1, 2, H, W), dtype=torch.float32, device="cuda")
        first = [(0, 1)]
        for k, m in first + [(i, batch) for i in range(1, n + 1, batch)]:
            a, b = int(ev.offsets[k]), int(ev.offsets[k + m])
            eb.check(eb.ebof_process_windows(s, m, _dev(ev.x[a:b]), _dev(ev.y[a:b]),
                                             _dev(ev.t[a:b]), None, int(ev.t_begin[k]), ev.dt,
                                             flow[k:k + m]))
        eb.check(eb.ebof_stream_sync(s, 1)[0])
        flows.append(flow.cpu().numpy())
        s.close()
    assert np.array_equal(flows[0], flows[1])
    assert np.abs(flows[0][1:]).max() > 0
