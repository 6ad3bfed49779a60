"""The SOR sweeps' three forms at every kind of halo.

A region's halo is 2 sweeps - 1 pixels and its interior 64 minus twice that, so
the sweep count sets where regions lie, the boxes of the tensor copies and their
offsets.  Calls of several frames, whose grids meet the rule that is under test:
at least a region per SM for the copy-ahead kernel (sor_tma_min_per_sm = 1), two
rows a strip within any number of waves (sor_row_waves), 64 x 64 regions with
neither.  Their flows are equal bit for bit, at widths and heights just under, at
and just over whole interiors, and the first is the oracle's within the fixed
0.05 px mean endpoint error of the parity tests.
"""
import numpy as np
import pytest

import oracle
from paper_2112_10591_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

NEVER = 1 << 20


@pytest.fixture(scope="module")
def eb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2112_10591_gb300 as m
    m.load()
    return m


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


# interiors: 62 (0 and 1 sweeps), 58, 54, 46, 18
@pytest.mark.parametrize("W,H,sor,batch", [
    (187, 125, 0, 16), (186, 124, 1, 28), (249, 187, 1, 8), (175, 117, 2, 16), (163, 109, 3, 16),
    (162, 161, 3, 18), (139, 93, 5, 16), (138, 137, 5, 18), (73, 91, 12, 6), (54, 37, 12, 20)])
@pytest.mark.parametrize("storage", [0, 1])
def test_sor_forms_agree_at_every_halo(eb, W, H, sor, batch, storage):
    R = 2 * sor - 1 if sor else 1
    tile = 64 - 2 * R
    regions = -(-W // tile) * -(-H // tile) * batch
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    assert regions >= sms  # the copy-ahead form's rule at level 0
    layouts = [{"sor_tma_min_per_sm": 1}, {"sor_tma_min_per_sm": NEVER, "sor_row_waves": 0}]
    if 32 - 2 * R >= 8:  # 64 x 32 regions have at least eight interior rows
        layouts.append({"sor_tma_min_per_sm": NEVER, "sor_row_waves": NEVER})
    ev = synth.translating_segments(width=W, height=H, n_windows=batch + 1, n_segments=14,
                                    events_per_window=max(600, W * H // 6), seed=W + sor)
    flows = []
    for layout in layouts:
        p = eb.ebof_default_params(W, H)
        p.var_sor, p.max_batch, p.storage = sor, batch, storage
        for k, v in layout.items():
            setattr(p, k, v)
        st, s = eb.ebof_stream_create(p, 0)
        eb.check(st)
        flow = torch.zeros((batch, 2, H, W), dtype=torch.float32, device="cuda")
        x, y, t, _, tb, te = ev.window(0)
        eb.check(eb.ebof_process_window(s, _dev(x), _dev(y), _dev(t), None, tb, te, flow[0]))
        a, b = int(ev.offsets[1]), int(ev.offsets[1 + batch])
        eb.check(eb.ebof_process_windows(s, batch, _dev(ev.x[a:b]), _dev(ev.y[a:b]),
                                         _dev(ev.t[a:b]), None, int(ev.t_begin[1]), ev.dt, flow))
        eb.check(eb.ebof_stream_sync(s, 1)[0])
        flows.append(flow.cpu().numpy())
        s.close()
    for layout, f in zip(layouts[1:], flows[1:]):
        assert np.array_equal(f, flows[0]), layout
    if storage == 0:
        w0, w1 = ev.window(0), ev.window(1)
        U = oracle.process_pair(W, H, (w0[0], w0[1], w0[2], w0[4], w0[5]),
                                (w1[0], w1[1], w1[2], w1[4], w1[5]), levels=p.levels,
                                patch=p.patch, var_sor=sor)[2]
        F = flows[0][0]
        assert np.hypot(F[0] - U[0], F[1] - U[1]).mean() <= 0.05
