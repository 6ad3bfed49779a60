"""The variational refinement's kernel forms against one another and the oracle.

Every layout setting tiles the same per-pixel arithmetic, so all of them give
the same flow bit for bit: at widths and heights around multiples of a SOR
region's interior (64 minus twice the halo 2 sweeps - 1), at odd sizes, with
regions that hold one level whole, and at sweep counts from none to the most
that a region's halo allows.  The flow is the oracle's within the fixed
0.05 px mean endpoint error of the parity tests.
"""
import numpy as np
import pytest

import oracle
from paper_2112_10591_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")

LAYOUTS = ({}, {"sor_tma_min_per_sm": 1}, {"sor_tma_min_per_sm": 1 << 20, "sor_row_waves": 0},
           {"sor_tma_min_per_sm": 1 << 20, "sor_row_waves": 64}, {"var_cluster_max": 16},
           {"coeff_cw_min_width": 1}, {"coeff_cw_min_width": 1, "coeff_cw_rows": 4},
           {"coeff_cw_min_width": 1 << 20, "coeff_cw_rows": 16})


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


@pytest.fixture(scope="module")
def eb():
    import paper_2112_10591_gb300 as m
    return m


@pytest.mark.parametrize("W,H,sor,batch", [
    (46, 46, 5, 1), (47, 93, 5, 1), (92, 45, 5, 1), (139, 47, 5, 1), (185, 138, 5, 3),
    (61, 33, 0, 1), (126, 63, 1, 1), (95, 70, 12, 1), (230, 131, 3, 2), (321, 247, 5, 8)])
def test_forms_agree_and_match_the_oracle(eb, W, H, sor, batch):
    ev = synth.translating_segments(width=W, height=H, n_windows=batch + 1, n_segments=14,
                                    events_per_window=max(600, W * H // 6), seed=W + H)
    flows = []
    for layout in LAYOUTS:
        p = eb.ebof_default_params(W, H)
        p.var_sor = sor
        p.max_batch = batch
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
    for layout, f in zip(LAYOUTS[1:], flows[1:]):
        assert np.array_equal(f, flows[0]), layout
    w0, w1 = ev.window(0), ev.window(1)
    U = oracle.process_pair(W, H, (w0[0], w0[1], w0[2], w0[4], w0[5]),
                            (w1[0], w1[1], w1[2], w1[4], w1[5]), levels=p.levels, patch=p.patch,
                            var_sor=sor)[2]
    F = flows[0][0]
    assert np.hypot(F[0] - U[0], F[1] - U[1]).mean() <= 0.05


@pytest.mark.parametrize("W,H,sor,outer", [
    (46, 46, 5, 2), (93, 47, 5, 1), (139, 185, 5, 5), (71, 353, 0, 3), (230, 131, 3, 4),
    (346, 260, 5, 5), (645, 479, 5, 5), (873, 645, 5, 2)])
def test_one_launch_a_level_is_a_launch_an_iteration(eb, W, H, sor, outer):
    """Windows one by one (small levels in one launch) and three a call (a
    launch per iteration): equal bit for bit, with levels of one region, of
    several, of more than a wave of them and of too many; twice, so that the
    second pass starts from the packets and counters of the first."""
    n = 3
    ev = synth.translating_segments(width=W, height=H, n_windows=2 * n + 1, n_segments=14,
                                    events_per_window=max(600, W * H // 8), seed=W + outer)
    flows = []
    for batch in (1, n):
        p = eb.ebof_default_params(W, H)
        p.var_sor, p.var_outer, p.max_batch = sor, outer, batch
        st, s = eb.ebof_stream_create(p, 0)
        eb.check(st)
        flow = torch.zeros((2 * n + 1, 2, H, W), dtype=torch.float32, device="cuda")
        for k in range(0, 2 * n + 1, batch if flows else 1):
            m = min(batch, 2 * n + 1 - k)
            a, b = int(ev.offsets[k]), int(ev.offsets[k + m])
            eb.check(eb.ebof_process_windows(s, m, _dev(ev.x[a:b]), _dev(ev.y[a:b]),
                                             _dev(ev.t[a:b]), None, int(ev.t_begin[k]), ev.dt,
                                             flow[k:k + m]))
        eb.check(eb.ebof_stream_sync(s, 1)[0])
        flows.append(flow.cpu().numpy())
        s.close()
    assert np.array_equal(flows[0], flows[1])
    assert np.abs(flows[0][-1]).max() > 0
