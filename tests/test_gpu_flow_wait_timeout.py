"""The copy-ahead SOR kernel when a region's flow comes too late.

The bound of that wait alone is set to 0 (ebof_debug_flow_wait_limit): the
coefficients arrive, the sweeps run, and the flow's wait runs out.  A block with
a further region reports it at that region's start, a block without one at its
end; both let the copies in flight land first.  ebof_stream_sync reports
EBOF_ERR_TIMEOUT and, after a reset, the flows equal a fresh stream's bit for
bit.
"""
import numpy as np
import pytest

from paper_2112_10591_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def eb():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2112_10591_gb300 as m
    m.load()
    return m


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


def _run(eb, s, ev, n):
    flow = torch.zeros((n, 2, ev.height, ev.width), dtype=torch.float32, device="cuda")
    x, y, t, _, tb, te = ev.window(0)
    assert eb.ebof_process_window(s, _dev(x), _dev(y), _dev(t), None, tb, te,
                                  flow[0]) == eb.EBOF_NO_PREVIOUS
    a, b = int(ev.offsets[1]), int(ev.offsets[1 + n])
    eb.check(eb.ebof_process_windows(s, n, _dev(ev.x[a:b]), _dev(ev.y[a:b]), _dev(ev.t[a:b]),
                                     None, int(ev.t_begin[1]), ev.dt, flow))
    return eb.ebof_stream_sync(s, 1)[0], flow


# regions of level 0 (48 a frame of 346 x 260) from one an SM on: 192 leave most
# blocks with one region, 336 give every block two or three
@pytest.mark.parametrize("n", [4, 7])
def test_a_late_flow_is_reported_and_the_stream_recovers(eb, n):
    ev = synth.translating_segments(n_windows=n + 1, seed=5)
    p = eb.ebof_default_params(ev.width, ev.height)
    p.max_batch, p.sor_tma_min_per_sm = n, 1
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    tile = 64 - 2 * (2 * p.var_sor - 1)
    assert -(-ev.width // tile) * -(-ev.height // tile) * n >= sms
    s, ref = (eb.ebof_stream_create(p, 0)[1] for _ in range(2))
    st, want = _run(eb, ref, ev, n)
    assert st == eb.EBOF_OK and float(want[-1].abs().max()) > 0
    for _ in range(2):
        assert eb.ebof_stream_reset(s) == eb.EBOF_OK
        assert eb.ebof_debug_flow_wait_limit(s, 0) == eb.EBOF_OK
        assert _run(eb, s, ev, n)[0] == eb.EBOF_ERR_TIMEOUT
        torch.cuda.synchronize()  # the context is intact
        assert eb.ebof_debug_flow_wait_limit(s, -1) == eb.EBOF_OK
        assert eb.ebof_stream_reset(s) == eb.EBOF_OK
        st, flow = _run(eb, s, ev, n)
        assert st == eb.EBOF_OK and torch.equal(flow, want)
    s.close()
    ref.close()
