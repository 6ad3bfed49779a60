"""The one-launch refinement of a level when its waits run out.

A wait bound of 0 (ebof_stream_set_wait_limit) ends the polls for the flow of
other regions at once: the blocks leave with work claimed and undone, the stream
reports EBOF_ERR_TIMEOUT, and the counters and tags that the launch leaves behind
serve the next launches: after a reset the flows equal a fresh stream's bit for
bit.  Levels of one region, of several and of more than a wave of them; launched
kernel by kernel (an export) and, with the bound set first, in a graph.
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


def _run(eb, s, ev, n, edge):
    flow = torch.zeros((n, 2, ev.height, ev.width), dtype=torch.float32, device="cuda")
    mask = torch.zeros((ev.height, ev.width), dtype=torch.uint8, device="cuda") if edge else None
    for k in range(n):
        x, y, t, _, tb, te = ev.window(k)
        st = eb.ebof_process_window(s, _dev(x), _dev(y), _dev(t), None, tb, te, flow[k],
                                    edge=mask)
        assert st == (eb.EBOF_NO_PREVIOUS if k == 0 else eb.EBOF_OK)
    return eb.ebof_stream_sync(s, 1)[0], flow


@pytest.mark.parametrize("W,H,outer", [(46, 46, 2), (139, 93, 5), (346, 260, 3), (640, 480, 2)])
def test_polls_that_run_out_are_reported_and_the_stream_recovers(eb, W, H, outer):
    n = 4
    ev = synth.translating_segments(width=W, height=H, n_windows=n, n_segments=14,
                                    events_per_window=max(600, W * H // 6), seed=W)
    p = eb.ebof_default_params(W, H)
    p.var_outer = outer
    s, ref = (eb.ebof_stream_create(p, 0)[1] for _ in range(2))
    st, want = _run(eb, ref, ev, n, True)
    assert st == eb.EBOF_OK and float(want[-1].abs().max()) > 0
    for _ in range(2):
        assert eb.ebof_stream_reset(s) == eb.EBOF_OK
        assert eb.ebof_stream_set_wait_limit(s, 0) == eb.EBOF_OK
        assert _run(eb, s, ev, n, True)[0] == eb.EBOF_ERR_TIMEOUT
        torch.cuda.synchronize()  # the context is intact
        assert eb.ebof_stream_sync(s, 1)[0] == eb.EBOF_OK
        assert eb.ebof_stream_set_wait_limit(s, -1) == eb.EBOF_OK
        assert eb.ebof_stream_reset(s) == eb.EBOF_OK
        st, flow = _run(eb, s, ev, n, True)
        assert st == eb.EBOF_OK and torch.equal(flow, want)
    s.close()
    ref.close()


def test_a_captured_bound_runs_out_too(eb):
    W, H, n = 139, 93, 4
    ev = synth.translating_segments(width=W, height=H, n_windows=n, n_segments=14,
                                    events_per_window=3000, seed=3)
    p = eb.ebof_default_params(W, H)
    s, other = (eb.ebof_stream_create(p, 0)[1] for _ in range(2))
    st, want = _run(eb, other, ev, n, False)
    assert st == eb.EBOF_OK
    assert eb.ebof_stream_set_wait_limit(s, 0) == eb.EBOF_OK
    assert _run(eb, s, ev, n, False)[0] == eb.EBOF_ERR_TIMEOUT
    assert eb.ebof_stream_reset(s) == eb.EBOF_OK
    assert _run(eb, s, ev, n, False)[0] == eb.EBOF_ERR_TIMEOUT
    # kernel by kernel at the default bound: the counters serve both
    assert eb.ebof_stream_set_wait_limit(s, -1) == eb.EBOF_OK
    assert eb.ebof_stream_reset(s) == eb.EBOF_OK
    st, flow = _run(eb, s, ev, n, True)
    assert st == eb.EBOF_OK and torch.equal(flow, want)
    s.close()
    other.close()
