"""Windows launched kernel by kernel, where a kernel may start before the one
ahead of it has ended, against the same windows from a captured graph, whose
kernels start one after another.

A call that exports the surface is launched kernel by kernel and one that does
not replays a graph; the arithmetic is the same, so the flows are equal bit for
bit.  The calls follow one another without a synchronisation, on the default
stream and on another, at sizes from a single level to several, with levels too
small for a patch and with windows without events.
"""
import numpy as np
import pytest

from paper_2112_10591_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


def _dev(a):
    return torch.from_numpy(np.ascontiguousarray(a)).to("cuda")


@pytest.mark.parametrize("storage", ["fp32", "fp16"])
@pytest.mark.parametrize("W,H,sor,other", [
    (16, 16, 5, False), (40, 33, 0, True), (97, 61, 5, True), (346, 260, 3, False),
    (1000, 700, 5, True)])
def test_kernel_by_kernel_is_the_graph(W, H, sor, other, storage):
    import paper_2112_10591_gb300 as eb
    n = 6
    ev = synth.translating_segments(width=W, height=H, n_windows=n, n_segments=10,
                                    events_per_window=max(300, W * H // 9), seed=W + H)
    wins = []
    for k in range(n):
        x, y, t, _, tb, te = ev.window(k)
        if k == 2:
            x, y, t = x[:0], y[:0], t[:0]
        wins.append((_dev(x), _dev(y), _dev(t), tb, te))
    cs = torch.cuda.Stream() if other else None
    flows = []
    for export in (False, True):
        p = eb.ebof_default_params(W, H)
        p.var_sor = sor
        p.storage = 1 if storage == "fp16" else 0
        st, s = eb.ebof_stream_create(p, 0)
        eb.check(st)
        flow = torch.zeros((n, 2, H, W), dtype=torch.float32, device="cuda")
        surface = torch.zeros((n, H, W), dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        for k, (x, y, t, tb, te) in enumerate(wins):
            eb.check(eb.ebof_process_window(s, x, y, t, None, tb, te, flow[k], None, None,
                                            surface[k] if export else None, cs))
        torch.cuda.synchronize()
        flows.append(flow.cpu().numpy())
        s.close()
    assert np.array_equal(flows[0], flows[1])
