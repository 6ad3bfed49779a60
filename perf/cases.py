"""Performance cases of the event-to-flow path: what its users call, and at which sizes.

Every case goes through the public entry points of paper_2112_10591_gb300
(the C ABI by its Python binding) on synthetic event streams: rigid objects
made of line segments that move and turn, plus uniform noise, as in the
package's own workloads.  A stream's windows form a ring (the objects' motion
over the ring adds up to zero), so a pass that feeds the whole ring leaves the
stream where it found it.

``exact`` restates the method in 64-bit torch from its definition: edge image,
Alg. 1 and Alg. 2, exact EDT, surface, and the Dense Inverse Search flow.
"""
import math

import numpy as np
import torch

import paper_2112_10591_gb300 as eb

DEVICE = "cuda:0"
WINDOW_US = 10_000
INF_D = 2147483647


# ------------------------------------------------------------------ the cases
def listed():
    return [
        # a small sensor's edge image to its distance transform and surface,
        # called on its own: the smallest call, where launches count
        {"name": "edt_346x260", "kind": "edt", "width": 346, "height": 260, "density": 0.22},
        # the same entry on a full-HD image
        {"name": "edt_1920x1080", "kind": "edt", "width": 1920, "height": 1080, "density": 0.3},
        # quality of a flow without ground truth, one 1280x720 window
        {"name": "fwl_1280x720", "kind": "fwl", "width": 1280, "height": 720, "density": 0.3},
        # one low-resolution camera in real time: each window in order
        {"name": "window_346x260", "kind": "window", "width": 346, "height": 260, "windows": 2,
         "density": 0.22},
        # one high-resolution camera in real time
        {"name": "window_1280x720", "kind": "window", "width": 1280, "height": 720, "windows": 2,
         "density": 0.3},
        # a cropped sensor with odd sizes, the 4-neighbour settings, and every
        # optional output (edge mask, squared distances, surface)
        {"name": "exports_613x397", "kind": "exports", "width": 613, "height": 397, "windows": 2,
         "density": 0.2, "connectivity": 4, "n_d": 2, "n_f": 3},
        # the flow block alone, on surfaces the caller computed
        {"name": "surface_641x479", "kind": "surface", "width": 641, "height": 479, "windows": 2,
         "density": 0.25},
        # throughput of one high-resolution stream, flows collected later
        {"name": "pipelined_1280x720", "kind": "pipelined", "width": 1280, "height": 720,
         "windows": 12, "density": 0.3},
        # the same from and to page-locked host memory
        {"name": "host_1280x720", "kind": "host", "width": 1280, "height": 720, "windows": 8,
         "density": 0.3},
        # recorded data in large batches: the largest call
        {"name": "windows_1280x720_x40", "kind": "windows", "width": 1280, "height": 720,
         "windows": 40, "density": 0.3},
        # a server's batch of one stream's backlog, FP16 storage
        {"name": "list_640x480_x8_fp16", "kind": "list", "width": 640, "height": 480,
         "windows": 8, "density": 0.3, "storage": "fp16"},
        # many cameras of two resolutions stepped together, FP16 storage, the
        # patch grids that the autotuner picks for them
        {"name": "multigroup_12+4_fp16", "kind": "multigroup", "width": 346, "height": 260,
         "streams": 12, "width2": 1280, "height2": 720, "streams2": 4, "windows": 2,
         "density": 0.3, "storage": "fp16", "patch": 8, "stride": 6, "patch2": 8, "stride2": 4},
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """A case of the same ranges: every entry point, sensor sizes from 64 px to
    1280x720 (EDT: to 4096 px), both storages, the options in use."""
    kind = rng.choice(["edt", "fwl", "window", "exports", "surface", "pipelined", "host",
                       "windows", "list", "multigroup"])
    c = {"kind": kind, "density": round(rng.uniform(0.05, 0.4), 3)}
    if kind in ("edt", "fwl"):
        top = 4096 if kind == "edt" else 1920
        c["width"] = _log(rng, 32, top)
        c["height"] = max(16, int(c["width"] * rng.uniform(0.4, 1.0)))
        return c
    c["width"] = _log(rng, 64, 1280)
    c["height"] = min(720, max(48, int(c["width"] * rng.uniform(0.5, 0.85))))
    c["storage"] = rng.choice(["fp32", "fp32", "fp16"])
    if rng.random() < 0.3:
        c["patch"] = rng.choice([8, 12])
        c["stride"] = rng.choice([4, 6])
    if rng.random() < 0.3:
        c.update(connectivity=4, n_d=rng.choice([1, 2]), n_f=rng.choice([3, 4]))
    c["windows"] = {"window": 2, "exports": 2, "surface": 2, "multigroup": 2,
                    "pipelined": rng.randint(4, 16), "host": rng.randint(3, 9),
                    "windows": _log(rng, 2, 32), "list": rng.randint(2, 8)}[kind]
    if kind == "multigroup":
        c["streams"] = rng.randint(2, 8)
        c["width2"] = _log(rng, 200, 1280)
        c["height2"] = min(720, max(120, int(c["width2"] * rng.uniform(0.5, 0.85))))
        c["streams2"] = rng.randint(1, 4)
    return c


def _options(case, second=False):
    """Every method parameter of a case (the library's defaults where the case
    names none)."""
    w = case["width2" if second else "width"]
    h = case["height2" if second else "height"]
    big = w >= 640
    conn = case.get("connectivity", 8)
    return {
        "width": w, "height": h, "connectivity": conn, "n_d": case.get("n_d", 1),
        "n_f": case.get("n_f", conn + 1), "alpha": 1.08, "levels": 5 if big else 3,
        "patch": case.get("patch2" if second else "patch", 12 if big else 8),
        "stride": case.get("stride2" if second else "stride", 4),
        "gn_iters": 12, "gn_damping": 0.1, "var_outer": 5, "var_sor": 5, "var_delta": 5.0,
        "var_gamma": 10.0, "var_alpha": 20.0, "sor_omega": 1.6,
        "storage": eb.EBOF_STORAGE_FP16 if case.get("storage") == "fp16"
        else eb.EBOF_STORAGE_FP32,
    }


def _params(opt, max_batch=1):
    p = eb.ebof_default_params(opt["width"], opt["height"])
    for k, v in opt.items():
        setattr(p, k, v)
    p.max_batch = max_batch
    return p


# ------------------------------------------------------------------- the data
def _events(W, H, windows, density, seed):
    """`windows` windows of 10 ms of a W x H stream as CUDA tensors: x, y
    (uint16), t (int64, sorted), p (int8) and the windows' offsets.  Objects
    are polygons of segments with a motion and a turn drawn anew per window
    (at most 1/64 of the width and 2 degrees), summing to zero over the ring;
    the windows hold 0.55 to 1.45 times density * W * H events, 3 % noise."""
    rng = np.random.default_rng([seed, W, H, windows])
    scale = W / 1280.0
    n_obj = max(3, int(round(12 * math.sqrt(W * H / 921600.0))))
    n_edge = 25 * n_obj
    centre = rng.random((n_obj, 2)) * [W, H]
    obj = rng.integers(0, n_obj, n_edge)
    r = rng.uniform(40.0, 200.0, n_edge) * scale * np.sqrt(rng.random(n_edge))
    phi = rng.uniform(0, 2 * math.pi, n_edge)
    p0 = centre[obj] + np.stack([r * np.cos(phi), r * np.sin(phi)], 1)
    ln, ang = rng.uniform(10.0, 120.0, n_edge) * scale, rng.uniform(0, 2 * math.pi, n_edge)
    p1 = p0 + np.stack([ln * np.cos(ang), ln * np.sin(ang)], 1)
    # +- 1/64 of the width: 20 px at 1280
    step = rng.uniform(-W / 64.0, W / 64.0, (windows, n_obj, 2))
    turn = np.deg2rad(rng.uniform(-2.0, 2.0, (windows, n_obj)))
    step -= step.mean(0)
    turn -= turn.mean(0)
    shift = np.concatenate([np.zeros((1, n_obj, 2)), np.cumsum(step, 0)])
    theta = np.concatenate([np.zeros((1, n_obj)), np.cumsum(turn, 0)])
    counts = np.maximum(1, (rng.uniform(0.55, 1.45, windows) * density * W * H)).astype(np.int64)

    dev = torch.device(DEVICE)
    g = torch.Generator(device=dev)
    g.manual_seed(int(rng.integers(1 << 40)))

    def up(a):
        return torch.from_numpy(np.ascontiguousarray(a)).to(dev)

    sign = up(np.where(np.arange(n_edge) % 2 == 0, 1, -1))
    p0, p1, obj, centre, shift, theta = map(up, (p0, p1, obj, centre, shift, theta))
    cdf = torch.cumsum(up(ln / ln.sum()), 0)
    n = int(counts.max()) * 2  # drawn per window: enough are on the image
    xs, ys, ts, ps, offsets = [], [], [], [], [0]
    for k in range(windows):
        e = torch.searchsorted(cdf, torch.rand(n, device=dev, generator=g,
                                               dtype=torch.float64)).clamp_(max=n_edge - 1)
        s = torch.rand(n, device=dev, generator=g, dtype=torch.float64)
        t = torch.randint(0, WINDOW_US, (n,), device=dev, generator=g)
        f = t.double() / WINDOW_US
        o = obj[e]
        th = torch.lerp(theta[k][o], theta[k + 1][o], f)
        sh = torch.lerp(shift[k][o], shift[k + 1][o], f[:, None])
        rel = torch.lerp(p0[e], p1[e], s[:, None]) - centre[o]
        c, sn = torch.cos(th), torch.sin(th)
        x = torch.floor(centre[o, 0] + c * rel[:, 0] - sn * rel[:, 1] + sh[:, 0] + 0.5).long()
        y = torch.floor(centre[o, 1] + sn * rel[:, 0] + c * rel[:, 1] + sh[:, 1] + 0.5).long()
        flip = torch.rand(n, device=dev, generator=g) < 0.1
        p = torch.where(flip, -sign[e], sign[e])
        noise = torch.rand(n, device=dev, generator=g) < 0.03
        x = torch.where(noise, torch.randint(0, W, (n,), device=dev, generator=g), x)
        y = torch.where(noise, torch.randint(0, H, (n,), device=dev, generator=g), y)
        keep = ((x >= 0) & (x < W) & (y >= 0) & (y < H)).nonzero()[:int(counts[k]), 0]
        keep = keep[torch.sort(t[keep], stable=True)[1]]
        xs.append(x[keep])
        ys.append(y[keep])
        ts.append(t[keep] + k * WINDOW_US)
        ps.append(p[keep])
        offsets.append(offsets[-1] + len(keep))
    return (torch.cat(xs).to(torch.int16).view(torch.uint16),
            torch.cat(ys).to(torch.int16).view(torch.uint16), torch.cat(ts),
            torch.cat(ps).to(torch.int8), offsets)


def _windows(ev):
    x, y, t, _, off = ev
    return [(x[a:b], y[a:b], t[a:b], k * WINDOW_US, (k + 1) * WINDOW_US)
            for k, (a, b) in enumerate(zip(off[:-1], off[1:]))]


def _edge_images(ev, W, H):
    """[windows][H][W] uint8: the pixels that an event of the window fell on."""
    out = torch.zeros((len(ev[4]) - 1, H, W), dtype=torch.uint8, device=DEVICE)
    flat = out.view(-1)
    x, y = ev[0].view(torch.int16).long(), ev[1].view(torch.int16).long()
    flat[(ev[2] // WINDOW_US) * (W * H) + y * W + x] = 1
    return out


def _smooth_surfaces(ev, W, H, alpha):
    """Surfaces as another front end computes them: exact Eq. 1, rounded to FP32."""
    d = _edt(_edge_images(ev, W, H))
    return (1.0 - torch.exp(-torch.sqrt(d.double()) / alpha)).float().contiguous()


def _streams_of(case, seed):
    """(options, [events of each stream]) of each group of a multigroup case."""
    got = []
    for second in (False, True):
        opt = _options(case, second)
        n = case["streams2" if second else "streams"]
        got.append((opt, [_events(opt["width"], opt["height"], case["windows"], case["density"],
                                  seed * 1000 + 100 * second + i) for i in range(n)]))
    return got


class _DeviceView:
    """A float32 device buffer of the library's, for torch.as_tensor (which keeps
    this object, and so the buffer's owners)."""

    def __init__(self, address, shape, owners):
        self.owners = owners
        self.__cuda_array_interface__ = {"data": (address, False), "shape": shape,
                                         "typestr": "<f4", "version": 3, "strides": None}


def _pinned(t):
    h = torch.empty(t.shape, dtype=t.dtype, pin_memory=True)
    h.copy_(t)
    return h


def _ok(status, what):
    if status < 0:
        raise eb.EbofError(status, what)
    return status


def prepare(case, seed):
    kind, dens = case["kind"], case["density"]
    dev = torch.device(DEVICE)
    torch.cuda.set_device(dev)
    s = {"kind": kind}
    if kind == "multigroup":
        s["groups"], s["steps"], s["out"] = [], [], []
        for opt, evs in _streams_of(case, seed):
            st, g = eb.ebof_group_create(_params(opt), len(evs), 0)
            _ok(st, "ebof_group_create")
            s["groups"].append(g)
            s["steps"].append([_windows(ev) for ev in evs])
        st, s["mg"] = eb.ebof_multigroup_create(s["groups"])
        _ok(st, "ebof_multigroup_create")
        last = case["windows"] - 1
        _ok(eb.ebof_multigroup_process(s["mg"], [[w[last] for w in g] for g in s["steps"]]),
            "ebof_multigroup_process")
        s["steps"] = [[[w[k] for w in g] for g in s["steps"]] for k in range(case["windows"])]
        for g in s["groups"]:
            s["out"].append(torch.as_tensor(
                _DeviceView(eb.ebof_group_flow(g, 0), (g.n, 2, g.params.height, g.params.width),
                            (g, s["mg"])), device=dev))
        return s

    opt = _options(case)
    W, H, K = opt["width"], opt["height"], case.get("windows", 1)
    s["W"], s["H"], s["K"] = W, H, K
    ev = _events(W, H, K, dens, seed)
    if kind == "edt":
        s["edge"] = _edge_images(ev, W, H)[0].contiguous()
        s["scratch"] = torch.empty((H, W), dtype=torch.int32, device=dev)
        s["edt"] = torch.empty((H, W), dtype=torch.int32, device=dev)
        s["surface"] = torch.empty((H, W), dtype=torch.float32, device=dev)
        return s
    if kind == "fwl":
        s["ev"] = ev
        s["flow"] = _some_flow(W, H, seed)
        s["scratch"] = torch.empty(eb.ebof_fwl_scratch_bytes(W, H), dtype=torch.uint8, device=dev)
        s["out"] = torch.empty(3, dtype=torch.float64, device=dev)
        return s

    batch = K if kind in ("windows", "list") else 1
    st, s["stream"] = eb.ebof_stream_create(_params(opt, batch), 0)
    _ok(st, "ebof_stream_create")
    wins = _windows(ev)
    flows = torch.zeros((K, 2, H, W), dtype=torch.float32, device=dev)
    s["flows"], s["flow"] = flows, list(flows.unbind(0))
    if kind == "surface":
        s["in"] = list(_smooth_surfaces(ev, W, H, opt["alpha"]).unbind(0))
        _ok(eb.ebof_process_surface(s["stream"], s["in"][-1], s["flow"][0]),
            "ebof_process_surface")
    else:
        x, y, t, tb, te = wins[-1]
        _ok(eb.ebof_process_window(s["stream"], x, y, t, None, tb, te, s["flow"][0]),
            "ebof_process_window")
    s["ev"], s["wins"] = ev, wins
    if kind == "exports":
        s["edge"] = [torch.empty((H, W), dtype=torch.uint8, device=dev) for _ in range(K)]
        s["edt"] = [torch.empty((H, W), dtype=torch.int32, device=dev) for _ in range(K)]
        s["surface"] = [torch.empty((H, W), dtype=torch.float32, device=dev) for _ in range(K)]
    if kind == "host":
        hx, hy, ht = _pinned(ev[0].view(torch.int16)), _pinned(ev[1].view(torch.int16)), \
            _pinned(ev[2])
        hx, hy, ht = hx.numpy().view(np.uint16), hy.numpy().view(np.uint16), ht.numpy()
        off = ev[4]
        s["wins"] = [(hx[a:b], hy[a:b], ht[a:b], k * WINDOW_US, (k + 1) * WINDOW_US)
                     for k, (a, b) in enumerate(zip(off[:-1], off[1:]))]
        s["flow"] = [torch.zeros((2, H, W), dtype=torch.float32, pin_memory=True)
                     for _ in range(K)]
    _ok(eb.ebof_stream_sync(s["stream"], 1)[0], "ebof_stream_sync")
    return s


def _some_flow(W, H, seed):
    """A smooth flow of a few px per window."""
    rng = np.random.default_rng([seed, W, H, 7])
    a = rng.uniform(-W / 64.0, W / 64.0, 6)
    y = torch.arange(H, device=DEVICE, dtype=torch.float64)[:, None] / H
    x = torch.arange(W, device=DEVICE, dtype=torch.float64)[None, :] / W
    u = a[0] + a[1] * torch.sin(5.0 * x + a[2]) * torch.cos(3.0 * y)
    v = a[3] + a[4] * torch.cos(4.0 * x) * torch.sin(6.0 * y + a[5])
    return torch.stack([u, v]).float().contiguous()


def run(s):
    kind = s["kind"]
    if kind == "edt":
        _ok(eb.ebof_edt(s["edge"], s["W"], s["H"], s["scratch"], s["edt"], s["surface"]),
            "ebof_edt")
        return {"edt": s["edt"], "surface": s["surface"]}
    if kind == "fwl":
        x, y, t, p, _ = s["ev"]
        st, out = eb.ebof_fwl(x, y, t, p, 0, WINDOW_US, s["flow"], s["W"], s["H"], s["scratch"],
                              s["out"])
        _ok(st, "ebof_fwl")
        return out
    if kind == "multigroup":
        for step in s["steps"]:
            _ok(eb.ebof_multigroup_process(s["mg"], step), "ebof_multigroup_process")
        return s["out"]
    stream = s["stream"]
    if kind == "windows":
        x, y, t, _, _ = s["ev"]
        _ok(eb.ebof_process_windows(stream, s["K"], x, y, t, None, 0, WINDOW_US, s["flows"]),
            "ebof_process_windows")
        return s["flows"]
    if kind == "list":
        _ok(eb.ebof_process_window_list(stream, s["wins"], s["flow"]),
            "ebof_process_window_list")
        return s["flows"]
    if kind == "surface":
        for a, f in zip(s["in"], s["flow"]):
            _ok(eb.ebof_process_surface(stream, a, f), "ebof_process_surface")
        return s["flows"]
    if kind == "exports":
        for k, (x, y, t, tb, te) in enumerate(s["wins"]):
            _ok(eb.ebof_process_window(stream, x, y, t, None, tb, te, s["flow"][k], s["edge"][k],
                                       s["edt"][k], s["surface"][k]), "ebof_process_window")
        return {"flow": s["flows"], "edge": s["edge"], "edt": s["edt"], "surface": s["surface"]}
    if kind == "window":
        for (x, y, t, tb, te), f in zip(s["wins"], s["flow"]):
            _ok(eb.ebof_process_window(stream, x, y, t, None, tb, te, f), "ebof_process_window")
        return s["flows"]
    if kind == "pipelined":
        for (x, y, t, tb, te), f in zip(s["wins"], s["flow"]):
            _ok(eb.ebof_process_window_async(stream, x, y, t, None, tb, te, f),
                "ebof_process_window_async")
        _ok(eb.ebof_stream_join(stream), "ebof_stream_join")
        return s["flows"]
    # host: page-locked buffers in and out; the flows are there after the sync
    for (x, y, t, tb, te), f in zip(s["wins"], s["flow"]):
        _ok(eb.ebof_process_window_host_async(stream, x, y, t, tb, te, f),
            "ebof_process_window_host_async")
    _ok(eb.ebof_stream_sync(stream, 1)[0], "ebof_stream_sync")
    return s["flow"]


# ------------------------------------------------------------------- the work
def _flow_flops(opt):
    """Arithmetic of one flow: the search's 25 per patch pixel and iteration,
    the densification's 25 per pixel and covering patch, and per pixel and
    outer iteration 150 for the linear system and 32 for an SOR sweep."""
    W, H, ps, st = opt["width"], opt["height"], opt["patch"], opt["stride"]
    total = 0.0
    for l in range(_levels(W, H, opt["levels"], ps)):
        w, h = W >> l, H >> l
        patches = len(_origins(w, ps, st)) * len(_origins(h, ps, st))
        total += patches * ps * ps * 25.0 * opt["gn_iters"]
        total += w * h * 25.0 * (ps / st) ** 2
        total += w * h * opt["var_outer"] * (150.0 + 32.0 * opt["var_sor"])
    return total


def work(case):
    """Bytes: events (x, y, t; p for the FWL) or images in, the previous
    window's image in and the new one out (the stream's state), results out."""
    kind = case["kind"]
    if kind == "multigroup":
        b = f = 0.0
        for second in (False, True):
            opt = _options(case, second)
            n = case["streams2" if second else "streams"] * case["windows"]
            P = opt["width"] * opt["height"]
            b += n * (12.0 * case["density"] * P + 4.0 * P + 8.0 * P)
            f += n * _flow_flops(opt)
        return {"bytes": b, "flops": f}
    opt = _options(case)
    P = opt["width"] * opt["height"]
    N = case["density"] * P
    if kind == "edt":
        return {"bytes": 9.0 * P, "flops": 12.0 * P}
    if kind == "fwl":
        return {"bytes": 13.0 * N + 8.0 * P, "flops": 30.0 * N + 6.0 * P}
    K = case["windows"]
    state = 4.0 * P if case.get("storage") == "fp16" else 8.0 * P
    source = 4.0 * P if kind == "surface" else 12.0 * N
    extra = 9.0 * P if kind == "exports" else 0.0
    return {"bytes": K * (source + state + 8.0 * P + extra),
            "flops": K * (_flow_flops(opt) + 30.0 * P)}


# ------------------------------------------------- the method in 64-bit torch
def _levels(W, H, levels, ps):
    n = 0
    while n < levels and (W >> n) >= ps and (H >> n) >= ps:
        n += 1
    return n


def _origins(n, ps, stride):
    return [min(k * stride, n - ps) for k in range((n - ps + stride - 1) // stride + 1)]


def _neighbours(E, conn):
    """Edge pixels among the 4 or 8 neighbours (outside the image: none)."""
    p = torch.nn.functional.pad(E.to(torch.int32), (1, 1, 1, 1))
    H, W = E.shape[1:]
    ring = [(0, 1), (2, 1), (1, 0), (1, 2)]
    if conn == 8:
        ring += [(0, 0), (0, 2), (2, 0), (2, 2)]
    return sum(p[:, a:a + H, b:b + W] for a, b in ring)


def _denoise_fill(E, opt):
    """Alg. 1, then Alg. 2 on its result."""
    E = torch.where(_neighbours(E, opt["connectivity"]) < opt["n_d"], torch.zeros_like(E), E)
    return torch.where(_neighbours(E, opt["connectivity"]) >= opt["n_f"], torch.ones_like(E), E)


def _edt(E):
    """Exact squared distance to the nearest edge pixel, int32 [F][H][W]."""
    F, H, W = E.shape
    big = 1 << 15  # above any distance here; its square still fits
    y = torch.arange(H, device=E.device, dtype=torch.int32)[None, :, None]
    up = torch.cummax(torch.where(E > 0, y, -big), 1)[0]
    dn = torch.flip(torch.cummin(torch.flip(torch.where(E > 0, y, big), [1]), 1)[0], [1])
    g = torch.minimum(y - up, dn - y).clamp(max=big)
    g2 = torch.where(g >= 16384, 1 << 30, g * g).reshape(F * H, W)
    x = torch.arange(W, device=E.device, dtype=torch.int32)
    x2 = (x[:, None] - x[None, :]) ** 2
    D = torch.empty((F * H, W), dtype=torch.int32, device=E.device)
    rows = max(1, (1 << 28) // (W * W))
    for a in range(0, F * H, rows):
        D[a:a + rows] = (g2[a:a + rows, None, :] + x2[None]).amin(2)
    D = D.reshape(F, H, W)
    return torch.where((E > 0).flatten(1).any(1)[:, None, None], D, INF_D)


def _surface(D, alpha):
    S = 1.0 - torch.exp(-torch.sqrt(D.double()) / alpha)
    return torch.where(D == INF_D, torch.ones_like(S), S)


def _bilinear(I, x, y):
    """Samples of I [F][H][W] at x, y [F][...], positions clamped to the image."""
    F, H, W = I.shape
    x, y = x.clamp(0, W - 1), y.clamp(0, H - 1)
    x0, y0 = torch.floor(x), torch.floor(y)
    fx, fy = x - x0, y - y0
    x0, y0 = x0.long(), y0.long()
    x1, y1 = (x0 + 1).clamp(max=W - 1), (y0 + 1).clamp(max=H - 1)
    f = (torch.arange(F, device=I.device) * (H * W)).reshape((F,) + (1,) * (x.dim() - 1))
    v = I.reshape(-1)

    def at(yy, xx):
        return v[f + yy * W + xx]

    return (1 - fy) * ((1 - fx) * at(y0, x0) + fx * at(y0, x1)) + \
        fy * ((1 - fx) * at(y1, x0) + fx * at(y1, x1))


def _diff(I, dim):
    """Central differences, replicated border."""
    n = I.shape[dim]
    k = torch.arange(n, device=I.device)
    return 0.5 * (I.index_select(dim, (k + 1).clamp(max=n - 1)) -
                  I.index_select(dim, (k - 1).clamp(min=0)))


def _search(I0, I0x, I0y, I1, Uc, opt):
    """Inverse search of every patch: patch flows [F][2][npy][npx]."""
    F, H, W = I0.shape
    ps, dev = opt["patch"], I0.device
    ox = torch.tensor(_origins(W, ps, opt["stride"]), device=dev)
    oy = torch.tensor(_origins(H, ps, opt["stride"]), device=dev)
    nx, ny = len(ox), len(oy)
    X, Y = ox.repeat(ny), oy.repeat_interleave(nx)
    q = torch.arange(ps * ps, device=dev)
    px, py = X[:, None] + (q % ps)[None], Y[:, None] + (q // ps)[None]
    at = py * W + px

    def patches(I):
        v = I.reshape(F, -1)[:, at]
        return v - v.mean(2, keepdim=True)

    T, gx, gy = patches(I0), patches(I0x), patches(I0y)
    h11, h12, h22 = (gx * gx).sum(2), (gx * gy).sum(2), (gy * gy).sum(2)
    ok = h11 * h22 - h12 * h12 > 1e-6 * ps ** 4
    mu = opt["gn_damping"] * (h11 + h22)
    a11, a22 = h11 + mu, h22 + mu
    det = torch.where(ok, a11 * a22 - h12 * h12, torch.ones_like(mu))
    if Uc is None:
        u0 = torch.zeros((F, nx * ny), device=dev, dtype=torch.float64)
        v0 = torch.zeros_like(u0)
    else:
        hc, wc = Uc.shape[2:]
        c = ((2 * Y + ps) // 4).clamp(0, hc - 1) * wc + ((2 * X + ps) // 4).clamp(0, wc - 1)
        u0, v0 = (2.0 * Uc.reshape(F, 2, -1)[:, :, c]).unbind(1)
    u, v = u0, v0
    for _ in range(opt["gn_iters"]):
        w = _bilinear(I1, px[None] + u[:, :, None], py[None] + v[:, :, None])
        r = w - w.mean(2, keepdim=True) - T
        b1, b2 = (gx * r).sum(2), (gy * r).sum(2)
        u = torch.where(ok, u - (a22 * b1 - h12 * b2) / det, u0)
        v = torch.where(ok, v - (a11 * b2 - h12 * b1) / det, v0)
    far = torch.hypot(u - u0, v - v0) > ps
    u, v = torch.where(far, u0, u), torch.where(far, v0, v)
    return torch.stack([u, v], 1).reshape(F, 2, ny, nx)


def _densify(I0, I1, up, opt):
    """Average of the patches that cover a pixel, by weight 1 / max(1, |residual|)."""
    F, H, W = I0.shape
    ps, dev = opt["patch"], I0.device
    num = torch.zeros((F, 2, H, W), device=dev, dtype=torch.float64)
    den = torch.zeros((F, H, W), device=dev, dtype=torch.float64)

    def covering(n):
        o = _origins(n, ps, opt["stride"])
        per = [[k for k, a in enumerate(o) if a <= x < a + ps] for x in range(n)]
        most = max(map(len, per))
        idx = torch.tensor([p + [0] * (most - len(p)) for p in per], device=dev)
        on = torch.tensor([[True] * len(p) + [False] * (most - len(p)) for p in per], device=dev)
        return idx, on

    ix, onx = covering(W)
    iy, ony = covering(H)
    x = torch.arange(W, device=dev, dtype=torch.float64)[None, None]
    y = torch.arange(H, device=dev, dtype=torch.float64)[None, :, None]
    for j in range(iy.shape[1]):
        for i in range(ix.shape[1]):
            uv = up[:, :, iy[:, j]][:, :, :, ix[:, i]]
            r = _bilinear(I1, x + uv[:, 0], y + uv[:, 1]) - I0
            lam = (1.0 / r.abs().clamp(min=1.0)) * (ony[:, j, None] & onx[None, :, i])[None]
            num += lam[:, None] * uv
            den += lam
    return num / den[:, None]


def _psi(s2):
    return 1.0 / (2.0 * torch.sqrt(s2 + 1e-6))


def _variational(I0, I0x, I0y, I1, U, opt):
    """Fixed-point iterations, each a red-black SOR solve from dU = 0."""
    F, H, W = I0.shape
    dev, om = I0.device, opt["sor_omega"]
    x = torch.arange(W, device=dev, dtype=torch.float64)[None, None]
    y = torch.arange(H, device=dev, dtype=torch.float64)[None, :, None]
    colour = ((x + y) % 2)[:, None] == 0
    pad = torch.nn.functional.pad

    def left(a):  # the neighbour's value, 0 outside the image
        return pad(a, (1, 0))[..., :-1]

    def right(a):
        return pad(a, (0, 1))[..., 1:]

    def above(a):
        return pad(a, (0, 0, 1, 0))[..., :-1, :]

    def below(a):
        return pad(a, (0, 0, 0, 1))[..., 1:, :]

    inside = [f(torch.ones((1, H, W), device=dev, dtype=torch.float64))
              for f in (left, right, above, below)]
    for _ in range(opt["var_outer"]):
        wx, wy = x + U[:, 0], y + U[:, 1]
        Iw = _bilinear(I1, wx, wy)
        Ix, Iy = _diff(Iw, 2), _diff(Iw, 1)
        Ixx, Ixy, Iyy = _diff(Ix, 2), _diff(Ix, 1), _diff(Iy, 1)
        Iz, Ixz, Iyz = Iw - I0, Ix - I0x, Iy - I0y
        nd = 1.0 / (Ix * Ix + Iy * Iy + 0.01)
        ng = 1.0 / (Ixx * Ixx + 2.0 * Ixy * Ixy + Iyy * Iyy + 0.01)
        on = (wx >= 0) & (wx <= W - 1) & (wy >= 0) & (wy <= H - 1)
        ad = torch.where(on, opt["var_delta"] * nd * _psi(nd * Iz * Iz), 0.0)
        ag = torch.where(on, opt["var_gamma"] * ng * _psi(ng * (Ixz * Ixz + Iyz * Iyz)), 0.0)
        dx = torch.zeros_like(U)
        dy = torch.zeros_like(U)
        dx[..., :-1] = U[..., 1:] - U[..., :-1]
        dy[:, :, :-1] = U[:, :, 1:] - U[:, :, :-1]
        a_s = opt["var_alpha"] * _psi((dx * dx + dy * dy).sum(1))
        w = [0.5 * (a_s + f(a_s)) * k
             for f, k in zip((left, right, above, below), inside)]
        sw = sum(w)
        a11 = ad * Ix * Ix + ag * (Ixx * Ixx + Ixy * Ixy) + sw
        a22 = ad * Iy * Iy + ag * (Ixy * Ixy + Iyy * Iyy) + sw
        a12 = ad * Ix * Iy + ag * (Ixx * Ixy + Ixy * Iyy)
        w = [k[:, None] for k in w]
        b = sum(k * (f(U) - U) for f, k in zip((left, right, above, below), w))
        b = b - torch.stack([ad * Ix * Iz + ag * (Ixx * Ixz + Ixy * Iyz),
                             ad * Iy * Iz + ag * (Ixy * Ixz + Iyy * Iyz)], 1)
        d = torch.zeros_like(U)
        for half in range(2 * opt["var_sor"]):
            r = b + w[0] * left(d) + w[1] * right(d) + w[2] * above(d) + w[3] * below(d)
            du = (1 - om) * d[:, 0] + om * (r[:, 0] - a12 * d[:, 1]) / a11
            dv = (1 - om) * d[:, 1] + om * (r[:, 1] - a12 * du) / a22
            d = torch.where(colour if half % 2 == 0 else ~colour, torch.stack([du, dv], 1), d)
        U = U + d
    return U


def _flow(S0, S1, opt):
    """Flow [F][2][H][W] from the surfaces S0 to S1 [F][H][W]."""
    F, H, W = S0.shape
    L = _levels(W, H, opt["levels"], opt["patch"])
    pyr = [(255.0 * S0, 255.0 * S1)]
    for _ in range(1, L):
        pyr.append(tuple(torch.nn.functional.avg_pool2d(a[:, None], 2)[:, 0] for a in pyr[-1]))
    U = None
    for I0, I1 in reversed(pyr):
        I0x, I0y = _diff(I0, 2), _diff(I0, 1)
        up = _search(I0, I0x, I0y, I1, U, opt)
        U = _variational(I0, I0x, I0y, I1, _densify(I0, I1, up, opt), opt)
    return U


def _flows_of_ring(S, opt):
    """Flow k from window k - 1 to window k of a ring of surfaces, a few at a time."""
    prev = torch.roll(S, 1, 0)
    n = max(1, (1 << 22) // (S.shape[1] * S.shape[2]))
    return torch.cat([_flow(prev[a:a + n], S[a:a + n], opt) for a in range(0, S.shape[0], n)])


def _exact_fwl(ev, flow, W, H):
    x, y = ev[0].view(torch.int16).long(), ev[1].view(torch.int16).long()
    p, tau = ev[3].double(), ev[2].double() / WINDOW_US
    at = y * W + x
    u = flow.double().reshape(2, -1)[:, at]
    plain = torch.zeros(W * H, device=x.device, dtype=torch.float64).index_add_(0, at, p)
    moved = torch.zeros_like(plain)
    xw, yw = x - u[0] * tau, y - u[1] * tau
    x0, y0 = torch.floor(xw), torch.floor(yw)
    for dy in (0, 1):
        for dx in (0, 1):
            X, Y = (x0 + dx).long(), (y0 + dy).long()
            w = p * (1 - (xw - X).abs()) * (1 - (yw - Y).abs())
            on = (X >= 0) & (X < W) & (Y >= 0) & (Y < H)
            moved.index_add_(0, (Y * W + X)[on], w[on])
    var = [(a * a).mean() - a.mean() ** 2 for a in (moved, plain)]
    return torch.stack([var[0] / var[1] if var[1] > 0 else torch.ones_like(var[0]), *var])


def exact(case, seed):
    kind, dens = case["kind"], case["density"]
    if kind == "multigroup":
        out = []
        for opt, evs in _streams_of(case, seed):
            flows = []
            for ev in evs:  # the pass ends with the flow to the last window
                E = _denoise_fill(_edge_images(ev, opt["width"], opt["height"]), opt)
                S = _surface(_edt(E), opt["alpha"])
                flows.append(_flow(S[-2:-1], S[-1:], opt))
            out.append(torch.cat(flows))
        return out
    opt = _options(case)
    W, H = opt["width"], opt["height"]
    ev = _events(W, H, case.get("windows", 1), dens, seed)
    if kind == "edt":
        D = _edt(_edge_images(ev, W, H))
        return {"edt": None, "surface": _surface(D, opt["alpha"])[0]}
    if kind == "fwl":
        return _exact_fwl(ev, _some_flow(W, H, seed), W, H)
    if kind == "surface":
        return _flows_of_ring(_smooth_surfaces(ev, W, H, opt["alpha"]).double(), opt)
    E = _denoise_fill(_edge_images(ev, W, H), opt)
    D = _edt(E)
    S = _surface(D, opt["alpha"])
    flows = _flows_of_ring(S, opt)
    if kind == "exports":
        return {"flow": flows, "edge": [None] * len(E), "edt": [None] * len(E),
                "surface": list(S.unbind(0))}
    if kind == "host":
        return list(flows.unbind(0))
    return flows
