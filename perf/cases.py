"""Performance cases: the work a user has this framework do, each through its
public entry points (binding.Plan, binding.Batch, learned.Conv,
learned.FastPath), with the inputs such a user holds and a 64-bit value of the
results in plain torch.

Kinds of cases:
  scan       Plan.execute: one scan, echo and image in device memory
  stream     Plan.execute_host_stream: a sequence of scans in pinned host memory
  batch      Batch.execute: uneven scans together
  exact_sum  Plan.execute_exact: the exact-sum hybrid used as a yardstick
  direct     Plan.execute_bp_direct: direct back-projection, the other yardstick
  conv       one convolution layer of the learned path: forward, input gradient,
             weight and bias gradients
  learned    FastPath.infer: cheap reconstruction, network, acceptance check
"""
import math
import random

import numpy as np
import torch

from paper_2109_02842_gb300 import binding, learned, workloads

C0 = 299792458.0

# The default plan of a scan; a case lists what differs.
SCAN = {"mode": 0, "radius": 0.6, "span": 120.0, "sections": 8, "per": 48, "tx": 0,
        "scans": 64, "pad": 128, "freqs": 64, "f0": 24e9, "f1": 34e9,
        "nx": 64, "ny": 64, "nz": 64, "ext": 0.4, "z_on_scan": False, "z_ext": 0.3,
        "precision": 0, "fp32": False, "points": 16}

# (input channels, output channels) of the network's layers
LAYERS = ((3, 16), (16, 16), (16, 32), (32, 32), (32, 64), (64, 64), (64, 128), (128, 128),
          (128, 64), (64, 32), (32, 16), (16, 2))


def _scan(kind, **kw):
    return dict(SCAN, kind=kind, **kw)


def listed():
    return [
        # the smallest scan (64 channels, 32 positions, 32^3 voxels): a quick
        # look while aligning an array, bound by launches and latency
        dict(_scan("scan", radius=0.5, span=60.0, sections=4, per=16, scans=32, pad=64, freqs=16,
                   f0=28e9, f1=33e9, nx=32, ny=32, nz=32, ext=0.2, z_ext=0.2), name="scan_small"),
        # an ordinary laboratory scan with transmit-receive pairs (120 pairs,
        # 51 frequencies, 64^3 voxels)
        dict(_scan("scan", mode=1, radius=1.0, span=33.0, sections=3, per=20, tx=2, freqs=51,
                   f0=30e9, f1=35e9, ext=0.2, z_ext=0.2), name="scan_multi_lab"),
        # the full-size monostatic scan of a body scanner
        dict(_scan("scan", scans=200, pad=200, nx=256, ny=256, nz=200, z_on_scan=True),
             name="scan_full"),
        # the full-size multistatic scan, BF16 intermediates
        dict(_scan("scan", mode=1, per=32, tx=4, scans=128, pad=128, nx=192, ny=192, nz=128,
                   z_on_scan=True, precision=1), name="scan_multi_bf16"),
        # a network analyser's 201-point sweep, odd array, odd image, heights
        # off the scan positions
        dict(_scan("scan", sections=5, per=23, scans=101, pad=216, freqs=201, nx=117, ny=93, nz=77,
                   z_ext=0.45), name="scan_sweep_odd"),
        # the plain FP32 kernels, asked for where BF16 products are not
        # wanted; odd sizes
        dict(_scan("scan", sections=7, per=31, scans=111, pad=225, freqs=57, nx=120, ny=101, nz=96,
                   z_ext=0.5, fp32=True), name="scan_fp32_odd"),
        # twelve uneven scans handed over together (a queue of a busy checkpoint)
        {"kind": "batch", "scenes": 12, "shapes": 1, "name": "batch_uneven"},
        # scans arriving in host memory one after another, images going back
        dict(_scan("stream", per=32, scans=128, pad=128, nx=192, ny=192, nz=128, z_on_scan=True),
             count=4, name="stream_host"),
        # the exact-sum hybrid and direct back-projection, run to check and to
        # time the method against (laboratory array, 64^3 voxels)
        dict(_scan("exact_sum", radius=1.0, span=33.0, sections=3, per=40, freqs=51, f0=30e9,
                   f1=35e9, ext=0.2, z_ext=0.2), name="exact_sum_lab"),
        dict(_scan("direct", radius=1.0, span=33.0, sections=3, per=40, scans=48, pad=96, freqs=51,
                   f0=30e9, f1=35e9, ext=0.2, z_ext=0.2), name="direct_lab"),
        # a training step's work in one full-resolution layer of the network
        {"kind": "conv", "cin": 16, "cout": 16, "d": 96, "h": 128, "w": 128, "relu": True,
         "name": "conv_train"},
        # an image from the cheap reconstruction and the network
        dict(_scan("learned", radius=0.5, span=60.0, sections=4, per=16, scans=32, pad=64,
                   freqs=64, f0=28e9, f1=33e9, nx=128, ny=128, nz=96, ext=0.2, z_ext=0.2),
             name="learned_infer"),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _smooth(n):
    """The smallest 2^a 3^b 5^c >= n."""
    while True:
        r = n
        for p in (2, 3, 5):
            while r % p == 0:
                r //= p
        if r == 1:
            return n
        n += 1


def _draw_scan(rng, kind, limit, **fixed):
    """A scan whose channels x pixels x bins (times frequencies and the like
    for the exact sums, see _terms) stay below `limit`."""
    while True:
        c = _scan(kind)
        c["mode"] = 1 if rng.random() < 0.3 else 0
        c["radius"] = round(rng.uniform(0.5, 1.0), 3)
        c["span"] = round(rng.uniform(30.0, 120.0), 1)
        c["sections"] = rng.randint(3, 12)
        c["per"] = rng.randint(8, 32) if c["mode"] else rng.randint(16, 48)
        c["tx"] = rng.randint(1, 4) if c["mode"] else 0
        c["scans"] = _log_int(rng, 24, 256)
        c["pad"] = _smooth(c["scans"] * rng.choice((1, 2)))
        c["freqs"] = _log_int(rng, 16, 201)
        c["f0"] = rng.choice((24e9, 26.5e9, 28e9, 30e9))
        c["f1"] = c["f0"] + rng.choice((5e9, 8e9, 10e9))
        c["ext"] = round(rng.uniform(0.2, 0.4), 3)
        least = int(c["ext"] / 0.007) + 1
        c["nx"] = _log_int(rng, least, 256)
        c["ny"] = _log_int(rng, least, 256)
        c["nz"] = _log_int(rng, 16, 200)
        c["z_on_scan"] = rng.random() < 0.5
        if c["z_on_scan"]:
            c["nz"] = min(c["nz"], c["scans"])
        c["z_ext"] = round(0.005 * c["scans"] * rng.uniform(0.5, 1.0), 4)
        c["points"] = rng.randint(4, 24)
        if kind == "scan":
            c["precision"] = rng.choice((0, 0, 0, 1, 2))
            c["fp32"] = rng.random() < 0.2
        c.update(fixed)
        # direct back-projection keeps a running FP32 sum over every channel,
        # position and frequency: it is a yardstick for laboratory sizes
        if kind == "direct" and _channels(c) * c["scans"] * c["freqs"] > 3.5e5:
            continue
        if _terms(c) * (4 if c["fp32"] else 1) <= limit:
            return c


def draw(rng):
    kind = rng.choice(("scan", "scan", "scan", "scan", "conv", "conv", "batch", "stream",
                       "exact_sum", "direct", "learned"))
    if kind == "scan":
        return _draw_scan(rng, kind, 5.0e9)
    if kind == "stream":
        return _draw_scan(rng, kind, 1.0e9, count=rng.randint(2, 5))
    if kind == "batch":
        return {"kind": "batch", "scenes": rng.randint(2, 14), "shapes": rng.randint(2, 1 << 20)}
    if kind == "exact_sum":
        return _draw_scan(rng, kind, 3.2e9)
    if kind == "direct":
        return _draw_scan(rng, kind, 7.0e10)
    if kind == "learned":
        return _scan("learned", radius=0.5, span=60.0, sections=rng.randint(3, 6),
                     per=rng.randint(12, 24), scans=32, pad=64, freqs=rng.randint(24, 96), f0=28e9,
                     f1=33e9, nx=8 * rng.randint(6, 16), ny=8 * rng.randint(6, 16),
                     nz=8 * rng.randint(2, 12), ext=0.2, z_ext=0.2)
    cin, cout = rng.choice(LAYERS)
    while True:
        d, h, w = (_log_int(rng, 4, n) for n in (96, 160, 160))
        if rng.random() < 0.5:        # the network's levels halve 128 x 128 x 96
            s = rng.choice((1, 2, 4, 8))
            d, h, w = _log_int(rng, 4, 96 // s), 128 // s, 128 // s
        if d * h * w * max(cin, 16) * max(cout, 16) <= 1.0e9:
            return {"kind": "conv", "cin": cin, "cout": cout, "d": d, "h": h, "w": w,
                    "relu": cout != 2}


# ---- sizes ---------------------------------------------------------------------------
def _channels(c):
    return c["sections"] * c["per"] * (c["tx"] if c["mode"] else 1)


def _terms(c):
    """Multiply-adds of the path: a channel, a pixel and a k_z bin (hybrid), times
    the frequencies (its exact sum); a channel, a voxel, a position and a
    frequency (direct)."""
    pix = float(c["nx"] * c["ny"])
    if c["kind"] == "direct":
        return _channels(c) * pix * c["nz"] * c["scans"] * c["freqs"]
    return _channels(c) * pix * c["pad"] * (c["freqs"] if c["kind"] == "exact_sum" else 1)


def _batch_shapes(case):
    """The scenes of a batch: 4-12 sections, 16-48 elements each, 64-256
    positions, 32-96 frequencies, images of 64^3-160^3 voxels."""
    r = random.Random(case["shapes"])
    out = []
    for _ in range(case["scenes"]):
        n, g = r.randint(64, 256), r.randint(64, 160)
        out.append(_scan("scan", sections=r.randint(4, 12), per=r.randint(16, 48), scans=n,
                         pad=_smooth(2 * n), freqs=r.randint(32, 96), nx=g, ny=g, nz=g,
                         z_ext=0.005 * n))
    return out


def _layers_of_net():
    """(cin, cout, level, relu) of the network's layers in order."""
    c = (16, 32, 64, 128)
    out = [(3, c[0], 0, True), (c[0], c[0], 0, True)]
    for k in (1, 2, 3):
        out += [(c[k - 1], c[k], k, True), (c[k], c[k], k, True)]
    for k in (2, 1, 0):
        out += [(c[k + 1], c[k], k, True), (c[k], c[k], k, True)]
    return out + [(c[0], 2, 0, False)]


def work(case):
    if case["kind"] == "batch":
        parts = [work(s) for s in _batch_shapes(case)]
        return {k: sum(p[k] for p in parts) for k in ("bytes", "flops")}
    if case["kind"] == "conv":
        v = case["d"] * case["h"] * case["w"]
        cin, cout = case["cin"], case["cout"]
        flops = 2.0 * 27 * cin * cout * v * (2 if cin == 3 else 3)
        # x, w, y, gy in; out, gx, gw out
        return {"bytes": v * (2 * cin + 2 * cout + 4 * cout + 2 * cout + (0 if cin == 3 else 4 * cin))
                + 27 * cin * cout * 6.0, "flops": flops}
    c = case
    cell = 8.0 * (_channels(c) * c["scans"] * c["freqs"] + c["nx"] * c["ny"] * c["nz"])
    if c["kind"] == "learned":
        v = c["nx"] * c["ny"] * c["nz"]
        half = dict(c, kind="scan", freqs=(c["freqs"] + 1) // 2)
        flops = sum(2.0 * 27 * a * b * v / 8 ** lev for a, b, lev, _ in _layers_of_net())
        w = work(half)
        return {"bytes": w["bytes"] + 8.0 * v, "flops": w["flops"] + flops}
    if c["kind"] == "exact_sum" or c["kind"] == "direct":
        return {"bytes": cell, "flops": 8.0 * _terms(c)}
    # the method: two weights of six taps and a complex multiply-add a term,
    # the two transforms over z, the range profiles
    return {"bytes": cell * c.get("count", 1), "flops": 48.0 * _terms(c) * c.get("count", 1)}


# ---- inputs --------------------------------------------------------------------------
def _geometry(c):
    """(elements [n][2], section of each, tx index, rx index): chords of a circle,
    elements cell-centred on each chord; transmitters then receivers of a
    chord, pairs within a chord."""
    span = math.radians(c["span"])
    phi = -span / 2 + span * np.arange(c["sections"] + 1) / c["sections"]
    joint = np.stack([c["radius"] * np.sin(phi), -c["radius"] * np.cos(phi)], 1)
    xy, sec, tx, rx = [], [], [], []
    for s in range(c["sections"]):
        for n in ([c["tx"]] if c["mode"] else []) + [c["per"]]:
            t = (np.arange(n) + 0.5) / n
            xy.append(joint[s] + t[:, None] * (joint[s + 1] - joint[s]))
            sec += [s] * n
        if c["mode"]:
            base = s * (c["tx"] + c["per"])
            for i in range(c["tx"]):
                for j in range(c["per"]):
                    tx.append(base + i)
                    rx.append(base + c["tx"] + j)
    chord = float(np.linalg.norm(joint[1] - joint[0]))
    return np.concatenate(xy), np.array(sec), np.array(tx, int), np.array(rx, int), chord


def _axes(c):
    """z positions of the scan and the voxel centres (start, step, count)."""
    dz = 0.005
    z0 = -(c["scans"] - 1) / 2 * dz
    g = {}
    for a in ("x", "y"):
        d = c["ext"] / c["n" + a]
        g[a + "0"], g["d" + a], g["n" + a] = -c["ext"] / 2 + d / 2, d, c["n" + a]
    if c["z_on_scan"]:
        g["z0"], g["dz"] = z0, dz
    else:
        g["dz"] = c["z_ext"] / c["nz"]
        g["z0"] = -c["z_ext"] / 2 + g["dz"] / 2
    g["nz"] = c["nz"]
    return z0, dz, g


def _freqs(c):
    return np.linspace(c["f0"], c["f1"], c["freqs"])


def _workload(c):
    xy, sec, tx, rx, chord = _geometry(c)
    z0, dz, g = _axes(c)
    return workloads.Workload("scan", c["mode"], c["radius"], c["sections"], chord, xy, sec, tx, rx,
                              z0, dz, c["scans"], c["pad"], _freqs(c), g)


def _channel_xy(c):
    xy, _, tx, rx, _ = _geometry(c)
    t = xy[tx] if c["mode"] else xy
    r = xy[rx] if c["mode"] else xy
    return (torch.tensor(t, dtype=torch.float64, device="cuda"),
            torch.tensor(r, dtype=torch.float64, device="cuda"))


def _echo(c, seed):
    """complex64 [channel][position][frequency]: point scatterers, 30 dB noise."""
    rng = np.random.default_rng([seed, c["points"]])
    z0, dz, _ = _axes(c)
    half = min(0.15, 0.45 * c["ext"])
    zs = (z0, z0 + dz * (c["scans"] - 1))
    pts = np.stack([rng.uniform(-half, half, c["points"]), rng.uniform(-half, half, c["points"]),
                    rng.uniform(zs[0], zs[1], c["points"])], 1)
    amp = rng.uniform(0.5, 1.0, c["points"])
    t, r = _channel_xy(c)
    z = z0 + dz * torch.arange(c["scans"], dtype=torch.float64, device="cuda")
    k = torch.tensor(2 * math.pi * _freqs(c) / C0, device="cuda")
    echo = torch.zeros((t.shape[0], c["scans"], c["freqs"]), dtype=torch.complex64, device="cuda")
    for p, a in zip(pts, amp):
        rt = torch.sqrt(((t - t.new_tensor(p[:2])) ** 2).sum(1)[:, None] + (z - p[2]) ** 2)
        rr = torch.sqrt(((r - r.new_tensor(p[:2])) ** 2).sum(1)[:, None] + (z - p[2]) ** 2)
        ph = torch.remainder((rt + rr)[:, :, None] * k, 2 * math.pi).float()
        echo += torch.polar(torch.full_like(ph, float(a)), -ph)
    power = float(torch.mean(torch.view_as_real(echo) ** 2)) * 2
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    noise = torch.randn(echo.shape, dtype=torch.complex64, device="cuda", generator=g)
    return echo + math.sqrt(power * 1e-3) * noise


def _plan(c):
    w = _workload(c)
    if not c["fp32"]:
        return binding.Plan.from_workload(w, precision=c["precision"])
    try:
        return binding.Plan.from_workload(w, precision=c["precision"], block_config=3)
    except binding.PolylineError:      # an x step too wide for the two-pixel kernel
        return binding.Plan.from_workload(w, precision=c["precision"], block_config=1)


def _conv_inputs(case, seed):
    """x, the layer's saved output y, its gradient, weights and bias. Activations
    are non-negative with half of them zero, as after a ReLU."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    v, cin, cout = case["d"] * case["h"] * case["w"], case["cin"], case["cout"]

    def normal(*shape):
        return torch.randn(shape, device="cuda", generator=g)

    x = normal(v, cin)
    x = (x if cin == 3 else x.clamp_min(0)).bfloat16()
    y = normal(v, cout).clamp_min(0).bfloat16()
    gy = normal(v, cout).bfloat16().float()
    w = normal(cout, 27 * cin) * math.sqrt(2.0 / (27 * cin))
    b = 0.1 * normal(cout)
    return x, y, gy, w, b


def _net_weights(seed):
    """[(w [cout][27 cin], b [cout])] of every layer: He-scaled, the head small,
    so that the correction is a few per cent of the image, as after training."""
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    out = []
    for cin, cout, _, relu in _layers_of_net():
        std = math.sqrt((2.0 if relu else 0.002) / (27 * cin))
        out.append((torch.randn((cout, 27 * cin), device="cuda", generator=g) * std,
                    torch.randn(cout, device="cuda", generator=g) * (2e-3 if relu else 1e-5)))
    return out


def _fill(layer, w, b):
    layer.w[:, :w.shape[1]].copy_(w)
    layer.b.copy_(b)
    layer.wb.copy_(layer.w.to(torch.bfloat16))


def prepare(case, seed):
    kind = case["kind"]
    if kind == "batch":
        scenes = _batch_shapes(case)
        return {"kind": kind, "batch": binding.Batch([_workload(s) for s in scenes]),
                "echos": [_echo(s, seed + 101 * i) for i, s in enumerate(scenes)]}
    if kind == "conv":
        x, y, gy, w, b = _conv_inputs(case, seed)
        layer = learned.Conv(case["cin"], case["cout"], case["relu"], np.random.default_rng(0))
        _fill(layer, w, b)
        return {"kind": kind, "layer": layer, "x": x, "y": y, "gy": gy,
                "dims": (case["d"], case["h"], case["w"])}
    if kind == "learned":
        net = learned.UNet3D(seed=0)
        for layer, (w, b) in zip(net.layers(), _net_weights(seed)):
            _fill(layer, w, b)
        path = learned.FastPath(_workload(case), net=net)
        return {"kind": kind, "path": path, "echo": path.cheap_echo(_echo(case, seed))}
    plan = _plan(case)
    if kind == "stream":
        echos = [_echo(case, seed + 101 * i).cpu().pin_memory() for i in range(case["count"])]
        images = [torch.empty(plan.image_shape, dtype=torch.complex64, pin_memory=True)
                  for _ in echos]
        return {"kind": kind, "plan": plan, "echos": echos, "images": images}
    return {"kind": kind, "plan": plan, "echo": _echo(case, seed)}


def run(state):
    kind = state["kind"]
    if kind == "scan":
        return state["plan"].execute(state["echo"])
    if kind == "exact_sum":
        return state["plan"].execute_exact(state["echo"])
    if kind == "direct":
        return state["plan"].execute_bp_direct(state["echo"])
    if kind == "batch":
        return state["batch"].execute(state["echos"])
    if kind == "stream":
        return state["plan"].execute_host_stream(state["echos"], state["images"])
    if kind == "learned":
        return state["path"].infer(state["echo"])
    layer = state["layer"]
    layer.gw.zero_()
    layer.gb.zero_()
    out = layer.forward(state["x"], state["dims"], out_bf16=layer.relu)
    gx = layer.backward(state["gy"], state["y"], state["x"], state["dims"],
                        need_gx=layer.cin != 3)
    return {"out": out, "gx": gx, "gw": layer.gw, "gb": layer.gb}


# ---- the results in 64 bits ------------------------------------------------------------
def _distances(xy, c):
    """[channel][pixel] distance in the plane, pixels x fastest."""
    _, _, g = _axes(c)
    px = g["x0"] + g["dx"] * torch.arange(c["nx"], dtype=torch.float64, device="cuda")
    py = g["y0"] + g["dy"] * torch.arange(c["ny"], dtype=torch.float64, device="cuda")
    d2 = (py[:, None] - xy[:, 1, None, None]) ** 2 + (px - xy[:, 0, None, None]) ** 2
    return torch.sqrt(d2).reshape(xy.shape[0], -1)


def _exact_hybrid(c, echo):
    """g(x, y, z) of the hybrid method: the transform over z, the exact sum over
    channels and frequencies k_m S e^{j kappa a} of each k_z bin and pixel, the
    inverse transform. The sum over frequencies is a band-limited function of the
    range a: it is taken at evenly spaced ranges (twice the Nyquist rate) and
    carried to the pixels' ranges with a 16-point Kaiser-Bessel kernel, whose
    error is below 1e-12."""
    n_pad, taps, over = c["pad"], 16, 2.0
    dev, f64 = "cuda", torch.float64
    z0, dz, g = _axes(c)
    k = torch.tensor(2 * math.pi * _freqs(c) / C0, device=dev)
    bins = torch.tensor(np.fft.fftfreq(n_pad, dz) * 2 * math.pi, device=dev)
    arg = (4 * k ** 2 - bins[:, None] ** 2) if c["mode"] == 0 else (k ** 2 - bins[:, None] ** 2 / 4)
    live = arg > 0
    kap = torch.sqrt(arg.clamp_min(0))
    lo, hi = float(kap[live].min()), float(kap[live].max())
    mid, band = (lo + hi) / 2, max(hi - lo, 1.0)
    step = 2 * math.pi / (over * band)
    t, r = _channel_xy(c)
    a = _distances(t, c)
    if c["mode"]:
        a = a + _distances(r, c)
    start = float(a.min()) - (taps / 2 + 1) * step
    rows = int((float(a.max()) - start) / step) + taps + 2
    beta = math.pi * taps * (1 - 1 / (2 * over))
    ranges = start + step * torch.arange(rows, dtype=f64, device=dev)
    S = torch.fft.fft(echo.to(torch.complex128), n=n_pad, dim=1).permute(1, 0, 2)
    off = torch.where(live, kap - mid, torch.zeros_like(kap))
    root = torch.sqrt(beta ** 2 - (off * step * taps / 2) ** 2)
    hat = taps * torch.sinh(root) / root
    S = S * torch.where(live, k / hat, torch.zeros_like(hat))[:, None, :]
    table = torch.empty((a.shape[0], rows, n_pad), dtype=torch.complex128, device=dev)
    for u in range(n_pad):
        table[:, :, u] = S[u] @ torch.exp(1j * off[u][:, None] * ranges)
    G = torch.zeros((a.shape[1], n_pad), dtype=torch.complex128, device=dev)
    where = torch.arange(taps, device=dev)
    for ch in range(a.shape[0]):
        x = (a[ch] - start) / step
        first = torch.floor(x).long() - taps // 2 + 1
        at = first[:, None] + where
        d = 2 * (x[:, None] - at) / taps
        weight = torch.i0(beta * torch.sqrt((1 - d * d).clamp_min(0)))
        got = torch.nn.functional.embedding_bag(
            at, torch.view_as_real(table[ch]).reshape(rows, 2 * n_pad), mode="sum",
            per_sample_weights=weight)
        G += torch.view_as_complex(got.view(-1, n_pad, 2)) * torch.exp(1j * mid * a[ch])[:, None]
    z = g["z0"] + g["dz"] * torch.arange(c["nz"], dtype=f64, device=dev)
    back = torch.exp(1j * (z[:, None] - z0) * bins) / n_pad
    return (back @ G.T).reshape(c["nz"], c["ny"], c["nx"])


def _exact_direct(c, echo):
    """g(x, y, z) = sum s k_m e^{j k_m R} over channels, positions and frequencies
    (evenly spaced: Horner's rule in e^{j dk R})."""
    z0, dz, g = _axes(c)
    k = 2 * math.pi * _freqs(c) / C0
    t, r = _channel_xy(c)
    dt, dr = _distances(t, c) ** 2, _distances(r, c) ** 2
    z = g["z0"] + g["dz"] * torch.arange(c["nz"], dtype=torch.float64, device="cuda")
    img = torch.zeros((c["nz"], c["ny"] * c["nx"]), dtype=torch.complex128, device="cuda")
    s = echo.to(torch.complex128) * torch.tensor(k, device="cuda")
    few = max(1, (1 << 25) // img.numel())
    for ch in range(dt.shape[0]):
        for n in range(0, c["scans"], few):
            at = z0 + dz * torch.arange(n, min(n + few, c["scans"]), dtype=torch.float64,
                                        device="cuda")
            h2 = (z - at[:, None])[:, :, None] ** 2
            R = torch.sqrt(dt[ch] + h2) + torch.sqrt(dr[ch] + h2)
            turn = torch.exp(1j * float(k[1] - k[0]) * R)
            acc = torch.zeros_like(turn)
            for m in range(len(k) - 1, -1, -1):
                acc.mul_(turn).add_(s[ch, n:n + few, m, None, None])
            img += (acc * torch.exp(1j * float(k[0]) * R)).sum(0)
    return img.reshape(c["nz"], c["ny"], c["nx"])


def _conv64(x, w, dims, cin):
    """3 x 3 x 3 convolution of channels-last [v][cin], zero padding, 64 bits."""
    xp = torch.nn.functional.pad(x.view(*dims, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    out = torch.zeros((x.shape[0], w.shape[0]), dtype=torch.float64, device="cuda")
    for tap in range(27):
        dz, dy, dx = tap // 9, tap // 3 % 3, tap % 3
        part = xp[dz:dz + dims[0], dy:dy + dims[1], dx:dx + dims[2]].reshape(-1, cin)
        out += part @ w[:, tap * cin:(tap + 1) * cin].T
    return out


def _exact_conv(case, seed):
    x, y, gy, w, b = _conv_inputs(case, seed)
    dims, cin, cout = (case["d"], case["h"], case["w"]), case["cin"], case["cout"]
    x, wd = x.double(), w.bfloat16().double()
    out = _conv64(x, wd, dims, cin) + b.double()
    gd = gy.double()
    if case["relu"]:
        out = out.clamp_min(0)
        gd = gd * (y > 0)
    flip = torch.empty((cin, 27 * cout), dtype=torch.float64, device="cuda")
    gw = torch.zeros((cout, (27 * cin + 15) // 16 * 16), dtype=torch.float64, device="cuda")
    xp = torch.nn.functional.pad(x.view(*dims, cin), (0, 0, 1, 1, 1, 1, 1, 1))
    for tap in range(27):
        dz, dy, dx = tap // 9, tap // 3 % 3, tap % 3
        part = xp[dz:dz + dims[0], dy:dy + dims[1], dx:dx + dims[2]].reshape(-1, cin)
        gw[:, tap * cin:(tap + 1) * cin] = gd.T @ part
        flip[:, (26 - tap) * cout:(27 - tap) * cout] = wd[:, tap * cin:(tap + 1) * cin].T
    gx = _conv64(gd, flip, dims, cout) if cin != 3 else None
    return {"out": out, "gx": gx, "gw": gw, "gb": gd.sum(0)}


def _exact_learned(c, seed):
    """The image of the network, its activations in 64 bits (the layers' BF16
    rounding is part of what a run's error is made of)."""
    half = dict(c, kind="scan", freqs=(c["freqs"] + 1) // 2)
    full_f = _freqs(c)[::2]
    half["f0"], half["f1"] = float(full_f[0]), float(full_f[-1])
    echo = _echo(c, seed)[:, :, ::2]
    cheap = _exact_hybrid(half, echo)
    dims = [(c["nz"] >> i, c["ny"] >> i, c["nx"] >> i) for i in range(4)]
    g = cheap.reshape(-1)
    s = g.abs().max()
    x = torch.stack([g.real / s, g.imag / s, g.abs() / s], 1)
    layers = [(w.bfloat16().double(), b.double()) for w, b in _net_weights(seed)]
    kinds = _layers_of_net()

    def conv(i, x):
        y = _conv64(x, layers[i][0], dims[kinds[i][2]], kinds[i][0]) + layers[i][1]
        return y.clamp_min(0) if kinds[i][3] else y

    skips = []
    for lev in range(4):
        if lev:
            d = dims[lev]
            x = x.view(d[0], 2, d[1], 2, d[2], 2, -1).mean((1, 3, 5)).reshape(-1, x.shape[1])
        x = conv(2 * lev + 1, conv(2 * lev, x))
        skips.append(x)
    for i, lev in enumerate((2, 1, 0)):
        x = x.view(*dims[lev + 1], -1)
        for ax in range(3):
            x = x.repeat_interleave(2, ax)
        x = conv(9 + 2 * i, conv(8 + 2 * i, x.reshape(-1, x.shape[-1])) + skips[lev])
    x = conv(14, x)
    gain = c["freqs"] / half["freqs"]
    return gain * cheap + (s * torch.view_as_complex(x.contiguous())).view(cheap.shape), cheap, None


def exact(case, seed):
    kind = case["kind"]
    if kind == "batch":
        return [_exact_hybrid(s, _echo(s, seed + 101 * i))
                for i, s in enumerate(_batch_shapes(case))]
    if kind == "conv":
        return _exact_conv(case, seed)
    if kind == "learned":
        return _exact_learned(case, seed)
    if kind == "stream":
        return [_exact_hybrid(case, _echo(case, seed + 101 * i)).cpu()
                for i in range(case["count"])]
    if kind == "direct":
        return _exact_direct(case, _echo(case, seed))
    return _exact_hybrid(case, _echo(case, seed))
