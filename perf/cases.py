"""Performance cases of the photoacoustic reconstruction library: the calls a user's program
makes, at the sizes of the library's own workloads, tests and batches.

Every case goes through the C-named entry points of the package.  Inputs are made from the
seed alone on the GPU with plain torch (phantoms, the data of a plain FP64 projection plus
noise, network tensors), so ``exact`` can rebuild them and compute the same outputs in 64
bits without the library.

Kinds of cases:
- ``forward``: y = K u.  Simulating data, the residual of an image.
- ``adjoint``: u = K^T y.  Backprojection, the gradient of the data term.
- ``solve``: one reconstruction (TV, TGV, directional TV, the dual-tree wavelet model).
- ``batch``: uneven reconstructions in one call.
- ``conv_fwd``, ``conv_bwd``: one 3x3 layer of the warm-start network and its two gradients.
- ``unet``: the whole network, forward and backward (the body of a training step).
"""
import math

import numpy as np
import torch

import paper_1707_02245_gb300 as P
from paper_1707_02245_gb300.warmstart import UNet

REGS = {"tv": P.PAT_TV, "tgv": P.PAT_TGV, "dtv": P.PAT_DTV, "dtcwt": P.PAT_WAV}
GAMMA = 0.95
BOX_U, BOX_V = 2.0, 4.0
GAP_EVERY = 10
PROBLEM = ("n", "n_det", "n_t", "arc", "reg", "alpha", "beta", "ratio")


# ---------------------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------------------

def listed():
    return [
        # the smallest projection: a 64^2 image seen by 64 detectors (preview, unit-scale data)
        dict(name="forward_64", kind="forward", n=64, n_det=64, n_t=128, m=256, arc=False),
        # simulating data on the fine grid of a 256^2 problem: 512^2 image, the densest array
        dict(name="forward_512", kind="forward", n=512, n_det=512, n_t=1024, m=256, arc=False),
        # backprojection of the benchmark geometry
        dict(name="adjoint_256", kind="adjoint", n=256, n_det=256, n_t=512, m=256, arc=False),
        # backprojection of a limited arc onto a grid that no tile size divides
        dict(name="adjoint_odd", kind="adjoint", n=181, n_det=37, n_t=333, m=200, arc=True),
        # a whole small TV reconstruction: discs, 200 iterations, where launches and set-up count
        dict(name="tv_64", kind="solve", reg="tv", n=64, n_det=64, n_t=128, m=256, arc=False, alpha=0.05, beta=1.0,
             ratio=1.0, iters=200),
        # the benchmark reconstruction: TGV 256^2 with the tuned primal-dual balance
        dict(name="tgv_256", kind="solve", reg="tgv", n=256, n_det=256, n_t=512, m=256, arc=False, alpha=0.02,
             beta=0.04, ratio=10.0, iters=200),
        # limited-angle compressive sampling with directional TV
        dict(name="dtv_arc_256", kind="solve", reg="dtv", n=256, n_det=32, n_t=512, m=256, arc=True, alpha=0.02,
             beta=1.0, ratio=1.0, iters=200),
        # the wavelet model (dual-tree complex transform, 4 levels)
        dict(name="dtcwt_256", kind="solve", reg="dtcwt", n=256, n_det=128, n_t=512, m=256, arc=False, alpha=0.02,
             beta=1.0, ratio=1.0, iters=100),
        # an uneven batch, the library's serving shape: sizes, arrays and regularisers mixed,
        # a tolerance set as in production (not reached within these iterations)
        dict(name="batch_mixed", kind="batch", m=256, iters=60, tol=1e-6,
             problems="128:32:256:0:tv:0.01:1:1 192:256:384:0:tgv:0.03:2:10 256:128:512:1:dtv:0.05:1:1 "
                      "384:64:768:0:tv:0.002:1:1 512:32:1024:0:tgv:0.02:2:10 128:512:256:0:dtv:0.09:1:1 "
                      "192:64:384:0:tv:0.005:1:1 255:33:509:1:tgv:0.02:0.04:10"),
        # the network's full-resolution layer (inference and training)
        dict(name="conv_fwd_256", kind="conv_fwd", batch=8, h=256, w=256, cin=32, cout=32, relu=True),
        # both gradients of a decoder layer on a concatenation
        dict(name="conv_bwd_128", kind="conv_bwd", batch=8, h=128, w=128, cin=192, cout=64),
        # forward and backward of the whole 4-level network, the body of a training step
        dict(name="unet_256", kind="unet", batch=8, h=256, w=256, base=32, levels=4),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _size(rng):
    """(n, n_det, n_t, arc): the grids and arrays of the library's workloads, odd ones among
    them, with the data of about two samples a pixel."""
    n = _log(rng, 48, 512)
    n_det = _log(rng, 8, 512)
    n_t = max(8, int(n * rng.uniform(1.5, 2.0)))
    return n, n_det, n_t, n_det <= 64 and rng.random() < 0.5


def _reg(rng, reg):
    """(alpha, beta, ratio)."""
    alpha = round(math.exp(rng.uniform(math.log(1e-3), math.log(0.1))), 6)
    return alpha, (2.0 if reg == "tgv" else 1.0), (10.0 if reg == "tgv" else 1.0)


def draw(rng):
    kind = rng.choice(["forward", "adjoint", "solve", "solve", "batch", "conv_fwd", "conv_bwd", "unet"])
    if kind in ("forward", "adjoint"):
        n, n_det, n_t, arc = _size(rng)
        return dict(kind=kind, n=n, n_det=n_det, n_t=n_t, m=rng.choice([128, 200, 256, 256]), arc=arc)
    if kind == "solve":
        n, n_det, n_t, arc = _size(rng)
        n_det = min(n_det, 256)
        reg = rng.choice(["tv", "tgv", "dtv", "dtcwt"])
        if reg == "dtcwt":
            n = max(64, min(256, n // 16 * 16))
            n_t = max(n_t, n)
        alpha, beta, ratio = _reg(rng, reg)
        return dict(kind=kind, reg=reg, n=n, n_det=n_det, n_t=n_t, m=256, arc=arc, alpha=alpha, beta=beta,
                    ratio=ratio, iters=_log(rng, 30, 200))
    if kind == "batch":
        text = []
        for _ in range(rng.randint(2, 8)):
            n, n_det, n_t, arc = _size(rng)
            n_det = min(n_det, 64 if n > 256 else 256)
            reg = rng.choice(["tv", "tgv", "dtv"])
            alpha, beta, ratio = _reg(rng, reg)
            text.append(f"{n}:{n_det}:{n_t}:{int(arc)}:{reg}:{alpha}:{beta}:{ratio}")
        return dict(kind=kind, m=256, iters=_log(rng, 25, 60), tol=1e-6, problems=" ".join(text))
    if kind == "unet":
        levels = rng.randint(2, 4)
        q = 2 ** (levels - 1)
        return dict(kind=kind, batch=rng.randint(1, 8), h=max(1, _log(rng, 24, 256) // q) * q,
                    w=max(1, _log(rng, 24, 256) // q) * q, base=rng.choice([8, 16, 32]), levels=levels)
    level = rng.randint(0, 3)   # a layer of the network: channels double as the sides halve
    c = 32 << level
    cin, cout = rng.choice([(c, c), (8 if level == 0 else c // 2, c), (3 * c if level < 3 else c, c)])
    side = _log(rng, 24, 256)
    return dict(kind=kind, batch=rng.randint(1, 8), h=max(3, side >> level), w=max(3, (side + rng.randint(-9, 9)) >> level),
                cin=cin, cout=cout, **({"relu": rng.random() < 0.7} if kind == "conv_fwd" else {}))


# ---------------------------------------------------------------------------------------
# inputs (plain torch; the same for every build of the library)
# ---------------------------------------------------------------------------------------

def _dev():
    return torch.device("cuda", torch.cuda.current_device())


def _gen(seed, salt=0):
    return torch.Generator(device=_dev()).manual_seed((int(seed) * 1000003 + salt) % (1 << 62))


def _detectors(n_det, arc):
    """Point detectors on a circle of radius 1.2: all round, or on a 90 degree arc."""
    if arc:
        a = math.pi / 2 * (np.arange(n_det) + 0.5) / n_det
    else:
        a = 2 * math.pi * (np.arange(n_det) + 0.5) / n_det
    return np.stack([1.2 * np.cos(a), 1.2 * np.sin(a)], 1)


def _dr(n_det, n_t, arc):
    """Radial step: n_t samples from zero to the farthest corner of the square."""
    det = _detectors(n_det, arc)
    corners = np.array([[-1.0, -1.0], [-1.0, 1.0], [1.0, -1.0], [1.0, 1.0]])
    return float(np.max(np.hypot(det[:, None, 0] - corners[:, 0], det[:, None, 1] - corners[:, 1]))) / n_t


def _phantom(n, seed, salt=0):
    """A tree of 40 random capsules 1 to 4 pixels (of a 256 grid) wide with decaying fluence, and 5 discs."""
    g = _gen(seed, 17 + salt)
    rnd = lambda *s: torch.rand(*s, generator=g, device=_dev(), dtype=torch.float64)  # noqa: E731
    x = (torch.arange(n, device=_dev(), dtype=torch.float64) + 0.5) * (2.0 / n) - 1
    X, Y = x[None, :], x[:, None]
    u = torch.zeros(n, n, device=_dev(), dtype=torch.float64)
    start, turn, length, width = 1.4 * rnd(40, 2) - 0.7, 2 * math.pi * rnd(40), 0.1 + 0.5 * rnd(40), (1 + 3 * rnd(40)) / 256
    for i in range(40):
        dx, dy = length[i] * torch.cos(turn[i]), length[i] * torch.sin(turn[i])
        t = (((X - start[i, 0]) * dx + (Y - start[i, 1]) * dy) / (length[i] ** 2)).clamp(0, 1)
        far = torch.hypot(X - start[i, 0] - t * dx, Y - start[i, 1] - t * dy)
        u = torch.maximum(u, ((width[i] - far) * n / 2 + 0.5).clamp(0, 1))
    u = u * torch.exp(-3 * (1 - X.abs()).clamp(min=0))
    c, rad, amp = 1.2 * rnd(5, 2) - 0.6, 0.05 + 0.15 * rnd(5), 0.25 + 0.25 * rnd(5)
    for i in range(5):
        u = u + amp[i] * ((rad[i] - torch.hypot(X - c[i, 0], Y - c[i, 1])) * n / 2 + 0.5).clamp(0, 1)
    return u


def _points(n, n_det, n_t, m, arc, d):
    """Continuous pixel coordinates (T x M) of the quadrature points of detector d, and the arc weights (T x 1)."""
    det = _detectors(n_det, arc)[d]
    r = (torch.arange(n_t, device=_dev(), dtype=torch.float64)[:, None] + 0.5) * _dr(n_det, n_t, arc)
    phi = 2 * math.pi * (torch.arange(m, device=_dev(), dtype=torch.float64) + 0.5) / m
    h = 2.0 / n
    return (det[0] + r * torch.cos(phi) + 1) / h - 0.5, (det[1] + r * torch.sin(phi) + 1) / h - 0.5, 2 * math.pi * r / m


def _taps(n, fx, fy):
    """[(pixel index clamped to the grid, weight, zero off the grid)] of the four bilinear taps."""
    i0, j0 = torch.floor(fx), torch.floor(fy)
    ax, ay = fx - i0, fy - j0
    out = []
    for di, wx in ((0, 1 - ax), (1, ax)):
        for dj, wy in ((0, 1 - ay), (1, ay)):
            i, j = (i0 + di).long(), (j0 + dj).long()
            on = (i >= 0) & (i < n) & (j >= 0) & (j < n)
            out.append((torch.where(on, j * n + i, 0), torch.where(on, wx * wy, 0.0)))
    return out


def _project(u, n_det, n_t, m, arc):
    """K u in 64 bits."""
    n = u.shape[0]
    y = torch.empty(n_det, n_t, device=_dev(), dtype=torch.float64)
    flat = u.double().reshape(-1)
    for d in range(n_det):
        fx, fy, w = _points(n, n_det, n_t, m, arc, d)
        y[d] = (sum(flat[i] * t for i, t in _taps(n, fx, fy)) * w).sum(1)
    return y


def _backproject(y, n, m, arc):
    """K^T y in 64 bits."""
    n_det, n_t = y.shape
    u = torch.zeros(n * n, device=_dev(), dtype=torch.float64)
    for d in range(n_det):
        fx, fy, w = _points(n, n_det, n_t, m, arc, d)
        for i, t in _taps(n, fx, fy):
            u.index_add_(0, i.reshape(-1), (t * w * y[d].double()[:, None]).reshape(-1))
    return u.reshape(n, n)


def _noise(y, seed, level, salt=0):
    z = torch.randn(y.shape, generator=_gen(seed, 29 + salt), device=_dev(), dtype=torch.float64)
    return y + level * y.abs().max() * z


def _data(c, seed, salt=0):
    """Noisy data of a phantom (5% of the clean data's maximum)."""
    return _noise(_project(_phantom(c["n"], seed, salt), c["n_det"], c["n_t"], c["m"], c["arc"]), seed, 0.05, salt).float()


def _fast_data(c, seed, salt=0):
    """Data for a backprojection without projecting: smooth profiles along time and detectors, plus noise."""
    k = torch.linspace(0, 1, c["n_t"], device=_dev(), dtype=torch.float64)[None, :]
    d = torch.linspace(0, 2 * math.pi, c["n_det"] + 1, device=_dev(), dtype=torch.float64)[:-1, None]
    a = torch.rand(12, 4, generator=_gen(seed, 31 + salt), device=_dev(), dtype=torch.float64)
    y = sum(a[i, 0] * torch.exp(-(((k - a[i, 1] - 0.2 * a[i, 2] * torch.sin(d + 6.3 * a[i, 3])) / 0.03) ** 2)) for i in range(12))
    return _noise(y, seed, 0.05, salt).float()


def _direction(n, seed, salt=0):
    """xi = grad w / sqrt(|grad w|^2 + eta^2) of the smoothed phantom (forward differences)."""
    w = _phantom(n, seed, salt)
    k = torch.exp(-0.5 * (torch.arange(-4, 5, device=_dev(), dtype=torch.float64) / 1.5) ** 2)
    k = k / k.sum()
    w = torch.nn.functional.conv2d(w[None, None], k[None, None, None, :], padding=(0, 4))
    w = torch.nn.functional.conv2d(w, k[None, None, :, None], padding=(4, 0))[0, 0]
    g = _grad(w)
    eta = 0.01 * (w.max() - w.min())
    return (g / torch.sqrt((g * g).sum(0) + eta * eta)).float().contiguous()


def _problems(c):
    """The problems of a solve or a batch, each a dict with the keys PROBLEM and m."""
    if c["kind"] == "solve":
        return [{k: c[k] for k in PROBLEM + ("m",)}]
    out = []
    for text in c["problems"].split():
        v = text.split(":")
        out.append(dict(n=int(v[0]), n_det=int(v[1]), n_t=int(v[2]), arc=v[3] == "1", reg=v[4], alpha=float(v[5]),
                        beta=float(v[6]), ratio=float(v[7]), m=c["m"]))
    return out


def _conv_inputs(c, seed):
    """Activations after a ReLU, He-normal weights, a small bias and an output gradient."""
    g = _gen(seed, 41)
    rnd = lambda *s: torch.randn(*s, generator=g, device=_dev())  # noqa: E731
    b, h, w, ci, co = (c[k] for k in ("batch", "h", "w", "cin", "cout"))
    x = rnd(b, h, w, ci).clamp(min=0).bfloat16()
    wt = (rnd(co, 3, 3, ci) * math.sqrt(2.0 / (9 * ci))).bfloat16()
    return x, wt, 0.1 * rnd(co), rnd(b, h, w, co).bfloat16()


UNET_CH = 8   # input and output channels of the warm-start network


def _unet_convs(c):
    """(cin, cout) of the network's convolutions in parameter order."""
    ch = [c["base"] << l for l in range(c["levels"])]
    convs, cin = [], UNET_CH
    for v in ch:
        convs += [(cin, v), (v, v)]
        cin = v
    for l in range(c["levels"] - 2, -1, -1):
        convs += [(ch[l + 1] + ch[l], ch[l]), (ch[l], ch[l])]
    return convs + [(ch[0], UNET_CH)]


def _unet_inputs(c, seed):
    g = _gen(seed, 43)
    rnd = lambda *s: torch.randn(*s, generator=g, device=_dev())  # noqa: E731
    shape = (c["batch"], c["h"], c["w"], UNET_CH)
    x = rnd(*shape).bfloat16()
    dy = rnd(*shape) / math.prod(shape)
    params = torch.cat([torch.cat([rnd(co * 9 * ci) * math.sqrt(2.0 / (9 * ci)), torch.zeros(co, device=_dev())])
                        for ci, co in _unet_convs(c)])
    return x, dy, params


# ---------------------------------------------------------------------------------------
# a pass
# ---------------------------------------------------------------------------------------

def _geometry(c):
    return P.Geometry(c["n"], _detectors(c["n_det"], c["arc"]), c["n_t"], 0.0, _dr(c["n_det"], c["n_t"], c["arc"]), c["m"])


def prepare(case, seed):
    c = case
    if c["kind"] == "forward":
        return dict(case=c, geo=_geometry(c), u=_phantom(c["n"], seed).float().contiguous(),
                    y=torch.empty(c["n_det"], c["n_t"], device=_dev()))
    if c["kind"] == "adjoint":
        return dict(case=c, geo=_geometry(c), y=_fast_data(c, seed).contiguous(), u=torch.empty(c["n"], c["n"], device=_dev()))
    if c["kind"] in ("solve", "batch"):
        s = dict(case=c, geo=[], f=[], prm=[], out=[])
        for k, p in enumerate(_problems(c)):
            nn, data = p["n"] ** 2, p["n_det"] * p["n_t"]
            s["geo"].append(_geometry(p))
            s["f"].append(_data(p, seed, k).contiguous())
            nx, ny = {"tv": (1, 2), "tgv": (3, 5), "dtv": (1, 2), "dtcwt": (1, 4)}[p["reg"]]
            out = dict(u=torch.empty(p["n"], p["n"], device=_dev()), x=torch.empty(nx * nn, device=_dev()),
                       y=torch.empty(data + ny * nn, device=_dev()))
            xi = _direction(p["n"], seed, k) if p["reg"] == "dtv" else None
            s["out"].append(out)
            s["prm"].append(P.make_params(reg=REGS[p["reg"]], alpha=p["alpha"], beta=p["beta"], gamma=GAMMA, xi=xi,
                                          iters=c["iters"], tol=c.get("tol", 0.0), gap_every=GAP_EVERY, box_u=BOX_U,
                                          box_v=BOX_V, step_ratio=p["ratio"], wavelet_levels=4,
                                          wavelet_kind=P.PAT_WAVELET_DTCWT, x_out=out["x"], y_out=out["y"]))
        return s
    if c["kind"] == "unet":
        x, dy, params = _unet_inputs(c, seed)
        net = UNet(base_ch=c["base"], levels=c["levels"], in_ch=UNET_CH, out_ch=UNET_CH)
        net.set_params(params.cpu().numpy())
        return dict(case=c, net=net, x=x, dy=dy, y=torch.empty(x.shape, device=_dev()),
                    grad=torch.empty(net.num_params, device=_dev()))
    x, w, bias, dy = _conv_inputs(c, seed)
    new = lambda *s: torch.empty(*s, device=_dev())  # noqa: E731
    return dict(case=c, x=x, w=w, bias=bias, dy=dy, y=new(dy.shape), dx=new(x.shape), dw=new(w.shape), db=new(c["cout"]))


def run(state):
    s, c = state, state["case"]
    stream = torch.cuda.current_stream()
    if c["kind"] == "forward":
        P.pat_forward(s["geo"].handle, s["u"], s["y"], stream)
        return s["y"]
    if c["kind"] == "adjoint":
        P.pat_adjoint(s["geo"].handle, s["y"], s["u"], stream)
        return s["u"]
    if c["kind"] == "solve":
        info = P.pat_reconstruct(s["geo"][0].handle, s["f"][0], s["prm"][0], s["out"][0]["u"], stream)
        return dict(s["out"][0], primal=info["primal"], gap=info["gap"], iters=info["iters_done"])
    if c["kind"] == "batch":
        infos = P.pat_reconstruct_batched([g.handle for g in s["geo"]], s["f"], s["prm"], [o["u"] for o in s["out"]], stream)
        return [dict(o, primal=i["primal"], gap=i["gap"], iters=i["iters_done"]) for o, i in zip(s["out"], infos)]
    if c["kind"] == "unet":
        b, h, w = c["batch"], c["h"], c["w"]
        s["net"].forward(s["x"], b, h, w, s["y"], stream)
        P.pat_unet_backward(s["net"].handle, s["dy"], s["grad"], stream)
        return dict(y=s["y"], grad=s["grad"])
    b, h, w, ci, co = (c[k] for k in ("batch", "h", "w", "cin", "cout"))
    if c["kind"] == "conv_fwd":
        P.pat_conv3x3_forward(s["x"], b, h, w, ci, s["w"], s["bias"], co, c["relu"], s["y"], stream)
        return s["y"]
    P.pat_conv3x3_backward_data(s["dy"], b, h, w, co, s["w"], ci, s["dx"], stream)
    P.pat_conv3x3_backward_weight(s["x"], s["dy"], b, h, w, ci, co, s["dw"], s["db"], stream)
    return dict(dx=s["dx"], dw=s["dw"], db=s["db"])


# ---------------------------------------------------------------------------------------
# what a pass cannot do without
# ---------------------------------------------------------------------------------------

def _on_grid(c):
    """Quadrature points whose taps touch the grid, from up to 16 of the detectors."""
    n, m, t = c["n"], c["m"], c["n_t"]
    det = _detectors(c["n_det"], c["arc"])
    pick = det[np.linspace(0, len(det) - 1, min(16, len(det))).astype(int)]
    r = (np.arange(t)[:, None] + 0.5) * _dr(c["n_det"], t, c["arc"])
    phi = 2 * math.pi * (np.arange(m) + 0.5) / m
    lim = 1 + 1.0 / n
    hits = sum(np.count_nonzero((np.abs(x + r * np.cos(phi)) < lim) & (np.abs(y + r * np.sin(phi)) < lim)) for x, y in pick)
    return hits / len(pick) * len(det)


# floating operations of a point in K and in K^T (position, taps, weights, sums), and of a
# pixel in the primal and dual steps of one iteration
K_FLOPS, KT_FLOPS = 15, 22
STEP_FLOPS = {"tv": 30, "tgv": 100, "dtv": 45, "dtcwt": 300}


def work(case):
    c = case
    if c["kind"] in ("forward", "adjoint"):
        return {"bytes": 4.0 * (c["n"] ** 2 + c["n_det"] * c["n_t"]),
                "flops": _on_grid(c) * (K_FLOPS if c["kind"] == "forward" else KT_FLOPS)}
    if c["kind"] in ("solve", "batch"):
        by = fl = 0.0
        for p in _problems(c):
            nn, data = p["n"] ** 2, p["n_det"] * p["n_t"]
            nx, ny = {"tv": (1, 2), "tgv": (3, 5), "dtv": (1, 2), "dtcwt": (1, 4)}[p["reg"]]
            by += 4.0 * (2 * data + nn * (1 + nx + ny + (2 if p["reg"] == "dtv" else 0)))
            fl += c["iters"] * (_on_grid(p) * (K_FLOPS + KT_FLOPS) + 4 * data + STEP_FLOPS[p["reg"]] * nn)
        return {"bytes": by, "flops": fl}
    if c["kind"] == "unet":
        px = c["batch"] * c["h"] * c["w"]
        level = [l for l in range(c["levels"]) for _ in (0, 1)] + [l for l in range(c["levels"] - 2, -1, -1) for _ in (0, 1)] + [0]
        one = [2.0 * 9 * ci * co * px / 4 ** l for (ci, co), l in zip(_unet_convs(c), level)]
        params = sum(9 * ci * co + co for ci, co in _unet_convs(c))
        return {"bytes": px * UNET_CH * (2.0 + 4 + 4) + 8.0 * params, "flops": 3 * sum(one) - one[0]}
    px, ci, co = c["batch"] * c["h"] * c["w"], c["cin"], c["cout"]
    if c["kind"] == "conv_fwd":
        return {"bytes": px * (2.0 * ci + 4 * co) + 18.0 * ci * co + 4 * co, "flops": 18.0 * px * ci * co}
    return {"bytes": px * (2.0 * ci + 2 * co + 4 * ci) + 54.0 * ci * co + 4 * co, "flops": 36.0 * px * ci * co}


# ---------------------------------------------------------------------------------------
# the same outputs in 64 bits, with plain torch
# ---------------------------------------------------------------------------------------

def _grad(u):
    g = torch.zeros((2,) + tuple(u.shape), device=u.device, dtype=u.dtype)
    g[0, :, :-1] = u[:, 1:] - u[:, :-1]
    g[1, :-1, :] = u[1:, :] - u[:-1, :]
    return g


def _minus_div(r):
    """The transpose of _grad."""
    o = torch.zeros_like(r[0])
    o[:, 1:] += r[0][:, :-1]
    o[:, :-1] -= r[0][:, :-1]
    o[1:, :] += r[1][:-1, :]
    o[:-1, :] -= r[1][:-1, :]
    return o


def _sym(v):
    """E v = (d_x v1, d_y v2, (d_y v1 + d_x v2) / sqrt 2) with backward differences d = -(forward)^T."""
    def back(a, dim):   # -(forward difference)^T
        z = torch.zeros_like(v)
        z[dim] = a
        return -_minus_div(z)
    return torch.stack([back(v[0], 0), back(v[1], 1), (back(v[0], 1) + back(v[1], 0)) / math.sqrt(2)])


def _sym_t(s):
    g11, g22, g12 = _grad(s[0]), _grad(s[1]), _grad(s[2])
    return torch.stack([-g11[0] - g12[1] / math.sqrt(2), -g22[1] - g12[0] / math.sqrt(2)])


def _ball(p, radius):
    norm = torch.sqrt((p * p).sum(0, keepdim=True))
    return p * torch.where(norm > radius, radius / norm.clamp(min=1e-300), torch.ones_like(norm))


class _SparseK:
    """K and K^T as sparse matrices in 64 bits."""

    def __init__(self, c):
        n, rows = c["n"], c["n_det"] * c["n_t"]
        cols, vals, counts = [], [], []
        for d in range(c["n_det"]):
            fx, fy, w = _points(n, c["n_det"], c["n_t"], c["m"], c["arc"], d)
            taps = _taps(n, fx, fy)
            i = torch.cat([t[0] for t in taps], 1)
            v = torch.cat([t[1] for t in taps], 1) * w
            keep = v != 0
            cols.append(i[keep])
            vals.append(v[keep])
            counts.append(keep.sum(1))
        cols, vals, counts = torch.cat(cols), torch.cat(vals), torch.cat(counts)
        row = torch.repeat_interleave(torch.arange(rows, device=_dev()), counts)
        zero = torch.zeros(1, device=_dev(), dtype=torch.int64)
        self.K = torch.sparse_csr_tensor(torch.cat([zero, counts.cumsum(0)]), cols, vals, (rows, n * n))
        order = torch.argsort(cols, stable=True)
        per = torch.bincount(cols, minlength=n * n)
        self.KT = torch.sparse_csr_tensor(torch.cat([zero, per.cumsum(0)]), row[order], vals[order], (n * n, rows))
        self.n = n

    def up(self, u):
        return self.K @ u.reshape(-1)

    def down(self, q):
        return (self.KT @ q).reshape(self.n, self.n)


class _Cwt:
    """The dual-tree complex wavelet transform W (4 planes) of n x n images, its transpose and
    its |W| sums, in 64 bits, with the closed-form 4-tap filters."""

    def __init__(self, n, levels):
        r3, r15 = math.sqrt(3.0), math.sqrt(15.0)
        h1 = [v / (4 * math.sqrt(2)) for v in (1 + r3, 3 + r3, 3 - r3, 1 - r3)]
        hq = [v / (8 * math.sqrt(2)) for v in (5 - r15, 5 + r15, 3 + r15, 3 - r15)]
        self.n, self.levels, self.mats = n, levels, []
        for l in range(levels):
            m = n >> l
            pair = []
            for tree in (0, 1):
                h = h1 if l == 0 else (hq if tree == 0 else hq[::-1])
                g = [(-1) ** i * h[len(h) - 1 - i] for i in range(len(h))]
                off = tree if l == 0 else 0
                a = np.zeros((m, m))
                for k in range(m // 2):
                    for i in range(len(h)):
                        a[k, (2 * k + i + off) % m] += h[i]
                        a[m // 2 + k, (2 * k + i + off) % m] += g[i]
                pair.append(torch.from_numpy(a).to(_dev()))
            self.mats.append(pair)
        low = torch.zeros(n, n, dtype=torch.bool, device=_dev())
        low[:n >> levels, :n >> levels] = True
        self.low = low

    def mix(self, t):
        """Tree planes aa, ab, ba, bb -> (Re z1, Im z1, Re z2, Im z2) at detail positions."""
        z = torch.stack([t[0] - t[3], t[1] + t[2], t[0] + t[3], t[2] - t[1]]) / math.sqrt(2)
        return torch.where(self.low, t, z)

    def unmix(self, z):
        t = torch.stack([z[0] + z[2], z[1] - z[3], z[1] + z[3], z[2] - z[0]]) / math.sqrt(2)
        return torch.where(self.low, z, t)

    def up(self, u):
        out = []
        for p in (0, 1):
            for q in (0, 1):
                t = u.clone()
                for l in range(self.levels):
                    m = self.n >> l
                    t[:m, :m] = self.mats[l][q] @ t[:m, :m] @ self.mats[l][p].T
                out.append(0.5 * t)
        return self.mix(torch.stack(out))

    def down(self, z):
        t4, u = self.unmix(z), 0
        for i, (p, q) in enumerate(((0, 0), (0, 1), (1, 0), (1, 1))):
            t = 0.5 * t4[i]
            for l in range(self.levels - 1, -1, -1):
                m = self.n >> l
                t[:m, :m] = self.mats[l][q].T @ t[:m, :m] @ self.mats[l][p]
            u = u + t
        return u

    def sums(self):
        """(row sums, column sums) of |W|.  Rows of one level, orientation and plane are circular
        shifts of each other by the level's step."""
        n = self.n
        rows, cols = torch.zeros(4, n, n, device=_dev(), dtype=torch.float64), torch.zeros(n, n, device=_dev(), dtype=torch.float64)
        bands = [(l, oy, ox) for l in range(1, self.levels + 1) for oy, ox in ((0, 1), (1, 0), (1, 1))] + [(self.levels, 0, 0)]
        for l, oy, ox in bands:
            m, step = n >> l, 1 << l
            for plane in range(4):
                e = torch.zeros(4, n, n, device=_dev(), dtype=torch.float64)
                e[plane, oy * m, ox * m] = 1
                w = self.down(e).abs()
                rows[plane, oy * m:oy * m + m, ox * m:ox * m + m] = w.sum()
                cols += w.reshape(m, step, m, step).sum((0, 2)).repeat(m, m)
        for a in (0, 2):   # the two rows of a complex coefficient share one step
            both = torch.maximum(rows[a], rows[a + 1])
            rows[a], rows[a + 1] = torch.where(self.low, rows[a], both), torch.where(self.low, rows[a + 1], both)
        return rows, cols

    def ball(self, z, radius):
        c1, c2 = _ball(z[:2], radius), _ball(z[2:], radius)
        return torch.where(self.low, z.clamp(-radius, radius), torch.cat([c1, c2]))

    def norm(self, z):
        c = torch.sqrt(z[0] ** 2 + z[1] ** 2) + torch.sqrt(z[2] ** 2 + z[3] ** 2)
        return torch.where(self.low, z.abs().sum(0), c).sum()


def _inv(s):
    return torch.where(s > 0, 1 / s.clamp(min=1e-300), torch.ones_like(s))


def _pdhg(p, f, xi, iters):
    """The primal-dual iteration with the alpha = 1 diagonal steps in 64 bits."""
    n, reg, alpha, ratio = p["n"], p["reg"], p["alpha"], p["ratio"]
    ab = alpha * p["beta"]
    A, f = _SparseK(p), f.double().reshape(-1)
    one = torch.ones(n, n, device=_dev(), dtype=torch.float64)
    krow, kcol = A.up(one), A.down(torch.ones_like(f))
    a = torch.zeros(n, n, device=_dev(), dtype=torch.float64)
    a[:, :-1] = 1
    b = a.T.contiguous()
    ex = a + a.flip(1)
    ey = ex.T
    W = _Cwt(n, 4) if reg == "dtcwt" else None
    if reg == "dtcwt":
        rows, cols = W.sums()
        sig_r, tau = _inv(rows), 1 / (kcol + cols)
    elif reg == "dtv":
        x64 = xi.double()
        d00, d01, d11 = 1 - GAMMA * x64[0] ** 2, -GAMMA * x64[0] * x64[1], 1 - GAMMA * x64[1] ** 2
        row0 = d00.abs() * a + d01.abs() * b + (d00 * a + d01 * b).abs()
        row1 = d01.abs() * a + d11.abs() * b + (d01 * a + d11 * b).abs()
        sig_r = _inv(torch.maximum(row0, row1))
        col = kcol + (d00 * a + d01 * b).abs() + (d01 * a + d11 * b).abs()
        col[:, 1:] += (d00.abs() + d01.abs())[:, :-1]
        col[1:, :] += (d01.abs() + d11.abs())[:-1, :]
        tau = 1 / col
    else:
        tau = 1 / (kcol + ex + ey)
        sig_r = _inv(2 * torch.maximum(a, b)) if reg == "tv" else 1 / (2 * torch.maximum(a, b) + 1)
    sig_s = 1 / torch.maximum(torch.maximum(ex, ey), (ex + ey) / math.sqrt(2))
    tau_v = torch.stack([1 / (1 + 2 * a + math.sqrt(2) * b), 1 / (1 + 2 * b + math.sqrt(2) * a)]) * ratio
    sig_q, tau, sig_r, sig_s = _inv(krow) / ratio, tau * ratio, sig_r / ratio, sig_s / ratio

    def D(g):   # D_xi g (its own transpose)
        return g - GAMMA * x64 * (x64 * g).sum(0) if reg == "dtv" else g

    up = W.up if W else lambda u: D(_grad(u))
    down = W.down if W else lambda r: _minus_div(D(r))
    ball = W.ball if W else _ball
    u, ub, q = torch.zeros_like(one), torch.zeros_like(one), torch.zeros_like(f)
    r = torch.zeros(4 if W else 2, n, n, device=_dev(), dtype=torch.float64)
    v, s = torch.zeros(2, n, n, device=_dev(), dtype=torch.float64), torch.zeros(3, n, n, device=_dev(), dtype=torch.float64)
    vb = v.clone()
    tgv = reg == "tgv"
    for _ in range(iters):
        q = (q + sig_q * (A.up(ub) - f)) / (1 + sig_q)
        r = ball(r + sig_r * (up(ub) - (vb if tgv else 0)), alpha)
        if tgv:
            s = _ball(s + sig_s * _sym(vb), ab)
            v1 = v - tau_v * (_sym_t(s) - r)
            vb, v = 2 * v1 - v, v1
        u1 = u - tau * (A.down(q) + down(r))
        ub, u = 2 * u1 - u, u1
    g = up(u) - (v if tgv else 0)
    pen = W.norm(g) if W else torch.sqrt((g * g).sum(0)).sum()
    if tgv:
        e = _sym(v)
        pen = pen + p["beta"] * torch.sqrt((e * e).sum(0)).sum()
    primal = 0.5 * ((A.up(u) - f) ** 2).sum() + alpha * pen
    dual = -(0.5 * (q * q).sum() + (q * f).sum()) - BOX_U * (A.down(q) + down(r)).abs().sum()
    if tgv:
        dual = dual - BOX_V * (_sym_t(s) - r).abs().sum()
    x = torch.cat([u.reshape(-1), v.reshape(-1)]) if tgv else u.reshape(-1)
    y = torch.cat([q, r.reshape(-1), s.reshape(-1)]) if tgv else torch.cat([q, r.reshape(-1)])
    return dict(u=u, x=x, y=y, primal=float(primal), gap=float(primal - dual), iters=iters)


def _unet_exact(c, seed):
    """The network in 64 bits without the 16-bit rounding of its activations.  Its parameter
    gradients have no such value: the stored activations' rounding decides which units are on."""
    x, dy, params = _unet_inputs(c, seed)
    F = torch.nn.functional
    convs, at, ws = _unet_convs(c), 0, []
    for ci, co in convs:
        w = params[at:at + co * 9 * ci].bfloat16().double().reshape(co, 3, 3, ci).permute(0, 3, 1, 2)
        ws.append((w, params[at + co * 9 * ci:at + co * 9 * ci + co].double()))
        at += co * 9 * ci + co
    k = iter(ws)

    def conv(t, act=True):
        w, b = next(k)
        o = F.conv2d(t, w, b, padding=1)
        return o.clamp(min=0) if act else o

    t, skips = x.double().permute(0, 3, 1, 2), []
    for l in range(c["levels"]):
        t = conv(conv(F.avg_pool2d(t, 2) if l else t))
        skips.append(t)
    for l in range(c["levels"] - 2, -1, -1):
        t = conv(conv(torch.cat([F.interpolate(t, scale_factor=2, mode="nearest"), skips[l]], 1)))
    return dict(y=conv(t, False).permute(0, 2, 3, 1).contiguous(), grad=None)


def exact(case, seed):
    c = case
    if c["kind"] == "forward":
        return _project(_phantom(c["n"], seed).float(), c["n_det"], c["n_t"], c["m"], c["arc"])
    if c["kind"] == "adjoint":
        return _backproject(_fast_data(c, seed), c["n"], c["m"], c["arc"])
    if c["kind"] in ("solve", "batch"):
        out = [_pdhg(p, _data(p, seed, k), _direction(p["n"], seed, k) if p["reg"] == "dtv" else None, c["iters"])
               for k, p in enumerate(_problems(c))]
        return out[0] if c["kind"] == "solve" else out
    if c["kind"] == "unet":
        return _unet_exact(c, seed)
    x, w, bias, dy = _conv_inputs(c, seed)
    xd, wd, dyd = x.double().permute(0, 3, 1, 2), w.double().permute(0, 3, 1, 2), dy.double().permute(0, 3, 1, 2)
    if c["kind"] == "conv_fwd":
        y = torch.nn.functional.conv2d(xd, wd, bias.double(), padding=1)
        return (y.clamp(min=0) if c["relu"] else y).permute(0, 2, 3, 1).contiguous()
    dx = torch.nn.functional.conv_transpose2d(dyd, wd, padding=1)
    xp = torch.nn.functional.pad(xd, (1, 1, 1, 1))
    dw = torch.stack([torch.stack([torch.einsum("nchw,nohw->oc", xp[:, :, i:i + c["h"], j:j + c["w"]], dyd)
                                   for j in range(3)], 1) for i in range(3)], 1)
    return dict(dx=dx.permute(0, 2, 3, 1).contiguous(), dw=dw, db=dyd.sum((0, 2, 3)))
