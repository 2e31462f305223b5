"""The work a user of this package has it do, as cases that can be timed and
checked: stepping lattices (2-D and 3-D, FP32 and FP16 storage, one lattice or
a sweep of them), the allocation-free step, and the surrogate's training and
prediction.  Every case goes through the public entry points
(include/inkjet.h, include/surrogate.h and their Python bindings).

``exact`` holds an independent FP64 statement of the same mathematics in plain
torch (whole-field operations on a padded lattice), used to see how far a
result is from the model itself.
"""
import ctypes as C
import math

import numpy as np
import torch

from paper_1702_04487_gb300 import inkjet as ij
from paper_1702_04487_gb300 import surrogate as sg

_c = C.CDLL(ij.library_path())  # the C entry points the bindings do not wrap

# ---------------------------------------------------------------------------
# Cases


def _lat(name, count, nx, ny, width, length, wall, steps, nz=0, half=0, tune=0, layout=-1):
    """`count` lattices of one handle, `steps` time steps, then every
    lattice's populations (and, of a single lattice, its newest record).
    layout >= 0: an uneven sweep, nozzle widths drawn by that number, lattice
    4 w x 30 w, nozzle length 4 w (nx .. length then only bound the sizes)."""
    c = dict(kind="lattice", count=count, nx=nx, ny=ny, nz=nz, width=width, length=length,
             wall=wall, steps=steps, half=half, tune=tune, layout=layout)
    return dict(c, name=name) if name else c


def listed():
    return [
        # One step between the caller's own buffers: a solver loop inside
        # another framework that owns all device memory; the smallest call.
        dict(name="noalloc_64x256", kind="noalloc", nx=64, ny=256, width=20, length=60, wall=4),
        # The 64 x 256 planar nozzle alone: a design study of one nozzle, ten
        # diagnostics periods between two looks at it; launch-bound.
        _lat("planar_64x256", 1, 64, 256, 20, 60, 4, 100),
        # The angle x surface-tension sweep at paper-like scale: 20 lattices
        # of 200 x 1600, launch shape tuned once as the README shows.
        _lat("sweep_20x200x1600", 20, 200, 1600, 50, 200, 10, 50, tune=1),
        # The same sweep in FP16 storage.
        _lat("sweep_20x200x1600_fp16", 20, 200, 1600, 50, 200, 10, 50, half=1, tune=1),
        # Uneven sweep, 256 instances in one launch, untuned: what the
        # surrogate service runs to make training data and to answer
        # rejected queries.
        _lat("uneven_256", 256, 192, 1440, 48, 192, 4, 100, layout=3),
        # A few lattices of odd width and height, untuned: a hand-made nozzle
        # whose sizes come from a drawing (odd widths copy by column).
        _lat("odd_4x251x1203", 4, 251, 1203, 61, 151, 11, 50),
        # The 3-D round nozzle, 60 and 120 degrees in one handle, FP32.
        _lat("round_2x128x128x640", 2, 128, 128, 24, 160, 10, 20, nz=640, tune=1),
        # The same in FP16 storage.
        _lat("round_2x128x128x640_fp16", 2, 128, 128, 24, 160, 10, 20, nz=640, half=1, tune=1),
        # Its quarter-size downscale alone, untuned: quick 3-D trials.
        _lat("round_32x32x160", 1, 32, 32, 6, 40, 3, 50, nz=160),
        # One gated surrogate query (an interactive caller).
        dict(name="predict_1", kind="predict", rows=1, members=5, hidden=256, train_rows=4096),
        # The largest batch the service is quoted on.
        dict(name="predict_65536", kind="predict", rows=65536, members=5, hidden=256,
             train_rows=4096),
        # Training the ensemble (default minibatch), 50 Adam steps.
        dict(name="train_256", kind="train", batch=256, members=5, hidden=256, train_rows=4096,
             steps=50),
    ]


def _log_int(rng, lo, hi):
    return max(lo, min(hi, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    kind = rng.choice(["noalloc", "2d", "2d", "2d", "3d", "3d", "uneven", "predict", "predict",
                       "train"])
    if kind == "uneven":
        n = _log_int(rng, 8, 256)
        return _lat("", n, 192, 1440, 48, 192, 4, 10 * rng.randint(2, 10),
                    layout=rng.randint(4, 10000))
    if kind in ("noalloc", "2d"):
        nx, ny = _log_int(rng, 48, 1200), _log_int(rng, 96, 4000)
        width = max(8, nx // rng.randint(3, 5))
        length = max(16, ny // rng.randint(4, 9))
        wall = max(2, min(10, nx // 20))
        if kind == "noalloc":
            return dict(kind="noalloc", nx=nx, ny=ny, width=width, length=length, wall=wall)
        half = rng.randint(0, 2) == 2
        if half:
            nx += nx % 2
        count = _log_int(rng, 1, max(1, min(64, 16000000 // (nx * ny))))
        return _lat("", count, nx, ny, width, length, wall, 10 * rng.randint(2, 8),
                    half=int(half), tune=rng.randint(0, 1))
    if kind == "3d":
        nx, ny = _log_int(rng, 24, 140), _log_int(rng, 24, 140)
        nz = _log_int(rng, 48, 640)
        half = rng.randint(0, 1)
        if half:
            nx += nx % 2
        m = min(nx, ny)
        radius, wall = max(4, m // 5), max(2, m // 14)
        return _lat("", rng.randint(1, 2), nx, ny, radius, max(8, nz // 4), wall,
                    10 * rng.randint(1, 2), nz=nz, half=half, tune=rng.randint(0, 1))
    net = dict(members=rng.choice([3, 5, 5, 8]), hidden=rng.choice([64, 128, 192, 256, 256]),
               train_rows=_log_int(rng, 512, 4096))
    if kind == "predict":
        return dict(kind="predict", rows=_log_int(rng, 1, 65536), **net)
    return dict(kind="train", batch=16 * _log_int(rng, 4, 64), steps=rng.randint(20, 60), **net)


# ---------------------------------------------------------------------------
# Lattice parameters and input states


def _sizes(case):
    """(nx, ny, nz, nozzle width or radius, length, wall) of every lattice."""
    if case["layout"] < 0:
        one = (case["nx"], case["ny"], case["nz"], case["width"], case["length"], case["wall"])
        return [one] * case["count"]
    r = np.random.default_rng(case["layout"])
    ws = r.integers(16, case["width"] + 1, case["count"])
    return [(4 * int(w), 30 * int(w), 0, int(w), 4 * int(w), case["wall"]) for w in ws]


def _params(size, rng, k, precision=0):
    """One lattice: angle, surface tension and drive drawn as in the sweeps."""
    nx, ny, nz, width, length, wall = size
    f0 = float(rng.uniform(1e-4, 2e-4))
    p = dict(nx=nx, ny=ny, geometry=1, nozzle_width=width, nozzle_length=length,
             wall_thickness=wall, rho_ink=10.0, rho_air=1.0, nu_ink=0.1, nu_air=0.05,
             sigma=0.01 * float(np.exp(rng.uniform(np.log(0.5), np.log(4.0)))), width_W=3.0,
             tau_phi=0.8, theta_deg=float(rng.uniform(30.0, 150.0)), F0=f0, F_neg=f0 / 2,
             T1=int(rng.integers(500, 1501)), T2=int(rng.integers(500, 1501)), diag_every=10,
             precision=precision, seed=k)
    return dict(p, dim=3, nz=nz) if nz else p


def _dirs(dim):
    """Directions (axial axis first, as the arrays are indexed), weights and
    the number of g directions, in the public order."""
    if dim == 2:
        xy = [(0, 0), (1, 0), (0, 1), (-1, 0), (0, -1), (1, 1), (-1, 1), (-1, -1), (1, -1)]
        return [(y, x) for x, y in xy], [4 / 9] + [1 / 9] * 4 + [1 / 36] * 4, 5
    d = [(0, 0, 0), (1, 0, 0), (-1, 0, 0), (0, 1, 0), (0, -1, 0), (0, 0, 1), (0, 0, -1)]
    for a, b in ((0, 1), (0, 2), (1, 2)):
        for sa, sb in ((1, 1), (-1, 1), (1, -1), (-1, -1)):
            v = [0, 0, 0]
            v[a], v[b] = sa, sb
            d.append(tuple(v))
    return [(z, y, x) for x, y, z in d], [1 / 3] + [1 / 18] * 6 + [1 / 36] * 12, 7


def _geometry(p):
    """(solid, wetting face, channel cross-section, distance of a column to
    the channel, shape) on the GPU."""
    dev = "cuda"
    x = torch.arange(p["nx"], device=dev, dtype=torch.float64)
    if p.get("dim", 2) == 2:
        a = torch.arange(p["ny"], device=dev)[:, None]
        w, t = p["nozzle_width"], p["wall_thickness"]
        c0 = (p["nx"] - w) // 2
        chan = ((x >= c0) & (x < c0 + w))[None]
        wall = (((x >= c0 - t) & (x < c0)) | ((x >= c0 + w) & (x < c0 + w + t)))[None]
        wet = ((x == c0 - 1) | (x == c0 + w))[None]
        beside = torch.maximum(c0 - x, x - (c0 + w - 1)).clamp(min=0.0)[None]
        shape = (p["ny"], p["nx"])
    else:
        a = torch.arange(p["nz"], device=dev)[:, None, None]
        y = torch.arange(p["ny"], device=dev, dtype=torch.float64)[:, None]
        r2 = (x - 0.5 * (p["nx"] - 1)) ** 2 + (y - 0.5 * (p["ny"] - 1)) ** 2
        r, t = p["nozzle_width"], p["wall_thickness"]
        inside = r2 < r * r
        ring = ~inside & (r2 < (r + t) ** 2)
        near = torch.zeros_like(inside)
        for dim in (0, 1):
            for s in (1, -1):
                near |= torch.roll(inside, s, dim)
        chan, wall, wet = inside[None], ring[None], (ring & near)[None]
        beside = (r2.sqrt() - r).clamp(min=0.0)[None]
        shape = (p["nz"], p["ny"], p["nx"])
    low = a < p["nozzle_length"]
    return ((low & wall).expand(shape), (low & wet).expand(shape), (low & chan).expand(shape),
            beside, shape)


def _waves(shape, rng, n=4):
    """A smooth random field of size about one, periodic in every axis."""
    out = torch.zeros(shape, device="cuda")
    for _ in range(n):
        arg = torch.zeros(1, device="cuda") + float(rng.uniform(0, 2 * np.pi))
        for ax, m in enumerate(shape):
            k = int(rng.integers(1, 4 if ax else 9))
            v = torch.arange(m, device="cuda", dtype=torch.float32) * (2 * np.pi * k / m)
            arg = arg + v.reshape([-1 if j == ax else 1 for j in range(len(shape))])
        out += torch.sin(arg)
    return out / n


def _constants(p):
    ri, ra, s, w = p["rho_ink"], p["rho_air"], p["sigma"], p["width_W"]
    phis, n0 = 0.5 * (ri - ra), 0.5 * (ri + ra)
    A, kappa = 3 * s / (8 * w * phis ** 4), 3 * s * w / (4 * phis ** 2)
    lo, hi, target = -1.0, 1.0, math.cos(math.radians(p["theta_deg"]))
    for _ in range(200):  # Cahn: cos(theta) = ((1 + o)^1.5 - (1 - o)^1.5) / 2
        o = 0.5 * (lo + hi)
        if 0.5 * ((1 + o) ** 1.5 - (1 - o) ** 1.5) < target:
            lo = o
        else:
            hi = o
    h = 0.5 * (lo + hi) * phis ** 2 * math.sqrt(2 * kappa * A)
    return dict(phis=phis, n0=n0, A=A, kappa=kappa, q=1 / (p["tau_phi"] + 0.5),
                gamma=0.04 / kappa, hk=h / kappa)


def _state(p, rng):
    """Populations (FP32, absolute) of a nozzle in mid-push: ink up to the
    exit with a diffuse meniscus, moving up the channel, with a smooth
    disturbance of velocity and density everywhere; solid cells 0."""
    dim = p.get("dim", 2)
    c, w, qg = _dirs(dim)
    k = _constants(p)
    solid, _, chan, beside, shape = _geometry(p)
    ax = torch.arange(shape[0], device="cuda", dtype=torch.float64)
    up = (ax - p["nozzle_length"]).reshape([-1] + [1] * (dim - 1))
    away = (beside ** 2 + up.clamp(min=0.0) ** 2).sqrt()
    phi = torch.where(beside > 0, torch.where(up < 0, -1.0, torch.tanh(-away / p["width_W"])),
                      torch.tanh(-up / p["width_W"])) * k["phis"]
    phi = phi.float()
    n = k["n0"] * (1 + 1e-3 * _waves(shape, rng))
    push = float(rng.uniform(0.01, 0.03))
    u = [0.004 * _waves(shape, rng) for _ in range(dim)]
    u[0] = u[0] + push * torch.exp(-(beside.float() / 4) ** 2) * torch.exp(
        -up.float().clamp(min=0.0) / 20)
    u2 = sum(v * v for v in u)
    fl = (~solid).float()
    f = torch.empty((len(c),) + tuple(shape), device="cuda")
    g = torch.empty((qg,) + tuple(shape), device="cuda")
    for i in range(len(c)):
        cu = sum(e * v for e, v in zip(c[i], u))
        f[i] = w[i] * n * (1 + 3 * cu + 4.5 * cu * cu - 1.5 * u2) * fl
        if 0 < i < qg:
            g[i] = phi * cu / (2 * k["q"]) * fl
    g[0] = (phi - g[1:].sum(0)) * fl
    return f, g


def _lattices(case, seed):
    rng = np.random.default_rng([seed, 17])
    return [_params(s, rng, k, case.get("half", 0)) for k, s in enumerate(_sizes(case))]


def _ptr(t, offset=0):
    return C.c_void_p(t.data_ptr() + 4 * offset)


def _ok(status):
    if status:
        raise RuntimeError("status %d: %s" % (status, ij.ij_last_error()))


# ---------------------------------------------------------------------------
# Surrogate inputs


def _rows(n, rng, spread=1.0):
    """Raw input rows of the sampler's ranges (idle time zero)."""
    x = np.zeros((n, 7))
    x[:, 0] = rng.uniform(90 - 70 * spread, 90 + 70 * spread, n)
    x[:, 1] = 0.0025 * np.exp(rng.uniform(-0.69 * spread, 0.69 * spread, n))
    x[:, 2] = 5e-4 * np.exp(rng.uniform(-1.5 * spread, 1.5 * spread, n))
    x[:, 3] = np.floor(500 + 4000 * rng.random(n) * spread)
    x[:, 4] = np.floor(500 + 4000 * rng.random(n) * spread)
    x[:, 6] = rng.integers(16, 49, n)
    return x.astype(np.float32)


def _outcomes(x, rng):
    """Smooth outcomes of the size the lattices give."""
    x = x.astype(np.float64)
    tc = np.sqrt(10 * x[:, 6] ** 3 / x[:, 1])
    y = np.empty((len(x), 4))
    y[:, 0] = tc * (1.2 + x[:, 0] / 300) * (5e-4 / x[:, 2]) ** 0.3
    y[:, 1] = 0.01 + 0.02 * np.tanh(x[:, 2] * x[:, 3]) - 4e-5 * x[:, 0]
    y[:, 2] = 1.5 * x[:, 6] ** 2 * (1 + 0.2 * np.sin(x[:, 0] / 30))
    y[:, 3] = np.floor(1.5 + np.sin(x[:, 4] / 900))
    y[:, :3] *= 1 + 0.01 * rng.standard_normal((len(x), 3))
    return y.astype(np.float32)


def _net_shapes(hidden):
    return [(hidden, 16)] + [(hidden, hidden)] * 3 + [(16, hidden)]


def _weights(case, rng, differ):
    """Parameter vectors of the members: He-uniform weights, members apart by
    `differ` of the bound (1: independent), padding zero."""
    shapes = _net_shapes(case["hidden"])
    base, out = None, []
    for _ in range(case["members"]):
        v = []
        for l, (o, i) in enumerate(shapes):
            fan = 7 if l == 0 else i
            wt = np.zeros((o, i))
            wt[:4 if l == 4 else o, :fan] = rng.uniform(-1, 1, (4 if l == 4 else o, fan)) * \
                math.sqrt(6 / fan)
            b = np.zeros(o)
            b[:4 if l == 4 else o] = rng.uniform(-0.1, 0.1, 4 if l == 4 else o)
            v += [wt.ravel(), b]
        v = np.concatenate(v)
        base = v if base is None else base
        out.append((v if differ == 1 else base + differ * v).astype(np.float32))
    return out


def _surrogate_inputs(case, seed):
    rng = np.random.default_rng([seed, 23])
    x = _rows(case["train_rows"], rng)
    y = _outcomes(x, rng)
    if case["kind"] == "train":
        return x, y, _weights(case, rng, 1), None
    par = _weights(case, rng, 0.02)
    # queries: nine tenths inside the sampler's ranges, the rest beyond them
    n = case["rows"]
    far = n // 10
    q = np.concatenate([_rows(n - far, rng, 0.98), _rows(far, rng, 1.4)]) if far else _rows(n, rng)
    return x, y, par, np.ascontiguousarray(q[rng.permutation(n)])


# ---------------------------------------------------------------------------


def prepare(case, seed):
    if case["kind"] in ("predict", "train"):
        x, y, par, q = _surrogate_inputs(case, seed)
        s = sg.Surrogate(members=case["members"], hidden=case["hidden"], seed=seed % 1000003,
                         batch=case.get("batch", 256))
        s.set_data(x, y)
        for m, v in enumerate(par):
            s.set_params(m, v)
        if case["kind"] == "predict":
            s.set_gate(0.03, 0.06)
        return dict(kind=case["kind"], s=s, q=q, steps=case.get("steps", 0))
    rng = np.random.default_rng([seed, 29])
    if case["kind"] == "noalloc":
        p = _params((case["nx"], case["ny"], 0, case["width"], case["length"], case["wall"]), rng, 0)
        f, g = _state(p, rng)
        n0 = _constants(p)["n0"]
        fluid = (f[0] != 0).float()
        for i, w in enumerate(_dirs(2)[1]):  # the stored layout: f_i - w_i n0
            f[i] -= float(np.float32(w) * np.float32(n0)) * fluid
        return dict(kind="noalloc", p=ij.make_params(p), t=int(rng.integers(0, 500)), f=f, g=g,
                    fo=torch.empty_like(f), go=torch.empty_like(g),
                    status=torch.zeros(1, dtype=torch.int32, device="cuda"))
    plist = _lattices(case, seed)
    h = ij.ij_create(plist)
    nf, ng = (19, 7) if case["nz"] else (9, 5)
    cells = [p["nx"] * p["ny"] * p.get("nz", 1) for p in plist]
    for k, p in enumerate(plist):
        f, g = _state(p, rng)
        _ok(_c.ij_set_state(h.ptr, C.c_int(k), _ptr(f), _ptr(g), C.c_longlong(0), C.c_int(1)))
    del f, g
    if case["tune"]:
        ij.ij_autotune(h)
    at = np.concatenate([[0], np.cumsum(cells)])
    total = int(at[-1])
    return dict(kind="lattice", h=h, count=len(plist), steps=case["steps"],
                f=torch.empty(nf * total, device="cuda"), g=torch.empty(ng * total, device="cuda"),
                at_f=[int(nf * a) for a in at], at_g=[int(ng * a) for a in at])


def run(state):
    if state["kind"] == "predict":
        mean, sd, accept = state["s"].predict(state["q"])
        return dict(mean=mean, sd=sd, accept=accept)
    if state["kind"] == "train":
        s = state["s"]
        loss = s.train(state["steps"])
        return dict(loss=loss, params=[s.get_params(m) for m in range(s.members)])
    if state["kind"] == "noalloc":
        stream = C.c_void_p(torch.cuda.current_stream().cuda_stream)
        _ok(_c.ij_step_noalloc(C.byref(state["p"]), C.c_longlong(state["t"]), _ptr(state["f"]),
                               _ptr(state["g"]), _ptr(state["fo"]), _ptr(state["go"]), None,
                               _ptr(state["status"]), stream))
        return dict(f=state["fo"], g=state["go"], status=state["status"])
    h = state["h"]
    ij.ij_step(h, state["steps"])
    for k in range(state["count"]):
        _ok(_c.ij_get_state(h.ptr, C.c_int(k), _ptr(state["f"], state["at_f"][k]),
                            _ptr(state["g"], state["at_g"][k]), C.c_int(1)))
    out = dict(f=state["f"], g=state["g"])
    if state["count"] == 1:
        out["record"] = ij.ij_observe(h, 0, phi=False)[0]
    return out


def work(case):
    if case["kind"] in ("predict", "train"):
        H, K = case["hidden"], case["members"]
        params = 16 * H + 3 * H * H + 16 * H + 4 * H + 16
        mac = 7 * H + 3 * H * H + 4 * H
        if case["kind"] == "predict":
            n = case["rows"]
            # queries in, answers out, the members' BF16 weights and the
            # training points of the gate once; the distance of every query
            # to every training point is part of the answer
            return dict(bytes=n * (28 + 36) + K * params * 2 + case["train_rows"] * 28,
                        flops=2.0 * n * K * mac + 21.0 * n * case["train_rows"])
        # per step: parameters, moments (read and written) and a minibatch
        return dict(bytes=case["steps"] * K * (params * 24 + case["batch"] * 46) + K * params * 4,
                    flops=6.0 * case["steps"] * K * case["batch"] * mac)
    if case["kind"] == "noalloc":
        n = case["nx"] * case["ny"]
        return dict(bytes=n * 112, flops=n * 330)
    cells = sum(s[0] * s[1] * max(1, s[2]) for s in _sizes(case))
    if case["nz"]:
        per, out, flops = (108, 54 + 104) if case["half"] else (208, 104 + 104), 0, 640
    else:
        per, out, flops = (60, 30 + 56) if case["half"] else (112, 56 + 56), 0, 330
    per, out = per
    return dict(bytes=cells * (per * case["steps"] + out), flops=cells * flops * case["steps"])


# ---------------------------------------------------------------------------
# The model in FP64


def _shift(a, c, back=False):
    """a at x + c (back: at x - c), periodic."""
    s = [(e if back else -e) for e in c]
    dims = [d for d, e in enumerate(s) if e]
    return torch.roll(a, [s[d] for d in dims], dims) if dims else a


def _pad(a):
    """Three more planes at both axial ends, repeating the end plane."""
    return torch.cat([a[:1]] * 3 + [a] + [a[-1:]] * 3)


def _exact_lattice(p, f, g, t0, steps):
    """(f, g, newest record) after `steps` steps from time t0."""
    dim = p.get("dim", 2)
    c, w, qg = _dirs(dim)
    Q, k = len(c), _constants(p)
    opp = [c.index(tuple(-e for e in v)) for v in c]
    solid0, wet0, chan0, _, shape = _geometry(p)
    solid, wet, chan = _pad(solid0), _pad(wet0), _pad(chan0)
    f, g = f.double(), g.double()
    phis, n0, q, tphi = k["phis"], k["n0"], k["q"], p["tau_phi"]
    faces = [v for v in c if sum(map(abs, v)) == 1]
    edges = [v for v in c if sum(map(abs, v)) == 2]
    fluid = (~solid).double()
    cf = sum(_shift(fluid, v) for v in faces)
    ce = sum(_shift(fluid, v) for v in edges)
    from_solid = [_shift(solid, v, True) for v in c]
    rec = None
    for s in range(steps):
        t = t0 + s
        F0 = p["F0"] if t < p["T1"] else (-p["F_neg"] if t < p["T1"] + p["T2"] else 0.0)
        fp = [_pad(v) for v in f]
        gp = [_pad(v) for v in g]
        phi = sum(gp)
        fo = phi * fluid
        by_face = sum(_shift(fo, v) for v in faces) / cf.clamp(min=1) + k["hk"] * wet.double()
        by_edge = sum(_shift(fo, v) for v in edges) / ce.clamp(min=1)
        hat = torch.where(solid, torch.where(cf > 0, by_face, by_edge), phi)
        lap = torch.zeros_like(phi)
        grad = [torch.zeros_like(phi) for _ in range(dim)]
        for i in range(1, Q):
            nb = _shift(hat, c[i])
            lap += 6 * w[i] * (nb - hat)
            for a in range(dim):
                if c[i][a]:
                    grad[a] += 3 * w[i] * c[i][a] * nb
        mu = 4 * k["A"] * phi * (phi ** 2 - phis ** 2) - k["kappa"] * lap
        ink = (0.5 * (phi / phis + 1)).clamp(0, 1)
        F = [mu * d for d in grad]
        F[0] = F[0] + F0 * ink * chan
        n = sum(fp)
        n = torch.where(solid, torch.full_like(n, n0), n)
        u = [(sum(c[i][a] * fp[i] for i in range(Q) if c[i][a]) + 0.5 * F[a]) / n
             for a in range(dim)]
        if t % 10 == 0:
            rec = _record(p, k, t, phi[3:-3], n[3:-3], u[0][3:-3], solid0)
        om = 1 / (0.5 + 3 * (p["nu_air"] + ink * (p["nu_ink"] - p["nu_air"])))
        u2 = sum(v * v for v in u)
        uF = sum(a * b for a, b in zip(u, F))
        p3 = 3 * (phi * mu + n / 3)
        rest = torch.zeros_like(phi)
        fs = [None] * Q
        for i in range(1, Q):
            cu = sum(e * v for e, v in zip(c[i], u) if e)
            cF = sum(e * v for e, v in zip(c[i], F) if e)
            eq = w[i] * (p3 + n * (3 * cu + 4.5 * cu ** 2 - 1.5 * u2))
            fo = (1 - om / 2) * w[i] * (3 * cF - 3 * uF + 9 * cu * cF)
            rest += om * eq + fo
            fs[i] = fp[i] + om * (eq - fp[i]) + fo
        fs[0] = fp[0] + om * (n - fp[0]) - rest
        move = [None] * qg
        ges = torch.zeros_like(phi)
        for i in range(1, qg):
            ge = 0.5 * k["gamma"] * mu + phi * sum(e * v for e, v in zip(c[i], u) if e) / (2 * q)
            ges += ge
            move[i] = q * gp[i] + (ge - gp[i]) / tphi
        g0 = gp[0] + (phi - ges - gp[0]) / tphi
        inner = slice(3, -3)
        f = torch.stack([torch.where(from_solid[i], fs[opp[i]], _shift(fs[i], c[i], True))[inner]
                         if i else fs[0][inner] for i in range(Q)])
        g = torch.stack([((1 - q) * gp[i] + torch.where(from_solid[i], move[opp[i]], _shift(
            move[i], c[i], True)))[inner] if i else g0[inner] for i in range(qg)])
        f[:, solid0] = 0
        g[:, solid0] = 0
    return f, g, rec


def _record(p, k, t, phi, n, u, solid):
    """The diagnostics record of one state (before any breakup)."""
    fl = (~solid).double()
    e = (phi / k["phis"]).clamp(0, 1) * fl
    cross = tuple(range(1, phi.dim()))
    w, m, pr = (v.sum(cross).cpu().numpy() for v in (e, e * n, e * n * u))
    A, L = len(w), p["nozzle_length"]
    need = p["nozzle_width"] if p.get("dim", 2) == 2 else math.pi * p["nozzle_width"] ** 2
    run = w > 0.5
    ink = np.where(run, w, 0.0)
    above = np.concatenate([np.cumsum(ink[::-1])[::-1][1:], [0.0]])
    rows = [y for y in range(L - L // 2, A) if above[y] > need]
    neck = min((w[y] for y in rows), default=1e30)
    starts = [y for y in range(A) if run[y] and (y == 0 or not run[y - 1])]
    r = dict(step=float(t), mass_n=float((n * fl).sum()), mass_phi=float((phi * fl).sum()),
             mom_y=float((n * u * fl).sum()), neck=float(neck),
             breakup_step=float(t) if neck < 0.01 else -1.0, droplet_volume=0.0,
             droplet_centroid_y=0.0, droplet_velocity=0.0,
             satellites=float(max(0, sum(y >= L for y in starts) - 1)), runs=float(len(starts)),
             head_y=-1.0, tail_y=-1.0)
    if starts:
        a = starts[-1]
        b = a
        while b < A and run[b]:
            b += 1
        vol = w[a:b].sum()
        r.update(droplet_volume=float(vol),
                 droplet_centroid_y=float((np.arange(a, b) * w[a:b]).sum() / vol),
                 droplet_velocity=float(pr[a:b].sum() / m[a:b].sum()),
                 head_y=float(b - 1 + (w[b - 1] - 0.5) / (w[b - 1] - w[b])) if b < A else A - 1.0,
                 tail_y=float(a - (w[a] - 0.5) / (w[a] - w[a - 1])) if a > 0 else 0.0)
    return r


def _mix64(z):
    m = (1 << 64) - 1
    z = (z + 0x9E3779B97F4A7C15) & m
    z = ((z ^ (z >> 30)) * 0xBF58476D1CE4E5B9) & m
    z = ((z ^ (z >> 27)) * 0x94D049BB133111EB) & m
    return z ^ (z >> 31)


def _columns(a, logs):
    """Transformed columns (log where the bit is set, then z-score), their
    mean and scale."""
    a = a.astype(np.float64)
    a = np.stack([np.log(a[:, d]) if logs >> d & 1 else a[:, d] for d in range(a.shape[1])], 1)
    mean, sd = a.mean(0), a.std(0)
    sd = np.where(sd > 1e-12, sd, 1.0)
    return (a - mean) / sd, mean, sd


def _unpack(v, hidden):
    out, at = [], 0
    for o, i in _net_shapes(hidden):
        out.append(v[at:at + o * i].reshape(o, i))
        out.append(v[at + o * i:at + o * i + o])
        at += o * i + o
    return out


def _forward(x, layers):
    for l in range(5):
        x = x @ layers[2 * l].T + layers[2 * l + 1]
        if l < 4:
            x = torch.nn.functional.gelu(x)
    return x


def _exact_surrogate(case, seed):
    x, y, par, q = _surrogate_inputs(case, seed)
    H = case["hidden"]
    cfg = sg.DEFAULT_CONFIG
    X, xm, xs = _columns(x, cfg["log_inputs"])
    T, ym, ys = _columns(y, cfg["log_outputs"])

    def pad(a):
        return torch.nn.functional.pad(torch.tensor(a, device="cuda"), (0, 9))

    if case["kind"] == "predict":
        q = q.astype(np.float64)
        q = np.stack([np.log(q[:, d]) if cfg["log_inputs"] >> d & 1 else q[:, d]
                      for d in range(7)], 1)
        Z = pad((q - xm) / xs)
        ys_t, ym_t = torch.tensor(ys, device="cuda"), torch.tensor(ym, device="cuda")
        outs = []
        for v in par:
            layers = _unpack(torch.tensor(v, device="cuda").double(), H)
            o = _forward(Z, layers)[:, :4] * ys_t + ym_t
            for d in range(4):
                if cfg["log_outputs"] >> d & 1:
                    o[:, d] = o[:, d].exp()
            outs.append(o)
        o = torch.stack(outs)
        return dict(mean=o.mean(0), sd=o.std(0, unbiased=False), accept=None)
    X, T = pad(X), torch.tensor(T, device="cuda")
    n, B, S = len(x), case["batch"], case["steps"]
    wt = torch.tensor(cfg["out_weight"], device="cuda", dtype=torch.float64)
    key = (seed % 1000003) ^ 0x5EED
    losses, params = [], []
    for m, v in enumerate(par):
        v = torch.tensor(v, device="cuda").double()
        m1, m2 = torch.zeros_like(v), torch.zeros_like(v)
        for s in range(S):
            rows = torch.tensor([_mix64(key ^ _mix64((m << 56) ^ (s << 24) ^ r)) % n
                                 for r in range(B)], device="cuda")
            a = v.clone().requires_grad_(True)
            out = _forward(X[rows], _unpack(a, H))[:, :4]
            loss = (wt * (out - T[rows]) ** 2).sum() / (4 * B)
            (gr,) = torch.autograd.grad(loss, a)
            # padding has no gradient: the padded inputs are zero, the padded
            # outputs are not in the loss
            m1 = cfg["beta1"] * m1 + (1 - cfg["beta1"]) * gr
            m2 = cfg["beta2"] * m2 + (1 - cfg["beta2"]) * gr * gr
            lr = cfg["lr"] * 0.5 * (1 + math.cos(math.pi * s / S))
            hat1, hat2 = m1 / (1 - cfg["beta1"] ** (s + 1)), m2 / (1 - cfg["beta2"] ** (s + 1))
            v = v - lr * hat1 / (hat2.sqrt() + cfg["eps"])
        losses.append(float(loss))
        params.append(v)
    return dict(loss=sum(losses) / len(losses), params=params)


def exact(case, seed):
    if case["kind"] in ("predict", "train"):
        return _exact_surrogate(case, seed)
    rng = np.random.default_rng([seed, 29])
    if case["kind"] == "noalloc":
        p = _params((case["nx"], case["ny"], 0, case["width"], case["length"], case["wall"]), rng, 0)
        f, g = _state(p, rng)
        fluid = (f[0] != 0).double()
        t = int(rng.integers(0, 500))
        ref = [float(np.float32(w) * np.float32(_constants(p)["n0"])) for w in _dirs(2)[1]]
        a = torch.stack([(f[i] - r * fluid.float()).double() + w * _constants(p)["n0"] * fluid
                         for i, (r, w) in enumerate(zip(ref, _dirs(2)[1]))])
        fo, go, _ = _exact_lattice(p, a, g, t, 1)
        fo = torch.stack([fo[i] - w * _constants(p)["n0"] * fluid
                          for i, w in enumerate(_dirs(2)[1])])
        return dict(f=fo, g=go, status=None)
    cells = sum(s[0] * s[1] * max(1, s[2]) for s in _sizes(case))
    if cells * case["steps"] > 5e8 or case["count"] * case["steps"] > 4000:
        return None  # about a minute or more of whole-field operations
    fs, gs = [], []
    for p in _lattices(case, seed):
        f, g = _state(p, rng)
        f, g, rec = _exact_lattice(p, f, g, 0, case["steps"])
        fs.append(f.reshape(-1))
        gs.append(g.reshape(-1))
    out = dict(f=torch.cat(fs), g=torch.cat(gs))
    if case["count"] == 1:
        out["record"] = rec
    return out
