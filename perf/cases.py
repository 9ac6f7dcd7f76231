"""Performance cases of the library: modelling, gradients, inner solves, frequency slices and
the preconditioner network, through the public entry points.

The sizes are the workloads of ``synth.py`` and of the benchmark (101 x 101, 201 x 201,
801 x 241, 1201 x 301, 400^3) with records short enough to time, plus odd and ragged sizes in
between.  Every input is made from the seed alone, on the GPU, without the library.

Kinds (what a user has the library do):

* ``forward``  : seismograms of point sources (``Context.forward``).
* ``gradient`` : adjoint-state gradient and misfit of one model (``Context.gradient``).
* ``saddle``   : saddle-point gradient and objective at an extended source.
* ``cg``       : the ESI (or WRI) normal equation, a fixed number of Algorithm 1 iterations.
* ``dscg``     : the same system in data space.  ``fdcg``: its frequency-domain form.
* ``dtft``     : forward modelling with on-the-fly frequency slices in FP16.
* ``pc_apply`` / ``pc_grad``: the preconditioner network, inference and training gradient.
"""
import math
import os

import numpy as np
import torch
import torch.nn.functional as F

from paper_2211_06300_gb300 import esi, synth

DT = {"f32": torch.float32, "f64": torch.float64}
W = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)


def listed():
    return [
        # the two-layer reflection test: one FP64 shot, the smallest call, latency alone
        dict(name="forward_small_f64", kind="forward", nz=101, ny=1, nx=101, ns=1, nt=500, nrec=101,
             dx=10.0, dt=1e-3, dtype="f64", off=False),
        # one point of the misfit-landscape scan: misfit and gradient of a single FP32 shot
        dict(name="gradient_landscape", kind="gradient", nz=201, ny=1, nx=201, ns=1, nt=1200,
             nrec=241, dx=10.0, dt=1e-3, dtype="f32", ckpt="f32", every=20, off=False),
        # observed data of a 2D line: 16 shots, a receiver on every column
        dict(name="forward_line", kind="forward", nz=241, ny=1, nx=801, ns=16, nt=1500, nrec=801,
             dx=12.5, dt=1e-3, dtype="f32", off=False),
        # the inner solve of the ESI step: 16 shots, diagonal preconditioner
        dict(name="esi_cg", kind="cg", nz=241, ny=1, nx=801, ns=16, nt=400, nrec=801, dx=12.5,
             dt=1e-3, dtype="f32", solver="diag", iters=5, lam=10.0, off=False),
        # the WRI inner solve on a ragged grid, receivers between the nodes
        dict(name="wri_cg_odd", kind="cg", nz=187, ny=1, nx=333, ns=5, nt=600, nrec=150, dx=12.5,
             dt=1e-3, dtype="f32", solver="wri", iters=6, lam=2e4, off=True),
        # the same ESI system solved in data space
        dict(name="data_space_cg", kind="dscg", nz=241, ny=1, nx=801, ns=16, nt=500, nrec=801,
             dx=12.5, dt=1e-3, dtype="f32", iters=4, lam=10.0, off=False),
        # ... and at four frequencies
        dict(name="frequency_cg", kind="fdcg", nz=241, ny=1, nx=801, ns=16, nt=500, nrec=801,
             dx=12.5, dt=1e-3, dtype="f32", iters=3, lam=10.0, nf=4, off=False),
        # the outer loop's gradient and objective at the inner solution
        dict(name="saddle_gradient", kind="saddle", nz=241, ny=1, nx=801, ns=16, nt=400, nrec=801,
             dx=12.5, dt=1e-3, dtype="f32", beta=0.5, off=False),
        # a survey's gradient: 64 shots of uneven apertures, BF16 checkpoints
        dict(name="gradient_survey", kind="gradient", nz=301, ny=1, nx=1201, ns=64, nt=400, nrec=501,
             dx=12.5, dt=1e-3, dtype="f32", ckpt="bf16", every=20, off=False),
        # a 3D volume's wavefield at five frequencies (the largest arrays)
        dict(name="dtft_volume", kind="dtft", nz=400, ny=400, nx=400, ns=1, nt=128, nrec=25600,
             dx=10.0, dt=0.8e-3, dtype="f32", nf=5, off=False),
        # a ragged 3D volume's gradient, two shots
        dict(name="gradient_volume_odd", kind="gradient", nz=150, ny=131, nx=187, ns=2, nt=150,
             nrec=900, dx=10.0, dt=0.8e-3, dtype="f32", ckpt="bf16", every=20, off=True),
        # the learned preconditioner applied to the images of a residual
        dict(name="pc_apply", kind="pc_apply", h=121, w=401, n=304),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


# cell updates of the largest listed case of a kind, and space-time elements of a field
_MOST = {"forward": 4.6e9, "gradient": 2.7e10, "cg": 1.3e10, "dscg": 1.6e10, "fdcg": 1.6e10,
         "saddle": 1.2e9, "dtft": 8.1e9}


def _modellings(case):
    k = case["kind"]
    if k == "gradient":
        return 3
    if k == "cg":
        return 1 + 2 * case["iters"] + (1 if case["solver"] == "wri" else 0)
    if k == "dscg":
        return 2 * (case["iters"] + 1) + 1
    if k == "fdcg":
        return 1 + 4 * case["iters"]
    return 1


def draw(rng):
    kind = rng.choice(["forward", "forward", "gradient", "gradient", "cg", "cg", "dscg", "fdcg",
                       "saddle", "dtft", "volume", "pc_apply", "pc_grad"])
    if kind.startswith("pc_"):
        return dict(kind=kind, h=_log(rng, 31, 151), w=_log(rng, 51, 601),
                    n=_log(rng, 4, 16) if kind == "pc_grad" else _log(rng, 8, 200))
    c = dict(kind=kind, nz=_log(rng, 64, 301), ny=1, nx=_log(rng, 64, 1201), ns=_log(rng, 1, 24),
             nt=_log(rng, 100, 1200), nrec=_log(rng, 16, 600), dx=rng.choice([10.0, 12.5]), dt=1e-3,
             dtype="f32", off=rng.random() < 0.3)
    if kind == "volume" or (kind == "dtft" and rng.random() < 0.5):
        c.update(kind=rng.choice(["forward", "gradient"]) if kind == "volume" else "dtft",
                 nz=_log(rng, 48, 260), ny=_log(rng, 48, 260), nx=_log(rng, 48, 260),
                 ns=_log(rng, 1, 3), nt=_log(rng, 64, 200), dx=10.0, dt=0.8e-3)
    kind = c["kind"]
    if kind == "forward" and c["ny"] == 1 and rng.random() < 0.35:
        c.update(dtype="f64", nz=_log(rng, 64, 160), nx=_log(rng, 64, 200), ns=_log(rng, 1, 4),
                 nt=_log(rng, 100, 600))
    if kind == "gradient":
        c.update(ckpt=rng.choice(["f32", "f16", "bf16"]), every=rng.choice([10, 20, 50]),
                 ns=_log(rng, 1, 64) if c["ny"] == 1 else c["ns"])
    if kind == "cg":
        c.update(solver=rng.choice(["diag", "diag", "none", "wri"]), iters=rng.randint(2, 6))
    if kind in ("dscg", "fdcg"):
        c.update(iters=rng.randint(1, 3))
    if kind in ("fdcg", "dtft"):
        c.update(nf=rng.randint(1, 6))
    if kind == "saddle":
        c.update(beta=10.0 ** rng.uniform(-2, 1))
    cells = c["nz"] * c["ny"] * c["nx"]
    field = kind in ("cg", "dscg", "saddle")
    if field:   # space-time vectors of all shots
        c["ns"] = max(1, min(c["ns"], int(1.2e9 / (cells * c["nt"]))))
    most = _MOST[kind] / _modellings(c)
    c["ns"] = max(1, min(c["ns"], int(most / (cells * c["nt"]))))
    c["nt"] = max(64, min(c["nt"], int(most / (cells * c["ns"]))))
    if kind in ("cg", "dscg", "fdcg"):
        lam = 10.0 * (c["nt"] / 400.0) ** 2
        c["lam"] = 2000.0 * lam if c.get("solver") == "wri" else lam
    return c


# ------------------------------------------------------------------------------------ inputs
def _shape(case):
    return (case["nz"], case["nx"]) if case["ny"] == 1 else (case["nz"], case["ny"], case["nx"])


def _rng(seed, salt):
    return np.random.default_rng([int(seed) & 0x7FFFFFFF, salt])


def _model(case, seed, smooth):
    """Layers with dips and Gaussian anomalies (smooth: a velocity gradient in their place)."""
    r = _rng(seed, 1)
    shape = _shape(case)
    ax = [torch.arange(n, dtype=torch.float64, device="cuda") for n in shape]
    z = ax[0].reshape((-1,) + (1,) * (len(shape) - 1))
    lat = ax[-1].reshape((1,) * (len(shape) - 1) + (-1,)) - shape[-1] / 2
    v = torch.zeros(shape, dtype=torch.float64, device="cuda")
    if smooth:
        v += 1700.0 + 2200.0 * z / shape[0]
    else:
        v += 1700.0
        for k in range(1, 8):
            depth = shape[0] * (k / 8 + 0.03 * r.uniform(-1, 1)) + math.tan(0.12 * r.uniform(-1, 1)) * lat
            v += 350.0 * (z >= depth)
    for _ in range(5):
        r2 = 0.0
        for a, n in enumerate(shape):
            d = (ax[a] - r.uniform(0.15, 0.85) * n) * case["dx"]
            r2 = r2 + (d * d).reshape((1,) * a + (-1,) + (1,) * (len(shape) - 1 - a))
        v += 200.0 * r.choice([-1.0, 1.0]) * torch.exp(r2 * (-0.5 / 100.0 ** 2))
    return v.to(DT[case["dtype"]]).contiguous()


NB = 20


def _geometry(case, seed):
    """Shots evenly spaced near the top; receivers in a line (2D) or a grid (3D) at that depth;
    apertures of uneven length where there are many shots; off: between the nodes."""
    r = _rng(seed, 2)
    dx, nx, ns = case["dx"], case["nx"], case["ns"]
    zr = (NB + 2 + (0.4 if case["off"] else 0.0)) * dx
    src = np.zeros((ns, 3))
    cols = np.linspace(NB + 2, nx - 1 - NB - 2, ns + 2)[1:-1]
    cols = np.round(cols) + r.integers(-1, 2) + (0.3 if case["off"] else 0.0)
    src[:, 0], src[:, 2] = cols * dx, (NB + 2) * dx
    recs = []
    if case["ny"] > 1:
        src[:, 1] = (case["ny"] // 2) * dx
        n = max(2, int(math.sqrt(case["nrec"])))
        step = 2 if 2 * n + 4 < min(nx, case["ny"]) else 1
        n = min(n, (min(nx, case["ny"]) - 4) // step)
        f = 0.35 if case["off"] else 0.0
        gx = (np.arange(n) * step + (nx - n * step) // 2 + f) * dx
        gy = (np.arange(n) * step + (case["ny"] - n * step) // 2 + f) * dx
        mx, my = np.meshgrid(gx, gy)
        grid = np.stack([mx.ravel(), my.ravel(), np.full(mx.size, zr)], axis=1)
        recs = [grid] * ns
    else:
        for s in range(ns):
            n = min(case["nrec"], nx - 1)
            if case["nrec"] >= nx:   # every column
                n, lo = nx, 0
            else:
                if ns > 16:
                    n = int(r.integers(max(1, (2 * n) // 5), min(nx - 1, (8 * n) // 5) + 1))
                lo = int(min(max(0, round(cols[s]) - n // 2), nx - 1 - n))
            x = (lo + np.arange(n) + (0.35 if case["off"] and n < nx else 0.0)) * dx
            recs.append(np.stack([x, np.zeros(n), np.full(n, zr)], axis=1))
    off = np.zeros(ns + 1, dtype=np.int64)
    off[1:] = np.cumsum([len(a) for a in recs])
    return synth.Geometry(src, off, np.concatenate(recs))


def _wavelets(case, seed):
    r = _rng(seed, 3)
    f = (14.0 if case["dx"] < 12 else 8.0) * r.uniform(0.9, 1.1, case["ns"])
    w = np.stack([synth.ricker(case["nt"], case["dt"], x, delay=min(1.5 / x, 0.3 * case["nt"] * case["dt"]))
                  for x in f])
    return torch.tensor(w, dtype=DT[case["dtype"]], device="cuda")


def _traces(case, geom, seed):
    """Observed data: a direct arrival and two reflections with moveout, and some noise."""
    r = _rng(seed, 4)
    nt, dt = case["nt"], case["dt"]
    fp = 14.0 if case["dx"] < 12 else 8.0
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)
    out = torch.empty(nt * int(geom.rec_offset[-1]), dtype=torch.float64, device="cuda")
    t = torch.arange(nt, dtype=torch.float64, device="cuda")[:, None] * dt
    events = [(1600.0 + 400.0 * k, (0.1 + 0.25 * k) * nt * dt, r.uniform(0.3, 1.0) / (1 + k)) for k in range(3)]
    for s in range(case["ns"]):
        rec = torch.tensor(geom.receivers(s) - geom.src_xyz[s], device="cuda")
        d = rec.norm(dim=1)[None, :]
        a = torch.zeros((nt, rec.shape[0]), dtype=torch.float64, device="cuda")
        for v, t0, amp in events:
            p = (math.pi * fp * (t - torch.sqrt(t0 * t0 + (d / v) ** 2))) ** 2
            a += amp * 1e-2 / torch.sqrt(1.0 + d / 100.0) * (1 - 2 * p) * torch.exp(-p)
        a += 1e-5 * torch.randn(a.shape, generator=g, dtype=torch.float64, device="cuda")
        o = nt * int(geom.rec_offset[s])
        out[o:o + a.numel()] = a.reshape(-1)
    return out.to(DT[case["dtype"]])


def _field(case, geom, seed):
    """An extended source: a few wavelets in time on patches around each source."""
    r = _rng(seed, 5)
    nt, shape = case["nt"], _shape(case)
    q = torch.empty((case["ns"], nt) + shape, dtype=DT[case["dtype"]], device="cuda")
    z = torch.arange(shape[0], dtype=torch.float64, device="cuda")[:, None] * case["dx"]
    x = torch.arange(shape[-1], dtype=torch.float64, device="cuda")[None, :] * case["dx"]
    for s in range(case["ns"]):
        acc = None
        for _ in range(3):
            cx, cz = geom.src_xyz[s, 0] + r.uniform(-300, 300), geom.src_xyz[s, 2] + r.uniform(0, 300)
            sig = r.uniform(60.0, 400.0)
            patch = torch.exp(((z - cz) ** 2 + (x - cx) ** 2) * (-0.5 / sig ** 2)).reshape(1, -1)
            w = synth.ricker(nt, case["dt"], r.uniform(5, 12), delay=r.uniform(0.2, 0.6) * nt * case["dt"])
            term = torch.tensor(w, device="cuda").reshape(-1, 1) * 1e-3
            acc = term.to(q.dtype) * patch.to(q.dtype) if acc is None else acc.addcmul_(term.to(q.dtype), patch.to(q.dtype))
        q[s] = acc.reshape((nt,) + shape)
    return q


def _images(case, seed):
    """Smooth band-limited BF16 images with an amplitude of their own each."""
    g = torch.Generator(device="cuda").manual_seed(int(seed) & 0x7FFFFFFF)
    n, h, w = case["n"], case["h"], case["w"]
    x = torch.randn((n, 16, (h + 7) // 8 + 1, (w + 7) // 8 + 1), generator=g, device="cuda")
    x = F.interpolate(x, size=(h, w), mode="bilinear", align_corners=False)
    x += 0.1 * torch.randn(x.shape, generator=g, device="cuda")
    x *= torch.exp(torch.randn((n, 1, 1, 1), generator=g, device="cuda"))
    return x.permute(0, 2, 3, 1).contiguous().to(torch.bfloat16)


def _weights():
    root = os.path.dirname(os.path.abspath(esi.__file__))
    return torch.tensor(np.load(os.path.join(root, "pc_weights.npy")), dtype=torch.float32, device="cuda")


def _frequencies(case, seed):
    r = _rng(seed, 6)
    return [float(f) for f in np.linspace(2.0, 12.0, case["nf"] + 2)[1:-1] + r.uniform(-0.4, 0.4, case["nf"])]


def prepare(case, seed):
    kind = case["kind"]
    if kind.startswith("pc_"):
        st = dict(case=case, x=_images(case, seed), net=esi.PCNet(case["h"], case["w"], case["n"]))
        st["net"].set_params(_weights())
        if kind == "pc_grad":
            st["e"] = _images(case, seed + 7919)
        return st
    st = dict(case=case, geom=_geometry(case, seed))
    st["v"] = _model(case, seed, smooth=kind not in ("forward", "dtft"))
    st["ctx"] = esi.Context(st["v"], case["dx"], case["dt"], case["nt"], NB, st["geom"])
    if kind in ("forward", "gradient", "dtft") or case.get("solver") == "wri":
        st["wav"] = _wavelets(case, seed)
    if kind not in ("forward", "dtft"):
        st["dobs"] = _traces(case, st["geom"], seed)
    if kind == "saddle":
        st["q"] = _field(case, st["geom"], seed)
    if kind in ("cg", "dscg"):
        st["out"] = st["ctx"].empty_field()
        st["w"] = st["ctx"].empty_traces()
    if kind in ("fdcg", "dtft"):
        st["freqs"] = _frequencies(case, seed)
    return st


def run(st):
    case = st["case"]
    kind = case["kind"]
    if kind == "pc_apply":
        return st["net"].apply(st["x"])
    if kind == "pc_grad":
        return st["net"].grad(st["x"], st["e"])
    ctx = st["ctx"]
    if kind == "forward":
        return ctx.forward(wavelet=st["wav"])
    if kind == "gradient":
        return ctx.gradient(wavelet=st["wav"], dobs=st["dobs"], mode="adjoint", param="v",
                            ckpt_every=case["every"], ckpt=case["ckpt"])
    if kind == "saddle":
        return ctx.gradient(ext=st["q"], dobs=st["dobs"], mode="saddle", beta=case["beta"], param="v")
    if kind == "dtft":
        tr = ctx.empty_traces()
        u, scales = ctx.dft_extract(st["freqs"], wavelet=st["wav"], half=True, traces=tr)
        return u, scales, tr
    if kind == "cg":
        if case["solver"] == "wri":
            q, _ = ctx.wri_solve(st["wav"], st["dobs"], case["lam"], 0.0, case["iters"], out=st["out"])
        else:
            q, _ = ctx.cg_solve(st["dobs"], case["lam"], 0.0, case["iters"], precond=case["solver"],
                                out=st["out"])
        return q
    if kind == "dscg":
        q, _ = ctx.dscg_solve(st["dobs"], case["lam"], 0.0, case["iters"], out=st["out"], w_out=st["w"])
        return q, st["w"]
    q, _ = ctx.fdcg_solve(st["dobs"], st["freqs"], case["lam"], 0.0, case["iters"], precond="diag")
    return q


def work(case):
    """Cell updates of the modellings (FP adds and multiplies of the stencil and the update),
    the vector operations of a solve, and each input and output once."""
    if case["kind"].startswith("pc_"):
        px, px2, px3, px4 = [case["n"] * math.ceil(case["h"] / k) * math.ceil(case["w"] / k) for k in (1, 2, 4, 8)]
        f = 2 * 9 * (2 * px * 16 * 32 + 32 * 32 * (2 * px2 + 2 * px3 + px4))
        if case["kind"] == "pc_grad":
            return {"bytes": 2 * 32.0 * px, "flops": 3.0 * f}
        return {"bytes": (32.0 + 64.0) * px, "flops": float(f)}
    es = 8 if case["dtype"] == "f64" else 4
    nd = 2 if case["ny"] == 1 else 3
    cells = case["nz"] * case["ny"] * case["nx"]
    ns, nt, kind = case["ns"], case["nt"], case["kind"]
    field = float(ns) * cells * nt
    flops = field * _modellings(case) * (8 * nd + 11)
    tr = es * ns * nt * float(min(case["nrec"], case["nx"] if nd == 2 else case["nrec"]))
    b = es * cells + tr
    if kind == "gradient":
        flops += field * 2
        b += es * cells
    elif kind == "saddle":
        flops += field * 6
        b += es * (field + cells)
    elif kind == "cg":
        flops += field * case["iters"] * 12
        b += es * field
    elif kind == "dscg":
        flops += field * (case["iters"] + 2)
        b += es * field + tr
    elif kind == "fdcg":
        flops += field * (1 + 4 * case["iters"]) * 4 * case["nf"]
        b += es * 2.0 * case["nf"] * ns * cells
    elif kind == "dtft":
        flops += field * 4 * case["nf"]
        b += 4.0 * case["nf"] * ns * cells
    return {"bytes": b, "flops": flops}


# ------------------------------------------------------------------------------ 64-bit values
class _Ref:
    """The discrete method in plain FP64 torch operations, all shots of a chunk at once."""

    def __init__(self, v, case, geom):
        d = self.d = v.double()
        self.shape, self.nd = tuple(d.shape), d.dim()
        dx, dt, nt = case["dx"], case["dt"], case["nt"]
        self.dx, self.dt, self.nt, self.geom, self.ns = dx, dt, nt, geom, geom.ns
        self.cc = d * d * (dt * dt / (dx * dx))
        kmax = 3.0 * float(d.max()) * math.log(1e3) / (2.0 * NB * dx) * dt / 2.0
        kap = torch.zeros(self.shape, dtype=torch.float64, device=d.device)
        for a, n in enumerate(self.shape):
            i = torch.arange(n, dtype=torch.float64, device=d.device)
            r = torch.clamp(torch.maximum(NB - i, i - (n - 1 - NB)), min=0.0) / NB
            kap += (kmax * r * r).reshape((1,) * a + (-1,) + (1,) * (self.nd - 1 - a))
        self.al = 1.0 / (1.0 + kap)
        self.ga = (1.0 - kap) * self.al
        self.alc = self.al * self.cc
        self.psh = tuple(n + 8 for n in self.shape)
        self.src = self._nodes(geom.src_xyz, np.arange(self.ns))
        shot = np.repeat(np.arange(self.ns), np.diff(geom.rec_offset))
        self.rec = self._nodes(geom.rec_xyz, shot)
        nr = np.diff(geom.rec_offset)[shot]
        first = geom.rec_offset[:-1][shot]
        self.tr0 = torch.tensor(nt * first + np.arange(len(shot)) - first, device=d.device)
        self.trs = torch.tensor(nr, device=d.device)

    def _nodes(self, xyz, shot):
        """Flat indices into the padded states [ns][...] of a point's nodes and their weights."""
        pos = np.asarray(xyz, dtype=np.float64)[:, [2, 0] if self.nd == 2 else [2, 1, 0]] / self.dx
        base = np.floor(pos).astype(np.int64)
        frac = pos - base
        idx, wts = [], []
        for c in range(2 ** self.nd):
            w, i = np.ones(len(pos)), np.asarray(shot, dtype=np.int64).copy()
            for a in range(self.nd):
                bit = (c >> a) & 1
                w = w * (frac[:, a] if bit else 1.0 - frac[:, a])
                i = i * self.psh[a] + np.minimum(base[:, a] + bit, self.shape[a] - 1) + 4
            idx.append(i)
            wts.append(w)
        dev = self.cc.device
        return torch.tensor(np.stack(idx, 1), device=dev), torch.tensor(np.stack(wts, 1), device=dev)

    def zeros(self):
        return torch.zeros((self.ns,) + self.psh, dtype=torch.float64, device=self.cc.device)

    def inner(self, p, axis=None, k=0):
        s = [slice(None)] + [slice(4, 4 + n) for n in self.shape]
        if axis is not None:
            s[axis + 1] = slice(4 + k, 4 + k + self.shape[axis])
        return p[tuple(s)]

    def step(self, cur, old, q=None, pts=None, amp=None):
        """old becomes the new state; returns S = L + dx^2 q (point amplitudes amp at pts)."""
        full = torch.zeros_like(cur)
        S = self.inner(full)
        torch.mul(self.inner(cur), self.nd * W[0], out=S)
        for a in range(self.nd):
            for k in range(1, 5):
                S.add_(self.inner(cur, a, k), alpha=W[k]).add_(self.inner(cur, a, -k), alpha=W[k])
        if q is not None:
            S.add_(q, alpha=self.dx * self.dx)
        if pts is not None:
            full.view(-1).index_add_(0, pts[0].reshape(-1), (pts[1] * amp[:, None]).reshape(-1))
        u, o = self.inner(cur), self.inner(old)
        o.copy_(u + self.ga * (u - o) + self.alc * S)
        return S

    def forward(self, wav=None, ext=None, each=None):
        tr = torch.zeros(self.nt * int(self.geom.rec_offset[-1]), dtype=torch.float64, device=self.cc.device)
        cur, old = self.zeros(), self.zeros()
        for n in range(self.nt):
            amp = None if wav is None else wav[:, n] * self.dx ** (2 - self.nd)
            q = None if ext is None else ext(n)
            S = self.step(cur, old, q, None if wav is None else self.src, amp)
            cur, old = old, cur
            tr[self.tr0 + n * self.trs] = (cur.view(-1)[self.rec[0]] * self.rec[1]).sum(1)
            if each is not None:
                each(n, S, cur, q)
        return tr

    def adjoint(self, tr, each):
        cur, old = self.zeros(), self.zeros()
        for n in range(self.nt - 1, -1, -1):
            self.step(cur, old, None, self.rec, tr[self.tr0 + n * self.trs] * self.dx * self.dx)
            cur, old = old, cur
            each(n, self.inner(cur))

    def adjoint_field(self, tr):
        f = torch.empty((self.ns, self.nt) + self.shape, dtype=torch.float64, device=self.cc.device)

        def put(n, lam):
            f[:, n] = lam
        self.adjoint(tr, put)
        return f

    def b2(self):
        ax = [torch.arange(n, dtype=torch.float64, device=self.cc.device) * self.dx for n in self.shape]
        r2 = torch.zeros((self.ns,) + self.shape, dtype=torch.float64, device=self.cc.device)
        for a, c in enumerate([2, 0] if self.nd == 2 else [2, 1, 0]):
            x = torch.tensor(self.geom.src_xyz[:, c], device=self.cc.device).reshape((-1,) + (1,) * self.nd)
            r2 += (ax[a].reshape((1,) * (a + 1) + (-1,) + (1,) * (self.nd - 1 - a)) - x) ** 2
        return (torch.sqrt(r2) + self.dx) ** 2

    def to_v(self, G, extra=1.0):
        c = self.cc * self.dx ** 2
        return extra * G / (c * self.dx ** 2) * 2.0 * torch.sqrt(c) * self.dt


def _dots(a, b):
    return (a * b).flatten(1).sum(1)


def _col(x, like):
    return x.reshape((-1,) + (1,) * (like.dim() - 1))


def _pcg(A, b, M, iters):
    x = torch.zeros_like(b)
    r, z = b, M(b)
    p, rho = z.clone(), _dots(r, z)
    for k in range(iters):
        ap = A(p)
        al = _col(rho / _dots(p, ap), p)
        x += al * p
        r = r - al * ap
        if k + 1 < iters:
            z = M(r)
            new = _dots(r, z)
            p = z + _col(new / rho, p) * p
            rho = new
    return x


def _exact_chunk(case, v, geom, wav, dobs, q, freqs):
    R = _Ref(v, case, geom)
    kind, nt = case["kind"], case["nt"]
    if kind == "forward":
        return (R.forward(wav=wav),)
    if kind == "gradient":
        hist = torch.empty((nt, R.ns) + R.shape, dtype=torch.float64, device=v.device)
        res = R.forward(wav=wav, each=lambda n, S, u, q_: hist[n].copy_(S)) - dobs
        G = torch.zeros(R.shape, dtype=torch.float64, device=v.device)
        R.adjoint(res, lambda n, lam: G.add_((lam * hist[n]).sum(0)))
        return R.to_v(G), float(0.5 * (res * res).sum())
    if kind == "saddle":
        b2, G = R.b2(), torch.zeros(R.shape, dtype=torch.float64, device=v.device)
        pen = [0.0]

        def each(n, S, u, qn):
            G.add_((b2 * qn * S).sum(0))
            pen[0] = pen[0] + (b2 * qn * qn).sum()
        res = R.forward(ext=lambda n: q[:, n].double(), each=each) - dobs
        J = 0.5 * (res * res).sum() + 0.5 * case["beta"] * pen[0]
        return R.to_v(G, -case["beta"]), float(J)
    if kind == "dtft":
        U = torch.zeros((R.ns, len(freqs)) + R.shape + (2,), dtype=torch.float64, device=v.device)

        def fold(n, S, u, q_):
            for m, f in enumerate(freqs):
                ph = 2 * math.pi * f * (n + 1) * case["dt"]
                U[:, m, ..., 0].add_(R.inner(u), alpha=math.cos(ph))
                U[:, m, ..., 1].add_(R.inner(u), alpha=math.sin(ph))
        tr = R.forward(wav=wav, each=fold)
        top = U.flatten(2).abs().amax(2)
        scale = top / 32768.0
        U /= torch.where(scale > 0, scale, 1.0).reshape(scale.shape + (1,) * (R.nd + 1))
        return U, scale.reshape(R.ns, -1).cpu().numpy(), tr
    lam = case["lam"]
    if kind == "cg":
        wri = case["solver"] == "wri"
        w = torch.full((R.ns, 1) + R.shape, lam, dtype=torch.float64, device=v.device) if wri else lam * R.b2().unsqueeze(1)
        b = R.adjoint_field(dobs - R.forward(wav=wav) if wri else dobs)
        A = lambda p: R.adjoint_field(R.forward(ext=lambda n: p[:, n])).addcmul_(w, p)  # noqa: E731
        return (_pcg(A, b, (lambda r: r / w) if case["solver"] == "diag" else (lambda r: r), case["iters"]),)
    if kind == "dscg":
        w = lam * R.b2().unsqueeze(1)
        seg = torch.tensor(np.repeat(np.arange(R.ns), np.diff(geom.rec_offset) * nt), device=v.device)

        def K(e):
            f = R.adjoint_field(e) / w
            return R.forward(ext=lambda n: f[:, n])

        def dot(a, b):
            return torch.zeros(R.ns, dtype=torch.float64, device=v.device).index_add_(0, seg, a * b)
        x = torch.zeros_like(dobs)
        r = K(dobs)
        p, rr = r.clone(), dot(r, r)
        for k in range(case["iters"]):
            ap = p + K(p)
            al = (rr / dot(p, ap))[seg]
            x = x + al * p
            r = r - al * ap
            new = dot(r, r)
            p = r + (new / rr)[seg] * p
            rr = new
        return R.adjoint_field(dobs - x) / w, x
    # frequency domain: complex slices [ns][nf][...]
    ph = 2 * math.pi * torch.tensor(freqs, dtype=torch.float64, device=v.device)[:, None] * \
        torch.arange(nt, dtype=torch.float64, device=v.device)[None, :] * case["dt"]
    E = torch.polar(torch.ones_like(ph), ph)
    G = (E @ E.conj().T) / nt
    w = lam * R.b2().unsqueeze(1)

    def fold(tr, unit):
        out = torch.zeros((R.ns, len(freqs)) + R.shape, dtype=torch.complex128, device=v.device)

        ec = E.cpu().numpy()

        def each(n, lamn):
            for m in range(len(freqs)):
                z = complex(ec[m, n]) * unit
                o = torch.view_as_real(out[:, m])
                o[..., 0].add_(lamn, alpha=z.real)
                o[..., 1].add_(lamn, alpha=z.imag)
        R.adjoint(tr, each)
        return out

    def A(p):
        pr = torch.view_as_complex(p)
        out = torch.zeros_like(pr)
        ec = E.cpu().numpy() / nt
        for part in range(2):
            def src(n):
                s = 0.0
                for m in range(len(freqs)):
                    z = complex(ec[m, n]).conjugate()
                    c, d = (z.real, -z.imag) if part == 0 else (z.imag, z.real)
                    s = s + p[:, m, ..., 0] * c + p[:, m, ..., 1] * d
                return s
            out += fold(R.forward(ext=src), 1.0 if part == 0 else 1j)
        out += w * torch.einsum("mk,sk...->sm...", G, pr)
        return torch.view_as_real(out)
    b = torch.view_as_real(fold(dobs, 1.0)).contiguous()
    return (_pcg(A, b, lambda r: r / w.unsqueeze(-1), case["iters"]),)


def _exact_net(case, seed):
    P = _weights().double()
    layers, o = [], 0
    for ci, co in [(16, 32)] + [(32, 32)] * 5 + [(32, 16)]:
        k = 9 * ci * co
        layers.append((P[o:o + k].reshape(3, 3, ci, co).permute(3, 2, 0, 1).contiguous().requires_grad_(True),
                       P[o + k:o + k + co].clone().requires_grad_(True)))
        o += k + co

    def net(x):
        rho = x.flatten(1).square().mean(1).sqrt().reshape(-1, 1, 1, 1)
        conv = lambda t, i: F.conv2d(t, layers[i][0], layers[i][1], padding=1)  # noqa: E731
        pool = lambda t: F.avg_pool2d(F.pad(t, (0, t.shape[3] % 2, 0, t.shape[2] % 2)), 2)  # noqa: E731
        up = lambda t, s: t.repeat_interleave(2, 2).repeat_interleave(2, 3)[:, :, :s.shape[2], :s.shape[3]] + s  # noqa: E731
        e1 = F.relu(conv(x / torch.where(rho > 0, rho, 1.0), 0))
        e2 = F.relu(conv(pool(e1), 1))
        e3 = F.relu(conv(pool(e2), 2))
        bt = F.relu(conv(pool(e3), 3))
        d3 = F.relu(conv(up(bt, e3), 4))
        d2 = F.relu(conv(up(d3, e2), 5))
        return conv(up(d2, e1), 6) * rho
    x = _images(case, seed).double().permute(0, 3, 1, 2).contiguous()
    with torch.backends.cudnn.flags(enabled=False):
        if case["kind"] == "pc_apply":
            with torch.no_grad():
                return torch.cat([net(x[i:i + 16]) for i in range(0, case["n"], 16)]).permute(0, 2, 3, 1).contiguous()
        e = _images(case, seed + 7919).double().permute(0, 3, 1, 2)
        z = x + net(x)
        ze, zz, ee = (z * e).flatten(1).sum(1), z.square().flatten(1).sum(1), e.square().flatten(1).sum(1)
        loss = (1 - ze * ze / (zz * ee)).mean()
        flat = [t for wb in layers for t in wb]
        g = torch.autograd.grad(loss, flat)
    out = [t.permute(2, 3, 1, 0).reshape(-1) if t.dim() == 4 else t for t in g]
    return torch.cat(out), float(loss)


def exact(case, seed):
    kind = case["kind"]
    if kind.startswith("pc_"):
        return _exact_net(case, seed)
    geom = _geometry(case, seed)
    v = _model(case, seed, smooth=kind not in ("forward", "dtft"))
    wav = _wavelets(case, seed).double() if kind in ("forward", "gradient", "dtft") or case.get("solver") == "wri" else None
    dobs = _traces(case, geom, seed).double() if kind not in ("forward", "dtft") else None
    q = _field(case, geom, seed) if kind == "saddle" else None
    freqs = _frequencies(case, seed) if kind in ("fdcg", "dtft") else None
    # shots in chunks whose space-time vectors fit
    field = 8.0 * case["nt"] * v.numel()
    chunk = max(1, min(case["ns"], int(3e10 / (field * (1 if kind in ("gradient", "dtft") else 1.5)))))
    if kind in ("forward", "saddle", "fdcg", "dtft"):
        chunk = case["ns"]
    parts, nt = [], case["nt"]
    for lo in range(0, case["ns"], chunk):
        hi = min(case["ns"], lo + chunk)
        o0, o1 = nt * int(geom.rec_offset[lo]), nt * int(geom.rec_offset[hi])
        parts.append(_exact_chunk(case, v, geom.select(range(lo, hi)), None if wav is None else wav[lo:hi],
                                  None if dobs is None else dobs[o0:o1],
                                  None if q is None else q[lo:hi], freqs))
    if kind in ("gradient", "saddle"):
        return sum(p[0] for p in parts), sum(p[1] for p in parts)
    if kind == "dtft":
        return parts[0]
    whole = tuple(parts[0][k] if len(parts) == 1 else torch.cat([p[k] for p in parts]) for k in range(len(parts[0])))
    return whole if kind == "dscg" else whole[0]
