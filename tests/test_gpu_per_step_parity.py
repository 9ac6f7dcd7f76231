"""Parity of the 2D per-step kernel with the FP64 oracle, in every variant of it.

Small 2D problems run their time loops on chip, so the parity cases of the other files no longer
reach this kernel.  It runs loops of fewer than eight steps, and FP32 loops of more cells than the
on-chip loops take two rows a thread of; both are used here, and the launch counts show that each
step was a launch (two where the shots run in two chains).  Grids of several 64 x 32 tiles with
ragged ends; sources and receivers off the nodes, across tile edges and in the last row and
column.  Bounds as in the other parity cases: FP64 1e-12 relative L2 (10 times that for the
frequency-domain and data-space solutions), FP32 1e-4 (1e-3 for the plain CG's solution and ten
times 1e-4 for the frequency-domain and data-space ones)."""
import numpy as np
import pytest

import oracle
from oracle import outer
from paper_2211_06300_gb300 import synth
from test_gpu_parity import TOL, _ctx, _dev, _orc

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


class Case:
    """A problem with the oracle's shots to compare, inputs, and the launches a loop of nt steps
    takes at least."""

    def __init__(self, shape, ns, nt, prec, compare, chains):
        rng = np.random.default_rng(shape[1] + nt)
        nz, nx = shape
        dx, ext = 10.0, (nx - 1) * 10.0
        self.prec, self.tol, self.nt, self.ns, self.shape = prec, TOL[prec], nt, ns, shape
        v = synth.dipping_layers(shape, dx, 5, nlayers=4, vmin=1500, vmax=2600, nanom=2, sigma=40.0)
        # the first source beside the corner of four tiles, the others anywhere
        sx = np.concatenate([[636.0], rng.uniform(60.0, ext - 60.0, ns - 1)])
        sz = np.concatenate([[316.0], rng.uniform(40.0, (nz - 5) * 10.0, ns - 1)])
        recs, rz = [], []
        for s in range(ns):
            n = 5 + 4 * (s % 3)   # around the source, then the last column and row
            recs.append(np.concatenate([sx[s] + rng.uniform(-30.0, 30.0, n), [ext, 3.0]]))
            rz.append(np.concatenate([np.clip(sz[s] + rng.uniform(-30.0, 30.0, n), 0.0, (nz - 1) * dx),
                                      [15.0, (nz - 1) * dx]]))
        self.geom = synth.surface_line(ns, sx, 0.0, recs, 0.0)
        self.geom.src_xyz[:, 2] = sz
        self.geom.rec_xyz[:, 2] = np.concatenate(rz)
        p = dict(dx=dx, dt=1e-3, nt=nt, nb=6)
        self.vref = float(v.max())
        self.o, self.shots = _orc(v, self.geom, p, vref=self.vref)
        self.c = _ctx(v, self.geom, p, prec, vref=self.vref)
        self.compare, self.loop = compare, nt * chains
        self.off = self.geom.rec_offset
        self.wav = rng.standard_normal((ns, nt))
        self.q = rng.standard_normal((ns, nt, nz * nx))
        self.e = rng.standard_normal(nt * int(self.off[-1]))

    def dev(self, a, field=False):
        return _dev(a.reshape((self.ns, self.nt) + self.shape) if field else a, self.prec)

    def of(self, traces, s):
        return np.asarray(traces)[self.nt * self.off[s]:self.nt * self.off[s + 1]].reshape(self.nt, -1)

    def call(self, loops, f):
        """f(), whose `loops` time loops must have taken a launch a step (and chain)."""
        n0 = self.c.launches
        out = f()
        assert self.c.launches - n0 >= loops * self.loop
        return out

    def close_to(self, got, ref, factor=1.0):
        got = got.double().cpu().numpy() if torch.is_tensor(got) else got
        err = oracle.rel_l2(np.asarray(got).reshape(np.asarray(ref).shape), ref)
        assert err <= factor * self.tol, err


def _make(kind):
    if kind == "two chains":
        # 36 shots of 4 x 5 tiles: more blocks than the chip holds; 70 steps: captured, and a block
        # of 64 and one of 6 in the DTFT
        return Case((131, 221), 36, 70, "f32", (0, 17, 18, 35), 2)
    return Case((45, 83), 3, 7, kind, (0, 1, 2), 1)


KINDS = ["f64", "f32", "two chains"]


@pytest.mark.parametrize("kind", KINDS)
def test_modelling(kind):
    t = _make(kind)
    c, o = t.c, t.o
    w, q, e = t.dev(t.wav), t.dev(t.q, True), t.dev(t.e)
    freqs = [6.0, 17.0, 33.0]
    for wv, qx in ((w, None), (None, q), (w, q)):
        tr = t.call(1, lambda: c.forward(wavelet=wv, ext=qx)).double().cpu().numpy()
        out, _ = t.call(1, lambda: c.dft_extract(freqs, wavelet=wv, ext=qx))
        for s in t.compare:
            ref = o.forward(t.shots[s], wavelet=None if wv is None else t.wav[s],
                            q_ext=None if qx is None else t.q[s], freqs=freqs)
            t.close_to(t.of(tr, s), ref["traces"])
            u = out[s].double().cpu().numpy().reshape(len(freqs), -1, 2)
            t.close_to(u[..., 0] + 1j * u[..., 1], ref["dft"])
    f, wo = t.call(1, lambda: c.adjoint(e, want_wavelet=True))
    f1, _ = t.call(1, lambda: c.adjoint(e))
    _, w1 = t.call(1, lambda: c.adjoint(e, want_field=False, want_wavelet=True))
    assert torch.equal(f, f1) and torch.equal(wo, w1)
    for s in t.compare:
        ref = o.adjoint(t.shots[s], t.of(t.e, s), want_src=True)
        t.close_to(f[s], ref["out"])
        t.close_to(wo[s], ref["src"])
    c.close()


@pytest.mark.parametrize("kind", KINDS)
def test_gradients(kind):
    t = _make(kind)
    c, o = t.c, t.o
    w, q, e = t.dev(t.wav), t.dev(t.q, True), t.dev(t.e)
    for wv, qx in ((w, None), (None, q), (w, q)):
        J_ref, g_ref = 0.0, 0.0
        for s, sh in enumerate(t.shots):
            J, g = o.misfit_gradient(sh, t.of(t.e, s), wavelet=None if wv is None else t.wav[s],
                                     q_ext=None if qx is None else t.q[s], param="v")
            J_ref, g_ref = J_ref + J, g_ref + g
        for every in (3, 40):
            g, J = t.call(2 if every < t.nt else 1,
                          lambda: c.gradient(wavelet=wv, ext=qx, dobs=e, ckpt_every=every))
            t.close_to(g, g_ref)
            assert abs(J - J_ref) <= t.tol * J_ref
    beta = 0.37
    ref = sum(o.saddle_gradient(sh, t.q[s], beta, param="v") for s, sh in enumerate(t.shots))
    J_ref = sum(outer.esi_objective(o, sh, t.q[s], t.of(t.e, s), beta) for s, sh in enumerate(t.shots))
    g, _ = t.call(1, lambda: c.gradient(ext=q, mode="saddle", beta=beta))
    g2, J = t.call(1, lambda: c.gradient(ext=q, dobs=e, mode="saddle", beta=beta))
    t.close_to(g, ref)
    t.close_to(g2, ref)
    assert abs(J - J_ref) <= t.tol * J_ref
    ref = sum(o.wri_gradient(sh, t.q[s], t.wav[s], beta, param="v") for s, sh in enumerate(t.shots))
    J_ref = sum(o.wri_objective(sh, t.q[s], t.of(t.e, s), t.wav[s], beta)
                for s, sh in enumerate(t.shots))
    g, _ = t.call(1, lambda: c.gradient(wavelet=w, ext=q, mode="wri", beta=beta))
    g2, J = t.call(1, lambda: c.gradient(wavelet=w, ext=q, dobs=e, mode="wri", beta=beta))
    t.close_to(g, ref)
    t.close_to(g2, ref)
    assert abs(J - J_ref) <= t.tol * J_ref
    c.close()


@pytest.mark.parametrize("kind", KINDS)
def test_solves(kind):
    t = _make(kind)
    c, o = t.c, t.o
    w, e = t.dev(t.wav), t.dev(t.e)
    lam, n = 0.05, 3
    plain = 1.0 if t.prec == "f64" else 10.0
    runs = {
        "none": (2, plain, lambda: c.cg_solve(e, lam, 0.0, n),
                 lambda sh, d, s: o.cg(sh, d, lam, 0.0, n)),
        "diag": (2, 1.0, lambda: c.cg_solve(e, lam, 0.0, n, precond="diag"),
                 lambda sh, d, s: o.pcg(sh, d, lam, 0.0, n, minv=1.0 / (lam * o.annihilator(sh.src_xyz) ** 2))),
        "wri": (2, 1.0, lambda: c.cg_solve(e, lam, 0.0, n, wri_wavelet=w),
                lambda sh, d, s: o.wri_cg(sh, d, t.wav[s], lam, 0.0, n)),
        "data": (2, 10.0, lambda: c.dscg_solve(e, lam, 0.0, n),
                 lambda sh, d, s: o.ds_cg(sh, d, lam, 0.0, n)),
        "freq": (4, 10.0, lambda: c.fdcg_solve(e, [8.0, 15.5, 23.0], lam, 0.0, n),
                 lambda sh, d, s: o.fd_cg(sh, d, lam, [8.0, 15.5, 23.0], 0.0, n)),
    }
    for name, (loops, factor, gpu, ref) in runs.items():
        q, rep = t.call(loops * n, gpu)
        for s in t.compare:
            r = ref(t.shots[s], t.of(t.e, s), s)
            assert rep["iters"][s] == r["iters"] == n, name
            assert np.allclose(rep["rel_res"][s], r["rel_res"], rtol=factor * t.tol, atol=0), (name, s)
            got = q[s].double().cpu().numpy()
            if name == "freq":
                got = got[..., 0] + 1j * got[..., 1]
            t.close_to(got, r["qbar"] if name == "freq" else r["q"] if name == "data" else r["x"], factor)
    c.close()
