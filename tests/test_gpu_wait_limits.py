"""A bounded device wait that runs out is reported by every kind of call.

ESI_LOOP_POLLS=0 (read when a context is created) lets the tiles of the on-chip loops give up on
their neighbours' rims after one look, so the wait runs out in every loop of more than one tile
and the kernel returns.  Calls that synchronise fail at once, calls that only enqueue return and
the context's next call, or esi_synchronize, reports it."""
import numpy as np
import pytest

from paper_2211_06300_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

NT, SHAPE = 24, (101, 101)


def _ctx(groups=1, dtype=torch.float32):
    from paper_2211_06300_gb300 import esi
    ns = 2
    geom = synth.surface_line(ns, [300.0, 700.0], 60.0, [np.arange(0.0, 1000.0, 50.0)] * ns, 20.0)
    c = esi.Context(torch.full(SHAPE, 2000.0, dtype=dtype, device="cuda"), 10.0, 1e-3, NT, 8, geom)
    if groups > 1:
        c.set_shot_groups(groups)
    return c


def _inputs(c):
    wav = torch.ones((c.ns, NT), dtype=c.dtype, device="cuda")
    d = torch.ones(NT * c.total_rec, dtype=c.dtype, device="cuda")
    q = torch.ones((c.ns, NT) + SHAPE, dtype=c.dtype, device="cuda")
    return wav, d, q


ENQUEUED = {
    "forward": lambda c, w, d, q: c.forward(wavelet=w),
    "adjoint": lambda c, w, d, q: c.adjoint(d),
    "normal_apply": lambda c, w, d, q: c.normal_apply(q, 1.0),
    "dft": lambda c, w, d, q: c.dft_extract([5.0], wavelet=w),
    "vjp": lambda c, w, d, q: c.gradient(wavelet=w, adj_src=d, ckpt_every=12),
    "saddle": lambda c, w, d, q: c.gradient(ext=q, mode="saddle", beta=1.0),
}
SYNCHRONISING = {
    "dft_half": lambda c, w, d, q: c.dft_extract([5.0], wavelet=w, half=True),
    "misfit": lambda c, w, d, q: c.gradient(wavelet=w, dobs=d, ckpt_every=12),
    "objective": lambda c, w, d, q: c.gradient(ext=q, dobs=d, mode="saddle", beta=1.0),
    "cg": lambda c, w, d, q: c.cg_solve(d, lam=1.0, tol=0.0, max_iter=2),
    "dscg": lambda c, w, d, q: c.dscg_solve(d, lam=1.0, tol=0.0, max_iter=2),
    "fdcg": lambda c, w, d, q: c.fdcg_solve(d, [5.0], lam=1.0, tol=0.0, max_iter=2),
}


def _raises_timeout(f):
    from paper_2211_06300_gb300 import esi
    with pytest.raises(esi.EsiError) as ei:
        f()
    assert ei.value.status == esi.ESI_ERR_TIMEOUT and "rims" in str(ei.value)


@pytest.mark.parametrize("groups", [1, 2])
@pytest.mark.parametrize("name", sorted(ENQUEUED))
def test_a_call_that_enqueues_is_reported_later(name, groups, monkeypatch):
    monkeypatch.setenv("ESI_LOOP_POLLS", "0")
    c = _ctx(groups)
    args = _inputs(c)
    ENQUEUED[name](c, *args)
    _raises_timeout(c.synchronize)
    _raises_timeout(lambda: c.forward(wavelet=args[0]))
    c.close()


@pytest.mark.parametrize("name", sorted(SYNCHRONISING))
def test_a_call_that_synchronises_reports_it(name, monkeypatch):
    monkeypatch.setenv("ESI_LOOP_POLLS", "0")
    c = _ctx()
    _raises_timeout(lambda: SYNCHRONISING[name](c, *_inputs(c)))
    _raises_timeout(c.synchronize)
    c.close()


def test_waits_that_end_are_not_reported():
    c = _ctx()
    w, d, q = _inputs(c)
    for f in (*ENQUEUED.values(), *SYNCHRONISING.values()):
        f(c, w, d, q)
        c.synchronize()
    c.close()
