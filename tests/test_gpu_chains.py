"""Time loops in two concurrent chains of launches (2D FP32 steps of more blocks than the chip
holds at once), against contexts of so few of the same shots that their loops run in one.

Shots are independent systems and every launch works on them alike, so the results of a shot are
equal to the bit; the gradient adds them up over the shots.  The record is longer than one part
of a captured loop and ends in an odd remainder; segments of 9 steps are launched directly."""
import numpy as np
import pytest

from paper_2211_06300_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _ctx(v, nt, src, recs, shots):
    from paper_2211_06300_gb300 import esi
    geom = synth.surface_line(len(shots), [src[s] for s in shots], 60.0, [recs[s] for s in shots], 20.0)
    return esi.Context(torch.tensor(v, dtype=torch.float32, device="cuda"), 10.0, 1e-3, nt, 12, geom)


@pytest.mark.parametrize("nz,nx,ns", [(241, 801, 7), (90, 1601, 9)])
def test_two_chains_give_the_bits_of_one(nz, nx, ns):
    nt, lam = 259, 10.0
    rng = np.random.default_rng(nz)
    v = 1500.0 + 1000.0 * rng.random((nz, nx))
    src = rng.uniform(0, (nx - 1) * 10.0, ns)
    recs = [rng.uniform(0, (nx - 1) * 10.0, 11 + 30 * (s % 3)) for s in range(ns)]
    wav = torch.tensor(rng.standard_normal((ns, nt)), dtype=torch.float32, device="cuda")
    q = torch.randn((ns, nt, nz, nx), device="cuda") * 1e-3
    freqs = [4.0, 9.0, 15.0]

    def run(shots):
        c = _ctx(v, nt, src, recs, shots)
        w, e = wav[shots].contiguous(), q[shots].contiguous()
        tr = c.forward(wavelet=w, ext=e)
        d = 1.1 * c.forward(wavelet=w) + 0.01
        qc, _ = c.cg_solve(d, lam=lam, tol=0.0, max_iter=2, precond="diag")
        sl, _ = c.dft_extract(freqs, wavelet=w)
        qf, _ = c.fdcg_solve(d, freqs, lam=lam, tol=0.0, max_iter=2)
        g, J = c.gradient(wavelet=w, dobs=d, ckpt_every=9)
        gs, Js = c.gradient(ext=e, dobs=d, mode="saddle", beta=0.5)
        c.close()
        return tr, qc, sl, qf, g, gs, J, Js

    whole = run(list(range(ns)))
    parts = [run(list(range(0, ns // 2))), run(list(range(ns // 2, ns)))]
    assert torch.equal(whole[0].flatten(), torch.cat([p[0].flatten() for p in parts]))
    for k in (1, 2, 3):
        assert torch.isfinite(whole[k]).all()
        assert torch.equal(whole[k], torch.cat([p[k] for p in parts]))
    for k in (4, 5):   # FP32 sums over the shots in another grouping
        ref = parts[0][k].double() + parts[1][k].double()
        assert (whole[k].double() - ref).norm() <= ns * 2.0 ** -23 * sum(p[k].double().norm() for p in parts)
    for k in (6, 7):
        assert whole[k] == pytest.approx(parts[0][k] + parts[1][k], rel=1e-5)
