"""Frequency-domain solves on the per-step kernel, with and without programmatic dependent
launches (ESI_PDL=0 orders every launch behind the completion of the one in front of it).

A step reads its extended source before it waits for the launch in front of it.  The synthesis
writes a block's sources right before the block's first step, which therefore must not be a
dependent launch.  Both orders run the same operations, so the solutions are equal to the bit.
The records hold several blocks and end in a short one; 31 steps or fewer are launched without a
captured graph."""
import numpy as np
import pytest

from paper_2211_06300_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape,ns,nt", [((241, 801), 7, 259), ((241, 801), 7, 31),
                                         ((24, 24, 40), 2, 131)])
def test_frequency_domain_solve_does_not_depend_on_the_launch_order(shape, ns, nt, monkeypatch):
    from paper_2211_06300_gb300 import esi
    rng = np.random.default_rng(nt)
    v = 1500.0 + 1000.0 * rng.random(shape)
    ext = (shape[-1] - 1) * 10.0
    src = rng.uniform(0, ext, ns)
    recs = [rng.uniform(0, ext, 20 + 10 * (s % 3)) for s in range(ns)]
    geom = synth.surface_line(ns, src, 60.0, recs, 20.0)
    d = torch.tensor(rng.standard_normal(nt * int(geom.rec_offset[-1])), dtype=torch.float32,
                     device="cuda")
    out = []
    for pdl in ("1", "0"):
        monkeypatch.setenv("ESI_PDL", pdl)
        c = esi.Context(torch.tensor(v, dtype=torch.float32, device="cuda"), 10.0, 1e-3, nt, 8, geom)
        n0 = c.launches
        q, rep = c.fdcg_solve(d, [4.0, 9.0, 15.0], lam=10.0, tol=0.0, max_iter=2)
        assert c.launches - n0 > 4 * 2 * nt   # four modellings an iteration, a launch a step
        assert torch.isfinite(q).all()
        out.append((q, rep["rel_res"]))
        c.close()
    assert torch.equal(out[0][0], out[1][0])
    for a, b in zip(out[0][1], out[1][1]):
        assert np.array_equal(a, b)
