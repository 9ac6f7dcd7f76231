"""Point sources of the on-chip 2D loops whose lists are long: many contributions to one node,
many nodes in one tile, receivers at one place, counts around the loads a thread keeps in flight.

The back-propagation of a record that is zero but for its last seven samples starts with the
seven steps of a record of those samples alone, which the per-step kernel runs (a loop of fewer
than eight steps): equal to the bit.  And a long list must not slow the loop: back-propagating
2000 traces a shot may take six times as long as modelling them (once it took 26 times, FP64 ten)."""
import time

import numpy as np
import pytest

from paper_2211_06300_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _geom(nz, nx, ns, n, kind):
    rng = np.random.default_rng(n)
    if kind == "line":       # between the rows and columns: up to dozens of traces a node
        x, z = np.linspace(0, (nx - 1) * 10.0, n), np.full(n, 22.5)
    elif kind == "nodes":    # one trace a node
        k = rng.permutation(nz * nx)[:n]
        x, z = (k % nx) * 10.0, (k // nx) * 10.0
    else:                    # all at one place, and a few elsewhere
        x, z = np.full(n, 37.5), np.full(n, 52.5)
        x[:3], z[:3] = [0.0, (nx - 1) * 10.0, 60.0], [0.0, (nz - 1) * 10.0, 30.0]
    g = synth.surface_line(ns, rng.uniform(0, (nx - 1) * 10.0, ns), 60.0, [x] * ns, 0.0)
    g.rec_xyz[:, 2] = np.concatenate([z] * ns)
    return g


def _ctx(nz, nx, nt, geom, dtype):
    from paper_2211_06300_gb300 import esi
    v = 1500.0 + 1000.0 * np.random.default_rng(nx).random((nz, nx))
    return esi.Context(torch.tensor(v, dtype=dtype, device="cuda"), 10.0, 1e-3, nt, 8, geom)


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nz,nx,ns,n,kind", [(97, 130, 20, 2000, "line"), (45, 83, 3, 300, "line"),
                                             (45, 83, 3, 100, "line"), (45, 83, 3, 200, "line"),
                                             (60, 70, 30, 4200, "nodes"), (60, 70, 2, 4200, "nodes"),
                                             (45, 83, 2, 385, "place"), (45, 83, 1, 5, "place")])
def test_long_lists_give_the_bits_of_the_per_step_kernel(nz, nx, ns, n, kind, dtype):
    nt, last = 24, 7
    geom = _geom(nz, nx, ns, n, kind)
    rng = np.random.default_rng(7)
    e7 = rng.standard_normal((ns, last, n))
    e = np.zeros((ns, nt, n))
    e[:, nt - last:] = e7
    out = []
    for steps, data in ((nt, e), (last, e7)):
        c = _ctx(nz, nx, steps, geom, dtype)
        n0 = c.launches
        f, _ = c.adjoint(torch.tensor(data.ravel(), dtype=dtype, device="cuda"))
        assert (c.launches - n0 < last) == (steps == nt)   # one launch for all steps / one each
        out.append(f[:, steps - last:].clone())
        assert torch.isfinite(f).all()
        c.close()
    assert out[0].abs().max() > 0 and torch.equal(out[0], out[1])


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
def test_long_lists_do_not_slow_the_loop(dtype):
    nt = 200
    geom = _geom(97, 130, 20, 2000, "line")
    c = _ctx(97, 130, nt, geom, dtype)
    wav = torch.randn((20, nt), dtype=dtype, device="cuda")
    d = c.forward(wavelet=wav)

    def ms(f):
        ts = []
        for _ in range(5):
            torch.cuda.synchronize()
            t = time.perf_counter()
            f()
            torch.cuda.synchronize()
            ts.append((time.perf_counter() - t) * 1e3)
        return sorted(ts)[2]

    fwd = ms(lambda: c.forward(wavelet=wav, out=d))
    adj = ms(lambda: c.adjoint(d, want_field=False, want_wavelet=True))
    assert adj < 6 * fwd, (adj, fwd)
    c.close()
