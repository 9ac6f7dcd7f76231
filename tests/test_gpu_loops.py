"""The on-chip 2D time loops against the per-step kernel (esi_forward_noalloc runs it).

Both perform the same operations in the same order per cell, so the seismograms are equal to
the bit whatever the cut into tiles: grids narrower than a tile's rim, ragged last blocks, one
shot over the whole chip, more shots than one launch holds, receivers between the nodes (also
across tile edges) and on the last row and column."""
import numpy as np
import pytest

from paper_2211_06300_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

CASES = [  # nz, nx, shots, steps, sponge cells
    (5, 7, 1, 40, 1), (9, 300, 2, 40, 2), (300, 9, 2, 40, 2), (45, 83, 3, 90, 6),
    (101, 101, 1, 120, 20), (241, 801, 1, 60, 20), (241, 801, 16, 40, 20),
    (301, 1201, 9, 24, 20), (64, 1600, 3, 30, 8), (97, 130, 40, 33, 8), (45, 83, 3, 8, 6),
    # tiles of the whole width fit the shared memory, but no layout of the threads covers them
    (90, 1601, 9, 20, 12), (9, 1601, 100, 20, 2)]


@pytest.mark.parametrize("dtype", [torch.float32, torch.float64])
@pytest.mark.parametrize("nz,nx,ns,nt,nb", CASES)
def test_forward_equals_the_per_step_kernel(nz, nx, ns, nt, nb, dtype):
    from paper_2211_06300_gb300 import esi
    if 2 * ns * nz * ((nx + 31) // 32 * 32) * dtype.itemsize > 32 << 20:
        pytest.skip("above the per-step entry point's fixed array")
    dx, dt = 10.0, 1e-3
    rng = np.random.default_rng(nz * 1000 + nx)
    v = 1500.0 + 1000.0 * rng.random((nz, nx))
    src_x = rng.uniform(0, (nx - 1) * dx, ns)
    recs = [np.concatenate([rng.uniform(0, (nx - 1) * dx, 5 + 40 * (s % 3)), [0.0, (nx - 1) * dx]])
            for s in range(ns)]
    geom = synth.surface_line(ns, src_x, 0.4 * (nz - 1) * dx, recs, 0.0)
    geom.rec_xyz[:, 2] = rng.uniform(0, (nz - 1) * dx, len(geom.rec_xyz))
    geom.rec_xyz[::7, 2] = (nz - 1) * dx
    ctx = esi.Context(torch.tensor(v, dtype=dtype, device="cuda"), dx, dt, nt, nb, geom)
    wav = torch.tensor(rng.standard_normal((ns, nt)), dtype=dtype, device="cuda")
    q = torch.tensor(rng.standard_normal((ns, nt, nz, nx)) * 1e-3, dtype=dtype, device="cuda")
    for ext in (None, q):
        got = ctx.forward(wavelet=wav, ext=ext)
        ref = torch.full_like(got, float("nan"))
        ctx.forward_noalloc(ref, wavelet=wav, ext=ext)
        assert torch.isfinite(got).all()
        assert torch.equal(got, ref)
    ctx.close()
