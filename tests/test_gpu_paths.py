"""Which path the time loops of a 2D context take, by its launches: on chip (one launch for the
steps of every shot, or of as many as fit), a launch a step, or two chains of them.  The other
tests compare the paths with one another at these sizes, which shows nothing once a rule moves
both sides to the same one."""
import numpy as np
import pytest

from paper_2211_06300_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

F32, F64 = torch.float32, torch.float64
CASES = [  # nz, nx, shots, type, launches a step (0: on chip)
    (5, 7, 1, F32, 0), (9, 300, 2, F32, 0), (45, 83, 3, F32, 0), (101, 101, 1, F32, 0),
    (241, 801, 1, F32, 0), (241, 801, 2, F32, 0), (64, 1600, 3, F32, 0),
    (5, 7, 1, F64, 0), (45, 83, 3, F64, 0), (101, 101, 1, F64, 0), (241, 801, 1, F64, 0),
    (241, 801, 4, F64, 0), (97, 130, 40, F64, 0),
    (241, 801, 4, F32, 1), (241, 801, 5, F32, 1), (131, 221, 24, F32, 1), (1500, 1500, 1, F64, 1),
    (241, 801, 7, F32, 2), (90, 1601, 9, F32, 2), (241, 801, 16, F32, 2), (131, 221, 36, F32, 2)]


@pytest.mark.parametrize("nz,nx,ns,dtype,per_step", CASES)
def test_the_path_of_a_time_loop(nz, nx, ns, dtype, per_step):
    from paper_2211_06300_gb300 import esi
    nt = 40
    geom = synth.surface_line(ns, np.linspace(0.0, (nx - 1) * 10.0, ns), 20.0,
                              [np.linspace(0.0, (nx - 1) * 10.0, 5)] * ns, 20.0)
    c = esi.Context(torch.full((nz, nx), 2000.0, dtype=dtype, device="cuda"), 10.0, 1e-3, nt, 2, geom)
    n0 = c.launches
    c.forward(wavelet=torch.ones((ns, nt), dtype=dtype, device="cuda"))
    n = c.launches - n0
    if per_step:
        assert n == per_step * nt + 1   # and the last sample
    else:
        assert n <= ns + 1
    c.close()


@pytest.mark.parametrize("nz,nx,ns,dtype,per_step", [(45, 83, 3, F32, 0), (45, 83, 3, F64, 0),
                                                     (241, 801, 4, F32, 1), (241, 801, 7, F32, 2)])
def test_a_new_model_reaches_the_loops_and_costs_what_they_use(nz, nx, ns, dtype, per_step):
    """alpha c, which only the on-chip loops read, is worked out for contexts that have them: at
    creation and for every new model (the model's own kernel is the other launch)."""
    from paper_2211_06300_gb300 import esi
    nt = 40
    geom = synth.surface_line(ns, np.linspace(0.0, (nx - 1) * 10.0, ns), 20.0,
                              [np.linspace(0.0, (nx - 1) * 10.0, 5)] * ns, 20.0)
    rng = np.random.default_rng(nx)
    v = [torch.tensor(1500.0 + 1000.0 * rng.random((nz, nx)), dtype=dtype, device="cuda") for _ in range(2)]
    wav = torch.tensor(rng.standard_normal((ns, nt)), dtype=dtype, device="cuda")
    a, b = [esi.Context(x, 10.0, 1e-3, nt, 2, geom, vref=2500.0) for x in v]
    n = 1 if per_step else 2
    assert a.launches == n
    first = a.forward(wavelet=wav)
    n0 = a.launches
    a.set_velocity(v[1])
    assert a.launches - n0 == n
    second = a.forward(wavelet=wav)
    assert torch.equal(second, b.forward(wavelet=wav)) and not torch.equal(first, second)
    a.close()
    b.close()
