"""A solve's network holds what applying it needs: no decoder sums and no normalised input, which
only a weight gradient reads.  Per pixel of an image, BF16 channels: 64 bytes at full resolution,
192, 192 and 128 at 1/4, 1/16 and 1/64 of the pixels, 126 in all; with the gradient's
64 + 32 + 64 / 4 + 64 / 16 it would be 242."""
import numpy as np
import pytest

from paper_2211_06300_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def test_a_loaded_network_holds_no_training_buffers():
    from paper_2211_06300_gb300 import esi
    ns, nt, shape = 4, 128, (241, 801)
    geom = synth.surface_line(ns, np.linspace(500.0, 7000.0, ns), 20.0, [np.arange(0.0, 8000.0, 500.0)] * ns, 20.0)
    c = esi.Context(torch.full(shape, 2000.0, device="cuda"), 10.0, 1e-3, nt, 8, geom)
    params = torch.zeros(esi.PCNet.param_count(), device="cuda")
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    c.pc_load(params)
    torch.cuda.synchronize()
    used = free - torch.cuda.mem_get_info()[0]
    pixels = ns * (nt // 16) * 121 * 401
    # (2 %: levels rounded up to whole pixels; twenty allocations in granules of 2 MB)
    assert used < 1.02 * 126 * pixels + 20 * (2 << 20), used / pixels
    c.close()
