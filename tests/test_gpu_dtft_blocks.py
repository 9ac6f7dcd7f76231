"""The blocked DTFT across block ends: 3D runs keep their states in the stash's slots, so a block's
first steps read the last slots of the block before (65, 130 steps: a last block of one and of two
steps; 20: one short block; longer runs are captured in parts); more frequencies than the fold
holds at once; accumulators that hold an earlier run's values; an output at a multiple of an
element's size only.
Against the oracle, with the bounds of the other DTFT tests."""
import numpy as np
import pytest

import oracle
from test_gpu_parity import TOL, _ctx, _dev, _esi, _orc
from paper_2211_06300_gb300 import synth

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32", "f64"])
@pytest.mark.parametrize("nt,nf", [(20, 2), (65, 3), (130, 9), (321, 1)])
def test_dtft_over_block_ends_3d(prec, nt, nf):
    import ctypes
    shape, dx, dt, nb = (19, 21, 37), 10.0, 1e-3, 3
    v = synth.dipping_layers(shape, dx, 4, nlayers=3, vmin=1500, vmax=2500, nanom=1, sigma=40.0)
    gx, gy = np.meshgrid(np.arange(30.0, 330.0, 35.0), np.arange(30.0, 180.0, 35.0))
    rec = np.stack([gx.ravel(), gy.ravel(), np.full(gx.size, 45.0)], axis=1)
    geom = synth.Geometry(np.array([[180.0, 100.0, 40.0], [95.0, 62.0, 50.0]]),
                          np.array([0, len(rec), 2 * len(rec)], dtype=np.int64),
                          np.concatenate([rec, rec]))
    p = dict(dx=dx, dt=dt, nt=nt, nb=nb)
    o, shots = _orc(v, geom, p)
    wav = np.stack([synth.ricker(nt, dt, f, delay=min(1.5 / f, 0.3 * nt * dt)) for f in (22.0, 28.0)])
    freqs = list(np.linspace(6.0, 38.0, nf))
    ctx = _ctx(v, geom, p, prec)
    wd = _dev(wav, prec)
    ctx.dft_extract(freqs, wavelet=_dev(3.0 * wav, prec))   # leaves its values behind
    tr = ctx.empty_traces()
    out, _ = ctx.dft_extract(freqs, wavelet=wd, traces=tr)
    half, scales = ctx.dft_extract(freqs, wavelet=wd, half=True)
    esi = _esi()
    # the same slices through a pointer that is a multiple of an element's size only
    n = half.numel()
    buf = torch.empty(n + 1, dtype=torch.float16, device="cuda")
    sc = np.zeros(2 * nf, dtype=np.float32)
    fr = np.asarray(freqs, dtype=np.float64)
    ctx._check(ctx.L.esi_dft_extract(ctx.h, esi._ptr(wd), None,
                                     fr.ctypes.data_as(ctypes.POINTER(ctypes.c_double)), nf,
                                     esi._ptr(buf[1:]), esi.DFT_C32_HALF,
                                     sc.ctypes.data_as(ctypes.POINTER(ctypes.c_float)), None))
    assert torch.equal(buf[1:], half.reshape(-1)) and np.array_equal(sc, scales.ravel())
    for s, sh in enumerate(shots):
        ref = o.forward(sh, wavelet=wav[s], freqs=freqs)
        got = out[s].double().cpu().numpy().reshape(nf, -1, 2)
        assert oracle.rel_l2(got[..., 0] + 1j * got[..., 1], ref["dft"]) <= TOL[prec]
        assert oracle.rel_l2(ctx.traces_of(tr, s).double().cpu().numpy(), ref["traces"]) <= TOL[prec]
        h = half[s].float().cpu().numpy().reshape(nf, -1, 2) * scales[s][:, None, None]
        for m in range(nf):
            assert oracle.rel_l2(h[m, :, 0] + 1j * h[m, :, 1], ref["dft"][m]) <= 1e-3
