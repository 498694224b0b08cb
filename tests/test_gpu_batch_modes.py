"""A batch of planes with the normal fluctuation and without it (needs a GB300): one rasterization for
all of its events, and every event's frame as the plane's own forward gives it.

Both launches add the same patches, so the frames differ by the order of FP32 additions only; the
tolerances are those of the other batch comparisons.
"""
import dataclasses

import numpy as np
import pytest

from paper_2104_08265_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def W():
    from paper_2104_08265_gb300 import _build
    _build.build()
    from paper_2104_08265_gb300 import wcsim
    return wcsim


def kernels(fn):
    """Names of the kernels that fn launches (a profiler session now and then records none)."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    for _ in range(5):
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            fn()
            torch.cuda.synchronize()
        names = [e.name for e in p.events() if e.device_type == torch.autograd.DeviceType.CUDA]
        if names:
            return names
    pytest.skip("the profiler records no kernels here")


@pytest.mark.parametrize("tile", [None, (128, 16), (64, 32)])
def test_batch_with_and_without_fluctuation(W, tile):
    import torch
    rng = np.random.default_rng(2)
    planes = []
    for i, (n_w, n_t, n_imp) in enumerate([(40, 600, 10), (31, 501, 7), (64, 800, 5)]):
        g = S.Geometry(n_wires=n_w, n_imp=n_imp, n_ticks=n_t, pitch_mm=3.0)
        n_ft = {600: 600, 501: 504, 800: 800}[n_t]
        n_fw = 32 if n_w == 31 else n_w
        R = (rng.normal(size=(n_imp, n_fw, n_ft)) + 1j * rng.normal(size=(n_imp, n_fw, n_ft)))
        pl = W.Plane(g, S.DriftParams(fluctuate=(1, 0, 1)[i], seed=5 + i, plane_id=i),
                     torch.from_numpy(R.astype(np.complex64)).cuda(), n_fw=n_fw, n_ft=n_ft)
        if tile:
            pl.set_raster_tile(*tile)
        planes.append((g, pl))
    which = [0, 1, 2, 1, 0, 2, 2]
    dev = [W.DeviceDepos.from_host(S.track_depos(rng, 2, n, planes[k][0].n_wires * 3.0,
                                                 0.3 * planes[k][0].n_ticks))
           for k, n in zip(which, (1, 33, 300, 7, 64, 129, 500))]
    b = W.Batch([planes[k][1] for k in which], dev)
    got = [w.clone() for w in b.run()]
    for e, (k, d) in enumerate(zip(which, dev)):
        pl = planes[k][1]
        prm = pl.params
        pl.set_params(dataclasses.replace(prm, seed=prm.seed + e))
        ref = pl.run(d)
        pl.set_params(prm)
        assert ref.abs().max() > 0
        assert ((got[e] - ref).double().norm() / ref.double().norm()).item() <= 1e-5, e
        assert ((got[e] - ref).abs().max() / ref.abs().max()).item() <= 1e-4, e
    assert sum("rasterize" in n for n in kernels(b.run)) == 1
    for _, pl in planes:
        assert pl.check_flags() == 0
        pl.close()
