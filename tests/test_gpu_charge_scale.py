"""The normal fluctuation at charges far from an event's own (needs a GB300).

The variance of a bin times the squared radius of a normal leaves FP32's range at both ends (from
Q' = 2^122 up, and where Q' is far below one electron); the bins have to come out as the oracle's all the
same.  Tolerances as in the other grid comparisons: FP32 weights of a few ulp and normals good to 1e-6
stay far below relative L2 1e-5 and 1e-4 of the peak.
"""
import numpy as np
import pytest

from oracle import oracle as O
from paper_2104_08265_gb300 import synth as S

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def W():
    from paper_2104_08265_gb300 import _build
    _build.build()
    from paper_2104_08265_gb300 import wcsim
    return wcsim


@pytest.mark.parametrize("q", [1e-36, 1e-30, 1e-20, 6e3, 1e30, 2e37])
def test_fluctuation_at_any_charge(W, q):
    import torch
    g = S.Geometry(n_wires=48, n_imp=10, n_ticks=800, pitch_mm=3.0)
    prm = S.DriftParams(fluctuate=1, seed=77)
    rng = np.random.default_rng(5)
    n = 40
    td = rng.uniform(20.0, 200.0, n)
    d = S.Depos(p=rng.uniform(5.0, 139.0, n), t=rng.uniform(20.0, 380.0, n) - td, td=td,
                q=np.full(n, q, np.float32), id=np.arange(n, dtype=np.uint32))
    ref = O.rasterize(g, prm, d)
    pl = W.Plane(g, prm, np.zeros((g.n_imp, g.n_wires, g.n_ticks), np.complex64))
    grid = torch.zeros((g.n_rows, g.n_ticks), dtype=torch.float32, device="cuda")
    pl.rasterize(W.DeviceDepos.from_host(d), grid)
    got = grid.cpu().numpy().astype(np.float64)
    assert ref.any() and np.isfinite(got).all()
    s = ref.max()
    assert np.linalg.norm(got / s - ref / s) <= 1e-5 * np.linalg.norm(ref / s)
    assert np.abs(got - ref).max() <= 1e-4 * s
    pl.close()
