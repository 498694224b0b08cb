"""The rasterizer's split of the depos over warps and its two forms of the bin masses (a series
about the bin centres, erfc differences at the edges) against the FP64 oracle (needs a GB300).

Sigmas run from a point through both sides of the line between the two forms (about half a bin at
three sigma) to windows wider than one patch tile; depo counts sit on both sides of a warp's share
and of the rule that chooses it.  Tolerances as in the other grid comparisons: FP32 weights of a
few ulp each (6e-8) and a Box-Muller normal good to 1e-6 stay far below relative L2 1e-5 and
1e-4 of the peak.
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


@pytest.mark.parametrize("n_ticks", [800, 803])
@pytest.mark.parametrize("n,fluct", [(1, 1), (5, 0), (4099, 1), (40003, 0), (40003, 1)])
def test_masses_from_points_to_wide_windows(W, n, fluct, n_ticks):
    import torch
    g = S.Geometry(n_wires=48, n_imp=10, n_ticks=n_ticks, pitch_mm=3.0)
    prm = S.DriftParams(fluctuate=fluct, seed=0xA11 + n, DT_cm2_s=20.0, DL_cm2_s=12.0)
    rng = np.random.default_rng(n + n_ticks)
    # sigma_T = 0.3 mm x (0 .. 12 bins): log-uniform, with points and the line's neighbourhood
    bins = np.exp(rng.uniform(np.log(0.05), np.log(12.0), n))
    bins[rng.random(n) < 0.05] = 0.0
    near = rng.random(n) < 0.3
    bins[near] = rng.uniform(0.2, 0.8, n)[near]
    td = (0.3 * bins) ** 2 / (2 * prm.DT_cm2_s * 1e-4)
    d = S.Depos(p=rng.uniform(-3.0, 147.0, n), t=rng.uniform(-5.0, 0.5 * n_ticks, n) - td, td=td,
                q=rng.lognormal(np.log(6000), 0.3, n).astype(np.float32),
                id=rng.integers(0, 2**32, n, dtype=np.uint32))
    if n == 1:
        d.p[0], d.t[0], d.td[0] = 70.0, 100.0, 30.0
    ref = O.rasterize(g, prm, d)
    pl = W.Plane(g, prm, np.zeros((g.n_imp, g.n_wires, 800 if n_ticks == 800 else 810), np.complex64))
    grid = torch.zeros((g.n_rows, g.n_ticks), dtype=torch.float32, device="cuda")
    pl.rasterize(W.DeviceDepos.from_host(d), grid)
    got = grid.cpu().numpy().astype(np.float64)
    assert pl.check_flags() == 0 and ref.any()
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref)
    assert np.abs(got - ref).max() <= 1e-4 * ref.max()
    pl.close()
