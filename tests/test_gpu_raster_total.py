"""The rasterizer's total charge against the FP64 oracle (needs a GB300).

The series form of the bin masses takes exp2 from a hardware instruction that truncates, and the
rasterizer adds the measured mean of what that costs back (7.7e-8 of a patch).  Nothing but the total
shows it: a bin is good to several 1e-8, and those errors average out over patches.  With 20,000 patches,
each scale rounded once (at most 6e-8, spread evenly: 2.5e-10 of the total) and some 150 bins of a few
2^-24 each (smaller still), the total lies far closer than 3e-8; without the correction, or with that of
another instruction, it would be 7.7e-8 off.
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


@pytest.mark.parametrize("td_lo,td_hi", [(60.0, 400.0), (400.0, 2200.0)])
def test_total_charge_is_unbiased(W, td_lo, td_hi):
    import torch
    g = S.Geometry(n_wires=240, n_imp=10, n_ticks=6000, pitch_mm=4.7)
    prm = S.DriftParams()
    rng = np.random.default_rng(8)
    n = 20000
    td = rng.uniform(td_lo, td_hi, n)
    d = S.Depos(p=rng.uniform(20.0, 240 * 4.7 - 20.0, n), t=rng.uniform(60.0, 2900.0, n) - td, td=td,
                q=rng.lognormal(np.log(6000), 0.3, n).astype(np.float32), id=np.arange(n, dtype=np.uint32))
    ref = O.rasterize(g, prm, d).sum()
    pl = W.Plane(g, prm, np.zeros((g.n_imp, g.n_wires, g.n_ticks), np.complex64))
    grid = torch.zeros((g.n_rows, g.n_ticks), dtype=torch.float32, device="cuda")
    pl.rasterize(W.DeviceDepos.from_host(d), grid)
    assert abs(grid.double().sum().item() / ref - 1.0) <= 3e-8
    pl.close()
