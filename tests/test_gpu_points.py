"""Depos without diffusion placed just below a bin edge (needs a GB300).

Positions so little below an edge that their fraction rounds up to 1 in FP32 belong to the next bin by
the bin decision; all of a point's charge, and the whole of dL/dS there, has to sit in that bin.  The
weights are exactly 0 and 1, so the grid is compared to one rounding of Q' (relative 1e-6: expf, and at
most a few depos per bin) and the charge gradient likewise; positions inside bins are mixed in.
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


def points(g, n, seed):
    rng = np.random.default_rng(seed)
    x = rng.integers(1, g.n_rows - 1, n).astype(np.float64)
    k = rng.integers(1, g.n_ticks - 1, n).astype(np.float64)
    x += np.where(rng.random(n) < 0.6, -1e-10, rng.uniform(0.1, 0.9, n))
    k += np.where(rng.random(n) < 0.6, -1e-10, rng.uniform(0.1, 0.9, n))
    return S.Depos(p=x, t=k * g.tick_us, td=np.zeros(n), q=np.floor(rng.uniform(500, 9000, n)).astype(np.float32),
                   id=np.arange(n, dtype=np.uint32))


@pytest.mark.parametrize("fluct", [0, 2])
def test_points_below_an_edge_keep_their_charge(W, fluct):
    import torch
    g = S.Geometry(n_wires=40, n_imp=8, n_ticks=600, pitch_mm=8.0)          # bins of 1 mm
    prm = S.DriftParams(fluctuate=fluct, seed=11)
    d = points(g, 700, 3)
    f = (d.p - np.floor(d.p)).astype(np.float32)
    assert (f == 1.0).any() and (f < 1.0).any()
    ref = O.rasterize(g, prm, d)
    pl = W.Plane(g, prm, np.zeros((g.n_imp, g.n_wires, g.n_ticks), np.complex64))
    grid = torch.zeros((g.n_rows, g.n_ticks), dtype=torch.float32, device="cuda")
    dd = W.DeviceDepos.from_host(d)
    pl.rasterize(dd, grid)
    got = grid.cpu().numpy().astype(np.float64)
    assert abs(ref.sum() - d.q.sum(dtype=np.float64)) <= 1e-6 * ref.sum()
    assert np.abs(got - ref).max() <= 1e-6 * ref.max()
    if fluct == 0:
        dS = np.random.default_rng(4).normal(size=grid.shape).astype(np.float32)
        grads = pl.rasterize_adjoint(dd, torch.from_numpy(dS).cuda())
        want = O.depo_grads(g, prm, d, dS.astype(np.float64))["q"]
        assert np.abs(grads["q"].cpu().numpy() - want).max() <= 1e-6 * np.abs(want).max()
    pl.close()
