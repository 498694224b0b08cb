"""Tiles that the autotuner reports for the exact binomial can be set by hand (needs a GB300).

The rule by the number of depos gives the exact binomial tiles of few depos per warp, (8, 32) and
(16, 16), and the autotuner may keep the rule; its report has to be a tile that the setter takes, in
every mode, and the grids agree with the oracle's with it (the exact binomial's counts equal but at CDF
steps, at most 1e-4 of the draws off by one).
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


def check(W, pl, dd, ref, fluct, what):
    import torch
    grid = torch.zeros(ref.shape, dtype=torch.float32, device="cuda")
    pl.rasterize(dd, grid)
    got = grid.cpu().numpy()
    diff = got - ref
    if fluct == 2:
        assert np.abs(diff).max() <= 1 and np.count_nonzero(diff) <= max(2, 1e-4 * got.size), what
    else:
        assert np.linalg.norm(diff) <= 1e-5 * np.linalg.norm(ref), what
        assert np.abs(diff).max() <= 1e-4 * ref.max(), what


@pytest.mark.parametrize("fluct", [0, 1, 2])
def test_small_tiles_and_refusals(W, fluct):
    g = S.Geometry(n_wires=64, n_imp=10, n_ticks=800, pitch_mm=3.0)
    prm = S.DriftParams(fluctuate=fluct, seed=0x71 + fluct)
    pl = W.Plane(g, prm, np.zeros((g.n_imp, g.n_wires, g.n_ticks), np.complex64))
    d = S.track_depos(np.random.default_rng(fluct), 3, 211, g.n_wires * 3.0, 300.0)
    dd, ref = W.DeviceDepos.from_host(d), O.rasterize(g, prm, d)
    for tile in ((8, 32), (16, 16)):
        pl.set_raster_tile(*tile)
        check(W, pl, dd, ref, fluct, tile)
        b = W.Batch([pl, pl], [dd, dd])
        for w in b.run():
            assert not w.any()                        # the response is zero
    for tile in ((0, 0), (8, 8), (8, 16), (16, 8), (16, 32), (32, 16), (32, 32), (48, 8), (512, 8), (64, 4)):
        with pytest.raises(W.WcsimError):
            pl.set_raster_tile(*tile)
    assert pl.check_flags() == 0
    pl.close()


@pytest.mark.parametrize("n", [150, 3000])
def test_the_reported_tile_can_be_set(W, n):
    g = S.Geometry(n_wires=64, n_imp=10, n_ticks=800, pitch_mm=3.0)
    prm = S.DriftParams(fluctuate=2, seed=9)
    pl = W.Plane(g, prm, np.zeros((g.n_imp, g.n_wires, g.n_ticks), np.complex64))
    d = S.track_depos(np.random.default_rng(n), 3, n, g.n_wires * 3.0, 300.0)
    dd, ref = W.DeviceDepos.from_host(d), O.rasterize(g, prm, d)
    rep = pl.autotune(dd)
    check(W, pl, dd, ref, 2, rep)
    pl.set_raster_tile(rep["depos_per_block"], rep["lanes_per_depo"])
    check(W, pl, dd, ref, 2, rep)
    pl.close()
