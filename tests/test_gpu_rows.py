"""The in-place time-axis transforms over lengths of every kind of plan, against the FP64 oracle
(needs a GB300).

The lengths run through every first and last radix, one to five passes, even and odd groups (the
padded layouts between passes), both forms of the last forward pass and of the first inverse pass
(mirrored butterflies in pairs, or not), and every block size; the small planes take blocks
enlarged for few CTAs, the wide ones the plan's own and the paired inverse.  FP32 transforms of
N <= 13500 points stay below 1e-6 relative L2; the tolerances are those of the other frames.
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


def close(got, ref, what):
    got = np.asarray(got, ref.dtype)
    assert np.isfinite(got).all(), what
    assert np.linalg.norm(got - ref) <= 1e-5 * np.linalg.norm(ref), what
    assert np.abs(got - ref).max() <= 1e-4 * np.abs(ref).max(), what


def check(W, n_w, n_imp, n_t, n_ft, seed):
    import torch
    g = S.Geometry(n_wires=n_w, n_imp=n_imp, n_ticks=n_t, pitch_mm=3.0)
    rng = np.random.default_rng(seed)
    R = (rng.normal(size=(n_imp, n_w, n_ft)) + 1j * rng.normal(size=(n_imp, n_w, n_ft))).astype(np.complex64)
    grid = rng.normal(size=(g.n_rows, n_t)).astype(np.float32)
    grid[:: 3] = 0.0                                       # pairs with one zero row
    grid[: 4] = 0.0                                        # and two
    G = rng.normal(size=(n_w, n_t)).astype(np.float32)
    pl = W.Plane(g, S.DriftParams(), torch.from_numpy(R).cuda())
    what = "%d wires x %d impacts, %d of %d points" % (n_w, n_imp, n_t, n_ft)
    d_grid = torch.from_numpy(grid).cuda()
    wave = pl.convolve(d_grid).cpu().numpy()
    close(wave, O.convolve(g, R, grid.astype(np.float64)), what)
    dS, dR = pl.convolve_adjoint(torch.from_numpy(G).cuda(), d_grid, want_resp=True)
    rS, rR = O.convolve_adjoint(g, R, grid.astype(np.float64), G.astype(np.float64))
    close(dS.cpu().numpy(), rS, what + " dS")
    close(dR.cpu().numpy(), rR, what + " dR")
    assert pl.check_flags() == 0
    pl.close()


@pytest.mark.parametrize("n_ft", [1, 2, 3, 5, 7, 8, 14, 15, 16, 24, 25, 28, 35, 49, 60, 64, 70, 98,
                                  105, 128, 175, 243, 343, 400, 625, 686, 1000, 1536, 1575, 2000,
                                  3375, 4096, 6000, 6250, 8192, 9600, 12005, 12500, 13122, 13500])
def test_every_kind_of_length(W, n_ft):
    check(W, 5, 3, n_ft, n_ft, n_ft)
    if n_ft > 30:
        check(W, 4, 2, n_ft - 7, n_ft, n_ft + 1)           # padded, odd and even rows


@pytest.mark.parametrize("n_ft", [70, 98, 625, 1024, 1575, 2000, 3000])
def test_many_ctas_take_the_plans_own_block(W, n_ft):
    check(W, 256, 10, n_ft - 2, n_ft, n_ft)
