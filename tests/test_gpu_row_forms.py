"""Row transforms in place and between two buffers, over the CTA counts where the choice changes, against
the FP64 oracle (needs a GB300).

The forms are chosen by the rounds that the CTAs take, so planes of few and of many rows run the same
lengths both ways: the frame's inverse (plain, residual and ADC read-out), the spectra of S, the spectra
of dL/dM after either, the inverse of dL/dS.
Tolerances as in the other frames: FP32 transforms of these lengths stay below 1e-6 relative L2.
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


# 16 x 16 x 16 and 20 x 20 x 16 (no pairs, large radices), 25 x 16 x 10, 25 x 15 x 8; few rows, and as many
# as make the second round small
@pytest.mark.parametrize("n_ft", [512, 3000, 4000, 4096, 4800, 6400, 7200])
@pytest.mark.parametrize("n_w,n_imp", [(9, 3), (96, 10), (128, 10), (610, 1)])
def test_both_forms(W, n_w, n_imp, n_ft):
    import torch
    n_t = n_ft - (n_w + n_ft // 8) % 3                       # even and odd rows, padded or not
    g = S.Geometry(n_wires=n_w, n_imp=n_imp, n_ticks=n_t, pitch_mm=3.0)
    rng = np.random.default_rng(n_ft + n_w)
    n_fw = {9: 9, 96: 96, 128: 128, 610: 625}[n_w]
    R = (rng.normal(size=(n_imp, n_fw, n_ft)) + 1j * rng.normal(size=(n_imp, n_fw, n_ft))).astype(np.complex64)
    grid = rng.normal(size=(g.n_rows, n_t)).astype(np.float32)
    G = rng.normal(size=(n_w, n_t)).astype(np.float32)
    pl = W.Plane(g, S.DriftParams(), torch.from_numpy(R).cuda(), n_fw=n_fw, n_ft=n_ft)
    what = "%d wires x %d impacts, %d of %d points" % (n_w, n_imp, n_t, n_ft)
    d_grid = torch.from_numpy(grid).cuda()
    close(pl.convolve(d_grid).cpu().numpy(), O.convolve(g, R, grid.astype(np.float64)), what)
    dS, dR = pl.convolve_adjoint(torch.from_numpy(G).cuda(), d_grid, want_resp=True)
    rS, rR = O.convolve_adjoint(g, R, grid.astype(np.float64), G.astype(np.float64))
    close(dS.cpu().numpy(), rS, what + " dS")
    close(dR.cpu().numpy(), rR, what + " dR")
    assert pl.check_flags() == 0
    pl.close()


@pytest.mark.parametrize("n_ft", [1000, 4096, 7200])
@pytest.mark.parametrize("n_w", [8, 610])
def test_read_outs_of_both_forms(W, n_w, n_ft):
    import torch
    g = S.Geometry(n_wires=n_w, n_imp=1, n_ticks=n_ft - 2, pitch_mm=3.0)
    rng = np.random.default_rng(n_ft + n_w)
    n_fw = {8: 8, 610: 625}[n_w]
    R = (rng.normal(size=(1, n_fw, n_ft)) + 1j * rng.normal(size=(1, n_fw, n_ft))).astype(np.complex64)
    prm = S.DriftParams()
    pl = W.Plane(g, prm, torch.from_numpy(R).cuda(), n_fw=n_fw, n_ft=n_ft)
    d = S.track_depos(rng, 2, 60, n_w * 3.0, 0.3 * n_ft)
    dd = W.DeviceDepos.from_host(d)
    ref = O.run(g, prm, R, d)
    wave = pl.run(dd)
    close(wave.cpu().numpy(), ref, "run")
    target = torch.randn((n_w, g.n_ticks), device="cuda") * float(wave.abs().max())
    res, loss = pl.run_residual(dd, target)
    assert ((res - (wave - target)).double().norm() / (wave - target).double().norm()).item() <= 6e-6
    want = 0.5 * res.double().square().sum().item()
    assert abs(float(loss) - want) <= 1e-5 * want
    gain = 1000.0 / float(wave.abs().max())
    pl.set_digitizer(gain, 2048.0, 12)
    code = pl.run_adc(dd).cpu().numpy().view(np.uint16).astype(np.float64)
    # one code where the frame lies within its rounding of a threshold
    assert np.abs(code - O.digitize(ref, gain, 2048.0, 12)).max() <= 1
    assert pl.check_flags() == 0
    pl.close()
