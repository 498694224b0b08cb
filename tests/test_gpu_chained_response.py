"""New responses between chained forwards of a small plane (needs a GB300).

The wire pass starts copying the response before the kernel ahead of it is done; every forward after a
new response has to use the new one.  Frames of the same kernels differ by the order of FP32 additions
only (below 6e-6 relative L2); the old response would be an error of order one.
"""
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


@pytest.mark.parametrize("n_w", [64, 128, 100])
def test_forwards_after_a_new_response(W, n_w):
    import torch
    g = S.Geometry(n_wires=n_w, n_imp=10, n_ticks=512, pitch_mm=3.0)
    rng = np.random.default_rng(n_w)
    Rs = [torch.from_numpy((rng.normal(size=(10, n_w, 512)) + 1j * rng.normal(size=(10, n_w, 512)))
                           .astype(np.complex64)).cuda() for _ in range(2)]
    d = W.DeviceDepos.from_host(S.track_depos(rng, 2, 150, n_w * 3.0, 150.0))
    ref = []
    for R in Rs:
        p = W.Plane(g, S.DriftParams(), R)
        ref.append(p.run(d).clone())
        p.close()
    pl = W.Plane(g, S.DriftParams(), Rs[0])
    out = [torch.zeros_like(ref[0]) for _ in range(12)]
    torch.cuda.synchronize()
    for i, o in enumerate(out):
        if i % 3 == 0:
            pl.set_response(Rs[(i // 3) % 2])
        pl.run(d, out=o)
    for i, o in enumerate(out):
        r = ref[(i // 3) % 2]
        assert ((o - r).double().norm() / r.double().norm()).item() <= 6e-6, i
    pl.close()
