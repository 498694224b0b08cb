"""Forwards of small planes launched chained (each kernel put on the SMs while the one before it
still runs) against the same forwards launched one after the other (needs a GB300).

Changing the parameters makes the next forward an unchained one.  Both launch the same kernels, and
their frames differ only by the order of the FP32 atomic adds into the grid: a row bin takes some
hundred adds at most, each rounded to 2^-24 of the sum, and the signs of the errors are random, so
below 100 x 2^-24 = 6e-6 relative L2.  Stale data (the frames alternate between two events with
nothing in common) would be an error of order one.
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


def rel(a, b):
    return ((a - b).double().norm() / b.double().norm()).item()


# wire kernels: one warp per column, staged block, direct with 4 columns, direct with one; the
# last plane has more row pairs than small planes may have
@pytest.mark.parametrize("n_w, n_imp, n_fw, n_t, n_ft", [
    (128, 10, 128, 1024, 1024), (4, 2, 32, 16, 24), (100, 10, 100, 700, 735), (1200, 1, 1500, 200, 200),
    (600, 2, 3000, 64, 64), (500, 4, 512, 300, 300)])
def test_chained_forwards(W, n_w, n_imp, n_fw, n_t, n_ft):
    import torch
    g = S.Geometry(n_wires=n_w, n_imp=n_imp, n_ticks=n_t, pitch_mm=3.0)
    rng = np.random.default_rng(n_fw + n_ft)
    R = (rng.normal(size=(n_imp, n_fw, n_ft)) + 1j * rng.normal(size=(n_imp, n_fw, n_ft))).astype(np.complex64)
    prm = S.DriftParams()
    pl = W.Plane(g, prm, torch.from_numpy(R).cuda(), n_fw=n_fw, n_ft=n_ft)
    depos = [W.DeviceDepos.from_host(S.track_depos(rng, 2, n, n_w * 3.0, 0.3 * n_t)) for n in (19, 200)]
    target = torch.randn((n_w, n_t), device="cuda")
    ref = []
    for d in depos:
        pl.set_params(prm)                      # the next forward is unchained
        ref.append(pl.run(d).clone())
    out = [torch.zeros_like(ref[0]) for _ in range(12)]
    torch.cuda.synchronize()
    for i, o in enumerate(out):
        pl.run(depos[i & 1], out=o)
    for i, o in enumerate(out):
        assert rel(o, ref[i & 1]) <= 6e-6, (i, rel(o, ref[i & 1]))
    # a loss reset between two forwards, and depos written by the kernel before the forward
    res, loss = pl.run_residual(depos[0], target)
    assert rel(res, ref[0] - target) <= 6e-6
    assert abs(float(loss) - 0.5 * res.double().square().sum().item()) <= 1e-5 * abs(float(loss))
    pl.run(depos[1])
    depos[1].q.mul_(2.0)
    assert rel(pl.run(depos[1]), 2 * ref[1]) <= 6e-6
    depos[1].q.mul_(0.5)
    # captured behind a copy: plain launches
    src = depos[0].q.clone()
    o = torch.zeros_like(ref[0])
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=s):
        depos[0].q.copy_(src)
        pl.run(depos[0], out=o, stream=torch.cuda.current_stream())
    for _ in range(3):
        depos[0].q.zero_()
        graph.replay()
        assert rel(o, ref[0]) <= 6e-6
    assert pl.check_flags() == 0
    pl.close()
