"""Performance cases: the calls a user of this framework makes, with the sizes and options they
make them with.

Frames go from the 128-wire x 1024-tick plane to the 960-wire x 6000-tick plane and the
9600-tick planes of mixed batches, depo counts from about a thousand (a short track) to the
1,000,000 of a full event.  A case is a dict of plain values; `kind` names the entry point:

    run         Plane.run: depos in, waveforms out (fluctuation, renormalisation, noise, spectrum
                padding as the case says)
    event       Plane.run on the three planes (two induction, one collection) of one event
    batch       Batch.run: independent events on planes of mixed shapes, one call
    rasterize   Plane.rasterize into a zeroed grid
    convolve    Plane.convolve of a grid
    gradient    Plane.run, then Plane.backward (per-depo and global gradients)
    fit         fit.gpu_event_gradient: one event's loss and gradients of the fitted globals and
                of the response
    autograd    autograd.simulate under torch.autograd, gradients of every input

`exact` restates each of them in 64 bits with torch alone: the bin windows are the integer
decisions of the 32-bit sequence the interface documents, everything else is FP64.
"""
import math

import numpy as np
import torch

from paper_2104_08265_gb300 import autograd, fit, synth, wcsim

V, TICK, NSIGMA = 1.6, 0.5, 3.0          # mm/us, us, patch half-width in sigmas
DL, DT, TAU = 4.0, 8.8, 10000.0          # cm^2/s, cm^2/s, us
SHAPES = {"128x1024": (128, 1024), "480x2000": (480, 2000), "480x9600": (480, 9600),
          "800x6000": (800, 6000), "800x2000": (800, 2000), "960x6000": (960, 6000),
          "960x9600": (960, 9600)}


def listed():
    return [
        # the smallest frame anyone simulates: one test-stand plane, four short tracks, mean path
        _case("small_frame", "run", 128, 1024, 2000, pitch=3.0, td_max=500.0),
        # the benchmark's frame: one DUNE-like collection plane with 40 cosmic-like tracks
        _case("collection_plane", "run", 960, 6000, 100000, fluctuate=1),
        # a shorter readout window of an induction plane with everything on: fluctuation,
        # renormalised patches, electronics noise
        _case("induction_noise", "run", 800, 2000, 30000, fluctuate=1, renormalize=1, noise=1,
              response="induction", td_max=750.0),
        # a plane whose sizes fit nothing: odd wires, impacts and ticks, spectra padded a little
        _case("ragged_frame", "run", 347, 1531, 10000, n_imp=7, n_fw=350, n_ft=1575, fluctuate=1,
              td_max=570.0),
        # the exact binomial draw (the paper's CPU reference) on a modest event
        _case("binomial_plane", "run", 800, 6000, 20000, fluctuate=2, response="induction"),
        # a full event on three planes: long tracks and many short segments
        _case("full_event", "event", 960, 6000, 1000000, fluctuate=1),
        # a stream of small and middle events on planes of mixed shapes, simulated together
        _case("mixed_batch", "batch", 960, 9600, 0, fluctuate=1, events=12, lo=1000, hi=200000,
              shapes="480x2000 800x6000 960x9600 960x6000"),
        # the rasterization layer alone, as a user does who convolves elsewhere
        _case("raster_layer", "rasterize", 960, 6000, 300000),
        # the convolution layer alone, zero-padded so that nothing wraps around
        _case("convolve_padded", "convolve", 800, 6000, 50000, n_fw=960, n_ft=6250,
              response="induction"),
        # gradients of the depos themselves (charge, position, spread), response fixed
        _case("depo_gradients", "gradient", 960, 6000, 100000),
        # one step of the detector-parameter fit: loss, globals and the response spectrum
        _case("fit_step", "fit", 960, 6000, 100000),
        # the small plane inside a torch training loop
        _case("autograd_small", "autograd", 128, 1024, 2000, pitch=3.0, td_max=500.0),
    ]


def draw(rng):
    def log(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    kind = rng.choice(["run", "run", "run", "rasterize", "convolve", "gradient", "fit",
                       "autograd", "batch", "event"])
    if kind == "batch":
        shapes = rng.sample(sorted(SHAPES), rng.randint(1, 4))
        return _case("", "batch", 960, 9600, 0, fluctuate=rng.choice([0, 1]),
                     events=rng.randint(2, 6), lo=1000, hi=log(5000, 200000),
                     shapes=" ".join(shapes))
    if kind == "event":
        return _case("", "event", 960, rng.choice([2000, 6000]), log(20000, 900000), fluctuate=1)
    nw = rng.choice([128, 256, 480, 512, 640, 800, 960]) if rng.random() < 0.5 else log(96, 960)
    nt = rng.choice([1024, 2000, 6000, 9600]) if rng.random() < 0.5 else log(1000, 9600)
    fw, ft = _smooth(nw), _smooth(nt)
    if rng.random() < 0.3:
        fw, ft = _smooth(nw + 20), _smooth(nt + 200)
    fl = rng.choice([0, 1, 1, 2]) if kind == "run" else rng.choice([0, 1]) if kind == "rasterize" else 0
    n = log(1000, 20000) if fl == 2 else log(1000, 100000) if kind != "rasterize" else log(1000, 500000)
    return _case("", kind, nw, nt, n, n_imp=rng.choice([10, 10, 10, 5, 7]), n_fw=fw, n_ft=ft,
                 fluctuate=fl, renormalize=int(rng.random() < 0.25),
                 noise=int(kind == "run" and rng.random() < 0.25),
                 response=rng.choice(["collection", "induction"]),
                 td_max=rng.uniform(0.3, 0.75) * nt * TICK)


def _case(name, kind, n_wires, n_ticks, depos, n_imp=10, n_fw=0, n_ft=0, pitch=4.7, fluctuate=0,
          renormalize=0, noise=0, response="collection", td_max=2250.0, **more):
    c = dict(kind=kind, n_wires=n_wires, n_imp=n_imp, n_ticks=n_ticks, n_fw=n_fw or n_wires,
             n_ft=n_ft or n_ticks, pitch=pitch, depos=depos, fluctuate=fluctuate,
             renormalize=renormalize, noise=noise, response=response, td_max=td_max, **more)
    if name:
        c["name"] = name
    return c


def _smooth(n):
    """The smallest length >= n with no prime factor above 7 (an FFT size the planes take)."""
    while True:
        m = n
        for p in (2, 3, 5, 7):
            while m % p == 0:
                m //= p
        if m == 1:
            return n
        n += 1


# ------------------------------------------------------------------ inputs
def _charges(rng, n):
    return rng.lognormal(math.log(6000.0), 0.3, n).astype(np.float32)


def _tracks(rng, n, p_range, td_max):
    """n depos on straight tracks of up to 2500, ends uniform in pitch position x drift time."""
    per = min(2500, max(1, n // 4))
    k = -(-n // per)
    a, b = rng.uniform(0, p_range, (k, 2)), rng.uniform(0, td_max, (k, 2))
    f = (np.arange(per) + 0.5) / per
    p = (a[:, :1] + (a[:, 1:] - a[:, :1]) * f).ravel()[:n]
    td = (b[:, :1] + (b[:, 1:] - b[:, :1]) * f).ravel()[:n]
    return synth.Depos(p=p, t=np.zeros(n), td=td, q=_charges(rng, n), id=np.arange(n, dtype=np.uint32))


def _event(rng, n, n_ticks):
    """The three planes' depos of an event: 200 long tracks and short segments in a box."""
    box = np.array([0.6 * n_ticks * TICK * V * 1.25, 1200.0, 3000.0])
    n_seg = min(5000, n // 200)
    length = rng.uniform(5.0, 50.0, n_seg)
    k = np.maximum(1, np.round(length)).astype(int)
    which = np.repeat(np.arange(n_seg), k)[:n]
    first = np.concatenate([[0], np.cumsum(k)[:-1]])
    f = (np.arange(which.size) - first[which] + 0.5) / k[which] - 0.5
    d = rng.normal(size=(n_seg, 3))
    d /= np.linalg.norm(d, axis=1, keepdims=True)
    seg = rng.uniform(0, 1, (n_seg, 3))[which] * box + (f * length[which])[:, None] * d[which]
    m = n - which.size
    per = -(-m // 200)
    a, b = rng.uniform(0, 1, (200, 1, 3)) * box, rng.uniform(0, 1, (200, 1, 3)) * box
    trk = (a + (b - a) * ((np.arange(per) + 0.5) / per)[None, :, None]).reshape(-1, 3)[:m]
    x, y, z = np.clip(np.concatenate([seg, trk]), 0.0, box).T
    q = _charges(rng, n)
    out = []
    for nw, deg, kind in ((800, 35.7, "induction"), (800, -35.7, "induction"), (960, 0.0, "collection")):
        a = math.radians(deg)
        p = z * math.cos(a) + y * math.sin(a) + (1200.0 * math.sin(-a) if deg < 0 else 0.0)
        out.append((nw, kind, synth.Depos(p=p, t=np.zeros(n), td=x / V, q=q,
                                          id=np.arange(n, dtype=np.uint32))))
    return out


def _response(g, n_fw, n_ft, kind):
    """R_j(kw, kt), complex64 [n_imp][n_fw][n_ft] on the GPU: a Gaussian pulse (or its bipolar
    derivative) through a semi-Gaussian shaper over 200 ticks, falling off as exp(-|x|/pitch)
    over +-10 wires."""
    n = min(200, n_ft)
    t = np.arange(n) * g.tick_us
    h = (t / 0.5) ** 4 * np.exp(-t / 0.5)
    u = t - 10.0
    f = np.exp(-0.5 * u * u) * (1.0 if kind == "collection" else -u)
    ft = np.zeros(n_ft)
    ft[:n] = np.convolve(f, h / h.sum())[:n]
    prof = np.zeros((g.n_imp, n_fw))
    for j in range(g.n_imp):
        off = ((j + 0.5) / g.n_imp - 0.5) * g.pitch_mm
        for dw in range(-10, 11):
            prof[j, dw % n_fw] += math.exp(-abs(dw * g.pitch_mm - off) / g.pitch_mm)
    a = torch.fft.fft(torch.from_numpy(prof).cuda(), dim=1)
    b = torch.fft.fft(torch.from_numpy(ft).cuda())
    return torch.stack([torch.outer(r, b).to(torch.complex64) for r in a])


def _geometry(nw, n_imp, nt, pitch):
    return synth.Geometry(n_wires=nw, n_imp=n_imp, n_ticks=nt, pitch_mm=pitch, tick_us=TICK)


def _params(case, seed, plane_id=0):
    return synth.DriftParams(v_mm_per_us=V, DL_cm2_s=DL, DT_cm2_s=DT, lifetime_us=TAU,
                             nsigma=NSIGMA, fluctuate=case["fluctuate"], seed=0x5EED0000 + seed,
                             plane_id=plane_id, renormalize=case["renormalize"])


def _parts(case, seed):
    """The planes and host depos of a case: a list of (geometry, params, response kind, n_fw,
    n_ft, depos), one per plane or event."""
    rng = np.random.default_rng([20210408, seed])
    if case["kind"] == "event":
        return [(_geometry(nw, case["n_imp"], case["n_ticks"], case["pitch"]),
                 _params(case, seed, i), kind, nw, case["n_ticks"], d)
                for i, (nw, kind, d) in enumerate(_event(rng, case["depos"], case["n_ticks"]))]
    if case["kind"] == "batch":
        shapes, out = case["shapes"].split(), []
        for e in range(case["events"]):
            i = e % len(shapes)
            nw, nt = SHAPES[shapes[i]]
            n = int(math.exp(rng.uniform(math.log(case["lo"]), math.log(case["hi"]))))
            g = _geometry(nw, case["n_imp"], nt, case["pitch"])
            out.append((g, _params(case, seed, i), "induction" if i % 2 else "collection", nw, nt,
                        _tracks(rng, n, nw * g.pitch_mm, 0.75 * nt * TICK)))
        return out
    g = _geometry(case["n_wires"], case["n_imp"], case["n_ticks"], case["pitch"])
    d = _tracks(rng, case["depos"], g.n_wires * g.pitch_mm, case["td_max"])
    return [(g, _params(case, seed), case["response"], case["n_fw"], case["n_ft"], d)]


def _noise(case):
    """Amplitude spectrum of the electronics noise: white plus a rise at low frequency."""
    k = np.arange(case["n_ft"] // 2 + 1, dtype=np.float64)
    return (200.0 * (1.0 + 4.0 * np.exp(-k / 20.0))).astype(np.float32)


def _cotangent(case, seed):
    """dL/dM of a frame against data: white at the size of the electronics noise."""
    gen = torch.Generator(device="cuda").manual_seed(seed + 17)
    return 100.0 * torch.randn(case["n_wires"], case["n_ticks"], generator=gen, device="cuda")


def _target(case, seed):
    """The frame a fit aims at (made with other diffusion and lifetime), from 64 bits."""
    g, prm, kind, n_fw, n_ft, d = _parts(case, seed)[0]
    other = (6.0, 10.0, 8000.0)
    R = _response(g, n_fw, n_ft, kind)
    return _convolve64(g, R, _grid64(g, prm, _patches(g, prm, d, other))).float()


def prepare(case, seed):
    kind, parts = case["kind"], _parts(case, seed)
    resp, planes, depos = {}, [], []
    for g, prm, rk, n_fw, n_ft, d in parts:
        key = (g, rk, n_fw, n_ft)
        if kind == "batch" and key in resp:          # events of one plane type share the plane
            planes.append(resp[key])
        else:
            R = _response(g, n_fw, n_ft, rk)
            planes.append(wcsim.Plane(g, prm, R, n_fw=n_fw, n_ft=n_ft))
            resp[key] = planes[-1]
        depos.append(wcsim.DeviceDepos.from_host(d))
    s = {"kind": kind, "planes": planes, "depos": depos}
    if case["noise"]:
        planes[0].set_noise(_noise(case), seed=seed + 99)
    if kind == "batch":
        s["batch"] = wcsim.Batch(planes, depos)
    if kind in ("rasterize", "convolve"):
        g = parts[0][0]
        s["grid"] = torch.zeros(g.n_rows, g.n_ticks, device="cuda")
        if kind == "convolve":
            s["grid"].copy_(_grid64(g, parts[0][1], _patches(g, parts[0][1], parts[0][5])))
    if kind in ("gradient", "autograd"):
        s["cotangent"] = _cotangent(case, seed)
    if kind == "fit":
        s["target"] = _target(case, seed)
        s["fit"] = fit.gpu_event_gradient(planes[0], depos[0], s["target"])
        s["state"] = fit.FitState(DL, DT, TAU, R)
        s["params"] = parts[0][1]
    if kind == "autograd":
        for a in (depos[0].q, depos[0].p, depos[0].t, depos[0].td, R):
            a.requires_grad_()
        s["response"] = R
        s["globals"] = [torch.tensor(x, dtype=torch.float64, requires_grad=True) for x in (DL, DT, TAU)]
    return s


GRADS = ("q", "p", "t", "sigma_L", "sigma_T", "DL", "DT", "lifetime")


def run(state):
    kind, plane, depos = state["kind"], state["planes"][0], state["depos"][0]
    if kind in ("run", "event"):
        return [p.run(d) for p, d in zip(state["planes"], state["depos"])]
    if kind == "batch":
        return state["batch"].run()
    if kind == "rasterize":
        return plane.rasterize(depos, state["grid"].zero_())
    if kind == "convolve":
        return plane.convolve(state["grid"])
    if kind == "gradient":
        wave = plane.run(depos)
        grads = plane.backward(depos, state["cotangent"])
        return [wave] + [grads[k] for k in GRADS]
    if kind == "fit":
        loss, grads = state["fit"](state["state"], state["params"])
        return [loss, grads["DL"], grads["DT"], grads["lifetime"], grads["response"]]
    wave = autograd.simulate(plane, depos, *state["globals"], response=state["response"])
    wrt = [depos.q, depos.p, depos.t, depos.td, *state["globals"], state["response"]]
    return [wave.detach()] + list(torch.autograd.grad(wave, wrt, state["cotangent"]))


# ------------------------------------------------------------------ the same in 64 bits
def _philox(c0, c1, c2, c3, k0, k1):
    """Philox4x32-10 on int64 tensors holding 32-bit words."""
    m = 0xFFFFFFFF
    for _ in range(10):
        a, b = c0 * 0xD2511F53, c2 * 0xCD9E8D57
        c0, c1, c2, c3 = (((b >> 32) & m) ^ c1 ^ k0, b & m, ((a >> 32) & m) ^ c3 ^ k1, a & m)
        k0, k1 = (k0 + 0x9E3779B9) & m, (k1 + 0xBB67AE85) & m
    return c0, c1, c2, c3


def _normals(x0, x1):
    u0, u1 = (x0.double() + 0.5) * 2.0 ** -32, (x1.double() + 0.5) * 2.0 ** -32
    r = torch.sqrt(-2.0 * torch.log(u0))
    return r * torch.cos(2 * math.pi * u1), r * torch.sin(2 * math.pi * u1)


def _axis(x, hw, n):
    """The window decision of one axis in its documented 32-bit steps: clipped lo, hi and the
    unclipped ones."""
    i0 = np.floor(x)
    frac = (x - i0).astype(np.float32)
    lo = i0 + np.floor(frac - hw)
    hi = i0 + np.floor(frac + hw)
    return np.maximum(lo, 0), np.minimum(hi, n - 1), lo, hi


def _patches(g, prm, d, globals_=None):
    """Windows (integers, from the 32-bit decision) and 64-bit depo values on the GPU."""
    dl, dt, tau = globals_ or (prm.DL_cm2_s, prm.DT_cm2_s, prm.lifetime_us)
    f = np.float32
    dp = g.pitch_mm / g.n_imp
    td = d.td.astype(f)
    sp = np.sqrt(f(2.0 * (dt * 1e-4)) * td)
    st = np.sqrt(f(2.0 * (dl * 1e-4)) * td) * f(1.0 / prm.v_mm_per_us)
    xp = (d.p - g.p0_mm) * (1.0 / dp)
    xt = (d.t + d.td - g.t0_us) * (1.0 / g.tick_us)
    wp = _axis(xp, f(prm.nsigma) * sp * f(1.0 / dp), g.n_rows)
    wt = _axis(xt, f(prm.nsigma) * st * f(1.0 / g.tick_us), g.n_ticks)
    ok = (wp[0] <= wp[1]) & (wt[0] <= wt[1])
    idx = np.nonzero(ok)[0]

    def dev(a):
        return torch.from_numpy(np.ascontiguousarray(a[idx])).cuda().double()

    td64 = dev(d.td)
    return {"idx": torch.from_numpy(idx).cuda(), "n": len(d), "td": td64, "q": dev(d.q),
            "x": dev(xp), "y": dev(xt), "bin_p": dp, "bin_t": g.tick_us, "D": (dl, dt, tau),
            "sp": torch.sqrt(2e-4 * dt * td64), "sl": torch.sqrt(2e-4 * dl * td64),
            "v": prm.v_mm_per_us, "id": dev(d.id.astype(np.int64)).long(),
            "win": [dev(a).long() for a in wp[:2] + wt[:2]],
            "open": [dev(a) for a in wp[2:] + wt[2:]]}


def _weights(x, sigma, bin_, first, count, lo, hi):
    """Normal mass of bins first .. first + count - 1 (zero outside lo .. hi), [depos][count]."""
    e = first[:, None] + torch.arange(count + 1, device=x.device)
    u = (e - x[:, None]) * (bin_ / (math.sqrt(2.0) * sigma))[:, None]
    low = 0.5 * torch.erfc(-u)                      # both tails keep their relative precision
    up = 0.5 * torch.erfc(u)
    mass = torch.where(u[:, :-1] > 0, up[:, :-1] - up[:, 1:], low[:, 1:] - low[:, :-1])
    mass = torch.where(sigma[:, None] > 0, mass, 1.0)     # a point: its window is the one bin
    b = e[:, :-1]
    return torch.where((b >= lo[:, None]) & (b <= hi[:, None]), mass, 0.0)


def _chunks(p, size=40000):
    order = torch.argsort(p["td"])                  # patches of a chunk have similar sizes
    for i in range(0, order.numel(), size):
        yield order[i:i + size]


def _patch_axes(p, s, sp, sl, x, y):
    """Row weights, tick weights (on whole 4-tick groups), first rows and first ticks of depos s."""
    r_lo, r_hi, k_lo, k_hi = (w[s] for w in p["win"])
    nr = int((r_hi - r_lo).max()) + 1
    q_lo = k_lo >> 2
    nt = 4 * (int(((k_hi >> 2) - q_lo).max()) + 1)
    wp = _weights(x, sp, p["bin_p"], r_lo, nr, r_lo, r_hi)
    wt = _weights(y, sl / p["v"], p["bin_t"], 4 * q_lo, nt, k_lo, k_hi)
    return wp, wt, r_lo, 4 * q_lo


def _grid64(g, prm, p):
    grid = torch.zeros(g.n_rows * g.n_ticks, dtype=torch.float64, device="cuda")
    seed = prm.seed
    for s in _chunks(p):
        qa = p["q"][s] * torch.exp(-p["td"][s] / p["D"][2])
        wp, wt, r0, t0 = _patch_axes(p, s, p["sp"][s], p["sl"][s], p["x"][s], p["y"][s])
        scale = qa
        if prm.renormalize:
            lo_p, hi_p, lo_t, hi_t = (o[s] for o in p["open"])
            for lo, hi, x, sig, b in ((lo_p, hi_p, p["x"][s], p["sp"][s], p["bin_p"]),
                                      (lo_t, hi_t, p["y"][s], p["sl"][s] / p["v"], p["bin_t"])):
                c = b / (math.sqrt(2.0) * sig)
                scale = scale / (1.0 - 0.5 * (torch.erfc((x - lo) * c) + torch.erfc((hi + 1 - x) * c)))
        v = scale[:, None, None] * wp[:, :, None] * wt[:, None, :]
        rows = r0[:, None] + torch.arange(wp.shape[1], device="cuda")
        ticks = t0[:, None] + torch.arange(wt.shape[1], device="cuda")
        if prm.fluctuate == 1:
            quads = (ticks[:, ::4] >> 2)[:, None, :].expand(-1, wp.shape[1], -1)
            c = _philox(quads, rows[:, :, None].expand_as(quads), p["id"][s][:, None, None].expand_as(quads),
                        torch.full_like(quads, prm.plane_id), seed & 0xFFFFFFFF, seed >> 32)
            z = torch.stack(_normals(c[0], c[1]) + _normals(c[2], c[3]), dim=-1).reshape(v.shape)
            var = (v * (1.0 - v / qa[:, None, None])).clamp(min=0)
            v = torch.where(v > 0, (v + torch.sqrt(var) * z).clamp(min=0), 0.0)
        at = rows[:, :, None] * g.n_ticks + ticks[:, None, :]
        live = v != 0
        grid.index_add_(0, at[live], v[live])
    return grid.view(g.n_rows, g.n_ticks)


def _spectra(g, grid, j, n_fw, n_ft):
    return torch.fft.fft2(grid.view(g.n_wires, g.n_imp, g.n_ticks)[:, j].double(), s=(n_fw, n_ft))


def _convolve64(g, R, grid):
    acc = 0
    for j in range(g.n_imp):
        acc = acc + R[j].to(torch.complex128) * _spectra(g, grid, j, R.shape[1], R.shape[2])
    return torch.fft.ifft2(acc).real[:g.n_wires, :g.n_ticks]


def _noise64(case, seed):
    n, nw = case["n_ft"], case["n_wires"]
    k = torch.arange(n // 2 + 1, device="cuda").expand(nw, -1)
    w = torch.arange(nw, device="cuda")[:, None].expand_as(k)
    key = seed + 99
    c = _philox(k >> 1, w, torch.full_like(k, 0x4E4F4953), torch.zeros_like(k), key & 0xFFFFFFFF, key >> 32)
    odd = (k & 1) == 1
    zr, zi = _normals(torch.where(odd, c[2], c[0]), torch.where(odd, c[3], c[1]))
    real = (k == 0) | (2 * k == n)
    h = math.sqrt(0.5)
    xi = torch.complex(torch.where(real, zr, h * zr), torch.where(real, 0.0, h * zi))
    return torch.fft.irfft(torch.from_numpy(_noise(case)).cuda().double() * xi, n=n)[:, :case["n_ticks"]]


def _adjoint64(g, R, grid, G, want_resp):
    n_fw, n_ft = R.shape[1], R.shape[2]
    Gh = torch.fft.fft2(G.double(), s=(n_fw, n_ft))
    dS = torch.empty(g.n_wires, g.n_imp, g.n_ticks, dtype=torch.float64, device="cuda")
    dR = []
    for j in range(g.n_imp):
        back = torch.fft.ifft2(R[j].to(torch.complex128).conj() * Gh)
        dS[:, j] = back.real[:g.n_wires, :g.n_ticks]
        if want_resp:
            dR.append(_spectra(g, grid, j, n_fw, n_ft).conj() * Gh / (n_fw * n_ft))
    return dS.view(g.n_rows, g.n_ticks), (torch.stack(dR) if want_resp else None)


def _depo_grads64(g, prm, p, dS):
    """Per-depo gradients (windows fixed) by automatic differentiation, then the globals."""
    if prm.renormalize:
        raise NotImplementedError
    out = {k: torch.zeros(p["n"], dtype=torch.float64, device="cuda") for k in GRADS[:5]}
    dl, dt, tau = p["D"]
    dS = torch.nn.functional.pad(dS, (0, 4))        # 4-tick groups may reach past the last tick
    for s in _chunks(p, 20000):
        leaf = [a[s].clone().requires_grad_() for a in (p["q"], p["x"], p["y"], p["sl"], p["sp"])]
        q, x, y, sl, sp = leaf
        wp, wt, r0, t0 = _patch_axes(p, s, sp, sl, x, y)
        rows = r0[:, None] + torch.arange(wp.shape[1], device="cuda")
        ticks = t0[:, None] + torch.arange(wt.shape[1], device="cuda")
        at = rows.clamp(max=g.n_rows - 1)[:, :, None] * dS.shape[1] + ticks.clamp(max=g.n_ticks)[:, None, :]
        patch = dS.reshape(-1)[at]
        loss = (q * torch.exp(-p["td"][s] / tau) * torch.einsum("nr,nrt,nt->n", wp, patch, wt)).sum()
        gq, gx, gy, gsl, gsp = torch.autograd.grad(loss, leaf)
        for k, v in zip(GRADS[:5], (gq, gx / p["bin_p"], gy / p["bin_t"], gsl, gsp)):
            out[k][p["idx"][s]] = v
    at = {k: out[k][p["idx"]] for k in GRADS[:5]}
    out["DL"] = (at["sigma_L"] * p["sl"]).sum() / (2 * dl)
    out["DT"] = (at["sigma_T"] * p["sp"]).sum() / (2 * dt)
    out["lifetime"] = (at["q"] * p["q"] * p["td"]).sum() / tau ** 2
    return out


def exact(case, seed):
    kind = case["kind"]
    if case["fluctuate"] == 2 or (case["renormalize"] and kind in ("gradient", "fit", "autograd")):
        return None
    out = []
    for e, (g, prm, rk, n_fw, n_ft, d) in enumerate(_parts(case, seed)):
        if kind == "batch":
            prm = synth.DriftParams(**{**prm.__dict__, "seed": prm.seed + e})
        p = _patches(g, prm, d)
        grid = _grid64(g, prm, p)
        if kind == "rasterize":
            return grid
        if kind == "convolve":
            grid = grid.float()
        R = _response(g, n_fw, n_ft, rk)
        wave = _convolve64(g, R, grid)
        if case["noise"]:
            wave = wave + _noise64(case, seed)
        if kind == "convolve":
            return wave
        if kind in ("run", "event", "batch"):
            out.append(wave)
            continue
        G = wave - _target(case, seed) if kind == "fit" else _cotangent(case, seed)
        dS, dR = _adjoint64(g, R, grid, G, kind != "gradient")
        gr = _depo_grads64(g, prm, p, dS)
        if kind == "gradient":
            return [wave] + [gr[k] for k in GRADS]
        if kind == "fit":
            return [0.5 * float((G * G).sum())] + [float(gr[k]) for k in GRADS[5:]] + [dR]
        td = torch.from_numpy(d.td).cuda()
        q = torch.from_numpy(d.q).cuda().double()
        g_td = (gr["t"] + gr["sigma_L"] * torch.sqrt(2e-4 * DL / td) / 2
                + gr["sigma_T"] * torch.sqrt(2e-4 * DT / td) / 2 - gr["q"] * q / TAU)
        return [wave, gr["q"], gr["p"], gr["t"], g_td] + [gr[k].cpu() for k in GRADS[5:]] + [dR]
    return out


# ------------------------------------------------------------------ work
def work(case):
    """Bytes: depos, the Hermitian half of the response (the whole of it where it is replaced or
    differentiated) and the outputs, once each.  FLOPs: the transforms' 5 N log2 N (half for real
    data), the response products, and about 10 per patch bin."""
    kind, total, flops = case["kind"], 0.0, 0.0
    if kind == "event":
        planes = [(w, case["n_ticks"], case["depos"]) for w in (800, 800, 960)]
    elif kind == "batch":
        shapes = case["shapes"].split()
        mean = (case["hi"] - case["lo"]) / math.log(case["hi"] / case["lo"])
        planes = [SHAPES[shapes[e % len(shapes)]] + (mean,) for e in range(case["events"])]
    else:
        planes = [(case["n_wires"], case["n_ticks"], case["depos"])]
    for i, (nw, nt, n) in enumerate(planes):
        single = kind not in ("event", "batch")
        fw, ft, ni = (case["n_fw"], case["n_ft"], case["n_imp"]) if single else (nw, nt, case["n_imp"])
        nh = ft // 2 + 1
        half, full, frame, grid = 8.0 * ni * fw * nh, 8.0 * ni * fw * ft, 4.0 * nw * nt, 4.0 * nw * ni * nt
        shared = kind == "batch" and i >= len(case["shapes"].split())
        rows = 2.5 * nw * ft * math.log2(ft)                # one impact's time transforms
        cols = 5.0 * nh * fw * math.log2(max(2, fw))        # one impact's wire transforms
        conv = (ni + 1) * (rows + cols) + 8.0 * ni * nh * fw
        bins = 10.0 * 135 * n
        total += {"rasterize": 32 * n + grid, "convolve": grid + half + frame,
                  "gradient": 64 * n + half + 2 * frame, "fit": 32 * n + 2 * full + frame,
                  "autograd": 72 * n + 2 * full + 2 * frame}.get(kind, 32 * n + frame + (0 if shared else half))
        flops += {"rasterize": bins, "convolve": conv, "gradient": 2 * conv + 3 * bins,
                  "fit": 2 * conv + 3 * bins, "autograd": 2 * conv + 3 * bins}.get(kind, conv + bins)
    return {"bytes": total, "flops": flops}
