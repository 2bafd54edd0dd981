"""Cases by which the speed of this package is measured, through its public entry points.

Each case is one call, or the few calls, that a program makes once its model,
source and receivers are in place: a forward run, a gradient, a batch of
shots, an inversion iteration.  Media are equal layers with a smooth +-5 %
perturbation and a Gardner density, generated on the GPU from the seed; the
runs are bounded samples of the usual 500 to 3000 steps, so the receivers lie
around the source, within what the waves reach in the steps taken, and the
wavelet peaks inside them.

`exact` restates the scheme in 64 bits with plain torch operations, and takes
gradients of it by torch's own differentiation.
"""
import math
import random

import torch

from paper_2112_15071_gb300 import autograd, ews

DEV = "cuda"
C1, C2 = 9.0 / 8.0, -1.0 / 24.0
LAYERS = (2000.0, 3000.0, 4000.0, 5000.0, 6000.0)
VPVS = 1.73


def _case(name, call, nx, ny, nz, nt, boundary, width, source, nrec, storage="f32", surface=0,
          coarse=0, uneven=False, snapshots=0, shots=1, nmin=0, ckpt=0):
    c = dict(call=call, nx=nx, ny=ny, nz=nz, nt=nt, boundary=boundary, width=width, source=source,
             nrec=nrec, storage=storage, surface=surface, coarse=coarse, uneven=uneven,
             snapshots=snapshots, shots=shots, nmin=nmin, ckpt=ckpt)
    return dict(c, name=name) if name else c


def listed():
    return [
        # the smallest grid in use: a parity-sized cube, where launches and latency count
        _case("forward_64_sponge", "run", 64, 64, 64, 500, "sponge", 16, "moment", 8),
        # odd, ragged sizes with partial tiles on every axis; a point force in C-PML edges
        _case("forward_70x45x37_cpml", "run", 70, 45, 37, 150, "cpml", 6, "force", 5),
        # a middle level of a level-of-detail sweep: unequal spacing, fits the L2
        _case("forward_128x128x64_uneven", "run", 128, 128, 64, 200, "sponge", 16, "moment", 8,
              uneven=True),
        # the benchmark's forward run: C-PML edges, double couple, a receiver array
        _case("forward_256_cpml", "run", 256, 256, 256, 100, "cpml", 20, "moment", 256),
        # a surface recording with a free surface and wavefield snapshots for a film
        _case("surface_200x168x136_cpml", "run", 200, 168, 136, 100, "cpml", 16, "moment", 100,
              surface=19, snapshots=50),
        # the medium held on a coarser grid and interpolated in the passes
        _case("coarse_256_cpml", "run", 256, 256, 256, 60, "cpml", 20, "moment", 256, coarse=64),
        # the largest grid, plain and with 16-bit wavefields
        _case("forward_1024x1024x512", "run", 1024, 1024, 512, 24, "sponge", 20, "force", 1024),
        _case("forward_1024x1024x512_bf16", "run", 1024, 1024, 512, 24, "sponge", 20, "force",
              1024, storage="bf16"),
        # gradient of one shot on an inversion-sized grid, checkpoints every 50 steps
        _case("gradient_192", "gradient", 192, 192, 192, 150, "sponge", 20, "moment", 400, ckpt=50),
        # a differentiable layer in a training loop, on a small grid: forward and backward
        _case("autograd_48x44x40", "autograd", 48, 44, 40, 120, "sponge", 8, "moment", 16, ckpt=40),
        # many shots of uneven size in one launch
        _case("batch_12_shots", "batch", 224, 224, 224, 60, "sponge", 16, "moment", 64, shots=12,
              nmin=96),
        # one iteration of a multi-shot inversion: batched gradients and a line search
        _case("inversion_96_4_shots", "fwi", 96, 96, 96, 80, "sponge", 12, "moment", 64, shots=4,
              ckpt=40),
    ]


def draw(rng):
    def size(lo, hi):
        return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))

    call = rng.choice(["run", "run", "run", "run", "gradient", "batch", "autograd", "fwi"])
    top = {"run": 360, "gradient": 200, "autograd": 90, "batch": 160, "fwi": 100}[call]
    nx, ny, nz = size(24, top), size(24, top), size(24, top)
    if call == "batch":                       # cubes in steps of 8 cells, as the batch recipe has
        nx = ny = nz = max(48, nx // 8 * 8)
    boundary = rng.choice(["sponge", "sponge", "cpml", "cpml", "none"])
    if call in ("gradient", "autograd", "fwi") and boundary == "cpml":
        boundary = "sponge"                   # no gradients with C-PML
    width = rng.randint(4, min(20, min(nx, ny, nz) // 3))
    source = rng.choice(["moment", "force"])
    nt = int(max(24, min(400, 1.5e9 / (nx * ny * nz)))) + rng.randint(0, 9)
    kw = {}
    if call == "run":
        kw["storage"] = rng.choice(["f32", "f32", "f32", "bf16", "f16"])
        form = rng.choice(["plain", "plain", "plain", "surface", "coarse"])
        if form == "surface" and width + 3 < nz // 2:
            kw["surface"] = width + 3
        elif form == "coarse":
            kw["coarse"] = size(8, 64)
        kw["uneven"] = rng.random() < 0.3 and form == "plain"
        kw["snapshots"] = rng.choice([0, 0, max(10, nt // 2)])
    elif call in ("gradient", "autograd"):
        nt = min(nt, 150)
        kw["ckpt"] = rng.choice([0, 25, 50])
    elif call == "fwi":
        nt = min(nt, 100)
        kw.update(shots=rng.randint(2, 4), ckpt=50)
    elif call == "batch":
        nt = min(nt, 100)
        kw.update(shots=rng.randint(2, 10), nmin=max(40, nx // 16 * 8))
    return _case(None, call, nx, ny, nz, nt, boundary, width, source, rng.choice([4, 16, 64, 256]),
                 **kw)


# --- inputs -----------------------------------------------------------------


def _sizes(case):
    """Grid of each shot of a case: the same cubes for every seed."""
    n, full = case["shots"], (case["nx"], case["ny"], case["nz"])
    if case["call"] != "batch":
        return [full] * n
    lo, hi = case["nmin"], case["nx"]
    cubes = [lo + (hi - lo) * s // max(1, n - 1) // 8 * 8 for s in range(n)]
    return [(c, c, c) for c in cubes]


def _noise(shape, gen, cells=10):
    """Smooth noise with max |p| = 1: coarse white noise, interpolated."""
    small = [max(2, -(-n // cells)) for n in shape]
    p = torch.randn([1, 1] + small, generator=gen, device=DEV)
    p = torch.nn.functional.interpolate(p, size=list(shape), mode="trilinear", align_corners=True)
    return (p / p.abs().max())[0, 0]


def _medium(shape, gen, amp=0.05):
    """(vp, vs, rho) on [nz][ny][nx]: layers, perturbation, Gardner density."""
    nz = shape[0]
    layer = torch.clamp(torch.arange(nz, device=DEV) * len(LAYERS) // nz, max=len(LAYERS) - 1)
    vp = torch.tensor(LAYERS, device=DEV)[layer][:, None, None] * (1.0 + amp * _noise(shape, gen))
    vp = vp.contiguous()
    return vp, vp / VPVS, 310.0 * torch.sqrt(torch.sqrt(vp))


def _problem(case, shot, seed):
    """Everything one shot is made of, as plain values and tensors."""
    nx, ny, nz = _sizes(case)[shot]
    gen = torch.Generator(device=DEV).manual_seed(1000 * seed + shot)
    rng = random.Random(1000 * seed + shot)
    h = (10.0, 10.0, 10.0) if not case["uneven"] else (10.0, 16.0, 7.0)
    W, nt = case["width"], case["nt"]
    vpmax = LAYERS[-1] * 1.05
    dt = 0.5 * 0.495 * min(h) / vpmax
    f0 = LAYERS[0] * 0.95 / VPVS / (8.0 * max(h))
    t = torch.arange(nt, dtype=torch.float64) + (0.5 if case["source"] == "moment" else 0.0)
    a = (math.pi * f0 * dt * (t - 0.4 * nt)) ** 2
    wavelet = ((1.0 - 2.0 * a) * torch.exp(-a)).float()
    edge = W + 1.0 if case["boundary"] != "none" else 2.0
    n = (nx, ny, nz)
    lo = [edge, edge, max(edge, float(case["surface"]))]
    hi = [m - edge - 2.0 for m in n]
    src = [l + (u - l) * rng.uniform(0.45, 0.55) for l, u in zip(lo, hi)]
    reach = max(3.0, 0.2 * nt)
    rec = [[min(max(s + rng.uniform(-reach, reach), l), u) * d
            for s, l, u, d in zip(src, lo, hi, h)] for _ in range(case["nrec"])]
    if case["source"] == "moment":
        comp = [1e15 * rng.uniform(0.5, 1.0) for _ in range(3)] + [1e15 * rng.uniform(-1, 1) for _ in range(3)]
    else:
        comp = [1e10 * rng.uniform(0.5, 1.0) for _ in range(3)]
    shape = (nz, ny, nx)
    if case["coarse"]:
        shape = tuple(min(case["coarse"], m) for m in shape)
    return dict(n=n, h=h, dt=dt, nt=nt, f0=f0, shape=shape, gen=gen, wavelet=wavelet,
                src=[s * d for s, d in zip(src, h)], comp=comp, rec=rec)


def _lame(m):
    vp, vs, rho = m
    mu = rho * vs * vs
    return rho * vp * vp - 2.0 * mu, mu, rho


def _with_anomaly(m, shape):
    """The medium with a +5 % sphere in the middle: what was observed."""
    r = [torch.arange(n, device=DEV) - n // 2 for n in shape]
    inside = (r[0][:, None, None] ** 2 + r[1][:, None] ** 2 + r[2] ** 2) <= (min(shape) / 4.0) ** 2
    return m[0] * (1.0 + 0.05 * inside), m[1] * (1.0 + 0.05 * inside), m[2]


def _simulation(case, p):
    snap = case["snapshots"]
    sim = ews.Simulation(*p["n"], p["h"], boundary=case["boundary"], width=case["width"], f0=p["f0"],
                         storage=case["storage"], snapshot_every=snap, snapshot_mask=4 if snap else 0)
    if case["surface"]:
        sim.set_free_surface(case["surface"])
    sim.set_source(case["source"], p["src"], p["comp"], p["wavelet"].numpy())
    sim.set_receivers(p["rec"])
    return sim


def prepare(case, seed):
    state = dict(case=case, shots=[])
    shared = None
    for s in range(case["shots"]):
        p = _problem(case, s, seed)
        if case["call"] == "fwi":             # one model, a source of its own for every shot
            shared = shared or _medium(p["shape"], p["gen"])
            medium = shared
        else:
            medium = _medium(p["shape"], p["gen"])
        sim = _simulation(case, p)
        seis = torch.zeros((3, case["nrec"], p["nt"]), device=DEV)
        shot = dict(sim=sim, nt=p["nt"], dt=p["dt"], seis=seis)
        if case["call"] in ("gradient", "fwi"):
            sim.set_model_vel(*[a.contiguous() for a in _with_anomaly(medium, p["shape"])])
            sim.run(p["nt"], p["dt"], seis)
            shot["observed"] = seis.clone()
        if case["coarse"]:
            sim.set_model_coarse(*medium, from_velocities=True)
        elif case["call"] in ("run", "gradient", "batch"):
            sim.set_model_vel(*medium)
        else:
            state["model"] = [a.contiguous() for a in _lame(medium)]
            sim.set_model_lame(*state["model"])
        if case["call"] == "gradient":
            shot["grad"] = torch.zeros((3,) + p["shape"], device=DEV)
        if case["snapshots"]:
            shot["snaps"] = torch.zeros((p["nt"] // case["snapshots"],) + p["shape"], device=DEV)
        state["shots"].append(shot)
    if case["call"] == "autograd":            # the cotangent that a misfit would send back
        gen = torch.Generator(device=DEV).manual_seed(seed)
        state["back"] = torch.randn((3, case["nrec"], case["nt"]), generator=gen, device=DEV)
    return state


def run(state):
    case, shots = state["case"], state["shots"]
    call, s = case["call"], shots[0]
    if call == "run":
        s["sim"].run(s["nt"], s["dt"], s["seis"], s.get("snaps"))
        return [s["seis"], s["snaps"]] if "snaps" in s else [s["seis"]]
    if call == "gradient":
        misfit, g = s["sim"].gradient(s["nt"], s["dt"], s["observed"], case["ckpt"], s["grad"])
        return [misfit, g[0], g[1], g[2]]
    if call == "autograd":
        model = [a.detach().requires_grad_(True) for a in state["model"]]
        seis = autograd.seismograms(s["sim"], *model, s["nt"], s["dt"], case["ckpt"])
        seis.backward(state["back"])
        return [seis.detach()] + [a.grad for a in model]
    if call == "batch":
        ews.ews_batch([dict(sim=x["sim"], nt=x["nt"], dt=x["dt"], seis=x["seis"]) for x in shots])
        return [x["seis"] for x in shots]
    model = [a.clone() for a in state["model"]]
    j0, j1, _ = ews.ews_fwi_iteration(
        [dict(sim=x["sim"], nt=x["nt"], dt=x["dt"], observed=x["observed"]) for x in shots], *model,
        max_rel_step=0.02, ckpt_every=case["ckpt"])
    return [j0, j1] + model


# --- what a pass cannot do without ------------------------------------------


def work(case):
    """A time step reads and writes the 9 wavefields once and reads the medium
    once (84 bytes a cell in FP32), and the C-PML edges read and write 6
    memory variables a damped direction; a step of a gradient's reverse sweep
    does the same with the adjoint fields, reads the velocity history that the
    forward step wrote, and updates the gradient."""
    es = 4 if case["storage"] == "f32" else 2
    total = flops = 0.0
    for nx, ny, nz in _sizes(case):
        cells = nx * ny * nz
        step = cells * (18.0 * es + (0.0 if case["coarse"] else 12.0))
        if case["boundary"] == "cpml":
            step += 48.0 * sum(cells * min(1.0, 2.0 * case["width"] / n) for n in (nx, ny, nz))
        runs = {"run": 1, "batch": 1, "gradient": 1, "autograd": 2, "fwi": 4}[case["call"]]
        total += runs * case["nt"] * step
        flops += runs * case["nt"] * 160.0 * cells
        if case["call"] in ("gradient", "autograd", "fwi"):
            total += case["nt"] * cells * (84.0 + 24.0 + 24.0)
            flops += case["nt"] * 220.0 * cells
    return {"bytes": total, "flops": flops}


def tolerance(case):
    if case["storage"] == "bf16":
        return {"rel": 2e-2}
    if case["storage"] == "f16":
        return {"rel": 5e-3}
    if case["call"] in ("gradient", "autograd"):
        return {"rel": 3e-5, "max": 3e-3}
    if case["call"] == "fwi":
        return {"rel": 1e-4, "max": 1e-2}
    return {"rel": 1e-5, "max": 1e-3}


# --- the same in 64 bits ----------------------------------------------------


def _shift(f, ax, s):
    """f at index i + s along dimension ax, zero outside."""
    n = f.shape[ax]
    pad = [0, 0] * 3
    g = f.narrow(ax, max(s, 0), n - abs(s))
    pad[2 * (2 - ax) + (1 if s > 0 else 0)] = abs(s)
    return torch.nn.functional.pad(g, pad)


def _diff(f, ax, half, h, switched=None):
    """Eq. 4 difference to the half points (half) or to the integer points.
    switched: planes along z that take the 2nd-order difference."""
    b, c, a, d = (0, 1, -1, 2) if half else (-1, 0, -2, 1)
    inner = _shift(f, ax, c) - _shift(f, ax, b)
    out = (C1 / h) * inner + (C2 / h) * (_shift(f, ax, d) - _shift(f, ax, a))
    if switched is not None:
        out = torch.where(switched[:, None, None], inner / h, out)
    return out


def _clamped(a, ax):
    return torch.cat([a.narrow(ax, 1, a.shape[ax] - 1), a.narrow(ax, a.shape[ax] - 1, 1)], ax)


def _sampled(a, shape, off):
    """Coarse-grid array sampled at the grid's points shifted by off (z, y, x)."""
    for ax in range(3):
        m, n = a.shape[ax], shape[ax]
        c = (torch.arange(n, device=DEV, dtype=torch.float64) + off[ax] + 0.5) * m / n - 0.5
        c = c.clamp(0, m - 1)
        i0 = c.long().clamp(max=max(m - 2, 0))
        f = (c - i0).reshape([-1 if x == ax else 1 for x in range(3)])
        lo = a.index_select(ax, i0)
        a = lo + f * (a.index_select(ax, (i0 + 1).clamp(max=m - 1)) - lo)
    return a


OFF = dict(vx=(0.5, 0, 0), vy=(0, 0.5, 0), vz=(0, 0, 0.5), sxx=(0, 0, 0), syy=(0, 0, 0),
           szz=(0, 0, 0), sxy=(0.5, 0.5, 0), sxz=(0.5, 0, 0.5), syz=(0, 0.5, 0.5))


def _taps(q, pos, h, n):
    """(k, j, i indices, weights) of the 8 neighbours of a point on field q's grid."""
    idx, wts = [], []
    for a in range(3):
        u = pos[a] / h[a] - OFF[q][a]
        i0 = min(int(math.floor(u)), n[a] - 2)
        idx.append((i0, i0 + 1))
        wts.append((1.0 - (u - i0), u - i0))
    return [((k, j, i), wts[2][c] * wts[1][b] * wts[0][a]) for c, k in enumerate(idx[2])
            for b, j in enumerate(idx[1]) for a, i in enumerate(idx[0])]


def _gather(q, positions, h, n):
    taps = [_taps(q, p, h, n) for p in positions]
    k, j, i = (torch.tensor([[t[0][a] for t in r] for r in taps], device=DEV) for a in range(3))
    return (k, j, i), torch.tensor([[t[1] for t in r] for r in taps], device=DEV, dtype=torch.float64)


def _forward64(case, p, lam, mu, rho, vpmax):
    """(seismograms, snapshots) of one run in 64 bits, differentiable in lam, mu, rho."""
    (nx, ny, nz), (hx, hy, hz), dt, W = p["n"], p["h"], p["dt"], case["width"]
    shape, f64 = (nz, ny, nx), dict(device=DEV, dtype=torch.float64)
    ks = case["surface"]
    i2 = h2 = None
    if ks:
        z = torch.arange(nz, device=DEV)
        i2, h2 = (z >= ks - 1) & (z <= ks), (z >= ks - 2) & (z <= ks)
        lam, mu, rho = (torch.cat([1e-3 * a[ks:ks + 1].expand(ks, -1, -1), a[ks:]]) for a in (lam, mu, rho))
    if case["coarse"]:
        bx, by, bz = (1.0 / _sampled(rho, shape, o) for o in ((0, 0, 0.5), (0, 0.5, 0), (0.5, 0, 0)))
        mxy, mxz, myz = (_sampled(mu, shape, o) for o in ((0, 0.5, 0.5), (0.5, 0, 0.5), (0.5, 0.5, 0)))
        lam, mu = (_sampled(a, shape, (0, 0, 0)) for a in (lam, mu))
    else:
        bx, by, bz = (2.0 / (rho + _clamped(rho, ax)) for ax in (2, 1, 0))

        def mean4(a, b):
            u = mu + _clamped(mu, a)
            return 0.25 * (u + _clamped(u, b))

        mxy, mxz, myz = mean4(2, 1), mean4(2, 0), mean4(1, 0)
        if ks:
            mxz, myz = mxz.clone(), myz.clone()
            for m, ax in ((mxz, 2), (myz, 1)):
                u = 1.0 / mu + _clamped(1.0 / mu, ax)
                m[ks - 1] = 4.0 / (u[ks - 1] + u[ks])
    l2m = lam + 2.0 * mu
    gain = torch.ones(shape, **f64) if case["boundary"] == "sponge" else None
    pml = []
    for ax, (n, h) in enumerate(((nz, hz), (ny, hy), (nx, hx))):
        at = torch.arange(n, **f64)
        sh = [-1 if x == ax else 1 for x in range(3)]
        if case["boundary"] == "sponge":
            d = torch.minimum(at, n - 1 - at)
            gain = gain * torch.where(d < W, torch.exp(-(0.3 * (W - d) / W) ** 2), 1.0).reshape(sh)
        if case["boundary"] == "cpml":
            q = torch.where(at < W, (W - at) / W, torch.where(at >= n - W, (at - (n - 1 - W)) / W, -1.0))
            on, q = q >= 0, q.clamp(min=0)
            d0 = -3.0 * vpmax * math.log(1e-3) / (2.0 * W * h) * q * q
            al = math.pi * p["f0"] * (1.0 - q)
            b = torch.exp(-(d0 + al) * dt)
            a = torch.where(d0 + al > 0, d0 * (b - 1.0) / (d0 + al), 0.0)
            pml.append(((on * a).reshape(sh), (on * b).reshape(sh)))
    psi = {}

    def D(f, ax, half, key):
        out = _diff(f, ax, half, (hz, hy, hx)[ax], None if ax else (h2 if half else i2))
        if pml:
            a, b = pml[ax]
            psi[key] = a * out if key not in psi else b * psi[key] + a * out
            out = out + psi[key]
        return out

    F = {q: torch.zeros(shape, **f64) for q in OFF}
    w = p["wavelet"].double().tolist()
    vol = hx * hy * hz
    kind = case["source"]
    names = ("vx", "vy", "vz") if kind == "force" else ("sxx", "syy", "szz", "sxy", "sxz", "syz")
    spread = []
    for q, m in zip(names, p["comp"]):
        add = torch.zeros(shape, **f64)
        for at, wt in _taps(q, p["src"], p["h"], p["n"]):
            add[at] += wt * dt * m / vol * (1.0 if kind == "force" else -1.0)
        spread.append((q, add if gain is None else add * gain))
    recs = {q: _gather(q, p["rec"], p["h"], p["n"]) for q in ("vx", "vy", "vz")}
    traces, snaps = {q: [] for q in recs}, []
    damp = (lambda f: f * gain) if gain is not None else (lambda f: f)
    for n in range(p["nt"]):
        F["vx"] = damp(F["vx"] + dt * bx * (D(F["sxx"], 2, True, 0) + D(F["sxy"], 1, False, 1) + D(F["sxz"], 0, False, 2)))
        F["vy"] = damp(F["vy"] + dt * by * (D(F["sxy"], 2, False, 3) + D(F["syy"], 1, True, 4) + D(F["syz"], 0, False, 5)))
        F["vz"] = damp(F["vz"] + dt * bz * (D(F["sxz"], 2, False, 6) + D(F["syz"], 1, False, 7) + D(F["szz"], 0, True, 8)))
        if kind == "force":
            for (q, add), b in zip(spread, (bx, by, bz)):
                F[q] = F[q] + w[n] * b * add
        for q, (at, wt) in recs.items():
            traces[q].append((F[q][at] * wt).sum(1))
        exx, eyy, ezz = D(F["vx"], 2, False, 9), D(F["vy"], 1, False, 10), D(F["vz"], 0, False, 11)
        F["sxx"] = damp(F["sxx"] + dt * (l2m * exx + lam * (eyy + ezz)))
        F["syy"] = damp(F["syy"] + dt * (l2m * eyy + lam * (exx + ezz)))
        F["szz"] = damp(F["szz"] + dt * (l2m * ezz + lam * (exx + eyy)))
        F["sxy"] = damp(F["sxy"] + dt * mxy * (D(F["vx"], 1, True, 12) + D(F["vy"], 2, True, 13)))
        F["sxz"] = damp(F["sxz"] + dt * mxz * (D(F["vx"], 0, True, 14) + D(F["vz"], 2, True, 15)))
        F["syz"] = damp(F["syz"] + dt * myz * (D(F["vy"], 0, True, 16) + D(F["vz"], 1, True, 17)))
        if kind == "moment":
            for q, add in spread:
                F[q] = F[q] + w[n] * add
        if case["snapshots"] and (n + 1) % case["snapshots"] == 0:
            snaps.append(F["vz"])
    return torch.stack([torch.stack(traces[q], 1) for q in ("vx", "vy", "vz")]), snaps


def exact(case, seed):
    cells = case["nx"] * case["ny"] * case["nz"]
    if case["call"] == "fwi" or (case["call"] in ("gradient", "autograd") and cells * case["nt"] > 4e7):
        return None                           # differentiating it would not fit
    if case["call"] == "run" and cells > 1e8 and case["storage"] != "f32":
        return None                           # the same run as in 32 bits
    out = []
    for s in range(case["shots"]):
        p = _problem(case, s, seed)
        if case["call"] == "run" and cells > 1e8:
            return [_local64(case, p)]
        m = _medium(p["shape"], p["gen"])
        if case["call"] in ("gradient", "autograd"):
            return _exact_gradient(case, p, m, seed)
        lame = _lame([a.double() for a in m])
        seis, snaps = _forward64(case, p, *lame, float(m[0].max()))
        out.append(seis)
        if snaps:
            out.append(torch.stack(snaps))
    return out


def _local64(case, p):
    """A large grid in 64 bits: the block around the source that the waves
    can have crossed on their way to a receiver (4 cells a step at most), if
    it lies clear of the edges, where the damping would begin."""
    vp, vs, rho = _medium(p["shape"], p["gen"])
    reach = [int(max(3.0, 0.2 * p["nt"]) + 2 * p["nt"] + 8)] * 3
    first = [max(0, int(s / h) - r) for s, h, r in zip(p["src"], p["h"], reach)]
    last = [min(n, int(s / h) + r) for s, h, n, r in zip(p["src"], p["h"], p["n"], reach)]
    if any(f < case["width"] or l > n - case["width"] for f, l, n in zip(first, last, p["n"])):
        return None
    cut = tuple(slice(f, l) for f, l in zip(first[::-1], last[::-1]))
    block = [a[cut].double() for a in (vp, vs, rho)]
    move = [f * h for f, h in zip(first, p["h"])]
    q = dict(p, n=tuple(l - f for f, l in zip(first, last)), src=[s - m for s, m in zip(p["src"], move)],
             rec=[[x - m for x, m in zip(r, move)] for r in p["rec"]])
    return _forward64(dict(case, boundary="none"), q, *_lame(block), 0.0)[0]


def _exact_gradient(case, p, m, seed):
    def gradient(lame, of):
        lame = [a.detach().clone().requires_grad_(True) for a in lame]
        seis, _ = _forward64(case, p, *lame, float(m[0].max()))
        loss = of(seis)
        loss.backward()
        return seis.detach(), float(loss.detach()), [a.grad for a in lame]

    if case["call"] == "autograd":
        gen = torch.Generator(device=DEV).manual_seed(seed)
        back = torch.randn((3, case["nrec"], case["nt"]), generator=gen, device=DEV).double()
        seis, _, g = gradient([a.double() for a in _lame(m)], lambda s: (s * back).sum())
        return [seis] + g
    with torch.no_grad():
        true = [a.double() for a in _with_anomaly(m, p["shape"])]
        observed = _forward64(case, p, *_lame(true), float(m[0].max()))[0].float().double()
    _, loss, g = gradient(_lame([a.double() for a in m]), lambda s: 0.5 * p["dt"] * (s - observed).square().sum())
    return [loss] + g
