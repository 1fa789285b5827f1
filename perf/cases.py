"""Performance cases of the egh library: what its users have it do, through the public calls.

A user of the library runs a model update (Green functions, Hessians, factors, multipliers) once
per iteration of an inversion, or one of its stages on its own: the Green stage of a new model,
the Hessians of given transforms, the deblur of gathers against a resident factored set, several
survey patches factored together, the modelling of the synthetic data the residuals come from, and
the serving loop's requests from host memory.  Sizes are those of the repository's workloads (the
101x101 model, the 921x301 layered model, the 1701x351 salt model, the serving sets) and of their
slices; `draw` gives further cases of the same ranges.

`exact` restates the method in 64-bit torch arithmetic (leapfrog, eighth-order Laplacian, sponge;
transforms, Gram, solve and synthesis written out), with none of the library's code.
"""
import math

import numpy as np
import torch

from paper_2512_16642_gb300 import egh

DX = 10.0          # grid spacing of every workload (m)
DT = 1e-3          # time step (s)
ALPHA = 1e-2       # penalty relative to the mean diagonal (or the largest eigenvalue)
SPONGE_R = 1e-3
FP32, MIXED = 0, 1


# ---- cases ---------------------------------------------------------------------------------
def listed():
    return [
        # one model update of a small survey with the library's default precision (the smallest
        # whole call; latency and launches of the FD steps count)
        dict(name="update_small", kind="update", nz=101, nx=101, ns=20, nt=1000, nrec=21, nf=5,
             f0=3.0, f1=7.0, nsrc=11, prec=FP32),
        # one model update of the layered survey in mixed precision: the benchmark's workload and
        # the largest call
        dict(name="update_layered", kind="update", nz=301, nx=921, ns=20, nt=4000, nrec=231, nf=26,
             f0=3.0, f1=8.0, nsrc=115, prec=MIXED),
        # the cheaper update: band-limited source, every tenth level transformed, one random
        # receiver per subset, penalty from the largest eigenvalue
        dict(name="update_bandlimited", kind="bandlimited", nz=301, nx=921, ns=20, nt=2000, nrec=100,
             nall=231, nf=26, f0=3.0, f1=8.0, decim=10, nsrc=34, prec=MIXED),
        # the Green stage alone on the salt grid (40 frequencies, an odd number of receivers), as a
        # rank of a sharded update runs it: its transforms are exported for the exchange
        dict(name="green_salt", kind="green", nz=351, nx=1701, ns=20, nt=500, nrec=19, nf=40, f0=2.0,
             f1=10.0, prec=FP32),
        # synthetic data of a gather of shots (what the residuals are made from)
        dict(name="forward_shots", kind="forward", nz=301, nx=921, ns=20, nt=1000, nrec=231, nsrc=23),
        # Hessians and penalty of given transforms, default precision and mixed precision
        dict(name="hessian_fp32", kind="hessian", nz=301, nx=921, ns=20, nrec=231, nf=26, f0=3.0,
             f1=8.0, prec=FP32),
        dict(name="hessian_mixed", kind="hessian", nz=301, nx=921, ns=20, nrec=231, nf=26, f0=3.0,
             f1=8.0, prec=MIXED),
        # one shot deblurred against a resident set (the smallest call)
        dict(name="deblur_one", kind="deblur", nrec=231, nf=26, f0=3.0, f1=8.0, nsrc=1, nt=4000,
             prec=MIXED),
        # every shot of the layered survey at once
        dict(name="deblur_shots", kind="deblur", nrec=231, nf=26, f0=3.0, f1=8.0, nsrc=115, nt=4000,
             prec=MIXED),
        # default precision, more frequencies, an odd record length
        dict(name="deblur_fp32_odd", kind="deblur", nrec=161, nf=40, f0=2.0, f1=10.0, nsrc=57, nt=2813,
             prec=FP32),
        # three survey patches factored in one batch, then each patch's shots deblurred
        dict(name="patches", kind="patches", nrec=161, nrec2=257, nrec3=341, nf=40, f0=2.0, f1=10.0,
             nsrc=16, nt=3000, prec=MIXED),
        # requests of uneven size from pinned host memory against two resident sets
        dict(name="serving_mix", kind="serving", nrec=101, nf=20, nrec2=211, nf2=27, f0=2.0, f1=10.0,
             nreq=10, maxsrc=24, nt=4000, prec=MIXED),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["update", "update", "bandlimited", "green", "forward", "hessian", "hessian",
                       "deblur", "deblur", "deblur", "patches", "serving"])
    prec = rng.choice([FP32, MIXED])
    nf = rng.randint(5, 40)
    f0, f1 = round(rng.uniform(2.0, 3.0), 2), round(rng.uniform(7.0, 10.0), 2)
    freq = dict(nf=nf, f0=f0, f1=f1)
    if kind in ("update", "bandlimited", "green", "forward"):
        nz, nx = _log(rng, 61, 351), _log(rng, 81, 1701)
        c = dict(kind=kind, nz=nz, nx=nx, ns=20, nt=rng.randint(300, 2000), prec=prec)
        nrec = min(_log(rng, 5, 120), nx)
        # at most a third of the largest listed update's point-steps, and room for the transforms
        while nrec > 5 and (nrec * c["nt"] * (nz + 40) * (nx + 40) > 1e11
                            or nrec * nf * (nz + 40) * (nx + 104) * 8 > 12e9):
            nrec = max(5, nrec // 2)
        nsrc = max(1, min(nx, _log(rng, 1, 60)))
        if kind == "forward":
            while nsrc > 1 and nsrc * c["nt"] * (nz + 40) * (nx + 40) > 3e10:
                nsrc //= 2
            del c["prec"]
            return dict(c, nrec=nrec, nsrc=nsrc)
        if kind == "green":
            return dict(c, nrec=nrec, **freq)
        if kind == "bandlimited":
            return dict(c, nrec=nrec, nall=min(nx, 2 * nrec + rng.randint(0, 9)),
                        decim=rng.choice([1, 4, 7, 10]), nsrc=nsrc, **freq)
        return dict(c, nrec=nrec, nsrc=nsrc, **freq)
    if kind == "hessian":
        nz, nx, nrec = _log(rng, 61, 351), _log(rng, 81, 1701), _log(rng, 11, 341)
        while nrec * nf * (nz + 40) * (nx + 104) * 8 > 12e9:
            nrec = max(5, nrec * 2 // 3)
        return dict(kind=kind, nz=nz, nx=nx, ns=20, nrec=min(nrec, nx), prec=prec, **freq)
    if kind == "deblur":
        nrec, nsrc, nt = _log(rng, 11, 461), _log(rng, 1, 115), rng.randint(1000, 6000)
        freq["nf"] = min(nf, max(5, 13000 // nrec))  # the transforms it is made from stay below 10 GB
        while nrec * nsrc * nt * 4 > 5e8:
            nsrc = max(1, nsrc // 2)
        return dict(kind=kind, nrec=nrec, nsrc=nsrc, nt=nt, prec=prec, **freq)
    if kind == "patches":
        return dict(kind=kind, nrec=_log(rng, 51, 341), nrec2=_log(rng, 51, 341), nrec3=_log(rng, 51, 341),
                    nsrc=_log(rng, 1, 32), nt=rng.randint(1000, 4000), prec=prec, **freq)
    return dict(kind="serving", nrec=rng.randint(51, 151), nf=rng.randint(10, 27), nrec2=rng.randint(101, 231),
                nf2=rng.randint(10, 33), f0=f0, f1=f1, nreq=rng.randint(2, 12), maxsrc=rng.randint(2, 24),
                nt=rng.randint(2000, 4000), prec=prec)


# ---- inputs --------------------------------------------------------------------------------
def _freqs(c, key="nf"):
    return np.linspace(c["f0"], c["f1"], c[key])


def _model(c, seed):
    """Smooth start model: velocity growing with depth over horizontal layers, with a few smooth
    lenses; 1500-4500 m/s (the workloads' smoothed start models)."""
    g = np.random.default_rng([11, int(seed)])
    nz, nx = c["nz"], c["nx"]
    z = np.linspace(0.0, 1.0, nz)[:, None]
    x = np.linspace(0.0, 1.0, nx)[None, :]
    v = 1500.0 + (g.uniform(2300.0, 2700.0) * z + 60.0 * np.sin(2 * np.pi * g.uniform(2, 5) * z)) * np.ones_like(x)
    for _ in range(4):
        cz, cx, s = g.uniform(0.2, 0.9), g.uniform(0, 1), g.uniform(0.05, 0.2)
        v *= 1.0 + g.uniform(-0.06, 0.06) * np.exp(-((z - cz) ** 2 + (x - cx) ** 2) / (2 * s * s))
    return np.clip(v, 1500.0, 4500.0).astype(np.float32)


def _surface(n, nx):
    return np.zeros(n, np.int32), np.linspace(0, nx - 1, n).round().astype(np.int32)


def _ricker(nt, f=8.0):
    t = np.arange(nt) * DT - 1.0 / f
    a = (np.pi * f * t) ** 2
    w = (1.0 - 2.0 * a) * np.exp(-a)
    w[np.abs(w) < 1e-7] = 0.0
    return w[: max(1, int(np.flatnonzero(w)[-1]) + 1)].astype(np.float32)


def _traces(shape, c, seed, device="cuda"):
    """Band-limited Gaussian residuals of unit rms (seeded)."""
    g = torch.Generator(device="cuda").manual_seed(1000 + int(seed))
    x = torch.randn(shape, generator=g, device="cuda")
    n = shape[-1]
    f = torch.fft.rfftfreq(n, DT, device="cuda")
    X = torch.fft.rfft(x)
    X *= torch.clamp(1.0 - torch.clamp(torch.maximum(c["f0"] - f, f - c["f1"]), min=0.0) / 0.5, min=0.0)
    y = torch.fft.irfft(X, n=n)
    y /= y.square().mean().sqrt().clamp(min=1e-20)
    return y.contiguous() if device == "cuda" else y.cpu()


def _transform_planes(nrec, freqs, NZ, NX, rix, ns, seed, out):
    """Far-field 2D Green functions of a medium with two scatterers at every padded grid point,
    written into out[nrec][nf][2][NZ][PX] (columns beyond NX stay zero)."""
    g = np.random.default_rng([12, int(seed)])
    dev = out.device
    c = float(g.uniform(1800.0, 2600.0))
    z = torch.arange(NZ, device=dev, dtype=torch.float32)[:, None] * DX
    x = torch.arange(NX, device=dev, dtype=torch.float32)[None, :] * DX
    scat = [(float(g.uniform(0.3, 0.9)) * NZ * DX, float(g.uniform(0.1, 0.9)) * NX * DX, float(g.uniform(0.5, 2.0)))
            for _ in range(2)]

    def green(r, w):  # modulus and phase of the asymptotic -i/4 H0^(2)(w r / c)
        k = 2 * math.pi * w / c
        return torch.sqrt(1.0 / (8 * math.pi * k * r)), k * r + math.pi / 4

    rs = [torch.sqrt((z - sz) ** 2 + (x - sx) ** 2) + 0.5 * DX for sz, sx, _ in scat]
    xr = torch.from_numpy((np.asarray(rix) + ns) * DX).to(dev, torch.float32)[:, None, None]
    ds = [torch.sqrt((sx - xr) ** 2 + (sz - ns * DX) ** 2) + DX for sz, sx, _ in scat]
    step = max(1, int(2e7) // (NZ * NX))
    for i in range(0, nrec, step):
        r = torch.sqrt((z - ns * DX) ** 2 + (x - xr[i: i + step]) ** 2) + 0.5 * DX
        for k, w in enumerate(freqs):
            a, p = green(r, w)
            re, im = a * torch.cos(p), -a * torch.sin(p)
            for (_, _, s), rr, d in zip(scat, rs, ds):
                a1, p1 = green(d[i: i + step], w)
                a2, p2 = green(rr, w)
                amp, q = (50.0 * s) * a1 * a2, p1 + p2
                re += amp * torch.cos(q)
                im -= amp * torch.sin(q)
            out[i: i + step, k, 0, :, :NX] = re
            out[i: i + step, k, 1, :, :NX] = im


def _ctx(nz, nx, ns, nt, rix, freqs, prec):
    n = len(rix)
    return egh.Context(nz, nx, DX, DX, ns, SPONGE_R, DT, nt, np.zeros(n, np.int32), rix, freqs, precision=prec)


def _with_transforms(nz, nx, ns, nt, rix, freqs, prec, seed):
    """A context holding the synthetic transforms of its receivers."""
    ctx = _ctx(nz, nx, ns, nt, rix, freqs, prec)
    st = ctx.stats()
    buf = ctx.transform_buffer(len(rix), len(freqs))
    NZ, PX = st["nz_pad"], st["pitch"]
    planes = buf[..., : NZ * PX].unflatten(-1, (NZ, PX))
    _transform_planes(len(rix), freqs, NZ, st["nx_pad"], rix, ns, seed, planes)
    ctx.import_green(buf)
    return ctx


def _set_grid(nrec):
    """Grid of a set that only has to hold Hessians of a surface spread: a receiver every four
    columns, as in the layered workload (the Hessians' condition depends on the spacing)."""
    return 40, max(4 * nrec, 48), (4 * np.arange(nrec)).astype(np.int32)


def _factored(nrec, freqs, nt, prec, seed):
    nz, nx, rix = _set_grid(nrec)
    ctx = _with_transforms(nz, nx, 4, nt, rix, freqs, prec, seed)
    ctx.hessian(egh.EGH_MU_REL_MEANDIAG, ALPHA)
    ctx.factor()
    ctx.release_green()
    return ctx


def _serving_set(nrec, nf, seed):
    """Hermitian positive-definite Hessians A A^H / m + 0.05 mean diag I (as the serving tests')."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    m = 2 * nrec
    A = torch.complex(torch.randn((nf, nrec, m), generator=g, device="cuda"),
                      torch.randn((nf, nrec, m), generator=g, device="cuda")) / math.sqrt(m)
    Q = A @ A.mH
    Q = 0.5 * (Q + Q.mH)
    d = torch.diagonal(Q, dim1=1, dim2=2)
    d += 0.05 * d.real.mean()
    return Q.cpu().numpy()


def _requests(c, seed):
    g = np.random.default_rng([13, int(seed)])
    sizes = np.random.default_rng([14, c["nreq"], c["maxsrc"], c["nt"]])  # the mix is the case's
    out = []
    for i in range(c["nreq"]):
        which = int(sizes.integers(2))
        ns = int(sizes.integers(1, c["maxsrc"] + 1))
        nt = int(sizes.integers(c["nt"] // 2, c["nt"] + 1))
        nrec = c["nrec"] if which == 0 else c["nrec2"]
        out.append((which, _traces((ns, nrec, nt), c, int(g.integers(1 << 30)), device="cpu")))
    return out


def _receivers(c, seed):
    if c["kind"] != "bandlimited":
        return _surface(c["nrec"], c["nx"])[1]
    allx = _surface(c["nall"], c["nx"])[1]
    return allx[egh.sample_receivers(c["nall"], c["nrec"], int(seed))]


def prepare(case, seed):
    c = case
    k = c["kind"]
    s = dict(kind=k)
    if k in ("update", "bandlimited", "green"):
        s["vel"] = torch.from_numpy(_model(c, seed)).cuda()
        s["ctx"] = _ctx(c["nz"], c["nx"], c["ns"], c["nt"], _receivers(c, seed), _freqs(c), c["prec"])
        if k == "green":
            s["out"] = s["ctx"].transform_buffer(c["nrec"], c["nf"])
            return s
        s["resid"] = _traces((c["nsrc"], c["nrec"], c["nt"]), c, seed)
        s["mult"] = torch.empty_like(s["resid"])
        if k == "bandlimited":
            s["wav"], s["decim"] = _ricker(c["nt"]), c["decim"]
        return s
    if k == "forward":
        s["vel"] = torch.from_numpy(_model(c, seed)).cuda()
        s["ctx"] = _ctx(c["nz"], c["nx"], c["ns"], c["nt"], _receivers(c, seed), np.array([5.0]), FP32)
        s["src"] = _surface(c["nsrc"], c["nx"])
        w = np.zeros(c["nt"], np.float32)
        r = _ricker(c["nt"])
        w[: r.size] = r
        s["wav"] = w
        s["out"] = torch.empty((c["nsrc"], c["nrec"], c["nt"]), device="cuda")
        return s
    if k == "hessian":
        s["ctx"] = _with_transforms(c["nz"], c["nx"], c["ns"], 4000, _receivers(c, seed), _freqs(c), c["prec"], seed)
        return s
    if k == "deblur":
        s["ctx"] = _factored(c["nrec"], _freqs(c), c["nt"], c["prec"], seed)
        s["resid"] = _traces((c["nsrc"], c["nrec"], c["nt"]), c, seed)
        s["mult"] = torch.empty_like(s["resid"])
        return s
    if k == "patches":
        s["ctx"], s["resid"] = [], []
        for i, n in enumerate((c["nrec"], c["nrec2"], c["nrec3"])):
            nz, nx, rix = _set_grid(n)
            ctx = _with_transforms(nz, nx, 4, c["nt"], rix, _freqs(c), c["prec"], seed + 100 * i)
            ctx.hessian(egh.EGH_MU_REL_MEANDIAG, ALPHA)
            ctx.release_green()
            s["ctx"].append(ctx)
            s["resid"].append(_traces((c["nsrc"], n, c["nt"]), c, seed + 100 * i))
        s["mult"] = [torch.empty_like(r) for r in s["resid"]]
        s["batch"] = egh.Batch(s["ctx"])
        return s
    sv = egh.Server(2 << 30, slots=4, max_batch_sources=96, precision=c["prec"])
    s["ids"] = [sv.add_set(_serving_set(c["nrec"], c["nf"], seed), _freqs(c), DT, c["nt"], c["nt"]),
                sv.add_set(_serving_set(c["nrec2"], c["nf2"], seed + 1), _freqs(c, "nf2"), DT, c["nt"], c["nt"])]
    s["reqs"] = [(w, t.pin_memory(), torch.empty(t.shape, pin_memory=True)) for w, t in _requests(c, seed)]
    s["sv"] = sv
    return s


def run(state):
    s = state
    k = s["kind"]
    if k in ("update", "bandlimited"):
        ctx = s["ctx"]
        if k == "update":
            ctx.green(s["vel"])
            mu = ctx.hessian(egh.EGH_MU_REL_MEANDIAG, ALPHA)
        else:
            ctx.green_bandlimited(s["vel"], s["wav"], s["decim"])
            mu = ctx.hessian(egh.EGH_MU_REL_MAXEIG, ALPHA)
        ctx.factor()
        return {"mu": mu, "mult": ctx.deblur(s["resid"], s["mult"])}
    if k == "green":
        s["ctx"].green(s["vel"])
        s["ctx"].export_green(0, s["ctx"].nf, s["out"])
        return s["out"]
    if k == "forward":
        return s["ctx"].forward(s["vel"], s["src"][0], s["src"][1], s["wav"], s["out"])
    if k == "hessian":
        mu = s["ctx"].hessian(egh.EGH_MU_REL_MEANDIAG, ALPHA)
        return {"mu": mu, "Q": s["ctx"].get_hessian(False)}
    if k == "deblur":
        return s["ctx"].deblur(s["resid"], s["mult"])
    if k == "patches":
        s["batch"].factor()
        return [ctx.deblur(r, m) for ctx, r, m in zip(s["ctx"], s["resid"], s["mult"])]
    ids = [s["sv"].submit(s["ids"][w], r, m) for w, r, m in s["reqs"]]
    for i in ids:
        s["sv"].wait(i)
    return [m for _, _, m in s["reqs"]]


# ---- what a pass cannot do without ---------------------------------------------------------
def work(case):
    c = case
    k = c["kind"]
    pad = (c.get("nz", 0) + 2 * c.get("ns", 0)) * (c.get("nx", 0) + 2 * c.get("ns", 0))
    deb = lambda n, nf, ns, nt: dict(bytes=8.0 * n * ns * nt + 8.0 * nf * n * n,  # noqa: E731
                                     flops=8.0 * nf * n * ns * nt + 8.0 * nf * n * n * ns)
    # a point-step: 8 sums of neighbour pairs, 9 multiply-adds, 3 operations of the update
    step = 8.0 + 18.0 + 4.0
    if k == "forward":
        return dict(bytes=4.0 * c["nz"] * c["nx"] + 4.0 * c["nsrc"] * c["nrec"] * c["nt"],
                    flops=step * c["nsrc"] * c["nt"] * pad)
    if k in ("update", "bandlimited", "green"):
        n, nf = c["nrec"], c["nf"]
        fl = (step + 4.0 * nf / c.get("decim", 1)) * n * c["nt"] * pad
        if k == "green":
            return dict(bytes=4.0 * c["nz"] * c["nx"] + 8.0 * n * nf * pad, flops=fl)
        d = deb(n, nf, c["nsrc"], c["nt"])
        return dict(bytes=4.0 * c["nz"] * c["nx"] + 8.0 * n * c["nsrc"] * c["nt"],
                    flops=fl + 4.0 * nf * n * n * pad + 4.0 / 3.0 * nf * n ** 3 + d["flops"])
    if k == "hessian":
        n, nf = c["nrec"], c["nf"]
        return dict(bytes=8.0 * n * nf * pad + 8.0 * nf * n * n, flops=4.0 * nf * n * n * pad)
    if k == "deblur":
        return deb(c["nrec"], c["nf"], c["nsrc"], c["nt"])
    if k == "patches":
        w = dict(bytes=0.0, flops=0.0)
        for n in (c["nrec"], c["nrec2"], c["nrec3"]):
            d = deb(n, c["nf"], c["nsrc"], c["nt"])
            w["bytes"] += d["bytes"]
            w["flops"] += d["flops"] + 4.0 / 3.0 * c["nf"] * n ** 3
        return w
    w = dict(bytes=0.0, flops=0.0)
    sizes = np.random.default_rng([14, c["nreq"], c["maxsrc"], c["nt"]])
    for _ in range(c["nreq"]):
        which = int(sizes.integers(2))
        ns = int(sizes.integers(1, c["maxsrc"] + 1))
        nt = int(sizes.integers(c["nt"] // 2, c["nt"] + 1))
        d = deb(*((c["nrec"], c["nf"]) if which == 0 else (c["nrec2"], c["nf2"])), ns, nt)
        w["bytes"] += d["bytes"]
        w["flops"] += d["flops"]
    return w


# ---- the same results in 64 bits -----------------------------------------------------------
class _Wave:
    """The padded grid's leapfrog in 64 bits for a batch of sources."""

    C = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)

    def __init__(self, vel, ns, nb):
        v = np.pad(vel.astype(np.float64), ns, mode="edge")
        self.NZ, self.NX = v.shape
        eta = np.zeros_like(v)
        if ns:
            e0 = 1.5 * float(vel.max()) * math.log(1.0 / SPONGE_R) / (ns * DX)
            prof = []
            for n in v.shape:
                i = np.arange(n)
                d = np.maximum(np.maximum(ns - i, i - (n - 1 - ns)), 0)
                prof.append(e0 * (d / ns) ** 2)
            eta = prof[0][:, None] + prof[1][None, :]
        a = 0.5 * eta * DT
        d = torch.device("cuda")
        self.c1 = torch.from_numpy(2.0 / (1.0 + a)).to(d)
        self.c2 = torch.from_numpy((1.0 - a) / (1.0 + a)).to(d)
        self.c3 = torch.from_numpy(DT * DT * v * v / (1.0 + a)).to(d)
        self.u = [torch.zeros((nb, self.NZ + 8, self.NX + 8), dtype=torch.float64, device=d) for _ in range(2)]
        self.lap = torch.empty((nb, self.NZ, self.NX), dtype=torch.float64, device=d)
        self.b = torch.arange(nb, device=d)

    def inner(self, i):
        return self.u[i][:, 4:-4, 4:-4]

    def step(self):
        """u[1] is the current level; afterwards the next one (u[0]: the one before)."""
        p, u = self.u
        NZ, NX = self.NZ, self.NX
        lap = self.lap
        torch.mul(u[:, 4:-4, 4:-4], 2 * self.C[0] / (DX * DX), out=lap)
        for j in range(1, 5):
            w = self.C[j] / (DX * DX)
            for a, b in ((j, 0), (-j, 0), (0, j), (0, -j)):
                lap.add_(u[:, 4 + a: 4 + a + NZ, 4 + b: 4 + b + NX], alpha=w)
        lap *= self.c3
        q = p[:, 4:-4, 4:-4]
        q *= self.c2
        torch.sub(lap, q, out=q)
        q.addcmul_(self.c1, u[:, 4:-4, 4:-4])
        self.u = [u, p]

    def inject(self, pz, px, amp):
        """adds amp / (dx dz) at each batch entry's point of the current level."""
        self.u[1][self.b, pz + 4, px + 4] += self.c3[pz, px] * (amp / (DX * DX))


def _exact_green(c, vel, rix, freqs, wav, decim):
    """ghat [nrec][nf][NZ][NX] complex128."""
    n, nt, ns = len(rix), c["nt"], c["ns"]
    W = _Wave(vel, ns, n)
    d = W.lap.device
    pz = torch.full((n,), ns, device=d)
    px = torch.from_numpy(rix.astype(np.int64)).to(d) + ns
    levels = [t for t in range(nt) if t % decim == 0]
    f = torch.from_numpy(np.asarray(freqs)).to(d)
    out = torch.zeros((len(freqs), 2, n * W.NZ * W.NX), dtype=torch.float64, device=d)
    buf, held = torch.empty((16, n * W.NZ * W.NX), dtype=torch.float64, device=d), []

    def flush():
        t = torch.tensor(held, dtype=torch.float64, device=d) * DT
        ph = 2 * math.pi * torch.remainder(f[:, None] * t[None, :], 1.0)
        w = torch.stack([torch.cos(ph), -torch.sin(ph)], 1).reshape(2 * len(freqs), -1)
        out.view(2 * len(freqs), -1).addmm_(w, buf[: len(held)])
        held.clear()

    levels = set(levels)
    for t in range(nt):
        if t >= 2:
            W.step()
        if t >= 1:
            amp = (1.0 if t == 1 else 0.0) if wav is None else (float(wav[t - 1]) if t - 1 < len(wav) else 0.0)
            if amp:
                W.inject(pz, px, amp)
        if t in levels and t >= 1:
            buf[len(held)].view(n, W.NZ, W.NX).copy_(W.inner(1))
            held.append(float(t))
            if len(held) == buf.shape[0]:
                flush()
    if held:
        flush()
    g = torch.complex(out[:, 0], out[:, 1]).view(len(freqs), n, W.NZ, W.NX)
    if wav is not None:
        t = torch.arange(len(wav), dtype=torch.float64, device=d) * DT
        ph = 2 * math.pi * torch.remainder(f[:, None] * t[None, :], 1.0)
        S = (torch.complex(torch.cos(ph), -torch.sin(ph)) * torch.from_numpy(wav.astype(np.float64)).to(d)).sum(1)
        g *= (decim / S)[:, None, None, None]
    return g


def _gram(g):
    """sum_x g_i conj(g_j) per frequency; g [nf][nrec][points] complex128."""
    return torch.stack([a @ a.mH for a in g])


def _solve_back(Q, resid, freqs, nt_ref, weights=None):
    """Multipliers [ns][nrec][nt] of residuals against Q [nf][nrec][nrec] (complex128)."""
    d = Q.device
    r = resid.double().to(d)
    nt, nf = r.shape[-1], len(freqs)
    t = torch.arange(nt, dtype=torch.float64, device=d) * DT
    f = torch.from_numpy(np.asarray(freqs, np.float64)).to(d)
    ph = 2 * math.pi * torch.remainder(f[:, None] * t[None, :], 1.0)
    co, si = torch.cos(ph), torch.sin(ph)
    flat = r.reshape(-1, nt)
    D = torch.complex(flat @ co.T, -(flat @ si.T)).view(r.shape[0], r.shape[1], nf)
    X = torch.linalg.solve(Q, D.permute(2, 1, 0).contiguous())  # [nf][nrec][ns]
    df = np.gradient(np.asarray(freqs)) if nf > 1 else np.array([1.0 / (nt_ref * DT)])
    w = torch.from_numpy(2.0 * df * DT).to(d)
    X = (X * w[:, None, None]).permute(2, 1, 0).reshape(-1, nf)
    return (X.real @ co - X.imag @ si).view(r.shape)


def _eye(n, d):
    return torch.eye(n, dtype=torch.complex128, device=d)


def _exact_hessian(planes, mode="mean"):
    """(mu, Q) of transforms [nrec][nf][2][points] (any float type) in 64 bits."""
    n, nf = planes.shape[:2]
    H = torch.empty((nf, n, n), dtype=torch.complex128, device=planes.device)
    for k in range(nf):
        a = torch.complex(planes[:, k, 0].double(), planes[:, k, 1].double())
        H[k] = a @ a.mH
    mu = ALPHA * float(torch.diagonal(H, dim1=1, dim2=2).real.mean())
    return mu, H + mu * _eye(n, H.device)


def _synthetic(nz, nx, ns, rix, freqs, seed):
    NZ, NX = nz + 2 * ns, nx + 2 * ns
    out = torch.zeros((len(rix), len(freqs), 2, NZ, NX), device="cuda")
    _transform_planes(len(rix), freqs, NZ, NX, rix, ns, seed, out)
    return out.flatten(3)


def exact(case, seed):
    c = case
    k = c["kind"]
    pad = (c.get("nz", 0) + 2 * c.get("ns", 0)) * (c.get("nx", 0) + 2 * c.get("ns", 0))
    if k in ("update", "bandlimited", "green"):
        if c["nrec"] * c["nt"] * pad > 8e10 or c["nrec"] * c["nf"] * pad * 16 > 40e9:
            return None  # over about 20 seconds, or too large in 64 bits
        vel, rix, freqs = _model(c, seed), _receivers(c, seed), _freqs(c)
        wav, decim = (_ricker(c["nt"]), c["decim"]) if k == "bandlimited" else (None, 1)
        g = _exact_green(c, vel, rix, freqs, wav, decim)
        nf, n, NZ, NX = g.shape
        if k == "green":
            PX = max(64, (NX + 4 + 63) // 64 * 64)
            G = (NZ * PX + 255) // 256 * 256
            out = torch.zeros((n, nf, 2, G), dtype=torch.float64, device="cuda")
            o = out[..., : NZ * PX].unflatten(-1, (NZ, PX))[..., :NX]
            o[:, :, 0] = g.real.transpose(0, 1)
            o[:, :, 1] = g.imag.transpose(0, 1)
            return out
        H = _gram(g.flatten(2))
        del g
        if k == "update":
            mu = ALPHA * float(torch.diagonal(H, dim1=1, dim2=2).real.mean())
        else:
            mu = ALPHA * float(torch.linalg.eigvalsh(H)[:, -1].max())
        Q = H + mu * _eye(n, H.device)
        return {"mu": mu, "mult": _solve_back(Q, _traces((c["nsrc"], n, c["nt"]), c, seed), freqs, c["nt"])}
    if k == "forward":
        if c["nsrc"] * c["nt"] * pad > 8e10:
            return None
        W = _Wave(_model(c, seed), c["ns"], c["nsrc"])
        d = W.lap.device
        sx = torch.from_numpy(_surface(c["nsrc"], c["nx"])[1].astype(np.int64)).to(d) + c["ns"]
        rx = torch.from_numpy(_receivers(c, seed).astype(np.int64)).to(d) + c["ns"]
        sz = torch.full_like(sx, c["ns"])
        wav = _ricker(c["nt"]).astype(np.float64)
        out = torch.zeros((c["nsrc"], c["nrec"], c["nt"]), dtype=torch.float64, device=d)
        for n in range(c["nt"] - 1):
            if n > 0:
                W.step()
            if n < len(wav) and wav[n]:
                W.inject(sz, sx, float(wav[n]))
            out[:, :, n + 1] = W.inner(1)[:, c["ns"], :][:, rx]
        return out
    if k == "hessian":
        planes = _synthetic(c["nz"], c["nx"], c["ns"], _receivers(c, seed), _freqs(c), seed)
        mu, Q = _exact_hessian(planes)
        return {"mu": mu, "Q": torch.view_as_real(Q).cpu().numpy()[..., 0] + 1j * torch.view_as_real(Q).cpu().numpy()[..., 1]}
    if k in ("deblur", "patches"):
        outs = []
        for i, n in enumerate((c["nrec"],) if k == "deblur" else (c["nrec"], c["nrec2"], c["nrec3"])):
            nz, nx, rix = _set_grid(n)
            _, Q = _exact_hessian(_synthetic(nz, nx, 4, rix, _freqs(c), seed + 100 * i))
            outs.append(_solve_back(Q, _traces((c["nsrc"], n, c["nt"]), c, seed + 100 * i), _freqs(c), c["nt"]))
        return outs[0] if k == "deblur" else outs
    sets = [(torch.from_numpy(_serving_set(c["nrec"], c["nf"], seed)).cuda().to(torch.complex128), _freqs(c)),
            (torch.from_numpy(_serving_set(c["nrec2"], c["nf2"], seed + 1)).cuda().to(torch.complex128), _freqs(c, "nf2"))]
    return [_solve_back(sets[w][0], t, sets[w][1], c["nt"]).cpu() for w, t in _requests(c, seed)]
