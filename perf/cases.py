"""The work that a user of this library has it do, as measurable cases.

A case names its kind (the entry point it calls) and its sizes.  `listed()`
holds one case for each thing the workflow is used for, `draw()` more of the
same ranges, `prepare()` the arrays and the context that a program has in hand
before the call, `run()` one pass through the public entry points, `work()`
what that pass cannot do without, and `exact()` what it returns in 64 bits.
Grids, acquisitions and options are those of `inputs.py`, the tests and the
bench: 10 m cells, a 20-cell sponge, dt = 1 ms, sources and receivers near the
surface, a water layer over dipping layers, and snapshots every 4 steps.
"""
import math

import numpy as np
import torch
import torch.nn.functional as F

from paper_2001_06444_gb300 import rtm

D, DT, NB = 10.0, 1e-3, 20
SNAP = {"f32": rtm.SNAP_F32, "bf16": rtm.SNAP_BF16, "f16": rtm.SNAP_F16}
# the grids of the workflow's experiments and request stream (nx, nz)
GRIDS = ((201, 101), (851, 176), (1701, 351), (2401, 601))


def listed():
    return [
        # one shot modelled on the small two-layer grid: the shortest call, where a
        # user tries a survey geometry; nothing but launch latency
        dict(name="model_shot", kind="model", nx=201, nz=101, nshot=1, nt=1000),
        # the smallest migration (the first configuration: 201 x 101, one shot, 1000
        # steps, FP32 snapshots)
        dict(name="migrate_shot", kind="migrate", nx=201, nz=101, nshot=1, nt=1000, isnap=4,
             snap="f32", checkpoint=0),
        # the Monte Carlo loop at the precision sweep's size: 16 velocity samples x 2
        # shots in one call, half-precision snapshots
        dict(name="migrate_ensemble", kind="ensemble", nx=201, nz=101, nsample=16, nshot=2,
             nt=800, isnap=4, snap="f16"),
        # the request loop: requests of the mixed grids submitted together and polled
        # until the last is done, BF16 snapshots
        dict(name="serve_mixed", kind="serve", mix=7, nreq=6, nshot=8, nt=2000, snap="bf16"),
        # the survey: many shots of the full-size model, FP32 snapshots every 4 steps
        dict(name="migrate_survey", kind="migrate", nx=1701, nz=351, nshot=48, nt=2000, isnap=4,
             snap="f32", checkpoint=0),
        # the largest grid with the source wavefield recomputed from checkpoints (the
        # memory-lean mode)
        dict(name="migrate_lean", kind="migrate", nx=2401, nz=601, nshot=4, nt=1000, isnap=4,
             snap="f32", checkpoint=-1),
        # least-squares migration: Born modelling and its adjoint, two iterations
        dict(name="lsrtm", kind="lsrtm", nx=851, nz=176, nshot=4, nt=1000, isnap=4, niter=2),
        # the uncertainty stage: statistics of 64 full-size images, then both maps
        dict(name="ensemble_maps", kind="stats", n=64, nx=1701, nz=351),
        # seismograms into the codec at the paper's 1e-4 tolerance
        dict(name="compress_seismograms", kind="compress", what="seis", tol=1e-4, count=8,
             n0=5000, n1=1701),
        # migrated images back out of the codec
        dict(name="decompress_images", kind="decompress", what="image", tol=1e-4, count=64,
             n0=351, n1=1701),
        # one sampler iteration of the tomography: one proposed model, its 34 sources
        dict(name="traveltimes_step", kind="eikonal", nz=88, nx=426, nsample=1, nsrc=34,
             fields=False),
        # traveltimes of a whole velocity ensemble
        dict(name="traveltimes_ensemble", kind="eikonal", nz=88, nx=426, nsample=64, nsrc=34,
             fields=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def _points(nx, nz):
    return (nx + 2 * NB) * (nz + 2 * NB)


def draw(rng):
    kind = rng.choice(("model", "migrate", "migrate", "ensemble", "serve", "lsrtm", "stats",
                       "compress", "decompress", "eikonal", "eikonal"))
    nx = _log(rng, 150, 2401)
    nz = max(80, min(601, int(nx * rng.uniform(0.2, 0.5))))
    upd = float(_points(nx, nz))
    if kind == "model":
        nt = _log(rng, 500, 3000)
        return dict(kind=kind, nx=nx, nz=nz, nt=nt,
                    nshot=min(_log(rng, 1, 32), max(1, int(3e10 / (upd * nt)))))
    if kind == "migrate":
        nt = _log(rng, 500, 3000)
        return dict(kind=kind, nx=nx, nz=nz, nt=nt,
                    nshot=min(_log(rng, 1, 32), max(1, int(3e10 / (upd * nt)))),
                    isnap=rng.choice((1, 2, 3, 4, 4, 8)), snap=rng.choice(("f32", "bf16", "f16")),
                    checkpoint=rng.choice((0, 0, 0, -1)))
    if kind == "ensemble":
        nx, nz, nt = min(nx, 901), min(nz, 201), _log(rng, 400, 1500)
        ns = min(_log(rng, 2, 32), max(2, int(1e10 / (_points(nx, nz) * nt))))
        return dict(kind=kind, nx=nx, nz=nz, nsample=ns, nshot=rng.choice((1, 2, 3)), nt=nt,
                    isnap=rng.choice((1, 4, 4, 8)), snap=rng.choice(("f32", "bf16", "f16")))
    if kind == "serve":
        return dict(kind=kind, mix=rng.randrange(1000), nreq=rng.choice((3, 4, 5, 6)),
                    nshot=rng.choice((4, 5, 6, 7, 8)), nt=_log(rng, 600, 2000),
                    snap=rng.choice(("bf16", "f16")))
    if kind == "lsrtm":
        nx, nz = min(nx, 851), min(nz, 201)
        return dict(kind=kind, nx=nx, nz=nz, nshot=rng.choice((1, 2, 3, 4)),
                    nt=_log(rng, 500, 1000), isnap=rng.choice((2, 3, 4)), niter=rng.choice((1, 2)))
    if kind == "stats":
        return dict(kind=kind, n=_log(rng, 4, 128), nx=min(nx, 1701), nz=min(nz, 351))
    if kind in ("compress", "decompress"):
        what = rng.choice(("seis", "image", "velocity"))
        n0, n1 = (_log(rng, 500, 5000), nx) if what == "seis" else (nz, nx)
        return dict(kind=kind, what=what, tol=rng.choice((1e-4, 1e-1, 0.0)), n0=n0, n1=n1,
                    count=max(1, min(_log(rng, 1, 64), int(3.4e7 / (n0 * n1)))))
    nz = _log(rng, 40, 180)
    nx = _log(rng, 60, 520)
    return dict(kind=kind, nz=nz, nx=nx, nsample=_log(rng, 1, 48), nsrc=rng.randint(2, 34),
                fields=rng.random() < 0.3)


# ---------------------------------------------------------------- inputs --

_ctx = None


def _context():
    """The one context a program keeps; its budget leaves room for the arrays."""
    global _ctx
    if _ctx is None:
        _ctx = rtm.Context(0, budget_bytes=72 << 30)
    return _ctx


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed) % (1 << 62))


def _smooth_noise(g, n, nz, nx, cz, cx):
    """n smooth random fields of unit variance, cz x cx cells correlation."""
    a = torch.randn((n, 1, max(3, int(nz / cz) + 3), max(3, int(nx / cx) + 3)), generator=g,
                    device="cuda")
    a = F.interpolate(a, size=(nz, nx), mode="bicubic", align_corners=True)[:, 0]
    return a / a.flatten(1).std(dim=1)[:, None, None]


def _velocity(g, n, nz, nx, d, smooth):
    """n velocity models (m/s): water over dipping layers of 1600-3500 m/s, a 4700
    m/s basement, each sample perturbed by 4 % below the water; smoothed over a few
    cells (a migration velocity) if `smooth`."""
    z = torch.linspace(0, 1, nz, device="cuda")[:, None]
    x = torch.linspace(-1, 1, nx, device="cuda")[None, :]
    dip = 0.12 * (2 * torch.rand(12, generator=g, device="cuda") - 1)
    water = 0.13
    count = torch.zeros((nz, nx), device="cuda")
    for k in range(12):
        count += (z >= (water + (k + 1) * 0.07 + dip[k] * x).clamp(min=water)).float()
    v = torch.where(z < water, torch.full_like(count, 1500.0), 1600.0 + 158.0 * count)
    v = torch.where((count >= 12) & (z >= water), torch.full_like(v, 4700.0), v)[None]
    v = v * torch.where(z < water, torch.zeros_like(count),
                        0.04 * _smooth_noise(g, n, nz, nx, 300 / d, 300 / d)).add(1.0)
    if smooth:
        w = np.exp(-0.5 * (np.arange(-6, 7) / 3.0) ** 2)
        w = (w / w.sum()).tolist()
        p = F.pad(v[:, None], (0, 0, 6, 6), mode="replicate")[:, 0]
        v = sum(w[k] * p[:, k:k + nz] for k in range(13))
        p = F.pad(v[:, None], (6, 6, 0, 0), mode="replicate")[:, 0]
        v = sum(w[k] * p[:, :, k:k + nx] for k in range(13))
    return v.clamp(1450.0, 5400.0).float().contiguous()


def _seismograms(g, nshot, nt, nrec, src_ix, f, water):
    """Recorded-like data [nshot][nt][nrec]: exactly zero before the first arrival,
    then a direct wave, reflections on hyperbolas and a weak coda, decaying."""
    out = torch.empty((nshot, nt, nrec), device="cuda")
    t = (torch.arange(nt, device="cuda") * DT)[:, None]
    r = torch.arange(nrec, device="cuda")[None, :] * D
    t0 = 0.1 + 0.15 * nt * DT * torch.arange(9, device="cuda") / 2 * (
        0.8 + 0.4 * torch.rand(9, generator=g, device="cuda"))
    amp = 0.1 * (2 * torch.rand(9, generator=g, device="cuda") - 1)
    t0, amp = t0.tolist(), amp.tolist()
    for s in range(nshot):
        off = (r - float(src_ix[s]) * D).abs()
        first = off / 1500.0
        env = (off / 100.0 + 1.0).rsqrt()
        a = (math.pi * f * (t - first - 1.0 / f)) ** 2
        d = 0.3 * env * (1 - 2 * a) * torch.exp(-a)
        for k in range(9):
            v = 1600.0 + 200.0 * k
            a = (math.pi * f * (t - torch.sqrt(t0[k] ** 2 + (off / v) ** 2) - 1.0 / f)) ** 2
            d += amp[k] * env * (1 - 2 * a) * torch.exp(-a)
        coda = F.interpolate(torch.randn((1, 1, max(4, nt // 25), max(4, nrec // 3)), generator=g,
                                         device="cuda"), size=(nt, nrec), mode="bicubic")[0, 0]
        d += 2e-3 * coda * torch.exp(-1.5 * (t - first).clamp(min=0))
        out[s] = torch.where(t < first, torch.zeros_like(d), d)
    return out


def _images(g, n, nz, nx):
    """Migrated images: thin dipping reflectors weakening with depth, side lobes and
    low-level noise, one background shared by the samples."""
    z = torch.linspace(0, 1, nz, device="cuda")[:, None]
    base = _smooth_noise(g, 1, nz, nx, 3, 40)[0]
    img = base[None] + 0.35 * _smooth_noise(g, n, nz, nx, 3, 25)
    img = img + 0.02 * torch.randn((n, nz, nx), generator=g, device="cuda")
    return (img * torch.exp(-2.0 * z) * 0.5).float().contiguous()


def _ricker(f, nt):
    a = (np.pi * f * (np.arange(nt) * DT - 1.0 / f)) ** 2
    return ((1.0 - 2.0 * a) * np.exp(-a)).astype(np.float32)


class _Survey:
    """Grid, acquisition and wavelet as the binding takes them."""

    def __init__(self, nx, nz, nshot, nt, f=12.0):
        self.nx, self.nz, self.nshot, self.nt, self.f = nx, nz, nshot, nt, f
        if nshot == 1:
            self.sx = np.array([nx // 2], np.int32)
        else:
            self.sx = np.round(np.linspace(0.05, 0.95, nshot) * (nx - 1)).astype(np.int32)
        self.sz = np.full(nshot, 1, np.int32)
        self.rx, self.rz = np.arange(nx, dtype=np.int32), np.full(nx, 1, np.int32)
        self.wav = _ricker(f, nt)
        self.keep = rtm._Keep()
        self.grid = rtm.make_grid(nx, nz, NB, D, D, DT, nt)
        self.acq = rtm.make_acq(self.keep, self.sx, self.sz, self.rx, self.rz, self.wav)


def _requests(case):
    """(nx, nz, shots, frequency) of each request of a mix: small and middle grids
    mostly, one large one, shots up to the case's."""
    rng = np.random.RandomState(case["mix"])
    out = []
    for k in range(case["nreq"]):
        nx, nz = GRIDS[(0, 1, 2, 0, 1, 3)[k % 6]]
        most = case["nshot"] if nx < 1000 else max(1, case["nshot"] // 3)
        out.append((nx, nz, int(rng.randint(1, most + 1)), float(rng.uniform(10.0, 15.0))))
    return out


def prepare(case, seed):
    kind = case["kind"]
    g = _gen(seed)
    st = {"case": dict(case), "ctx": _context()}
    if kind in ("model", "migrate", "ensemble", "lsrtm"):
        nx, nz, nshot, nt = case["nx"], case["nz"], case["nshot"], case["nt"]
        s = st["survey"] = _Survey(nx, nz, nshot, nt)
        n = case.get("nsample", 1)
        st["vel"] = _velocity(g, n, nz, nx, D, kind != "model")
        if kind != "ensemble":
            st["vel"] = st["vel"][0].contiguous()
        if kind == "model":
            st["out"] = torch.zeros((nshot, nt, nx), device="cuda")
        else:
            st["seis"] = _seismograms(g, nshot, nt, nx, s.sx, s.f, 0.13)
            st["opts"] = rtm.Opts(case["isnap"], SNAP[case.get("snap", "f32")], 1e-6, 1,
                                  case.get("checkpoint", 0))
            st["out"] = torch.zeros((n, nz, nx) if kind == "ensemble" else (nz, nx), device="cuda")
    elif kind == "serve":
        st["reqs"] = []
        for nx, nz, nshot, f in _requests(case):
            s = _Survey(nx, nz, nshot, case["nt"], f)
            vel = _velocity(g, 1, nz, nx, D, True)[0].contiguous()
            seis = _seismograms(g, nshot, case["nt"], nx, s.sx, f, 0.13)
            img = torch.zeros((nz, nx), device="cuda")
            req = rtm.Request(s.grid, vel.data_ptr(), s.acq, seis.data_ptr(),
                              rtm.Opts(4, SNAP[case["snap"]], 1e-6, 1, 0), img.data_ptr())
            st["reqs"].append((req, s, vel, seis, img))
        torch.cuda.synchronize()  # the request loop's streams do not wait for this one
    elif kind == "stats":
        st["images"] = _images(g, case["n"], case["nz"], case["nx"])
        npix = case["nz"] * case["nx"]
        st["out"] = [torch.zeros(npix, dtype=t, device="cuda")
                     for t in (torch.float64, torch.float64, torch.float32, torch.float32,
                               torch.float64, torch.float64)]
    elif kind in ("compress", "decompress"):
        x = _codec_data(case, seed)
        stride = (rtm.compress_bound(case["n0"], case["n1"]) + 15) // 16 * 16
        st["stride"], st["data"] = stride, x
        st["streams"] = torch.zeros(case["count"] * stride, dtype=torch.uint8, device="cuda")
        if kind == "decompress":  # the streams a program has read from its files
            st["ctx"].compress(x, case["tol"], out=st["streams"], stride=stride)
            st["data"] = torch.zeros_like(x)
    else:
        st["vel"], st["src"], st["rec"] = _eikonal_inputs(case, seed)
        n = (case["nsample"], case["nsrc"])
        st["times"] = torch.zeros((*n, case["nx"]), device="cuda")
        st["fields"] = (torch.zeros((*n, case["nz"], case["nx"]), device="cuda")
                        if case["fields"] else None)
    return st


def _codec_data(case, seed):
    g = _gen(seed)
    n, n0, n1 = case["count"], case["n0"], case["n1"]
    if case["what"] == "seis":
        src = np.round(np.linspace(0.05, 0.95, n) * (n1 - 1)).astype(np.int32)
        return _seismograms(g, n, n0, n1, src, 12.0, 0.13)
    if case["what"] == "image":
        return _images(g, n, n0, n1)
    return _velocity(g, n, n0, n1, D, False)


def _eikonal_inputs(case, seed):
    """Velocities on the 40 m tomography grid, surface sources, a receiver at every
    surface node."""
    vel = _velocity(_gen(seed), case["nsample"], case["nz"], case["nx"], 40.0, False)
    sx = np.round(np.linspace(0.02, 0.98, case["nsrc"]) * (case["nx"] - 1)).astype(np.int32)
    rx = np.arange(case["nx"], dtype=np.int32)
    return vel, (np.zeros_like(sx), sx), (np.zeros_like(rx), rx)


# ------------------------------------------------------------------- run --


def run(st):
    case, ctx, kind = st["case"], st["ctx"], st["case"]["kind"]
    if kind == "model":
        s = st["survey"]
        return ctx.model(s.grid, st["vel"], s.acq, -1, st["out"])
    if kind == "migrate":
        s = st["survey"]
        return ctx.migrate(s.grid, st["vel"], s.acq, st["seis"], st["opts"], st["out"])
    if kind == "ensemble":
        s = st["survey"]
        return ctx.migrate_ensemble(s.grid, st["vel"], s.acq, st["seis"], st["opts"], st["out"])
    if kind == "lsrtm":
        s = st["survey"]
        misfit = ctx.lsrtm(s.grid, st["vel"], s.acq, st["seis"], st["opts"], case["niter"],
                           st["out"])
        return {"refl": st["out"], "misfit": misfit}
    if kind == "serve":
        tickets = [ctx.submit(r[0]) for r in st["reqs"]]
        for t in tickets:
            state, rc = ctx.poll(t, 60000)
            if state != rtm.REQ_DONE:
                raise RuntimeError(f"request {t}: state {state}, {ctx.last_error()}")
        return [r[4] for r in st["reqs"]]
    if kind == "stats":
        o = st["out"]
        ctx.ensemble_stats(st["images"], *o[:4])
        ctx.uncertainty_maps(o[0], o[1], o[4], o[5])
        return dict(zip(("mean", "std", "q05", "q95", "confidence", "ratio"), o))
    if kind == "compress":
        _, _, sizes = ctx.compress(st["data"], case["tol"], out=st["streams"], stride=st["stride"])
        return {"streams": st["streams"], "sizes": torch.tensor(sizes)}
    if kind == "decompress":
        return ctx.decompress(st["streams"], st["stride"], case["count"], case["n0"], case["n1"],
                              st["data"])
    iters = ctx.eikonal(st["vel"], 40.0, 40.0, *st["src"], *st["rec"], times=st["times"],
                        fields=st["fields"])
    out = {"times": st["times"], "iters": torch.tensor(iters)}
    if st["fields"] is not None:
        out["fields"] = st["fields"]
    return out


def _rtm_work(nx, nz, items, nt, isnap, esz, passes):
    """Wave propagation: 22 operations per padded update; what must cross memory is
    the velocity, the data, the image and one write and one read of each snapshot."""
    upd = _points(nx, nz) * float(nt) * items
    nsnap = nt // isnap if isnap else 0
    return {"bytes": 4.0 * items * nt * nx + 8.0 * nx * nz + 2.0 * esz * nsnap * items * nx * nz,
            "flops": 22.0 * upd * passes}


def work(case):
    kind = case["kind"]
    esz = {"f32": 4, "bf16": 2, "f16": 2}.get(case.get("snap", "f32"), 4)
    if kind == "model":
        return _rtm_work(case["nx"], case["nz"], case["nshot"], case["nt"], 0, 0, 1)
    if kind in ("migrate", "ensemble"):
        return _rtm_work(case["nx"], case["nz"], case["nshot"] * case.get("nsample", 1),
                         case["nt"], 0 if case.get("checkpoint", 0) else case["isnap"], esz, 2)
    if kind == "lsrtm":  # niter Born modellings and niter + 1 adjoints, two passes each
        w = _rtm_work(case["nx"], case["nz"], case["nshot"], case["nt"], case["isnap"], 4, 2)
        k = 2 * case["niter"] + 1
        return {"bytes": k * w["bytes"], "flops": k * w["flops"]}
    if kind == "serve":
        ws = [_rtm_work(nx, nz, ns, case["nt"], 4, esz, 2) for nx, nz, ns, _ in _requests(case)]
        return {k: sum(w[k] for w in ws) for k in ("bytes", "flops")}
    if kind == "stats":
        npix = float(case["nx"] * case["nz"])
        return {"bytes": npix * (4 * case["n"] + 24 + 16 + 16), "flops": npix * 8 * case["n"]}
    if kind in ("compress", "decompress"):
        n = float(case["count"] * case["n0"] * case["n1"])
        ratio = {"seis": 0.15, "image": 0.5, "velocity": 0.5}[case["what"]]
        return {"bytes": 4 * n * (1 + ratio), "flops": 20 * n}
    n = float(case["nz"] * case["nx"])
    p = case["nsample"] * case["nsrc"]
    return {"bytes": 4 * n * case["nsample"] + 4.0 * p * (n if case["fields"] else case["nx"]),
            "flops": 4 * 4 * 12 * n * p}


# ----------------------------------------------------------------- exact --

_A8 = (-205.0 / 72.0, 8.0 / 5.0, -1.0 / 5.0, 8.0 / 315.0, -1.0 / 560.0)


class _Wave64:
    """The symmetric sponge scheme in 64 bits over a batch of items."""

    def __init__(self, vel, nx, nz, src, rec, wav, nt):
        self.nx, self.nz, self.nt = nx, nz, nt
        self.rx, self.rz = rec
        v = F.pad(vel.double()[:, None], (NB, NB, NB, NB), mode="replicate")[:, 0]
        self.c = (v * DT) ** 2

        def g1(n):
            k = torch.arange(n, device="cuda", dtype=torch.float64)
            k = torch.minimum(k, n - 1 - k)
            return torch.where(k < NB, torch.exp(-(0.015 * (NB - k)) ** 2), torch.ones_like(k))
        g = g1(nz + 2 * NB)[:, None] * g1(nx + 2 * NB)[None, :]
        self.h, self.g2 = torch.sqrt(g), g * g
        self.src, self.wav = src, wav.astype(np.float64) / (D * D)
        self.B = vel.shape[0]
        self.items = torch.arange(self.B, device="cuda")

    def rest(self):
        z = torch.zeros((self.B, self.nz + 2 * NB, self.nx + 2 * NB), dtype=torch.float64,
                        device="cuda")
        return z, z.clone()

    def step(self, u, up):
        """2nd order in time, 8th in space, before any source term."""
        w = F.pad(self.h * u, (4, 4, 4, 4))
        n, m = u.shape[1], u.shape[2]
        lap = (2 * _A8[0]) * w[:, 4:4 + n, 4:4 + m]
        for k in range(1, 5):
            lap += _A8[k] * (w[:, 4 - k:4 - k + n, 4:4 + m] + w[:, 4 + k:4 + k + n, 4:4 + m] +
                             w[:, 4:4 + n, 4 - k:4 - k + m] + w[:, 4:4 + n, 4 + k:4 + k + m])
        return self.h * (2 * w[:, 4:4 + n, 4:4 + m] + self.c * lap / (D * D)) - self.g2 * up

    def phys(self, u):
        return u[:, NB:NB + self.nz, NB:NB + self.nx]

    def add_source(self, u, n):
        i, (sz, sx) = self.items, self.src
        u[i, sz + NB, sx + NB] += self.c[i, sz + NB, sx + NB] * self.wav[n]

    def record(self, u):
        return u[:, self.rz + NB, self.rx + NB]

    def forward(self, isnap=0, born=None, S=None):
        """Snapshots of the source wavefield (isnap > 0), or the traces; with born =
        (reflectivity, isnap) the field driven by the snapshots S instead."""
        u, up = self.rest()
        kept, traces = [], []
        for n in range(self.nt):
            un = self.step(u, up)
            if born is None:
                self.add_source(un, n)
            elif (n + 1) % born[1] == 0:
                self.phys(un).add_(self.phys(self.c) * born[0] * S[(n + 1) // born[1] - 1])
            u, up = un, u
            if isnap:
                if (n + 1) % isnap == 0:
                    kept.append(self.phys(u).clone())
            else:
                traces.append(self.record(u))
        return kept if isnap else torch.stack(traces, 1)

    def backward(self, data, isnap, S):
        """num and den of the imaging condition, data [B][nt][nrec]."""
        w, wp = self.rest()
        num = torch.zeros((self.B, self.nz, self.nx), dtype=torch.float64, device="cuda")
        den = torch.zeros_like(num)
        cr = self.record(self.c)
        for k in range(self.nt, 0, -1):
            wn = self.step(w, wp)
            wn[:, self.rz + NB, self.rx + NB] += cr * data[:, k - 1]
            w, wp = wn, w
            if k % isnap == 0:
                s = S[k // isnap - 1]
                num += s * self.phys(w)
                den += s * s
        return num, den


def _wave(vel, s, shots):
    dev = dict(device="cuda", dtype=torch.long)
    return _Wave64(vel, s.nx, s.nz, (torch.tensor(s.sz[shots], **dev),
                                     torch.tensor(s.sx[shots], **dev)),
                   (torch.tensor(s.rx, **dev), torch.tensor(s.rz, **dev)), s.wav, s.nt)


def _image64(vel, s, seis, isnap):
    """The filtered stack of all shots over one model."""
    total = torch.zeros((s.nz, s.nx), dtype=torch.float64, device="cuda")
    per = 8.0 * (s.nt // isnap) * s.nx * s.nz
    most = max(1, int(40e9 / max(per, 1.0)))
    for a in range(0, s.nshot, most):
        shots = np.arange(a, min(s.nshot, a + most))
        w = _wave(vel[None].expand(len(shots), -1, -1), s, shots)
        S = w.forward(isnap)
        num, den = w.backward(seis[shots].double(), isnap, S)
        add = 1e-6 * den.flatten(1).max(dim=1).values[:, None, None]
        dd = den + add
        total += torch.where(dd > 0, num / dd.clamp(min=1e-300), torch.zeros_like(num)).sum(0)
    p = F.pad(total[None, None], (1, 1, 1, 1), mode="replicate")[0, 0]
    return -((p[:-2, 1:-1] - 2 * total + p[2:, 1:-1]) + (p[1:-1, :-2] - 2 * total + p[1:-1, 2:])) \
        / (D * D)


def _eikonal64(vel, d, sz, sx):
    """The first-order upwind traveltimes of every (sample, source), by repeated
    sweeps of the whole grid until nothing changes."""
    n, nz, nx = vel.shape
    h = (d / vel.double())[:, None]
    inf = float("inf")
    T = torch.full((n, len(sx), nz, nx), inf, dtype=torch.float64, device="cuda")
    k = torch.arange(len(sx), device="cuda")
    T[:, k, torch.tensor(sz, device="cuda").long(), torch.tensor(sx, device="cuda").long()] = 0.0
    for it in range(1, 20 * (nz + nx)):
        p = F.pad(T, (1, 1, 1, 1), value=inf)
        a = torch.minimum(p[:, :, :-2, 1:-1], p[:, :, 2:, 1:-1])
        b = torch.minimum(p[:, :, 1:-1, :-2], p[:, :, 1:-1, 2:])
        del p
        lo, hi = torch.minimum(a, b), torch.maximum(a, b)
        del a, b
        one = lo + h
        diff = torch.where(one < hi, torch.zeros_like(lo), hi - lo)
        two = 0.5 * (2 * lo + diff + torch.sqrt((2 * h * h - diff * diff).clamp(min=0)))
        new = torch.minimum(T, torch.where(one <= hi, one, two))
        if it % 50 == 0 and torch.equal(new, T):
            return T
        T = new
    return T


def exact(case, seed):
    kind = case["kind"]
    if kind in ("compress", "decompress"):
        return None  # a lossy stream has no 64-bit value; bytes are compared as they are
    if kind in ("model", "migrate", "ensemble", "lsrtm", "serve"):
        points = sum(_points(nx, nz) * ns for nx, nz, ns, _ in _requests(case)) \
            if kind == "serve" else _points(case["nx"], case["nz"]) * case["nshot"] * \
            case.get("nsample", 1)
        passes = {"model": 1, "lsrtm": 2 * (2 * case.get("niter", 0) + 1)}.get(kind, 2)
        parts = case["nreq"] if kind == "serve" else case.get("nsample", 1)
        if passes * case["nt"] * (points * 1.2e-10 + parts * 4e-4) > 18:
            return None
    with torch.no_grad():
        st = prepare(case, seed)
        if kind == "model":
            s = st["survey"]
            return _wave(st["vel"][None].expand(s.nshot, -1, -1), s, np.arange(s.nshot)).forward()
        if kind == "migrate":
            return _image64(st["vel"], st["survey"], st["seis"], case["isnap"])
        if kind == "ensemble":
            return torch.stack([_image64(v, st["survey"], st["seis"], case["isnap"])
                                for v in st["vel"]])
        if kind == "serve":
            return [_image64(vel, s, seis, 4) for _, s, vel, seis, _ in st["reqs"]]
        if kind == "lsrtm":
            return _lsrtm64(st, case)
        if kind == "stats":
            x = st["images"].double().flatten(1)
            n = x.shape[0]
            mean, std = x.mean(0), x.std(0)
            h = (n - 1) * torch.tensor([0.05, 0.95], dtype=torch.float64)
            srt = x.sort(0).values
            q = []
            for v in h.tolist():
                i = int(math.floor(v))
                q.append(srt[i] + (v - i) * (srt[min(i + 1, n - 1)] - srt[i]))
            conf = (std.max() - std) / (std.max() - std.min())
            return dict(mean=mean, std=std, q05=q[0], q95=q[1], confidence=conf, ratio=std / mean)
        T = _eikonal64(st["vel"], 40.0, *st["src"])
        out = {"times": T[:, :, 0, :], "iters": None}
        if case["fields"]:
            out["fields"] = T
        return out


def _lsrtm64(st, case):
    s, isnap = st["survey"], case["isnap"]
    w = _wave(st["vel"][None].expand(s.nshot, -1, -1), s, np.arange(s.nshot))
    S = w.forward(isnap)
    r = st["seis"].double()
    m = torch.zeros((s.nz, s.nx), dtype=torch.float64, device="cuda")
    grad = w.backward(r, isnap, S)[0].sum(0)
    p, gamma, misfit = grad.clone(), (grad * grad).sum(), [float((r * r).sum())]
    for _ in range(case["niter"]):
        q = w.forward(born=(p, isnap), S=S)
        alpha = gamma / (q * q).sum()
        m += alpha * p
        r = r - alpha * q
        misfit.append(float((r * r).sum()))
        grad = w.backward(r, isnap, S)[0].sum(0)
        g2 = (grad * grad).sum()
        p = grad + g2 / gamma * p
        gamma = g2
    return {"refl": m, "misfit": misfit}
