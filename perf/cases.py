"""The projector's workloads as timed cases.

Each case is a call, or the few calls, that a program reconstructing from CT or
PET data makes in its inner loop, on a scene it meets in practice: Gaussians
fitted to a random ellipsoid phantom, measured data of that phantom.

``listed()`` names the cases, ``draw(rng)`` gives others of the same ranges,
``prepare`` makes a case's inputs and handles on the GPU, ``run`` makes one
pass through the public calls, ``work`` counts what the pass cannot do without
and ``exact`` is the same result from plain PyTorch in binary64.
"""
import math

import numpy as np
import torch

from paper_2602_01057_gb300 import rgrt, synth

DEV = "cuda"
SQRT_2PI = math.sqrt(2.0 * math.pi)
CUT = 9.0             # a pair counts within 3 sigma of the line
KAPPA2 = 7.0          # Epanechnikov support
# operations of a kept pair: the closed form (39), its adjoint (97.5), and per
# time-of-flight bin 4 and 8 more
FWD_OPS, ADJ_OPS, TOF_FWD, TOF_ADJ = 39.0, 97.5, 4.0, 8.0
# densest problem (rays x Gaussians) that exact() takes on
EXACT_PAIRS = 6e10
# nominal volume of the phantoms' support (CT units^3, PET mm^3)
SUPPORT = {"ct": 1.3, "pet": 8.5e5}


# ---------------------------------------------------------------------------
# the cases
# ---------------------------------------------------------------------------

def _ct(name, call, kind, n, views, rows, cols, **more):
    return dict(name=name, call=call, kind=kind, n=n, views=views, rows=rows, cols=cols, **more)


def _pet(name, call, n, angles, rows=63, cols=329, **more):
    c = dict(name=name, call=call, kind="pet", n=n, views=angles, rows=rows, cols=cols, scan_angles=288,
             arc_mode=0, tof=0)
    c.update(more)
    return c


def listed():
    return [
        # the smallest optimisation step: launches and latency count
        _ct("ct_parallel_step", "step", "parallel", 1000, 16, 64, 64),
        # a forward projection of compact-support kernels on a wide, ragged
        # detector (simulated data, a residual check)
        _ct("ct_parallel_epan_fwd", "forward", "parallel", 5000, 90, 97, 161, kernel="epanechnikov"),
        # a reconstruction's mini-batch: 8 of a cone-beam scan's views
        _ct("ct_cone_minibatch", "grad", "cone", 50_000, 8, 256, 256),
        # the full cone-beam gradient
        _ct("ct_cone_full", "grad", "cone", 50_000, 180, 256, 256),
        # a ragged scan through autograd, as one layer of a larger model
        _ct("ct_cone_autograd_odd", "autograd", "cone", 12_345, 7, 201, 333),
        # the full PET ring gradient with attenuation and background
        _pet("pet_ring_full", "grad", 200_000, 288, corrections=True),
        # a PET mini-batch on uncorrected (raw) radial positions
        _pet("pet_raw_minibatch", "grad", 100_000, 8, arc_mode=1, corrections=True),
        # one of 12 ordered subsets of a time-of-flight sinogram, 13 bins
        _pet("pet_tof_subset", "grad", 100_000, 24, tof=13),
        # the largest: every LOR of a 32-ring scanner up to ring difference 5
        _pet("pet3d_full", "grad", 200_000, 288, rows=32, kind="pet3d", max_ring_diff=5),
        # helical cone-beam CT: explicit rays, forward and adjoint by hand
        _ct("ct_helical_rays", "pair", "helical", 20_000, 24, 128, 128),
        # the reconstructed volume
        dict(name="voxels", call="voxelize", kind="volume", n=50_000, nx=256, ny=256, nz=256),
        # one step of many small uneven scans together
        dict(name="ct_batch_step", call="batch", kind="cone", n=5000, scans=24, views=40, side=96),
    ]


def _logu(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case of the listed ranges."""
    what = rng.choice(["parallel", "cone", "cone", "pet", "pet", "tof", "pet3d", "rays", "volume", "batch"])
    call = rng.choice(["grad", "forward", "autograd"])
    if what == "parallel":
        return dict(call=rng.choice(["step", "forward"]), kind="parallel", n=_logu(rng, 1000, 20_000),
                    views=_logu(rng, 16, 90), rows=_logu(rng, 64, 160), cols=_logu(rng, 64, 192),
                    kernel=rng.choice(["gaussian", "epanechnikov"]))
    if what == "cone":
        return dict(call=call, kind="cone", n=_logu(rng, 5000, 120_000), views=_logu(rng, 4, 180),
                    rows=_logu(rng, 96, 320), cols=_logu(rng, 96, 384))
    if what == "pet":
        return dict(call=call, kind="pet", n=_logu(rng, 50_000, 300_000), views=_logu(rng, 6, 288), rows=63,
                    cols=2 * rng.randint(130, 164) + 1, scan_angles=288, arc_mode=rng.randint(0, 1), tof=0,
                    corrections=bool(rng.randint(0, 1)))
    if what == "tof":
        return dict(call="grad", kind="pet", n=_logu(rng, 50_000, 200_000), views=_logu(rng, 6, 48),
                    rows=rng.choice([47, 63]), cols=2 * rng.randint(130, 164) + 1, scan_angles=288, arc_mode=0,
                    tof=rng.choice([9, 11, 13]))
    if what == "pet3d":
        return dict(call="grad", kind="pet3d", n=_logu(rng, 50_000, 200_000), views=_logu(rng, 6, 96),
                    rows=rng.randint(24, 32), cols=2 * rng.randint(130, 164) + 1, scan_angles=288, arc_mode=0,
                    tof=0, max_ring_diff=rng.randint(1, 5))
    if what == "rays":
        return dict(call="pair", kind="helical", n=_logu(rng, 5000, 50_000), views=_logu(rng, 8, 48),
                    rows=_logu(rng, 64, 192), cols=_logu(rng, 64, 192))
    if what == "volume":
        return dict(call="voxelize", kind="volume", n=_logu(rng, 5000, 200_000), nx=_logu(rng, 64, 300),
                    ny=_logu(rng, 64, 300), nz=_logu(rng, 64, 300))
    return dict(call="batch", kind="cone", n=_logu(rng, 1500, 8000), scans=rng.randint(8, 40),
                views=_logu(rng, 16, 48), side=rng.choice([64, 96, 128]))


# ---------------------------------------------------------------------------
# scenes
# ---------------------------------------------------------------------------

def _gen(seed):
    return torch.Generator(device=DEV).manual_seed(int(seed))


def _phantom(pet, seed):
    """Random ellipsoids as GPU tensors (axes, rotations, centres, densities)."""
    ph = synth.pet_phantom(seed) if pet else synth.ellipsoid_phantom(12, seed=1000 + seed)
    return {k: torch.from_numpy(np.asarray(v, np.float64)).to(DEV) for k, v in ph.items()}


def _inside(ph, x):
    """[n, k]: the point lies in the ellipsoid."""
    local = torch.einsum("nkj,kji->nki", x[:, None, :] - ph["centre"][None], ph["rot"])
    return ((local / ph["axes"]) ** 2).sum(-1) <= 1.0


def _gaussians(ph, n, seed, scale=1.0):
    """n Gaussians fitted to the phantom: centres distributed as its density,
    sizes around h = (support / n)^(1/3), random orientations, masses that
    match the density."""
    g = _gen(seed)
    vol = 4.0 / 3.0 * math.pi * ph["axes"].prod(1)

    def points(which):
        d = torch.randn(which.numel(), 3, generator=g, device=DEV, dtype=torch.float64)
        d = d / d.norm(dim=1, keepdim=True)
        r = torch.rand(which.numel(), 1, generator=g, device=DEV, dtype=torch.float64) ** (1.0 / 3.0)
        return ph["centre"][which] + torch.einsum("nij,nj->ni", ph["rot"][which], d * r * ph["axes"][which])

    k = vol.numel()
    probe = torch.arange(k, device=DEV).repeat_interleave(2048)
    cover = _inside(ph, points(probe)).sum(1).clamp(min=1).double()
    support = float((vol * (1.0 / cover).reshape(k, -1).mean(1)).sum())
    h = (support / n) ** (1.0 / 3.0)
    which = torch.multinomial(ph["density"] * vol, n, replacement=True, generator=g)
    mu = points(which)
    ls = math.log(h) + 0.3 * torch.randn(n, 3, generator=g, device=DEV, dtype=torch.float64)
    q = torch.randn(n, 4, generator=g, device=DEV, dtype=torch.float64)
    q = q / q.norm(dim=1, keepdim=True)
    dens = (_inside(ph, mu).double() * ph["density"]).sum(1)
    rho = scale * dens * h ** 3 / ((2.0 * math.pi) ** 1.5 * ls.sum(1).exp())
    return {k: v.float().contiguous() for k, v in dict(mu=mu, ls=ls, q=q, rho=rho).items()}


def _desc(c):
    """The geometry description the library takes."""
    V, H, W = c["views"], c["rows"], c["cols"]
    if c["kind"] == "parallel":
        return synth.geom_parallel(V, H, W, 2.0 / W, 2.0 / W, -2.0, 2.0)
    if c["kind"] == "cone":
        pitch = 1.5 * 256.0 / max(H, W) / synth.CT_MM_PER_UNIT
        return synth.geom_cone(V, H, W, pitch, pitch, 7.8125, 11.71875)
    # PET: every (288 / views)-th angle, an ordered subset
    ang = math.pi * np.floor(np.arange(V) * c["scan_angles"] / V) / c["scan_angles"]
    if c["kind"] == "pet3d":
        d = synth.geom_pet3d(V, W, H, 400.0, 576, 4.0, c["max_ring_diff"], c["arc_mode"])
    else:
        d = synth.geom_pet(V, W, H, 400.0, 576, 2.0, c["arc_mode"])
        if c["tof"]:
            d = synth.with_tof_bins(d, c["tof"], 47.0 * 13 / c["tof"], 31.85)
    return dict(d, angles=ang)


def _view_rays(c, d, v):
    """(o, d, ta, tb) in binary64 of view v, rows x cols rays each (3-D PET:
    view = (ring difference, angle); rows without a ring pair are NaN)."""
    H, W = c["rows"], c["cols"]
    f64 = dict(device=DEV, dtype=torch.float64)
    i = torch.arange(W, **f64) - 0.5 * (W - 1)
    j = torch.arange(H, **f64) - 0.5 * (H - 1)
    ez = torch.tensor([0.0, 0.0, 1.0], **f64)
    a = float(d["angles"][v % c["views"]])
    ca, sa = math.cos(a), math.sin(a)
    if c["kind"] in ("parallel", "cone", "helical"):
        ew, eu = torch.tensor([ca, sa, 0.0], **f64), torch.tensor([-sa, ca, 0.0], **f64)
        u, w = i * d["pitch_u"], j * d["pitch_v"]
        grid = u[None, :, None] * eu + w[:, None, None] * ez
        if c["kind"] == "parallel":
            o = grid
            return (o.reshape(-1, 3), ew.expand(H * W, 3), torch.full((H * W,), d["t_a"], **f64),
                    torch.full((H * W,), d["t_b"], **f64))
        s = -d["dso"] * ew + float(d["z"][v] if "z" in d else 0.0) * ez
        dv = (d["dsd"] * ew + grid).reshape(-1, 3)
        L = dv.norm(dim=1)
        return s.expand(H * W, 3), dv / L[:, None], torch.zeros_like(L), L
    eu, ew = torch.tensor([ca, sa, 0.0], **f64), torch.tensor([sa, -ca, 0.0], **f64)
    R = d["radius"]
    s = i * math.pi * R / d["n_crystals"] if d["arc_mode"] == 0 else R * torch.sin(i * math.pi / d["n_crystals"])
    h = (R * R - s * s).sqrt()
    delta = v // c["views"] - c["max_ring_diff"] if c["kind"] == "pet3d" else 0
    z1, z2 = j.clone() * d["pitch_v"], j.clone() * d["pitch_v"]
    if delta >= 0:
        z2 = z2 + delta * d["pitch_v"]
    else:
        z1 = z1 - delta * d["pitch_v"]
    if delta:
        z1[H - abs(delta):] = math.nan
    p1 = s[None, :, None] * eu - h[None, :, None] * ew + z1[:, None, None] * ez
    p2 = s[None, :, None] * eu + h[None, :, None] * ew + z2[:, None, None] * ez
    dv = (p2 - p1).reshape(-1, 3)
    L = dv.norm(dim=1)
    return (0.5 * (p1 + p2)).reshape(-1, 3), dv / L[:, None], -0.5 * L, 0.5 * L


def _n_views(c):
    return c["views"] * (2 * c.get("max_ring_diff", 0) + 1)


def _place(c, values):
    """Per-view values [views][bins x rows x cols] in the library's layout."""
    x = torch.stack(values)
    V, H, W, B = x.shape[0], c["rows"], c["cols"], max(1, c.get("tof", 0))
    x = x.reshape(V, B, H, W)
    return (x.permute(1, 2, 0, 3) if c["kind"] == "pet" else x).reshape(-1)


def _chords(c, d, ph, v):
    """Line integrals of the phantom along view v's rays."""
    o, dr, ta, tb = _view_rays(c, d, v)
    p = torch.einsum("nkj,kji->nki", o[:, None] - ph["centre"][None], ph["rot"]) / ph["axes"]
    e = torch.einsum("nj,kji->nki", dr, ph["rot"]) / ph["axes"]
    A, B, C = (e * e).sum(-1), (p * e).sum(-1), (p * p).sum(-1) - 1.0
    sq = (B * B - A * C).clamp(min=0).sqrt()
    out = ((2.0 * sq / A) * ph["density"]).sum(1).nan_to_num(0.0)
    if not c.get("tof"):
        return out
    # time of flight: the activity spread over the bins around the object
    k = torch.arange(c["tof"], device=DEV, dtype=torch.float64) - 0.5 * (c["tof"] - 1)
    w = torch.exp(-0.5 * (k * d["tof_spacing"] / 90.0) ** 2)
    return (w / (w.sum() * d["tof_spacing"]))[:, None] * out[None]


def _scan(c, seed):
    """Inputs of one scan: geometry description, Gaussians, measured data."""
    pet = c["kind"] in ("pet", "pet3d")
    ph = _phantom(pet, seed)
    g = _gen(seed + 17)
    if c["kind"] == "helical":
        pitch = 1.5 * 256.0 / max(c["rows"], c["cols"]) / synth.CT_MM_PER_UNIT
        th = 2.0 * math.pi * np.arange(c["views"]) / c["views"]
        z = th / (2.0 * math.pi)
        d = dict(kind="helical", angles=th, z=z - 0.5 * (z[0] + z[-1]), pitch_u=pitch, pitch_v=pitch, dso=7.8125,
                 dsd=11.71875)
    else:
        d = _desc(c)
    G = _gaussians(ph, c["n"], seed + 5)
    out = dict(desc=d, G=G, seed=seed)
    if c["call"] in ("forward",):
        return out
    if c["call"] in ("autograd", "pair"):
        R = _n_views(c) * c["rows"] * c["cols"] * max(1, c.get("tof", 0))
        out["w"] = torch.randn(R, generator=g, device=DEV)
        return out
    y = _place(c, [_chords(c, d, ph, v) for v in range(_n_views(c))])
    hp = dict(kappa=1.0, poisson_eps=1e-9)
    if pet:
        kappa = 15.0 * _n_views(c) * c["rows"] * c["cols"] / max(float(y.sum()), 1e-30)
        mean = kappa * y
        hp = dict(kappa=kappa, poisson_eps=0.5 if not c["tof"] else 0.05)
        if c.get("corrections"):
            out["mult"] = (0.2 + 0.8 * torch.rand(y.numel(), generator=g, device=DEV))
            out["add"] = (1.0 + torch.rand(y.numel(), generator=g, device=DEV))
            mean = mean * out["mult"] + out["add"]
        y = torch.poisson((mean + hp["poisson_eps"]).float(), generator=g)
    else:
        y = y.float() * (1.0 + 0.01 * torch.randn(y.numel(), generator=g, device=DEV))
    out.update(y=y.contiguous(), hp=hp, loss=rgrt.RGRT_LOSS_POISSON if pet else rgrt.RGRT_LOSS_L2)
    return out


# learning rates late in a schedule (the defaults divided by 100)
_LATE = dict(lr_mu=2e-6, lr_logscale=5e-5, lr_quat=1e-5, lr_rho=2e-5)


def _batch_scans(c, seed):
    """Uneven scans around the case's size (the sizes follow the case alone)."""
    r = np.random.default_rng(c["scans"])
    out = []
    for k in range(c["scans"]):
        n = int(c["n"] * math.exp(r.uniform(-1.0, 1.0)))
        s = dict(call="batch", kind="cone", n=n, views=max(4, int(c["views"] * r.uniform(0.6, 1.4))),
                 rows=c["side"], cols=c["side"])
        out.append((s, _scan(s, seed + 100 * k)))
    return out


def _grid(c):
    dims = (c["nx"], c["ny"], c["nz"])
    size = tuple(2.0 / n for n in dims)
    return dict(origin=tuple(-1.0 + 0.5 * s for s in size), size=size, dims=dims)


# ---------------------------------------------------------------------------
# one pass
# ---------------------------------------------------------------------------

def _empty_like(G):
    return [torch.empty_like(G[k]) for k in ("mu", "ls", "q", "rho")]


def prepare(case, seed):
    ctx = rgrt.Context(0)
    if case["call"] == "batch":
        scans = _batch_scans(case, seed)
        gs = [rgrt.Gaussians(ctx, *(s["G"][k] for k in ("mu", "ls", "q", "rho"))) for _, s in scans]
        geoms = [rgrt.Geometry(ctx, s["desc"]) for _, s in scans]
        return dict(case=case, ctx=ctx, gs=gs, geoms=geoms, batch=rgrt.Batch(ctx, gs, geoms),
                    ys=[s["y"] for _, s in scans], hp=rgrt.adam_params(**_LATE), t=0,
                    out=[_empty_like(s["G"]) for _, s in scans])
    if case["call"] == "voxelize":
        G = _gaussians(_phantom(False, seed), case["n"], seed + 5)
        gs = rgrt.Gaussians(ctx, *(G[k] for k in ("mu", "ls", "q", "rho")))
        return dict(case=case, ctx=ctx, gs=gs, vol=_grid(case),
                    out=torch.empty((case["nz"], case["ny"], case["nx"]), device=DEV))
    s = _scan(case, seed)
    G = s["G"]
    if case["kind"] == "helical":
        rays = [_view_rays(case, s["desc"], v) for v in range(case["views"])]
        o, d, ta, tb = (torch.cat([r[k] for r in rays]) for k in range(4))
        geom = rgrt.Geometry(ctx, dict(kind="rays", o=o.float().contiguous(), d=d.float().contiguous(),
                                       t=torch.stack([ta, tb], 1).float().contiguous()))
    else:
        geom = rgrt.Geometry(ctx, s["desc"])
    if "mult" in s:
        geom.set_corrections(s["mult"], s["add"])
    st = dict(case=case, ctx=ctx, geom=geom, scan=s, grads=_empty_like(G), loss=torch.zeros(1, device=DEV), t=0)
    if case["call"] == "autograd":
        st["leaves"] = [G[k].requires_grad_() for k in ("mu", "ls", "q", "rho")]
        return st
    st["gs"] = rgrt.Gaussians(ctx, *(G[k] for k in ("mu", "ls", "q", "rho")))
    if case.get("kernel", "gaussian") != "gaussian":
        st["gs"].set_kernel(case["kernel"])
    st["I"] = torch.empty(geom.n_rays, device=DEV)
    st["hp"] = rgrt.adam_params(**s.get("hp", {}), **_LATE)
    return st


def run(state):
    call, ctx = state["case"]["call"], state["ctx"]
    if call == "batch":
        state["t"] += 1
        losses = state["batch"].loss_step(state["ys"], rgrt.RGRT_LOSS_L2, state["hp"], state["t"])
        for g, o in zip(state["gs"], state["out"]):
            g.get(*o)
        cat = [torch.cat([o[k].reshape(-1) for o in state["out"]]) for k in range(4)]
        return dict(losses=losses, mu=cat[0], ls=cat[1], q=cat[2], rho=cat[3])
    if call == "voxelize":
        return rgrt.gaussians_voxelize(ctx, state["gs"], state["vol"], state["out"])
    geom, s = state["geom"], state["scan"]
    if call == "forward":
        return rgrt.project_forward(ctx, state["gs"], geom, state["I"])
    if call == "autograd":
        for p in state["leaves"]:
            p.grad = None
        I = rgrt.gaussian_project(*state["leaves"], geom)
        I.backward(s["w"])
        return dict(I=I.detach(), grads=[p.grad for p in state["leaves"]])
    if call == "pair":
        rgrt.project_forward(ctx, state["gs"], geom, state["I"])
        rgrt.project_backward(ctx, state["gs"], geom, s["w"], *state["grads"])
        return dict(I=state["I"], grads=state["grads"])
    if call == "step":
        state["t"] += 1
        rgrt.loss_step(ctx, state["gs"], geom, s["y"], s["loss"], state["hp"], state["t"], state["loss"])
        state["gs"].get(*state["grads"])
        return dict(loss=state["loss"], params=state["grads"])
    rgrt.loss_grad(ctx, state["gs"], geom, s["y"], s["loss"], state["hp"], state["loss"], *state["grads"])
    return dict(loss=state["loss"], grads=state["grads"])


# ---------------------------------------------------------------------------
# the work of one pass
# ---------------------------------------------------------------------------

def _pairs(c):
    """Expected kept pairs: the 3-sigma footprint of an average Gaussian."""
    n = c["n"]
    if c["call"] == "batch":
        V, H, W = c["scans"] * c["views"], c["side"], c["side"]
    else:
        V, H, W = _n_views(c), c["rows"], c["cols"]
    if c["kind"] in ("pet", "pet3d"):
        h2 = (SUPPORT["pet"] / n) ** (2.0 / 3.0)
        if c["kind"] == "pet3d":
            V = V * (H - 0.5 * c["max_ring_diff"]) * 4.0 / 128.0
        return 9.0 * math.pi * h2 * 1.1 * V * n / (2.18 * (4.0 if c["kind"] == "pet3d" else 2.0))
    h2 = (SUPPORT["ct"] / n) ** (2.0 / 3.0)
    pitch = 2.0 / W if c["kind"] == "parallel" else 2.0 / max(H, W)   # at the object
    cut = KAPPA2 if c.get("kernel") == "epanechnikov" else CUT
    return min(1.0, H / W) * cut * math.pi * h2 * 1.1 * V * n / pitch ** 2


def work(case):
    c = case
    if c["call"] == "voxelize":
        nv = c["nx"] * c["ny"] * c["nz"]
        pairs = 36.0 * math.pi * SUPPORT["ct"] * 1.15 * nv / 8.0      # 4/3 pi 27 h^3 n = 36 pi support
        return {"bytes": 44.0 * c["n"] + 4.0 * nv, "flops": 14.0 * pairs}
    pairs, bins = _pairs(c), max(0, c.get("tof", 0))
    fwd, adj = pairs * (FWD_OPS + TOF_FWD * bins), pairs * (ADJ_OPS + TOF_ADJ * bins)
    if c["call"] == "batch":
        n, R = c["n"] * c["scans"], c["scans"] * c["views"] * c["side"] ** 2
    else:
        n, R = c["n"], _n_views(c) * c["rows"] * c["cols"] * max(1, bins)
    rays = 32.0 * R if c["kind"] == "helical" else 0.0
    if c["call"] == "forward":
        return {"bytes": 44.0 * n + 4.0 * R, "flops": fwd}
    if c["call"] in ("autograd", "pair"):       # projections out, weights in, gradients out
        return {"bytes": 88.0 * n + 8.0 * R + rays, "flops": fwd + adj}
    if c["call"] in ("step", "batch"):          # data in; parameters and two moments read and written
        return {"bytes": 6 * 44.0 * n + 4.0 * R, "flops": fwd + adj}
    return {"bytes": 88.0 * n + 4.0 * R * (3 if c.get("corrections") else 1), "flops": fwd + adj}


# ---------------------------------------------------------------------------
# the same results in binary64
# ---------------------------------------------------------------------------

_SYM = ((0, 0), (0, 1), (0, 2), (1, 1), (1, 2), (2, 2))


def _precision(ls, q):
    """P = R diag(exp(-2 l)) R^T, packed (00, 01, 02, 11, 12, 22)."""
    w, x, y, z = (q / q.norm(dim=1, keepdim=True)).unbind(1)
    R = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y - w * z), 2 * (x * z + w * y),
                     2 * (x * y + w * z), 1 - 2 * (x * x + z * z), 2 * (y * z - w * x),
                     2 * (x * z - w * y), 2 * (y * z + w * x), 1 - 2 * (x * x + y * y)], 1).reshape(-1, 3, 3)
    P = torch.einsum("nik,nk,njk->nij", R, torch.exp(-2.0 * ls), R)
    return torch.stack([P[:, a, b] for a, b in _SYM], 1)


def _mul(P, x):
    """P x for packed symmetric P."""
    return torch.stack([P[:, 0] * x[:, 0] + P[:, 1] * x[:, 1] + P[:, 2] * x[:, 2],
                        P[:, 1] * x[:, 0] + P[:, 3] * x[:, 1] + P[:, 4] * x[:, 2],
                        P[:, 2] * x[:, 0] + P[:, 4] * x[:, 1] + P[:, 5] * x[:, 2]], 1)


def _sym(a, b):
    """Weights w with sum_e w_e P_e = a^T P b."""
    return torch.stack([a[:, i] * b[:, j] + (a[:, j] * b[:, i] if i != j else 0.0) for i, j in _SYM], 1)


def _kept(o, d, mu, P, cut):
    """(ray, Gaussian) indices of the pairs with m <= cut."""
    Pm = _mul(P, mu)
    mPm = (mu * Pm).sum(1)
    A = _sym(d, d) @ P.T
    m = torch.cat([_sym(d, o), -d], 1) @ torch.cat([P, Pm], 1).T
    m = m.square_().div_(A).neg_()
    del A
    m += torch.cat([_sym(o, o), -2.0 * o], 1) @ torch.cat([P, Pm], 1).T
    m += mPm[None]
    return torch.nonzero(m <= cut, as_tuple=True)


def _values(o, d, ta, tb, mu, P, rho, tof, epan):
    """Line integrals of the pairs (rows match); [bins, pairs] with time of flight."""
    e = o - mu
    Pd = _mul(P, d)
    A, B, C = (d * Pd).sum(1), (e * Pd).sum(1), (e * _mul(P, e)).sum(1)
    if epan:
        c = 1.0 - (C - B * B / A) / KAPPA2
        a = (KAPPA2 * c.clamp(min=0) / A).sqrt()
        s0, s1 = torch.maximum(ta + B / A, -a), torch.minimum(tb + B / A, a)
        s1 = torch.maximum(s0, s1)
        F = lambda s: s * (c - A * s * s / (3.0 * KAPPA2))  # noqa: E731
        return (rho * (F(s1) - F(s0)))[None]
    out = []
    for tc, sg in (tof or [(0.0, math.inf)]):
        tau = 0.0 if math.isinf(sg) else 1.0 / (sg * sg)
        A1, B1, C1 = A + tau, B - tau * tc, C + tau * tc * tc
        f = rho * torch.sqrt(math.pi / (2.0 * A1)) * torch.exp(-0.5 * (C1 - B1 * B1 / A1))
        w = torch.rsqrt(2.0 * A1)
        f = f * (torch.erf((A1 * tb + B1) * w) - torch.erf((A1 * ta + B1) * w))
        out.append(f * (math.sqrt(tau) / SQRT_2PI if tau else 1.0))
    return torch.stack(out)


def _project(c, s, want_I, grad_of):
    """Projections and, when grad_of(view, I) gives (loss, dL/dI), the loss and
    the parameter gradients."""
    d = s["desc"]
    G = {k: v.detach().double() for k, v in s["G"].items()}
    ls, q = G["ls"].requires_grad_(), G["q"].requires_grad_()
    P = _precision(ls, q)
    Pd, mu, rho = (x.detach().clone().requires_grad_() for x in (P, G["mu"], G["rho"]))
    epan = c.get("kernel") == "epanechnikov"
    tof = None
    if c.get("tof"):
        tof = [((k - 0.5 * (c["tof"] - 1)) * d["tof_spacing"], d["tof_sigma"]) for k in range(c["tof"])]
    bins = max(1, c.get("tof", 0))
    step = max(64, int(6e7 // c["n"]))
    Is, loss = [], 0.0
    for v in range(_n_views(c)):
        o, dr, ta, tb = _view_rays(c, d, v)
        if c["kind"] == "helical":      # the rays are handed over in binary32
            o, ta, tb = (x.float().double() for x in (o, ta, tb))
            dr = dr.float().double()
            dr = dr / dr.norm(dim=1, keepdim=True)
        shift = (o * dr).sum(1)         # from the point nearest the origin
        o, ta, tb = o - shift[:, None] * dr, ta + shift, tb + shift
        Iv = torch.zeros(bins, o.shape[0], device=DEV, dtype=torch.float64)
        for r0 in range(0, o.shape[0], step):
            sl = slice(r0, min(o.shape[0], r0 + step))
            rows, live = torch.arange(sl.start, sl.stop, device=DEV), ~torch.isnan(o[sl, 2])
            rows = rows[live]
            if rows.numel() == 0:
                continue
            ri, gi = _kept(o[rows], dr[rows], mu.detach(), Pd.detach(), KAPPA2 if epan else CUT)
            ri = rows[ri]
            with torch.set_grad_enabled(grad_of is not None):
                if tof:     # bin centres count from the chord's midpoint
                    off = shift[ri]
                    val = _values(o[ri] + off[:, None] * dr[ri], dr[ri], ta[ri] - off, tb[ri] - off, mu[gi], Pd[gi],
                                  rho[gi], tof, epan)
                else:
                    val = _values(o[ri], dr[ri], ta[ri], tb[ri], mu[gi], Pd[gi], rho[gi], None, epan)
                Iv.index_add_(1, ri, val.detach())
                if grad_of is not None:
                    lo, w = grad_of(v, Iv, rows)
                    loss += lo
                    (val * w[:, ri]).sum().backward()
            del val
        Is.append(Iv.reshape(-1))
    I = _place(c, Is) if want_I else None
    if grad_of is None:
        return I, None, None
    P.backward(Pd.grad)
    return I, loss, [mu.grad, ls.grad, q.grad, rho.grad]


def _per_view(c, x):
    """The library's layout back to [views][bins, rows x cols]."""
    V, H, W, B = _n_views(c), c["rows"], c["cols"], max(1, c.get("tof", 0))
    if c["kind"] == "pet":
        x = x.reshape(B, H, V, W).permute(2, 0, 1, 3)
    return x.reshape(V, B, H * W).double()


def _loss_of(c, s):
    y = _per_view(c, s["y"])
    mult = _per_view(c, s["mult"]) if "mult" in s else None
    add = _per_view(c, s["add"]) if "add" in s else None
    hp, poisson = s["hp"], s["loss"] == rgrt.RGRT_LOSS_POISSON
    kappa, eps = np.float32(hp["kappa"]).item(), np.float32(hp["poisson_eps"]).item()

    def f(v, I, rows):
        w = torch.zeros_like(I)
        m = mult[v][:, rows] if mult is not None else 1.0
        b = add[v][:, rows] if add is not None else 0.0
        x, yy = m * I[:, rows], y[v][:, rows]
        if poisson:
            lam = kappa * x + eps + b
            w[:, rows] = kappa * m * (1.0 - yy / lam)
            return float((lam - yy * lam.log()).sum()), w
        w[:, rows] = m * (x + b - yy)
        return float(0.5 * (x + b - yy).square().sum()), w

    return f


def _dead_rows_loss(c, s):
    """3-D PET rows without a ring pair: projections of 0 that the loss counts."""
    if c["kind"] != "pet3d" or s["loss"] != rgrt.RGRT_LOSS_POISSON:
        return 0.0
    y, eps, tot = _per_view(c, s["y"]), np.float32(s["hp"]["poisson_eps"]).item(), 0.0
    for v in range(_n_views(c)):
        k = abs(v // c["views"] - c["max_ring_diff"])
        if k:
            tail = y[v].reshape(c["rows"], c["cols"])[c["rows"] - k:]
            tot += float((eps - tail * math.log(eps)).sum())
    return tot


def _adam_first(p, g, lr):
    """The first Adam step from zero moments."""
    g = g.float().double()
    return p.double() - lr * g / (g.abs() + 1e-8)


def _exact_step(c, s):
    _, loss, grads = _project(c, s, False, _loss_of(c, s))
    lrs = [np.float32(_LATE[k]).item() for k in ("lr_mu", "lr_logscale", "lr_quat", "lr_rho")]
    return loss, [_adam_first(s["G"][k], g, lr) for k, g, lr in zip(("mu", "ls", "q", "rho"), grads, lrs)]


def _exact_volume(c, seed):
    G = _gaussians(_phantom(False, seed), c["n"], seed + 5)
    G = {k: v.double() for k, v in G.items()}
    P, vol = _precision(G["ls"], G["q"]), _grid(c)
    ax = [np.float32(vol["origin"][a]).item() + np.float32(vol["size"][a]).item() *
          torch.arange(vol["dims"][a], device=DEV, dtype=torch.float64) for a in range(3)]
    out = torch.zeros(c["nz"], c["ny"], c["nx"], device=DEV, dtype=torch.float64)
    reach = 3.01 * torch.exp(G["ls"].max(1).values)
    for k in range(c["nz"]):
        for j0 in range(0, c["ny"], 32):
            yy = ax[1][j0:j0 + 32]
            near = torch.nonzero(((G["mu"][:, 2] - ax[2][k]).abs() <= reach) & (G["mu"][:, 1] >= yy[0] - reach) &
                                 (G["mu"][:, 1] <= yy[-1] + reach)).reshape(-1)
            if near.numel() == 0:
                continue
            x = torch.stack([ax[0].repeat(yy.numel()), yy.repeat_interleave(c["nx"]),
                             ax[2][k].expand(yy.numel() * c["nx"])], 1)
            Pn, mn = P[near], G["mu"][near]
            Pm = _mul(Pn, mn)
            m = torch.cat([_sym(x, x), -2.0 * x], 1) @ torch.cat([Pn, Pm], 1).T + (mn * Pm).sum(1)
            f = torch.where(m <= CUT, torch.exp(-0.5 * m), torch.zeros_like(m))
            out[k, j0:j0 + 32] = (f @ G["rho"][near]).reshape(yy.numel(), c["nx"])
    return out


def exact(case, seed):
    c = case
    if c["call"] == "voxelize":
        return _exact_volume(c, seed) if c["n"] * float(c["nx"] * c["ny"] * c["nz"]) < 1e12 else None
    if c["call"] == "batch":
        if c["scans"] * c["views"] * c["side"] ** 2 * c["n"] > EXACT_PAIRS:
            return None
        losses, params = [], []
        for sc, s in _batch_scans(c, seed):
            loss, p = _exact_step(sc, s)
            losses.append(loss)
            params.append(p)
        cat = [torch.cat([p[k].reshape(-1) for p in params]) for k in range(4)]
        return dict(losses=np.array(losses), mu=cat[0], ls=cat[1], q=cat[2], rho=cat[3])
    if float(_n_views(c)) * c["rows"] * c["cols"] * c["n"] > EXACT_PAIRS:
        return None
    s = _scan(c, seed)
    if c["call"] == "forward":
        return _project(c, s, True, None)[0]
    if c["call"] in ("autograd", "pair"):
        w = _per_view(c, s["w"])
        I, _, g = _project(c, s, True, lambda v, I, rows: (0.0, w[v]))
        return dict(I=I, grads=g)
    if c["call"] == "step":
        if c.get("kernel", "gaussian") != "gaussian":
            return None
        loss, p = _exact_step(c, s)
        return dict(loss=torch.tensor([loss], dtype=torch.float64), params=p)
    _, loss, g = _project(c, s, False, _loss_of(c, s))
    return dict(loss=torch.tensor([loss + _dead_rows_loss(c, s)], dtype=torch.float64), grads=g)
