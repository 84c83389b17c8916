"""Adjoint of the parallel-ray geometries (Gaussian by Gaussian, adjoint.cu)
against the FP64 oracle at the sizes where its work split changes: partial
warps, one Gaussian, detectors narrower than a column pair, bands of a
rectangle larger than the staging buffer (rows, and columns past 512), one
Gaussian far larger than its neighbours, lanes per Gaussian from 2 to 16, and
the spatial order's one-CTA and several-CTA forms.

Tolerance 1e-4 relative L2 of the oracle's bracket, as the other gradients.
"""
import math

import numpy as np
import pytest

from paper_2602_01057_gb300 import synth

pytestmark = pytest.mark.gpu

GRAD_TOL = 1e-4


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_01057_gb300 import build, rgrt
    build.build()
    ctx = rgrt.Context(0)
    yield torch, rgrt, ctx
    ctx.close()


def _parallel(V, H, W, pitch):
    return synth.geom_parallel(V, H, W, pitch, pitch, -4.0, 4.0)


def _mixed():
    """Small Gaussians and one that covers the detector."""
    G = synth.gaussians_uniform(200, 33, half_box=0.9, log_sigma=math.log(0.02))
    G["ls"][77] = math.log(0.4)
    G["mu"][77] = 0.0
    return G


CASES = {
    "one": lambda: (synth.gaussians_uniform(1, 31, half_box=0.1, log_sigma=math.log(0.1)), _parallel(3, 16, 16, 0.05)),
    "partial_warp": lambda: (synth.gaussians_uniform(133, 32, log_sigma=math.log(0.06)), _parallel(3, 31, 45, 0.05)),
    "narrow": lambda: (synth.gaussians_uniform(65, 34, half_box=0.1, log_sigma=math.log(0.05)), _parallel(2, 40, 1, 0.05)),
    "rows_banded": lambda: (synth.gaussians_uniform(40, 35, log_sigma=math.log(0.01)), _parallel(2, 300, 130, 0.008)),
    "columns_banded": lambda: (synth.gaussians_uniform(40, 36, log_sigma=math.log(0.02)), _parallel(2, 9, 700, 0.004)),
    "outlier": lambda: (_mixed(), _parallel(3, 96, 96, 0.02)),
    "wide_8_lanes": lambda: (synth.gaussians_uniform(24, 37, half_box=0.3, log_sigma=math.log(0.1)), _parallel(2, 128, 128, 0.008)),
    "wide_16_lanes": lambda: (synth.gaussians_uniform(9, 38, half_box=0.2, log_sigma=math.log(0.2)), _parallel(1, 256, 256, 0.006)),
    "many": lambda: (synth.gaussians_uniform(17_001, 39, log_sigma=math.log(0.03)), _parallel(1, 40, 40, 0.05)),
    "ring_raw": lambda: (dict(synth.gaussians_uniform(300, 40, half_box=100.0, log_sigma=math.log(4.0))),
                         synth.geom_pet(7, 129, 21, 200.0, 288, 9.0, arc_mode=1)),
    "ring_tof_banded": lambda: (dict(synth.gaussians_uniform(60, 41, half_box=120.0, log_sigma=math.log(3.0))),
                                synth.with_tof_bins(synth.geom_pet(3, 281, 9, 400.0, 576, 20.0), 16, 40.0, 30.0)),
}


@pytest.mark.parametrize("kernel", ["gaussian", "epanechnikov"])
@pytest.mark.parametrize("name", list(CASES))
def test_parallel_adjoint_matches_oracle(env, oracle, name, kernel):
    torch, rg, ctx = env
    G, gd = CASES[name]()
    if kernel == "epanechnikov" and gd.get("n_tof"):
        pytest.skip("time of flight takes the Gaussian kernel")
    geom = rg.Geometry(ctx, gd)
    gs = rg.Gaussians(ctx, *[torch.from_numpy(np.ascontiguousarray(G[k])).cuda() for k in ("mu", "ls", "q", "rho")])
    gs.set_kernel(kernel)
    w = synth.random_weights(geom.n_rays, 5)
    n = gs.n
    outs = [torch.empty(s, device="cuda") for s in ((n, 3), (n, 3), (n, 4), (n,))]
    rg.project_backward(ctx, gs, geom, torch.from_numpy(w).cuda(), *outs)
    ref = oracle.backward(gd, dict(G, kernel=kernel), w)
    for key, o in zip(("mu", "ls", "q", "rho"), outs):
        got = o.cpu().numpy().astype(np.float64)
        clip = np.clip(got, ref["lo"][key], ref["hi"][key])
        e = np.linalg.norm(got - clip) / max(np.linalg.norm(ref[key]), 1e-30)
        assert e < GRAD_TOL, f"{key}: {e:.2e}"


def _tof():
    return synth.with_tof_bins(synth.geom_pet(2, 65, 5, 400.0, 288, 20.0), 5, 40.0, 30.0)


# one Gaussian well inside the field of view: (half-axis, geometry)
MASKED = {
    "parallel": lambda: (0.12, _parallel(2, 48, 48, 0.03)),
    "cone": lambda: (0.12, synth.geom_cone(2, 48, 48, 0.06, 0.06, 3.0, 6.0)),
    "ring": lambda: (20.0, synth.geom_pet(2, 65, 21, 400.0, 288, 9.0)),
    "ring_tof": lambda: (20.0, _tof()),
    "pet3d": lambda: (20.0, synth.geom_pet3d(2, 65, 9, 400.0, 288, 9.0, 2)),
}


@pytest.mark.parametrize("bad", [math.nan, math.inf])
@pytest.mark.parametrize("name", list(MASKED))
def test_non_finite_weight_outside_the_cut_adds_nothing(env, name, bad):
    """A NaN or infinite dL/dI where the Gaussian contributes nothing leaves its
    gradient as a zero there does.  Tolerance: both sum the same terms, up to
    the order of a few atomic additions in binary32."""
    torch, rg, ctx = env
    s, gd = MASKED[name]()
    geom = rg.Geometry(ctx, gd)
    f = dict(dtype=torch.float32, device="cuda")
    gs = rg.Gaussians(ctx, torch.tensor([[0.4 * s, -0.3 * s, 0.2 * s]], **f),
                      torch.log(torch.tensor([[s, 0.5 * s, 0.7 * s]], **f)),
                      torch.tensor([[0.9, 0.1, -0.3, 0.2]], **f), torch.tensor([1.0], **f))
    img = rg.project_forward(ctx, gs, geom, torch.empty(geom.n_rays, device="cuda"))
    empty = img.reshape(-1) == 0.0
    assert 0 < int(empty.sum()) < empty.numel()
    w = torch.from_numpy(synth.random_weights(geom.n_rays, 6)).cuda().reshape(-1)
    res = []
    for fill in (0.0, bad):
        outs = [torch.empty(sh, device="cuda") for sh in ((1, 3), (1, 3), (1, 4), (1,))]
        rg.project_backward(ctx, gs, geom, torch.where(empty, torch.full_like(w, fill), w), *outs)
        res.append(torch.cat([o.reshape(-1) for o in outs]).double().cpu())
    assert torch.linalg.norm(res[1] - res[0]) <= 1e-5 * torch.linalg.norm(res[0])


def _sizes(n, seed, ls, box=0.9, large=()):
    """n Gaussians, the first of them of other log-sizes: (count, log-size), ..."""
    G = synth.gaussians_uniform(n, seed, half_box=box, log_sigma=ls)
    at = 0
    for count, x in large:
        G["ls"][at:at + count] = x
        at += count
    p = np.random.default_rng(seed).permutation(n)
    return {k: v[p] for k, v in G.items()}


def _ring(V, W, H, bins=0, arc_mode=0):
    gd = synth.geom_pet(V, W, H, 400.0, 576, 9.0, arc_mode=arc_mode)
    return synth.with_tof_bins(gd, bins, 40.0, 30.0) if bins else gd


L = math.log
# sets large enough to be staged; in parts of 8,000 (view, Gaussian) pairs they are not
STAGED = {
    "rows_banded": lambda: (_sizes(40_000, 51, L(0.01)), _parallel(1, 300, 130, 0.008)),
    "columns_banded": lambda: (_sizes(40_000, 52, L(0.01)), _parallel(1, 9, 700, 0.004)),
    "one_column": lambda: (_sizes(40_000, 53, L(0.01)), _parallel(1, 300, 1, 0.008)),
    "views": lambda: (_sizes(12_000, 54, L(0.02)), _parallel(4, 61, 47, 0.03)),
    "outliers": lambda: (_sizes(40_000, 55, L(0.01), large=((20, L(0.08)), (5, L(0.3)))), _parallel(1, 200, 211, 0.01)),
    "ends": lambda: (_sizes(40_000, 56, L(0.01), large=((20, L(0.08)), (5, L(0.3)))),
                     synth.geom_parallel(1, 200, 211, 0.01, 0.01, -0.3, 0.2)),
    "ring": lambda: (_sizes(20_000, 57, L(4.0), 120.0, ((9, L(30.0)),)), _ring(2, 281, 21)),
    "ring_raw": lambda: (_sizes(20_000, 58, L(4.0), 120.0, ((9, L(30.0)),)), _ring(2, 281, 21, arc_mode=1)),
    "ring_5_bins": lambda: (_sizes(20_000, 59, L(4.0), 120.0, ((9, L(30.0)),)), _ring(2, 281, 21, 5)),
    "ring_16_bins": lambda: (_sizes(20_000, 60, L(4.0), 120.0, ((9, L(60.0)),)), _ring(2, 281, 21, 16)),
}


@pytest.mark.parametrize("kernel", ["gaussian", "epanechnikov"])
@pytest.mark.parametrize("name", list(STAGED))
def test_staged_and_direct_walks_agree(env, name, kernel):
    """A Gaussian's gradient takes nothing from the others, so a set's equals its
    parts' -- the set staged (with its large footprints in place), the small
    parts all in place.  Both decide every pair by the same roundings, only the
    sums' order differs: within 2e-6 of the norm (a few ulp of the terms)."""
    torch, rg, ctx = env
    G, gd = STAGED[name]()
    if kernel == "epanechnikov" and gd.get("n_tof"):
        pytest.skip("time of flight takes the Gaussian kernel")
    geom = rg.Geometry(ctx, gd)
    w = torch.from_numpy(synth.random_weights(geom.n_rays, 7)).cuda()

    def grads(G):
        gs = rg.Gaussians(ctx, *[torch.from_numpy(np.ascontiguousarray(G[k])).cuda() for k in ("mu", "ls", "q", "rho")])
        gs.set_kernel(kernel)
        outs = [torch.empty(s, device="cuda") for s in ((gs.n, 3), (gs.n, 3), (gs.n, 4), (gs.n, 1))]
        ctx.prof_reset()
        ctx.prof_enable(True)
        rg.project_backward(ctx, gs, geom, w, *outs)
        staged = ctx.prof_get("k_order")[0] > 0
        ctx.prof_enable(False)
        return [o.double() for o in outs], staged

    whole, staged = grads(G)
    assert staged
    n, step = G["rho"].size, 8000 // int(gd["n_views"])
    parts = []
    for a in range(0, n, step):
        part, staged = grads({k: v[a:a + step] for k, v in G.items()})
        assert not staged
        parts.append(part)
    for key, a, b in zip(("mu", "ls", "q", "rho"), whole, [torch.cat(x) for x in zip(*parts)]):
        e = float(torch.linalg.norm(a - b) / torch.linalg.norm(b))
        assert e < 2e-6, f"{key}: {e:.2e}"


def test_few_large_footprints_are_shared_out(env):
    """64 Gaussians over most of a 512 x 512 view (their boxes, walked by one warp
    each, took 50 times the forward): the gradient takes no more than five
    forward projections, best of five each."""
    torch, rg, ctx = env
    geom = rg.Geometry(ctx, _parallel(1, 512, 512, 2.0 / 512))
    G = synth.gaussians_uniform(64, 61, half_box=0.7, log_sigma=math.log(0.2))
    gs = rg.Gaussians(ctx, *[torch.from_numpy(np.ascontiguousarray(G[k])).cuda() for k in ("mu", "ls", "q", "rho")])
    img, w = torch.empty(geom.n_rays, device="cuda"), torch.rand(geom.n_rays, device="cuda")
    outs = [torch.empty(s, device="cuda") for s in ((64, 3), (64, 3), (64, 4), (64,))]

    def best(call):
        ms = []
        for _ in range(7):
            a, b = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            a.record()
            call()
            b.record()
            torch.cuda.synchronize()
            ms.append(a.elapsed_time(b))
        return min(ms[2:])

    fwd = best(lambda: rg.project_forward(ctx, gs, geom, img))
    assert best(lambda: rg.project_backward(ctx, gs, geom, w, *outs)) < 5.0 * fwd


def test_footprint_of_more_than_2_31_pixels(env):
    """One isotropic Gaussian over a detector whose pixels an int does not count:
    dL/drho is the weighted sum of the closed form at the few weighted pixels."""
    torch, rg, ctx = env
    side, sigma, pitch = 46_400, 1.0, 1e-4
    geom = rg.Geometry(ctx, synth.geom_parallel(1, side, side, pitch, pitch, -40.0, 40.0))
    f = dict(dtype=torch.float32, device="cuda")
    gs = rg.Gaussians(ctx, torch.zeros((1, 3), **f), torch.zeros((1, 3), **f),
                      torch.tensor([[1.0, 0.0, 0.0, 0.0]], **f), torch.ones(1, **f))
    rng = np.random.default_rng(62)
    row, col = rng.integers(0, side, (2, 500))
    wt = rng.uniform(0.5, 1.5, 500)
    w = torch.zeros(side * side, **f)
    w[torch.from_numpy(row * side + col).cuda()] = torch.from_numpy(wt).float().cuda()
    out = torch.empty(1, **f)
    rg.project_backward(ctx, gs, geom, w, None, None, None, out)
    u, v = (col - 0.5 * (side - 1)) * pitch, (row - 0.5 * (side - 1)) * pitch
    m = u * u + v * v          # a pair counts within 3 sigma of the line
    ref = float((wt * math.sqrt(2.0 * math.pi) * sigma * np.exp(-0.5 * m))[m <= 9.0].sum())
    assert abs(float(out) - ref) < 1e-4 * ref


@pytest.mark.parametrize("bad", [math.nan, math.inf])
@pytest.mark.parametrize("walk", ["direct", "staged"])
@pytest.mark.parametrize("name", [n for n in MASKED if n != "ring_tof"])
def test_non_finite_weight_outside_the_support_adds_nothing(env, name, walk, bad):
    """The same for the Epanechnikov kernel, a NaN or infinite dL/dI where no
    support reaches: one Gaussian, and (staged) one among 40,000 far smaller.
    The sums are of the same terms; 1e-5 as above."""
    torch, rg, ctx = env
    s, gd = MASKED[name]()
    n = 1
    G = {"mu": np.array([[0.4 * s, -0.3 * s, 0.2 * s]]), "ls": np.log([[s, 0.5 * s, 0.7 * s]]),
         "q": np.array([[0.9, 0.1, -0.3, 0.2]]), "rho": np.ones(1)}
    if walk == "staged":
        n, rng = 40_000, np.random.default_rng(63)
        G["mu"] = np.concatenate([G["mu"], rng.uniform(-s, s, (n - 1, 3))])
        G["ls"] = np.concatenate([G["ls"], np.full((n - 1, 3), math.log(0.02 * s))])
        G["q"] = np.concatenate([G["q"], rng.normal(size=(n - 1, 4))])
        G["rho"] = np.ones(n)
    geom = rg.Geometry(ctx, gd)
    gs = rg.Gaussians(ctx, *[torch.from_numpy(G[k]).float().cuda() for k in ("mu", "ls", "q", "rho")])
    gs.set_kernel("epanechnikov")
    img = rg.project_forward(ctx, gs, geom, torch.empty(geom.n_rays, device="cuda"))
    empty = img.reshape(-1) == 0.0
    assert 0 < int(empty.sum()) < empty.numel()
    w = torch.from_numpy(synth.random_weights(geom.n_rays, 6)).cuda().reshape(-1)
    res = []
    for fill in (0.0, bad):
        outs = [torch.empty(sh, device="cuda") for sh in ((n, 3), (n, 3), (n, 4), (n,))]
        rg.project_backward(ctx, gs, geom, torch.where(empty, torch.full_like(w, fill), w), *outs)
        res.append(torch.cat([o.reshape(-1) for o in outs]).double().cpu())
    assert torch.linalg.norm(res[1] - res[0]) <= 1e-5 * torch.linalg.norm(res[0])


def test_order_gives_way_to_the_budget(env):
    """The staged walk's spatial order is left out where the memory budget has no
    room for it: a budget for the set, one view's binning and the gradient
    accumulator admits the call, and the gradient is the same (sums in another
    order, 2e-6 as above).  Scratch is taken an eighth larger than asked."""
    torch, rg, ctx = env
    N, side = 400_000, 128
    gd = _parallel(1, side, side, 0.015)
    G = _sizes(N, 64, L(0.01))
    w = torch.rand(side * side, device="cuda")

    def grads(budget, keys=False):
        c = rg.Context(0, budget)
        gs = rg.Gaussians(c, *[torch.from_numpy(np.ascontiguousarray(G[k])).cuda() for k in ("mu", "ls", "q", "rho")])
        geom = rg.Geometry(c, gd)
        outs = [torch.empty(s, device="cuda") for s in ((N, 3), (N, 3), (N, 4), (N, 1))]
        c.prof_enable(True)
        rg.project_backward(c, gs, geom, w, *outs)
        ordered = c.prof_get("k_order")[0]
        K = rg.debug_tile_lists(c, gs, geom)[1].size if keys else 0
        gs.close()
        geom.close()
        c.close()
        return [o.double() for o in outs], ordered, K

    ref, ordered, K = grads(0, True)
    assert ordered == 1
    own = (44 + 80 + 48) * N + 1.125 * (16 * N + 64 * N + 17 * K)     # set; counts, boxes, accumulator, keys
    got, ordered, _ = grads(int(1.01 * own) + (1 << 20))
    assert ordered == 0
    for a, b in zip(got, ref):
        assert float(torch.linalg.norm(a - b) / torch.linalg.norm(b)) < 2e-6
