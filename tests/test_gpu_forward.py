"""Tile integration against the FP64 oracle where its work split changes: every
tile shape (threads from one warp with idle groups to four), ragged detectors,
lists shared by the CTAs of a cluster and lists of a single CTA, general-path
Gaussians in a shared list, and the adjoint's shared lists.

Tolerances: projections 1e-5, gradients 1e-4 relative L2 of the oracle's
brackets, as everywhere else.
"""
import math

import numpy as np
import pytest

from paper_2602_01057_gb300 import synth

pytestmark = pytest.mark.gpu

FWD_TOL, GRAD_TOL = 1e-5, 1e-4


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


def _geometry(kind, tile):
    if kind == "parallel":   # the segment ends inside some Gaussians
        return synth.geom_parallel(2, 37, 53, 0.05, 0.05, -0.8, 2.0, tile=tile), 1.0
    if kind == "cone":
        return synth.geom_cone(2, 37, 53, 0.08, 0.08, 4.0, 6.0, tile=tile), 1.0
    if kind == "tof":
        return synth.with_tof_bins(synth.geom_pet(2, 53, 21, 200.0, 160, 8.0, tile=tile), 5, 40.0, 30.0), 80.0
    return synth.geom_pet3d(2, 53, 13, 200.0, 160, 12.0, 2, tile=tile), 80.0


@pytest.mark.parametrize("n", [300, 6000])
@pytest.mark.parametrize("tile", [(8, 4), (8, 12), (16, 4), (16, 16), (32, 8)])
@pytest.mark.parametrize("kind", ["parallel", "cone", "tof", "pet3d"])
def test_forward_and_adjoint_tile_shapes(env, oracle, kind, tile, n):
    torch, rg, ctx = env
    gd, box = _geometry(kind, tile)
    G = synth.gaussians_uniform(n, 51, half_box=box, log_sigma=math.log(0.06 * box))
    geom = rg.Geometry(ctx, gd)
    gs = rg.Gaussians(ctx, *[torch.from_numpy(np.ascontiguousarray(G[k])).cuda() for k in ("mu", "ls", "q", "rho")])
    I = torch.full((geom.n_rays,), float("nan"), device="cuda")
    rg.project_forward(ctx, gs, geom, I)
    ref = oracle.forward(gd, G)
    got = I.cpu().numpy().astype(np.float64)
    clip = np.clip(got, ref["I_lo"], ref["I_hi"])
    assert np.linalg.norm(got - clip) < FWD_TOL * np.linalg.norm(clip)
    w = synth.random_weights(geom.n_rays, 5)
    outs = [torch.empty(s, device="cuda") for s in ((n, 3), (n, 3), (n, 4), (n,))]
    rg.project_backward(ctx, gs, geom, torch.from_numpy(w).cuda(), *outs)
    ref = oracle.backward(gd, G, w)
    for key, o in zip(("mu", "ls", "q", "rho"), outs):
        g = o.cpu().numpy().astype(np.float64)
        clip = np.clip(g, ref["lo"][key], ref["hi"][key])
        assert np.linalg.norm(g - clip) < GRAD_TOL * np.linalg.norm(ref[key]), key


@pytest.mark.parametrize("n", [1, 6, 4095, 4097, 16383, 16384, 16385])
def test_count_scan_sizes(env, n):
    """The scan of the tile counts by one CTA and by three launches (2 views:
    more than 32,768 counts): the projection is linear in the set, so the two
    halves of a set of tiny Gaussians add up to it (binary32 sums of fewer than
    100 terms a pixel: 1e-5 relative L2)."""
    torch, rg, ctx = env
    geom = rg.Geometry(ctx, synth.geom_parallel(2, 64, 64, 0.03, 0.03, -4.0, 4.0))
    G = synth.gaussians_uniform(n, 52, half_box=0.9, log_sigma=math.log(0.01))
    t = {k: torch.from_numpy(np.ascontiguousarray(G[k])).cuda() for k in ("mu", "ls", "q", "rho")}
    t["rho"] = t["rho"].abs()

    def forward(a, b):
        gs = rg.Gaussians(ctx, *[t[k][a:b].contiguous() for k in ("mu", "ls", "q", "rho")])
        return rg.project_forward(ctx, gs, geom, torch.empty(geom.n_rays, device="cuda")).double()
    whole, cuts = forward(0, n), sorted({0, n // 3, n})
    parts = sum(forward(a, b) for a, b in zip(cuts, cuts[1:]))
    assert torch.linalg.norm(whole - parts) <= 1e-5 * torch.linalg.norm(whole)
