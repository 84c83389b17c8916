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
