"""The batched form (many scans per step, persistent launches, CUDA graph)
against one-scan-at-a-time calls of the same library and against the FP64
oracle, and the autotuner."""
import math

import numpy as np
import pytest

from paper_2602_01057_gb300 import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2602_01057_gb300 import build, rgrt
    build.build()
    ctx = rgrt.Context(0)
    return torch, rgrt, ctx


def _scans(seed, k, tile=(16, 16)):
    rng = np.random.default_rng(seed)
    out = []
    for i in range(k):
        n = int(np.exp(rng.uniform(math.log(500), math.log(6000))))
        v = int(rng.integers(3, 12))
        side = int(rng.choice([32, 48, 64]))
        G, _ = synth.workload_c2(seed * 100 + i, n=n, n_views=v, side=side)
        gd = synth.geom_c2(n_views=v, side=side, tile=tile)
        out.append((G, gd))
    return out


def _dev(torch, G):
    return [torch.from_numpy(np.ascontiguousarray(G[k])).cuda() for k in ("mu", "ls", "q", "rho")]


def test_batch_forward_equals_single_scans(env):
    torch, rg, ctx = env
    scans = _scans(1, 7)
    gs = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    geoms = [rg.Geometry(ctx, gd) for _, gd in scans]
    b = rg.Batch(ctx, gs, geoms)
    outs = [torch.empty(g.n_rays, device="cuda") for g in geoms]
    for _ in range(2):            # the second call replays the captured graph
        b.forward(outs)
        for g, geom, o in zip(gs, geoms, outs):
            ref = torch.empty(geom.n_rays, device="cuda")
            rg.project_forward(ctx, g, geom, ref)
            torch.cuda.synchronize()
            assert torch.equal(o, ref)   # same tiles and pairs: fixed-point sums, identical


def test_batch_forward_matches_oracle(env, oracle):
    """The batched forward against the FP64 oracle: every ray of the first 4
    scans, a stratified 1/64 subsample (every 64th ray) of the others."""
    torch, rg, ctx = env
    scans = _scans(3, 8)
    gs = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    geoms = [rg.Geometry(ctx, gd) for _, gd in scans]
    b = rg.Batch(ctx, gs, geoms)
    outs = [torch.empty(g.n_rays, device="cuda") for g in geoms]
    b.forward(outs)
    torch.cuda.synchronize()
    for i, ((G, gd), o) in enumerate(zip(scans, outs)):
        I = o.cpu().numpy().astype(np.float64)
        if i < 4:
            ref = oracle.forward(gd, G)
        else:
            idx = np.arange(0, I.size, 64)
            ref = oracle.forward_rays(gd, G, idx)
            I = I[idx]
        clip = np.clip(I, ref["I_lo"], ref["I_hi"])
        err = np.linalg.norm(I - clip) / max(np.linalg.norm(clip), 1e-300)
        assert np.count_nonzero(ref["I"]) > 0
        assert err < 1e-5, (i, err)


def test_batch_loss_step_matches_single_scans(env):
    torch, rg, ctx = env
    scans = _scans(2, 5)
    hp = rg.adam_params()
    # measured data: projections of perturbed copies
    ys = []
    for G, gd in scans:
        geom = rg.Geometry(ctx, gd)
        gt = rg.Gaussians(ctx, *_dev(torch, synth.perturbed(G, 7, pos_std=0.01)))
        y = torch.empty(geom.n_rays, device="cuda")
        rg.project_forward(ctx, gt, geom, y)
        ys.append(y)
    gb = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    gsingle = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    geoms = [rg.Geometry(ctx, gd) for _, gd in scans]
    b = rg.Batch(ctx, gb, geoms)
    for t in (1, 2, 3):
        lb = b.loss_step(ys, rg.RGRT_LOSS_L2, hp, t)
        for i in range(len(scans)):
            ls = np.zeros(1, np.float32)
            rg.loss_step(ctx, gsingle[i], geoms[i], ys[i], rg.RGRT_LOSS_L2, hp, t, ls)
            assert lb[i] == pytest.approx(float(ls[0]), rel=1e-5, abs=1e-12)
    for i in range(len(scans)):
        a, c = gb[i].numpy(), gsingle[i].numpy()
        for k in ("mu", "ls", "q", "rho"):
            G0 = scans[i][0][k]
            da = a[k].astype(np.float64) - G0
            dc = c[k].astype(np.float64) - G0
            assert np.linalg.norm(da - dc) <= 1e-3 * np.linalg.norm(dc) + 1e-7, (i, k)


def test_batch_with_large_and_small_scans(env):
    """A scan large enough to fill the GPU for many waves (40 views of 256^2,
    10,240 tiles of 16 x 16) is projected with launches of its own inside the
    batch; the small ones share the persistent launches.  Forward and three
    optimisation steps against single-scan calls."""
    torch, rg, ctx = env
    G, _ = synth.workload_c2(31, n=5000, n_views=40, side=256)
    scans = [(G, synth.geom_c2(n_views=40, side=256))] + _scans(4, 3)
    gb = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    gsingle = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    geoms = [rg.Geometry(ctx, gd) for _, gd in scans]
    b = rg.Batch(ctx, gb, geoms)
    outs = [torch.empty(g.n_rays, device="cuda") for g in geoms]
    b.forward(outs)
    for g, geom, o in zip(gsingle, geoms, outs):
        ref = torch.empty(geom.n_rays, device="cuda")
        rg.project_forward(ctx, g, geom, ref)
        torch.cuda.synchronize()
        assert torch.equal(o, ref)
    hp = rg.adam_params()
    ys = []
    for (G, gd), geom in zip(scans, geoms):
        gt = rg.Gaussians(ctx, *_dev(torch, synth.perturbed(G, 9, pos_std=0.01)))
        y = torch.empty(geom.n_rays, device="cuda")
        rg.project_forward(ctx, gt, geom, y)
        ys.append(y)
    for t in (1, 2, 3):
        lb = b.loss_step(ys, rg.RGRT_LOSS_L2, hp, t)
        for i in range(len(scans)):
            ls = np.zeros(1, np.float32)
            rg.loss_step(ctx, gsingle[i], geoms[i], ys[i], rg.RGRT_LOSS_L2, hp, t, ls)
            assert lb[i] == pytest.approx(float(ls[0]), rel=1e-5, abs=1e-12)
    for i in range(len(scans)):
        a, c = gb[i].numpy(), gsingle[i].numpy()
        for k in ("mu", "ls", "q", "rho"):
            G0 = scans[i][0][k]
            da = a[k].astype(np.float64) - G0
            dc = c[k].astype(np.float64) - G0
            assert np.linalg.norm(da - dc) <= 1e-3 * np.linalg.norm(dc) + 1e-7, (i, k)
    assert b.info()["work_items"] == sum(g.n_rays // 256 for g in geoms[:1]) + sum(
        (gd["n_views"] * ((gd["n_cols"] + 15) // 16) * ((gd["n_rows"] + 15) // 16)) for _, gd in scans[1:])


def test_batch_replans_when_entries_outgrow_capacity(env):
    torch, rg, ctx = env
    scans = _scans(3, 3)
    gs = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    geoms = [rg.Geometry(ctx, gd) for _, gd in scans]
    b = rg.Batch(ctx, gs, geoms)
    cap0 = b.info()["key_capacity"]
    # grow every Gaussian 3x: far more (tile, Gaussian) entries than planned
    for (G, _), g in zip(scans, gs):
        ls = torch.from_numpy(np.ascontiguousarray(G["ls"] + math.log(3.0)).astype(np.float32)).cuda()
        g.set(ls=ls)
    outs = [torch.empty(g.n_rays, device="cuda") for g in geoms]
    b.forward(outs)
    info = b.info()
    assert info["replans"] >= 1 and info["key_capacity"] > cap0
    for g, geom, o in zip(gs, geoms, outs):
        ref = torch.empty(geom.n_rays, device="cuda")
        rg.project_forward(ctx, g, geom, ref)
        torch.cuda.synchronize()
        assert torch.equal(o, ref)


def test_batch_rejects_mixed_tiles(env):
    torch, rg, ctx = env
    (G1, gd1), (G2, gd2) = _scans(4, 2)
    gd2 = dict(gd2, tile_w=8, tile_h=8)
    gs = [rg.Gaussians(ctx, *_dev(torch, G)) for G in (G1, G2)]
    geoms = [rg.Geometry(ctx, gd) for gd in (gd1, gd2)]
    with pytest.raises(rg.RgrtError):
        rg.Batch(ctx, gs, geoms)


def test_autotune_returns_a_candidate(env):
    torch, rg, ctx = env
    G, _ = synth.workload_c2(5, n=4000, n_views=24, side=96)
    gd = synth.geom_c2(n_views=24, side=96)
    g = rg.Gaussians(ctx, *_dev(torch, G))
    tw, th, ms = rg.autotune_tile(ctx, g, gd, max_views=8)
    assert (tw, th) in {(16, 16), (16, 8), (8, 8), (32, 8)} and ms > 0


def test_batch_tile_lists_match_the_oracle(env, oracle):
    """The batch's own binning (device-side key count, padding keys past the
    step's entries, shared sort scratch) gives every scan the oracle's FP32
    tile sets -- scans small enough for the persistent launches and a scan
    large enough for launches of its own."""
    torch, rg, ctx = env
    scans = _scans(5, 5)
    G, _ = synth.workload_c2(77, n=20_000, n_views=90, side=256)
    scans.append((G, synth.geom_c2(n_views=90, side=256)))
    gs = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    geoms = [rg.Geometry(ctx, gd) for _, gd in scans]
    b = rg.Batch(ctx, gs, geoms)
    outs = [torch.empty(g.n_rays, device="cuda") for g in geoms]
    for rep in range(2):              # planning pass, then a graph replay
        b.forward(outs)
        for i, (G, gd) in enumerate(scans):
            start, gid = b.debug_tile_lists(i)
            rstart, rgid = oracle.tile_lists_fp32(gd, G, gd["tile_w"], gd["tile_h"])
            assert gid.size == rgid.size and gid.size > 0, (rep, i)
            assert np.array_equal(start, rstart), (rep, i)
            tile = np.repeat(np.arange(start.size - 1), np.diff(start))
            assert np.array_equal(gid[np.lexsort((gid, tile))], rgid), (rep, i)


@pytest.mark.parametrize("shared", [False, True])
@pytest.mark.parametrize("kind", ["parallel", "cone"])
def test_batch_bins_scans_side_by_side(env, kind, shared):
    """More scans than binning streams, of both ray kinds and uneven sizes, and
    scans that share one Gaussian set (one stream): two steps equal the scans'
    own projections, bit for bit."""
    torch, rg, ctx = env
    sizes = [(2, 33), (9, 64), (1, 8), (5, 48), (3, 96), (7, 40)]
    gds = [synth.geom_parallel(v, s, s, 2.0 / s, 2.0 / s, -4.0, 4.0) if kind == "parallel" else
           synth.geom_cone(v, s, s, 4.0 / s, 4.0 / s, 4.0, 8.0) for v, s in sizes]
    geoms = [rg.Geometry(ctx, gd) for gd in gds]
    gs = [rg.Gaussians(ctx, *_dev(torch, synth.gaussians_uniform(300 + 700 * (i % 4), 60 + i, log_sigma=math.log(0.05))))
          for i in range(1 if shared else len(sizes))]
    gs = gs * len(sizes) if shared else gs
    b = rg.Batch(ctx, gs, geoms)
    outs = [torch.empty(g.n_rays, device="cuda") for g in geoms]
    for _ in range(2):
        b.forward(outs)
        for g, geom, o in zip(gs, geoms, outs):
            ref = rg.project_forward(ctx, g, geom, torch.empty(geom.n_rays, device="cuda"))
            torch.cuda.synchronize()
            assert torch.equal(o, ref)


def test_batch_projection_follows_moved_gaussians(env):
    """A scan's lists are cut into as many parts as a projection of its own cuts
    them, also after its Gaussians have shrunk or grown across the rule's
    thresholds since the batch was planned: bit for bit at every size."""
    torch, rg, ctx = env
    gd = synth.geom_parallel(6, 64, 64, 2.0 / 64, 2.0 / 64, -4.0, 4.0)
    G = synth.gaussians_uniform(2500, 71, log_sigma=math.log(0.09))
    g, geom = rg.Gaussians(ctx, *_dev(torch, G)), rg.Geometry(ctx, gd)
    small = rg.Gaussians(ctx, *_dev(torch, synth.gaussians_uniform(50, 72)))
    b = rg.Batch(ctx, [g, small], [geom, geom])
    outs = [torch.empty(geom.n_rays, device="cuda") for _ in range(2)]
    lists = set()
    for shrink in (0.0, 0.7, 1.4, 2.1, 0.3):
        g.set(ls=torch.from_numpy(G["ls"] - np.float32(shrink)).cuda())
        b.forward(outs)
        ref = rg.project_forward(ctx, g, geom, torch.empty(geom.n_rays, device="cuda"))
        start, _ = b.debug_tile_lists(0)
        lists.add(int(math.log2(start[-1] / (start.size - 1))))
        torch.cuda.synchronize()
        assert torch.equal(outs[0], ref), shrink
    assert lists == {7, 8, 9}     # 2, 4 and 8 parts: average lists from 128, 256 and 512 entries


def test_parallel_batch_needs_no_scratch_per_scan(env):
    """A batch of parallel-beam scans keeps a scan's ids, ranges, images and
    gradients, and binning scratch for one scan at a time: a budget for these
    admits it, and its steps are those of a batch with room to spare (the terms
    of a sum in another order: within 1e-4 of a step's size)."""
    torch, rg, ctx = env
    n, N, V, side = 6, 40_000, 30, 64
    gd = synth.geom_parallel(V, side, side, 2.0 / side, 2.0 / side, -4.0, 4.0)
    sets = [synth.gaussians_uniform(N, 80 + i, log_sigma=math.log(0.012)) for i in range(n)]
    y = [torch.rand(V * side * side, device="cuda") for _ in range(n)]

    def steps(budget):
        c = rg.Context(0, budget)
        gs = [rg.Gaussians(c, *_dev(torch, G)) for G in sets]
        geom = rg.Geometry(c, gd)
        b = rg.Batch(c, gs, [geom] * n)
        cap = b.info()["key_capacity"]
        loss = [b.loss_step(y, t=t) for t in (1, 2)]
        out = [g.numpy() for g in gs]
        b.close()
        c.close()
        return cap, loss, out

    cap, loss, out = steps(0)
    E, T, R = N * V, V * (side // 16) ** 2, V * side * side
    per_scan = 4 * cap / n + 8 * T + 8 * R + (64 + 44) * N            # ids, ranges, image and dL/dI, gradients
    sets_bytes = (44 + 80 + 48 + 88) * N                               # parameters, records, Adam moments
    shared = 16 * E + 13 * 1.1 * cap / n                               # one scan's binning
    _, loss2, out2 = steps(int(1.03 * (n * (per_scan + sets_bytes) + shared)) + (1 << 20))
    for a, b in zip(loss, loss2):
        np.testing.assert_allclose(a, b, rtol=1e-5)
    for a, b, g in zip(out, out2, sets):
        for k in a:
            assert np.linalg.norm(a[k] - b[k]) <= 1e-4 * np.linalg.norm(a[k] - g[k]), k


def _parallel(v, side):
    return synth.geom_parallel(v, side, side, 2.0 / side, 2.0 / side, -4.0, 4.0)


def test_parallel_batch_steps_match_single_scans(env):
    """Optimisation steps of parallel-ray scans: more small ones than streams, of
    uneven sizes, both walks of the adjoint (few pairs in place; 17,001 Gaussians
    staged, with the order's scratch), a large scan among them and a ring.
    Losses and parameters follow the scans' own steps as far as the cone beam's
    do above: 1e-5 of a loss, 1e-3 of a parameter's way."""
    torch, rg, ctx = env
    scans = [(synth.gaussians_uniform(n, 90 + i, log_sigma=math.log(s)), gd) for i, (n, s, gd) in enumerate([
        (300, 0.06, _parallel(5, 33)), (17_001, 0.02, _parallel(4, 64)), (1, 0.2, _parallel(2, 16)),
        (2_500, 0.03, _parallel(90, 256)), (900, 0.05, _parallel(9, 48)), (40_000, 0.015, _parallel(9, 64)),
        (33, 0.1, _parallel(1, 80))])]
    ring = synth.gaussians_uniform(5_000, 98, half_box=120.0, log_sigma=math.log(5.0))
    scans.append((ring, synth.geom_pet(12, 129, 21, 400.0, 288, 9.0)))
    hp = rg.adam_params()
    geoms = [rg.Geometry(ctx, gd) for _, gd in scans]
    ys = []
    for (G, gd), geom in zip(scans, geoms):
        gt = rg.Gaussians(ctx, *_dev(torch, synth.perturbed(G, 7, pos_std=0.01)))
        ys.append(rg.project_forward(ctx, gt, geom, torch.empty(geom.n_rays, device="cuda")))
    gb = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    own = [rg.Gaussians(ctx, *_dev(torch, G)) for G, _ in scans]
    b = rg.Batch(ctx, gb, geoms)
    assert b.info()["work_items"] > 16_000          # the large scan's tiles among them
    for t in (1, 2, 3):
        lb = b.loss_step(ys, rg.RGRT_LOSS_L2, hp, t)
        for i, (g, geom, y) in enumerate(zip(own, geoms, ys)):
            ls = np.zeros(1, np.float32)
            rg.loss_step(ctx, g, geom, y, rg.RGRT_LOSS_L2, hp, t, ls)
            assert lb[i] == pytest.approx(float(ls[0]), rel=1e-5, abs=1e-12), (t, i)
    for i, (G, _) in enumerate(scans):
        a, c = gb[i].numpy(), own[i].numpy()
        for k in a:
            d = np.linalg.norm((a[k].astype(np.float64) - c[k]).ravel())
            assert d <= 1e-3 * np.linalg.norm((c[k].astype(np.float64) - G[k]).ravel()), (i, k)


@pytest.mark.parametrize("kind", ["parallel", "cone"])
def test_step_of_scans_that_share_a_set(env, kind):
    """Two scans of one set in a batch: both gradients are taken at the step's
    start, then Adam is applied for one scan after the other (the two updates
    recomputed in binary64 from the scans' own gradients; 1e-3 of the way)."""
    torch, rg, ctx = env
    gds = [_parallel(5, 48), _parallel(3, 64)] if kind == "parallel" else \
        [synth.geom_cone(v, s, s, 4.0 / s, 4.0 / s, 4.0, 8.0) for v, s in ((5, 48), (3, 64))]
    G = synth.gaussians_uniform(700, 99, log_sigma=math.log(0.06))
    geoms = [rg.Geometry(ctx, gd) for gd in gds]
    gt = rg.Gaussians(ctx, *_dev(torch, synth.perturbed(G, 8, pos_std=0.01)))
    ys = [rg.project_forward(ctx, gt, q, torch.empty(q.n_rays, device="cuda")) for q in geoms]
    hp = rg.adam_params()
    g = rg.Gaussians(ctx, *_dev(torch, G))
    grads = []
    for geom, y in zip(geoms, ys):
        o = {k: torch.empty(G[k].shape, device="cuda") for k in G}
        rg.loss_grad(ctx, g, geom, y, rg.RGRT_LOSS_L2, hp, None, o["mu"], o["ls"], o["q"], o["rho"])
        grads.append({k: v.double().cpu().numpy() for k, v in o.items()})
    rg.Batch(ctx, [g, g], geoms).loss_step(ys, rg.RGRT_LOSS_L2, hp, 1)
    got = g.numpy()
    for k, lr in (("mu", hp.lr_mu), ("ls", hp.lr_logscale), ("q", hp.lr_quat), ("rho", hp.lr_rho)):
        p, m, v = G[k].astype(np.float64), 0.0, 0.0
        for d in grads:
            m = hp.beta1 * m + (1.0 - hp.beta1) * d[k]
            v = hp.beta2 * v + (1.0 - hp.beta2) * d[k] ** 2
            p = p - lr / (1.0 - hp.beta1) * m / (np.sqrt(v / (1.0 - hp.beta2)) + hp.eps)
        assert np.linalg.norm(got[k] - p) <= 1e-3 * np.linalg.norm(p - G[k]), k
