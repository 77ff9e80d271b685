"""Adjoint to every Gaussian parameter (gs_render_backward with parameter
gradients, config 'differentiation check') vs the FP64 oracle's analytic
adjoint, which finite differences pin (tests/test_oracle_pins.py).  Bar:
per parameter group, ||g_gpu - g_oracle|| / ||g_oracle|| <= 1e-3."""
import numpy as np
import pytest

import oracle as O
from paper_2408_10154_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2408_10154_gb300 as gs
    from paper_2408_10154_gb300 import autograd, build
    build.build()
    O.build()
    ctx = gs.Context(0)
    yield gs, autograd, ctx
    ctx.close()


def dev(a, dtype=torch.float32):
    return torch.as_tensor(np.ascontiguousarray(a)).to(device="cuda", dtype=dtype).contiguous()


GROUPS = (("means", "means4", 3), ("log_scales", "log_scales4", 3), ("quats", "quats4", 4), ("logits", "logits", 1),
          ("rgb", "rgb4", 3))


def check(env, gd, cams, poses, seed, subset=None):
    gs, autograd, ctx = env
    og = O.Gaussians.from_dict(gd)
    g = gs.Gaussians.from_numpy(gd)
    rng = np.random.default_rng(seed)
    P = dev(poses.reshape(-1, 12))
    out = gs.gs_render(ctx, g, P, cams)
    cr = [rng.standard_normal((3, int(c[5]), int(c[4]))).astype(np.float32) for c in cams]
    cd = [rng.standard_normal((int(c[5]), int(c[4]))).astype(np.float32) for c in cams]
    ca = [rng.standard_normal((int(c[5]), int(c[4]))).astype(np.float32) for c in cams]
    piv = np.stack([O.centroid(og).astype(np.float32)] * len(cams))
    cat = lambda xs: dev(np.concatenate([x.reshape(-1) for x in xs]))
    pg, gr = gs.gs_render_backward(ctx, g, P, cams, out["t_final"], out["last"], cat(cr), cat(cd), cat(ca),
                                   dev(piv), params=True)
    ref = {k: 0.0 for k, _, _ in GROUPS}
    for c, cam in enumerate(cams):
        b = O.backward(og, poses[c].astype(np.float32).astype(np.float64), cam, cr[c].astype(np.float64),
                       cd[c].astype(np.float64), ca[c].astype(np.float64), pivot=piv[c].astype(np.float64))
        for k, _, _ in GROUPS:
            ref[k] = ref[k] + b[k]
        tw = b["twist"]
        assert np.linalg.norm(pg[c].cpu().numpy() - tw) <= 1e-3 * np.linalg.norm(tw)
    idx = np.arange(og.n) if subset is None else subset
    for k, key, K in GROUPS:
        got = gr[key].cpu().numpy()
        got = got[idx] if key == "logits" else got[idx, :K]
        want = ref[k][idx]
        err = np.linalg.norm(got - want) / np.linalg.norm(want)
        assert err <= 1e-3, (k, err)


def test_parameter_adjoint_500_exhaustive(env):
    c = synth.small_case(500, 64, 48, 56.0, n_views=2, seed=1003, ls_mean=-3.0)
    poses = np.stack([synth.random_rigid(np.random.default_rng(3), 3.0, 0.03) for _ in range(2)])
    check(env, c["gaussians"], c["cams"], poses, 4)


def test_parameter_adjoint_300k_subset(env):
    # the differentiation-check workload at full size (300k Gaussians,
    # 1200x680), one keyframe, a random 1 % of the Gaussians compared
    c = synth.diff_check_300k()
    rng = np.random.default_rng(1003)
    sub = rng.choice(c["gaussians"]["means4"].shape[0], 3000, replace=False)
    poses = np.stack([synth.random_rigid(rng, 5.0, 0.05)])
    check(env, c["gaussians"], c["cams"][:1], poses, 5, subset=np.sort(sub))


def test_autograd_function_matches_render_backward(env):
    gs, autograd, ctx = env
    c = synth.small_case(300, 48, 32, 40.0, n_views=1, seed=8)
    g = gs.Gaussians.from_numpy(c["gaussians"])
    leaves = [t.clone().requires_grad_(True) for t in (g.means4, g.log_scales4, g.quats4, g.logits, g.rgb4)]
    gg = gs.Gaussians(*leaves)
    P = dev(np.eye(3, 4).reshape(1, 12))
    rgb, depth, alpha = autograd.rasterize(ctx, gg, P, c["cams"])
    w = torch.randn_like(rgb)
    (w * rgb).sum().backward()
    out = gs.gs_render(ctx, g, P, c["cams"])
    _, gr = gs.gs_render_backward(ctx, g, P, c["cams"], out["t_final"], out["last"], w, torch.zeros_like(depth),
                                  torch.zeros_like(alpha), params=True)
    for leaf, key in zip(leaves, ("means4", "log_scales4", "quats4", "logits", "rgb4")):
        assert torch.equal(leaf.grad, gr[key])


@pytest.mark.parametrize("n,W,H,f,views", [(500, 64, 48, 56.0, 2), (3000, 160, 120, 140.0, 3)])
def test_saved_forward_equals_render_and_backward(env, n, W, H, f, views):
    # gs_render_saved + gs_render_backward_saved (the adjoint from the kept
    # projection and tile lists, no second binning) against gs_render +
    # gs_render_backward: the same renders and gradients, bit for bit
    gs, autograd, ctx = env
    c = synth.small_case(n, W, H, f, n_views=views, seed=n, ls_mean=-3.0)
    g = gs.Gaussians.from_numpy(c["gaussians"])
    rng = np.random.default_rng(n)
    poses = np.stack([synth.random_rigid(rng, 3.0, 0.03) for _ in range(views)])
    P = dev(poses.reshape(-1, 12))
    out = gs.gs_render(ctx, g, P, c["cams"])
    o2, sv = gs.gs_render_saved(ctx, g, P, c["cams"])
    for k in ("rgb", "depth", "alpha"):
        assert torch.equal(out[k], o2[k]), k
    npx = sum(int(cam[4]) * int(cam[5]) for cam in c["cams"])
    cr, cd, ca = (dev(rng.standard_normal(3 * npx)), dev(rng.standard_normal(npx)), dev(rng.standard_normal(npx)))
    piv = dev(np.stack([O.centroid(O.Gaussians.from_dict(c["gaussians"]))] * views))
    pg1, gr1 = gs.gs_render_backward(ctx, g, P, c["cams"], out["t_final"], out["last"], cr, cd, ca, piv, params=True)
    for _ in range(2):  # the saved state serves more than one adjoint
        pg2, gr2 = gs.gs_render_backward_saved(ctx, sv, cr, cd, ca, piv, params=True)
        assert torch.equal(pg1, pg2)
        for k in gr1:
            assert torch.equal(gr1[k], gr2[k]), k
    sv.close()


def test_parameter_adjoint_list_lengths(env):
    # records over 1 to 3,225 tiles of a 1200x680 frame, both sides of the
    # length where the sum over a record's tiles changes hands (32) and of
    # its staging (64), two cameras, Gaussian counts around a block of 128
    rng = np.random.default_rng(77)
    for n in (1, 127, 129):
        gd = synth.gaussians_box(n, rng, center=(0.0, 0.0, 2.5), half=1.2, ls_mean=-2.5, ls_std=0.1)
        gd["log_scales4"][:, :3] = rng.uniform(-5.5, 0.6, (n, 1)) + rng.normal(0.0, 0.2, (n, 3))
        gd["logits"][:] = rng.normal(-3.0, 0.5, n)
        cams = np.stack([synth.camera(600.0, 600.0, 600.0, 340.0, 1200, 680, np.eye(3, 4)),
                         synth.camera(300.0, 300.0, 150.0, 90.0, 301, 181, np.eye(3, 4))])
        poses = np.stack([synth.random_rigid(rng, 3.0, 0.03) for _ in cams])
        check(env, gd, cams, poses, n)


def test_parameter_adjoint_ignores_earlier_calls(env):
    # list entries behind a tile's last contributor hold no gradient of an
    # earlier call on the context: near-opaque layers hide many of them
    gs, _, ctx = env
    rng = np.random.default_rng(78)
    g1 = synth.gaussians_box(4000, rng, half=0.8, ls_mean=-2.5)
    g2 = synth.gaussians_box(3000, rng, half=0.8, ls_mean=-2.3)
    g2["logits"][:] = 7.0
    cams = synth.circle_cameras(2, 0.25, (0.0, 0.0, 2.5), 320, 240, 250.0)
    P = dev(np.stack([np.eye(3, 4).reshape(12)] * 2))

    def grads(c, gd, scale):
        g = gs.Gaussians.from_numpy(gd)
        out = gs.gs_render(c, g, P, cams)
        cr, cd = torch.full_like(out["rgb"], scale), torch.full_like(out["depth"], scale)
        return gs.gs_render_backward(c, g, P, cams, out["t_final"], out["last"], cr, cd, params=True)[1]

    fresh = gs.Context(0)
    want = grads(fresh, g2, 1.0)
    for _ in range(2):
        grads(ctx, g1, 1e6)
        got = grads(ctx, g2, 1.0)
        for k in want:
            assert torch.equal(got[k], want[k]), k
    fresh.close()


def test_saved_forward_repeats_at_the_smallest_budget(env):
    # a repeated forward (whose lists are sized by what the shape had before)
    # needs no more scratch than the first
    gs, _, _ = env
    c = synth.small_case(2500, 120, 88, 100.0, n_views=2, seed=79, ls_mean=-3.0)
    g = gs.Gaussians.from_numpy(c["gaussians"])
    P = dev(np.tile(np.eye(3, 4).reshape(1, 12), (2, 1)))
    want, sv = gs.gs_render_saved(gs.Context(0), g, P, c["cams"])
    sv.close()

    def passes(budget, times):
        ctx = gs.Context(0, budget)
        try:
            for _ in range(times):
                out, saved = gs.gs_render_saved(ctx, g, P, c["cams"])
                saved.close()
                assert all(torch.equal(out[k], want[k]) for k in want)
            return True
        except gs.GsError:
            return False
        finally:
            ctx.close()

    lo, hi = 1 << 12, 1 << 26
    assert not passes(lo, 1) and passes(hi, 1)
    while hi - lo > 256:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if passes(mid, 1) else (mid, hi)
    assert passes(hi, 3)


def test_lists_too_short_for_the_next_scene(env):
    # a scene whose duplicates exceed what the context's lists hold is
    # composited again once they are counted, and a smaller one behind it
    # keeps no more than its own lists: outputs and gradients as on a fresh
    # context, before and after
    gs, _, _ = env
    rng = np.random.default_rng(80)
    few = synth.gaussians_box(900, rng, half=1.2, ls_mean=-5.0, ls_std=0.2)
    many = {k: v.copy() for k, v in few.items()}
    many["log_scales4"][:, :3] += 4.2
    many["logits"][:] = -3.0
    cams = synth.circle_cameras(2, 0.25, (0.0, 0.0, 2.5), 640, 480, 500.0)
    P = dev(np.stack([np.eye(3, 4).reshape(12)] * 2))
    npx = 2 * 640 * 480
    cr, cd = dev(rng.standard_normal(3 * npx)), dev(rng.standard_normal(npx))

    def render(ctx, gd):
        out = gs.gs_render(ctx, gs.Gaussians.from_numpy(gd), P, cams)
        return [out[k] for k in ("rgb", "depth", "alpha", "t_final", "last")]

    def step(ctx, gd):
        out, sv = gs.gs_render_saved(ctx, gs.Gaussians.from_numpy(gd), P, cams)
        pg, gr = gs.gs_render_backward_saved(ctx, sv, cr, cd, params=True)
        sv.close()
        return [out[k] for k in ("rgb", "depth", "alpha")] + [pg] + [gr[k] for k in sorted(gr)]

    for f in (render, step):
        want = {}
        for name, gd in (("few", few), ("many", many)):
            fresh = gs.Context(0)
            want[name] = f(fresh, gd)
            fresh.close()
        ctx = gs.Context(0)
        for name, gd in (("few", few), ("many", many), ("few", few), ("few", few), ("many", many)):
            got = f(ctx, gd)
            for k, (x, y) in enumerate(zip(got, want[name])):
                assert torch.equal(x, y), (f.__name__, name, k)
        ctx.close()
