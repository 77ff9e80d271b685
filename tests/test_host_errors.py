"""Host code of the library over a CUDA runtime without a GPU (fake_cudart.c,
linked with the library's own objects): a launch that the runtime refuses is
reported by the call that made it, a saved forward's adjoint takes the scratch
of its own duplicates, and the binding's marshalling costs no more than the
plain ctypes arrays."""
import ctypes
import os
import shutil
import subprocess
import time

import numpy as np
import pytest
import torch

HERE = os.path.dirname(os.path.abspath(__file__))


@pytest.fixture(scope="module")
def fake_lib(tmp_path_factory):
    if shutil.which("nvcc") is None and not os.path.exists("/usr/local/cuda/bin/nvcc"):
        pytest.skip("nvcc not available")
    from paper_2408_10154_gb300 import build
    build.build()
    d = tmp_path_factory.mktemp("fake")
    obj, so = str(d / "fake_cudart.o"), str(d / "libgsreg_fake.so")
    subprocess.run(["gcc", "-std=gnu11", "-w", "-fPIC", "-c", os.path.join(HERE, "fake_cudart.c"), "-o", obj], check=True)
    objs = [os.path.join(build.BUILD, s.replace(".cu", ".o")) for s in build.SOURCES]
    subprocess.run(["g++", "-shared", "-Wl,-Bsymbolic", "-Wl,-z,defs", "-o", so, *objs, obj], check=True)
    return so


@pytest.fixture
def fake(fake_lib, monkeypatch):
    """(package module, fake runtime) with the binding on the fake library."""
    from paper_2408_10154_gb300 import build, gsreg
    monkeypatch.setattr(build, "LIB", fake_lib)
    monkeypatch.setattr(gsreg, "_lib", None)
    monkeypatch.setattr(gsreg, "_stream", lambda: None)
    monkeypatch.setattr(gsreg, "_ptr", lambda t: None if t is None else t.data_ptr())
    rt = gsreg.load()
    rt.fake_pool_bytes.restype = ctypes.c_size_t
    rt.fake_refuse(-1)
    rt.fake_dups(0)
    yield gsreg, rt
    rt.fake_refuse(-1)


class Image:
    """A host tensor that the binding takes for a device tensor."""

    def __init__(self, *shape):
        self.t, self.is_cuda, self.is_contiguous = torch.zeros(shape), True, lambda: True
        self.data_ptr = self.t.data_ptr


def scene(gs, n=70):
    z = lambda k: torch.zeros((n, k))
    g = gs.Gaussians(z(4), z(4), z(4), torch.zeros(n), z(4))
    cam = np.array([30, 30, 16, 16, 32, 32, 1, 0, 0, 0, 0, 1, 0, 0, 0, 0, 1, 0], np.float32)
    return g, torch.eye(3, 4).reshape(1, 12), cam[None], (cam, Image(3, 32, 32), Image(32, 32))


def calls(gs, ctx):
    g, P, cams, view = scene(gs)
    few = gs.Gaussians(*[t[:40].contiguous() for t in (g.means4, g.log_scales4, g.quats4, g.logits, g.rgb4)])

    def saved():
        _, sv = gs.gs_render_saved(ctx, g, P, cams)
        try:
            gs.gs_render_backward_saved(ctx, sv, params=True)
        finally:
            sv.close()

    return {
        "render": lambda: gs.gs_render(ctx, g, P, cams),
        "saved": saved,
        "loss": lambda: gs.gs_loss(ctx, cams, torch.zeros(3 * 1024), torch.zeros(1024), torch.zeros(3 * 1024),
                                   torch.zeros(1024)),
        "register": lambda: gs.gs_register(ctx, g, g, [view], [view], 2),
        "batch": lambda: gs.gs_register_batch(ctx, [(g, g, [view], [view])], 2),
        "overlap": lambda: gs.gs_overlap_ratio(ctx, few, few, np.eye(3, 4)),
        "transform": lambda: gs.gs_transform(ctx, g, np.eye(3, 4)),
        "transform_batch": lambda: gs.gs_transform_batch(ctx, [g, g], np.stack([np.eye(3, 4)] * 2)),
    }


@pytest.mark.parametrize("name", ["render", "saved", "loss", "register", "batch", "overlap", "transform",
                                  "transform_batch"])
def test_a_refused_launch_is_reported(fake, name):
    # every launch of a call in turn, on a first call and on the later ones
    # of a context (which take what the first left)
    gs, rt = fake
    for warm in (0, 2):
        n = 0
        while True:
            ctx = gs.Context(0)
            call = calls(gs, ctx)[name]
            for _ in range(warm):
                call()
            rt.fake_refuse(n)
            try:
                call()
                reported = False
            except gs.GsError as e:
                reported = True
                assert e.status == 3, e  # GS_ERR_CUDA
            launched = rt.fake_launches()
            rt.fake_refuse(-1)
            ctx.close()
            if launched <= n:
                break
            assert reported, (warm, n)
            n += 1
        assert n > 0 and not reported


def test_counting_grids_are_cleared_behind_a_refused_launch(fake):
    # a repeated render clears nothing (each list build leaves the counting
    # grids clear), but the one behind a call whose list build was refused does
    gs, rt = fake
    ctx = gs.Context(0)
    render = calls(gs, ctx)["render"]

    def memsets():
        before = rt.fake_memsets()
        render()
        return rt.fake_memsets() - before

    memsets()
    usual = memsets()
    for n in (2, 3):  # tables, projection, then the ranges and the placement
        rt.fake_refuse(n)
        with pytest.raises(gs.GsError):
            render()
        rt.fake_refuse(-1)
        assert memsets() == usual + 1
        assert memsets() == usual
    ctx.close()


def train(gs, ctx, adjoint=True):
    g, P, cams, _ = scene(gs)
    _, sv = gs.gs_render_saved(ctx, g, P, cams)
    try:
        if adjoint:
            gs.gs_render_backward_saved(ctx, sv, params=True)
    finally:
        sv.close()


def test_a_repeated_training_step_fits_the_first_ones_budget(fake):
    # the lists of a repeated pass are sized by a guess; its adjoint's slots
    # are those of the duplicates it has
    gs, rt = fake
    rt.fake_dups(400_000)

    def passes(budget, times):
        ctx = gs.Context(0, budget)
        try:
            for _ in range(times):
                train(gs, ctx)
            return True
        except gs.GsError as e:
            assert e.status == 2, e  # GS_ERR_OOM
            return False
        finally:
            ctx.close()

    lo, hi = 1 << 16, 1 << 28
    assert not passes(lo, 1) and passes(hi, 1)
    while hi - lo > 256:
        mid = (lo + hi) // 2
        lo, hi = (lo, mid) if passes(mid, 1) else (mid, hi)
    assert passes(hi, 3)


def test_a_pass_with_many_duplicates_does_not_inflate_later_ones(fake):
    gs, rt = fake

    def after(dups):
        """scratch of the adjoint, and bytes of the saved forward, of a pass
        with 100,000 duplicates behind passes with dups of them"""
        ctx = gs.Context(0)
        for d in dups:
            rt.fake_dups(d)
            train(gs, ctx, adjoint=False)
        rt.fake_dups(100_000)
        g, P, cams, _ = scene(gs)
        before, pool = ctx.bytes(), rt.fake_pool_bytes()
        _, sv = gs.gs_render_saved(ctx, g, P, cams)
        pool = rt.fake_pool_bytes() - pool
        lists = ctx.bytes()
        gs.gs_render_backward_saved(ctx, sv, params=True)
        scratch = ctx.bytes() - lists
        assert lists == before or not dups
        sv.close()
        ctx.close()
        return scratch, pool

    alone = after([])
    many = after([3_000_000, 3_000_000])
    assert many[0] == alone[0]
    # (a block that is at most half as long again, and 64 Ki entries, is kept)
    assert many[1] <= alone[1] + 4 * (50_000 + 65_536)


@pytest.mark.parametrize("n", [1, 2, 4, 8, 24])
def test_transform_batch_marshalling_cost(fake, n):
    # the host time of a call on a few maps, against the same call through
    # one ctypes array per argument (best of many, in turn)
    gs, rt = fake
    ctx = gs.Context(0)
    maps, Ts = [scene(gs, 8)[0] for _ in range(n)], np.stack([np.eye(3, 4)] * n)

    def plain():
        arr = (gs.gs_gaussians_t * n)(*[g.c_struct() for g in maps])
        Th = np.ascontiguousarray(np.asarray(Ts, np.float64).reshape(n, 12))
        outs = [(torch.empty_like(g.means4), torch.empty_like(g.quats4)) for g in maps]
        om = (ctypes.c_void_p * n)(*[m.data_ptr() for m, _ in outs])
        oq = (ctypes.c_void_p * n)(*[q.data_ptr() for _, q in outs])
        ctx.check(rt.gs_transform_batch(ctx.handle, arr, n, Th.ctypes.data_as(ctypes.c_void_p), om, oq, None))
        return [gs.Gaussians(m, g.log_scales4, q, g.logits, g.rgb4) for g, (m, q) in zip(maps, outs)]

    def best(f):
        t = time.perf_counter()
        for _ in range(20):
            f()
        return time.perf_counter() - t

    times = [(best(lambda: gs.gs_transform_batch(ctx, maps, Ts)), best(plain)) for _ in range(60)]
    ctx.close()
    assert min(t for t, _ in times) <= 1.1 * min(t for _, t in times)
