"""Tile lists of caller-made records (gs_bin) against numpy: list lengths
around the hand-overs of the per-tile sort (registers, shared memory, chunks
merged in global memory) and frames around those of the list ranges (rows
wider than a warp, more rows than threads, grids in shared or in global
memory).  Keys, values, ranges and counts are exact."""
import numpy as np
import pytest

from paper_2408_10154_gb300 import synth

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def env():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_2408_10154_gb300 as gs
    from paper_2408_10154_gb300 import build
    build.build()
    c = gs.Context(0)
    yield gs, c
    c.close()


def check(env, cams, n, rects, z):
    """rects [cams * n, 4] tile rectangles (x0, x1, y0, y1; empty: x0 == x1)."""
    gs, ctx = env
    rec = np.zeros((len(rects), 12), np.float32)
    rec[:, 6] = z
    bits = rec.view(np.uint32)
    x0, x1, y0, y1 = [rects[:, k].astype(np.uint32) for k in range(4)]
    bits[:, 7], bits[:, 11] = x0 | (x1 << 16), y0 | (y1 << 16)
    cnt = ((x1 - x0) * (y1 - y0)).astype(np.int32)
    keys, vals, ranges = gs.gs_bin(ctx, torch.tensor(rec).cuda(), torch.tensor(cnt).cuda(), cams, n)
    tiles, base = [], 0
    for k, cam in enumerate(np.asarray(cams)):
        TX, TY = (int(cam[4]) + 15) // 16, (int(cam[5]) + 15) // 16
        for r in range(k * n, (k + 1) * n):
            if cnt[r]:
                ys, xs = np.meshgrid(np.arange(y0[r], y1[r]), np.arange(x0[r], x1[r]), indexing="ij")
                t = base + (ys * TX + xs).reshape(-1)
                tiles.append(np.stack([t, np.full(len(t), r)], 1))
        base += TX * TY
    tr = np.concatenate(tiles).astype(np.int64) if tiles else np.zeros((0, 2), np.int64)
    zb = bits[:, 6][tr[:, 1]].astype(np.int64)
    order = np.lexsort((tr[:, 1], zb, tr[:, 0]))
    tr, zb = tr[order], zb[order]
    np.testing.assert_array_equal(keys.cpu().numpy(), (tr[:, 0] << 32) | zb)
    np.testing.assert_array_equal(vals.cpu().numpy(), tr[:, 1].astype(np.int32))
    lens = np.bincount(tr[:, 0], minlength=base)
    end = np.cumsum(lens)
    want = np.where(lens[:, None] > 0, np.stack([end - lens, end], 1), 0)
    np.testing.assert_array_equal(ranges.cpu().numpy(), want)


@pytest.mark.parametrize("n", [1, 2, 33, 129, 256, 257, 511, 513, 1024, 4095, 4096, 4097, 8193, 20000])
def test_list_lengths(env, n):
    # two tiles hold every record, two more half of them; depths with ties
    rng = np.random.default_rng(n)
    cams = np.stack([synth.camera(30.0, 30.0, 32.0, 8.0, 64, 16, np.eye(3, 4))])
    rects = np.tile([0, 2, 0, 1], (n, 1))
    rects[rng.random(n) < 0.5, 1] = 4
    check(env, cams, n, rects, np.round(rng.uniform(0.3, 5.0, n), 2))


@pytest.mark.parametrize("sizes", [[(16, 16)], [(500, 20), (1, 1), (513, 300)], [(32, 9000)], [(520, 9000), (40, 40)],
                                   [(1200, 680), (1199, 681)]])
def test_frame_shapes(env, sizes):
    rng = np.random.default_rng(sum(w + h for w, h in sizes))
    n = 400
    cams = np.stack([synth.camera(50.0, 50.0, w / 2, h / 2, w, h, np.eye(3, 4)) for w, h in sizes])
    rects = []
    for w, h in sizes:
        TX, TY = (w + 15) // 16, (h + 15) // 16
        a, b = rng.integers(0, TX + 1, (n, 2)), rng.integers(0, TY + 1, (n, 2))
        small = rng.random(n) < 0.9  # most cover a few tiles, some the frame
        a[small, 1] = np.minimum(a[small, 0] + rng.integers(0, 3, small.sum()), TX)
        b[small, 1] = np.minimum(b[small, 0] + rng.integers(0, 3, small.sum()), TY)
        r = np.concatenate([np.sort(a, 1), np.sort(b, 1)], 1)
        r[(r[:, 0] == r[:, 1]) | (r[:, 2] == r[:, 3])] = 0
        rects.append(r)
    check(env, cams, n, np.concatenate(rects), rng.uniform(0.3, 5.0, n * len(sizes)).astype(np.float32))


@pytest.mark.parametrize("n,large", [(1, 1.0), (3, 1.0), (257, 0.5), (300, 1.0), (2000, 0.05), (311_297, 0.002)])
def test_records_of_many_tiles(env, n, large):
    # records of more than four tiles share their block's threads: none, one
    # and all of a block, runs around 1,024 tiles, one and two records a thread
    rng = np.random.default_rng(n)
    w, h = 16 * 33, 16 * 32
    cams = np.stack([synth.camera(50.0, 50.0, w / 2, h / 2, w, h, np.eye(3, 4))])
    x, y = rng.integers(0, 33, n), rng.integers(0, 32, n)
    rects = np.stack([x, np.minimum(x + rng.integers(1, 3, n), 33), y, np.minimum(y + rng.integers(1, 3, n), 32)], 1)
    big = np.flatnonzero(rng.random(n) < large)
    rects[big, 0], rects[big, 2] = rng.integers(0, 2, (2, len(big)))
    rects[big, 1], rects[big, 3] = rng.integers(7, 34, len(big)), rng.integers(2, 33, len(big))
    rects[big, 3] = np.maximum(rects[big, 3], rects[big, 2] + 1)
    rects[big[::3]] = [0, 33, 0, 32]
    check(env, cams, n, rects, np.round(rng.uniform(0.3, 5.0, n), 3))
