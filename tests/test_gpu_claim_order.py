"""Claim order of camera traces: costly tiles first, ties in raster order, and
the same paths whatever the order.  Shard r of c traces the pixels at positions
r, r + c, ... of the order, so one shard per pixel reads the order back."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_01137_gb300 as m
    from paper_1902_01137_gb300 import build
    build.build()
    ctx = m.Context(0)
    yield m, ctx
    ctx.close()


def test_costly_pixels_first_traces_the_same_paths(env):
    # one warp, so the launch has fewer lanes than paths and is given an order;
    # eight paths a pixel, an oblique camera, tiles cut at the edges
    m, ctx = env
    sp = scenes.blobs_small(0)
    sc = m.Scene.from_spec(ctx, sp)
    for cam in (scenes.nadir_camera(sp, 37, 21),
                scenes.CameraSpec((1.0, -4.0, 6.0), (3.2, 3.2, 0.8), (0.0, 0.0, 1.0), 50.0, 45, 30)):
        for kw in (dict(), dict(count_events=1)):
            kw.update(seed=5, grid_size=1, block_size=32)
            a = sc.trace_camera(cam, 8, **kw)
            b = sc.trace_camera(cam, 8, pixel_order=m.MCRT_ORDER_RASTER, **kw)
            np.testing.assert_allclose(a.mean, b.mean, rtol=1e-12, atol=0)
            np.testing.assert_allclose(a.se, b.se, rtol=1e-9, atol=1e-15)
            for k in ("paths", "tentative", "real", "ground", "leaf_steps", "sun_tentative", "sun_rays"):
                assert a.counters.get(k) == b.counters.get(k), k
    sc.close()


def _pixels_at(sc, cam, ranks):
    """The pixel at each of these positions of the claim order."""
    out = []
    for r in ranks:
        mean = sc.trace_camera(cam, 64, seed=1, shard_index=int(r), shard_count=cam.width * cam.height).mean
        y, x = np.nonzero(mean)
        assert len(y) == 1
        out.append((int(y[0]), int(x[0])))
    return out


@pytest.mark.parametrize("tx,ty", [(1, 1), (2, 1), (5, 3), (9, 7), (128, 128)])
def test_tiles_are_sorted_by_cost(env, tx, ty):
    """One voxel column behind each tile of 8 x 8 pixels, seen from so far up
    that its rays stay in it: a tile's cost is its column's extinction (two
    neighbours in the order differ by 5e-5 or more, their rays' lengths by FP32
    rounding).  Half of the columns are empty: equal costs, in raster order."""
    m, ctx = env
    n = tx * ty
    r = np.random.default_rng(n)
    k = np.where(r.uniform(size=n) < 0.5, 0.1 + 0.8 * r.permutation(n) / n, 0.0).astype(np.float32).reshape(ty, tx)
    sc = m.Scene(ctx, np.repeat(k[None], 2, axis=0), 1.0, 1.0, 1.0, levels=1, albedo=0.9)
    far = 1e4 * max(tx, ty)
    cam = scenes.CameraSpec((0.5 * tx, 0.5 * ty, 2.0 + far), (0.5 * tx, 0.5 * ty, 0.0), (0.0, 1.0, 0.0),
                            2.0 * np.degrees(np.arctan(0.5 * tx / (far + 1.0))), 8 * tx, 8 * ty)
    ranks = np.arange(n) if n < 100 else np.unique(np.concatenate([[0, 1, n - 2, n - 1], r.integers(0, n, 60)]))
    got = [(y // 8, x // 8) for y, x in _pixels_at(sc, cam, 64 * ranks)]
    sc.close()
    order = sorted(range(n), key=lambda t: (-float(k[t // tx, t % tx]), t))
    assert got == [(order[q] // tx, order[q] % tx) for q in ranks]
