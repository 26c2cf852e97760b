"""Lanes without a path take over sun rays from other lanes of their warp,
and small launches spread their paths over the warps.  Neither may change a
result: every path's score is the same sum whatever lane traced its sun
rays.  Path counts sit at the edges of a warp and of one path per warp."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu

OPTS = {"ratio": {}, "delta": dict(sun_mode=1), "decomp": dict(sun_mode=2), "order3": dict(max_order=3),
        "octree": dict(grid=1, finest_level=1)}


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_01137_gb300 as m
    from paper_1902_01137_gb300 import build
    build.build()
    ctx = m.Context(0)
    sp = scenes.blobs_small(0)
    flat, hilly = m.Scene.from_spec(ctx, sp), m.Scene.from_spec(ctx, sp)
    hilly.set_heightfield(scenes.heightfield(128, 0.3, seed=1)[:96, :], sp.ground_albedo)
    for sc in (flat, hilly):
        sc.build_octree()
    yield m, ctx, sp, flat, hilly
    flat.close()
    hilly.close()
    ctx.close()


def _same(a, b):
    # FP64 sums of at most 2^17 FP32 scores in another order: 2^17 2^-53 < 2e-11
    np.testing.assert_allclose(a.mean, b.mean, rtol=2e-11, atol=1e-15)


@pytest.mark.parametrize("ground", ["flat", "hilly"])
@pytest.mark.parametrize("opts", sorted(OPTS))
@pytest.mark.parametrize("n", [1, 31, 33, 4865, 20000])
def test_helped_flux_paths_score_the_same(env, n, opts, ground):
    m, ctx, sp, flat, hilly = env
    sc = flat if ground == "flat" else hilly
    # one warp: full until its queue runs dry; every lane of every warp spread thin
    one = sc.trace_flux(n, seed=5, grid_size=1, block_size=32, chunk=1, **OPTS[opts])
    _same(sc.trace_flux(n, seed=5, chunk=1, **OPTS[opts]), one)


@pytest.mark.parametrize("shape", [(1, 1, 1), (7, 5, 3), (64, 48, 2)])
def test_helped_images_are_the_same(env, shape):
    m, ctx, sp, flat, hilly = env
    w, h, spp = shape
    cam = scenes.nadir_camera(sp, w, h)
    for sc in (flat, hilly):
        _same(sc.trace_camera(cam, spp, seed=6, chunk=1),
              sc.trace_camera(cam, spp, seed=6, grid_size=1, block_size=32, chunk=1))


@pytest.mark.parametrize("dalpha", [0, 1])
def test_helped_batch_items_are_the_same(env, dalpha):
    m, ctx, sp, flat, hilly = env
    items = [(flat, 0.0, 30.0, 0.0, 33, 1), (flat, 0.2, 70.0, 40.0, 2001, 2), (flat, 0.01, 10.0, 0.0, 1, 3)]
    _same(m.trace_batch(ctx, items, chunk=1, batch_dalpha=dalpha),
          m.trace_batch(ctx, items, chunk=1, grid_size=1, block_size=32, batch_dalpha=dalpha))


@pytest.mark.parametrize("size", [(8, 8), (9, 7), (37, 21), (1000, 8), (8200, 3), (1024, 1024), (1025, 1024)])
def test_claim_order_covers_the_image(env, size):
    # 1, 2 (one ragged), 15, 125, 1025 and 16,384 tiles are sorted on the device, more on the host;
    # a pixel left out or taken twice would change its sum
    m, ctx, sp, flat, hilly = env
    cam = scenes.nadir_camera(sp, *size)
    kw = dict(seed=7, chunk=1) if size[0] * size[1] > 200000 else dict(seed=7, chunk=1, grid_size=1, block_size=32)
    a = flat.trace_camera(cam, 1, pixel_order=m.MCRT_ORDER_COST, **kw)
    b = flat.trace_camera(cam, 1, pixel_order=m.MCRT_ORDER_RASTER, **kw)
    np.testing.assert_array_equal(a.mean, b.mean)


def test_heights_from_any_memory_are_the_same(env):
    # in place from device memory, through a copy from the host and from an address between floats
    import ctypes
    import torch
    m, ctx, sp, flat, hilly = env
    hh = np.ascontiguousarray(scenes.heightfield(64, 0.2, seed=2)[:48, :], dtype=np.float32)
    ny, nx = hh.shape
    raw = torch.zeros(hh.nbytes + 2, dtype=torch.uint8, device="cuda")
    raw[2:] = torch.from_numpy(hh.view(np.uint8).reshape(-1)).cuda()
    xy = np.random.default_rng(0).uniform(0, 3, (500, 2)).astype(np.float32)
    got = []
    for how in ("host", "device", "between"):
        sc = m.Scene.from_spec(ctx, sp)
        if how == "between":
            p = ctypes.c_void_p(raw.data_ptr() + 2)
            m._check(m._load().mcrt_scene_set_ground_heightfield(sc.h, p, nx, ny, m.MCRT_MEM_DEVICE, 0.1), ctx.h)
        else:
            sc.set_heightfield(hh if how == "host" else torch.from_numpy(hh).cuda(), 0.1)
        got.append(np.concatenate([np.ravel(a) for a in sc.terrain_height(xy)]))
        sc.close()
    np.testing.assert_array_equal(got[0], got[1])
    np.testing.assert_array_equal(got[0], got[2])
