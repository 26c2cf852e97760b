"""Sun rays taken over by idle lanes, in the variants where most can go wrong:
the learned passes (an owner that stops at a learned vertex waits for its
helpers), Rayleigh clear air and BF16 voxels.  A path's score is the same sum
whatever lane traced its sun rays."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu

ONE_WARP = dict(grid_size=1, block_size=32, chunk=1)


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
    f32 = m.Scene.from_spec(ctx, sp)
    bf16 = m.Scene.from_spec(ctx, sp, storage=m.MCRT_STORAGE_BF16)
    air = m.Scene.from_spec(ctx, sp)
    m.mcrt_scene_set_clear_sky_phase(ctx.h, air.h, m.MCRT_PHASE_RAYLEIGH)
    prop = m.Proposal(ctx, seed=3)
    for sc in (f32, bf16, air):
        sc.build_octree()
    yield m, sp, dict(f32=f32, bf16=bf16, rayleigh=air), prop
    for o in (f32, bf16, air, prop):
        o.close()
    ctx.close()


def _same(a, b):
    # FP64 sums of at most 2^17 FP32 scores in another order: 2^17 2^-53 < 2e-11
    np.testing.assert_allclose(a.mean, b.mean, rtol=2e-11, atol=1e-15)


@pytest.mark.parametrize("opts", [dict(), dict(grid=1, finest_level=1), dict(sun_mode=1)],
                         ids=["pyramid", "merged", "delta"])
@pytest.mark.parametrize("scene", ["bf16", "rayleigh"])
@pytest.mark.parametrize("n", [1, 33, 4865])
def test_fluxes_score_the_same(env, n, scene, opts):
    m, sp, scs, prop = env
    _same(scs[scene].trace_flux(n, seed=5, chunk=1, **opts), scs[scene].trace_flux(n, seed=5, **ONE_WARP, **opts))


@pytest.mark.parametrize("scene", ["f32", "bf16"])
@pytest.mark.parametrize("learned", [1, 3, 8])
@pytest.mark.parametrize("n", [1, 33, 4865])
def test_learned_fluxes_score_the_same(env, n, learned, scene):
    m, sp, scs, prop = env
    kw = dict(seed=6, proposal=prop, n_learned=learned)
    _same(scs[scene].trace_flux(n, chunk=1, **kw), scs[scene].trace_flux(n, **ONE_WARP, **kw))


@pytest.mark.parametrize("scene", ["f32", "bf16", "rayleigh"])
def test_images_score_the_same(env, scene):
    m, sp, scs, prop = env
    cam = scenes.nadir_camera(sp, 37, 21)
    kw = dict(seed=7) if scene == "rayleigh" else dict(seed=7, proposal=prop, n_learned=4)
    _same(scs[scene].trace_camera(cam, 3, chunk=1, **kw), scs[scene].trace_camera(cam, 3, **ONE_WARP, **kw))
