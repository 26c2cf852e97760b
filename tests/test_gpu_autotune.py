"""The launch shapes that the batch autotuner tries."""
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
    sc = m.Scene.from_spec(ctx, scenes.blobs_small(0))
    sc.trace_flux(100, seed=1)                 # (its leaf map, a launch of its own)
    yield m, ctx, sc
    sc.close()
    ctx.close()


def _tuned(env, paths, fraction, **opts):
    m, ctx, sc = env
    items = m.make_batch_items([(sc, 0.0, 30.0, 0.0, paths, 1), (sc, 0.1, 60.0, 0.0, paths // 2, 2)])
    before = ctx.launches
    o, best = m.mcrt_autotune_batch(ctx.h, items, fraction, m.Scene._opts(**opts))
    assert best > 0.0
    return o, ctx.launches - before


def test_full_warps_are_tuned_around_the_default_wait(env):
    # 2 block sizes x 4 chunks x 4 waits, twice each (one launch a trace)
    o, launches = _tuned(env, 2_000_000, 1.0)
    assert launches == 2 * 32
    assert o.rare_batch in (12, 16, 20, 24) and o.chunk in (1, 2, 4, 8) and o.block_size in (64, 128)


def test_the_callers_own_shape_is_tried(env):
    o, launches = _tuned(env, 2_000_000, 1.0, grid_size=1000, block_size=96, rare_batch=18)
    assert launches == 2 * 33
    assert (o.grid_size, o.block_size, o.rare_batch) == (1000, 96, 18) or \
        (o.grid_size == 0 and o.block_size in (64, 128) and o.rare_batch in (12, 16, 20, 24))


def test_a_sample_too_thin_to_wait_keeps_the_default_wait(env):
    # a sample of some 3 paths a warp says nothing about the wait of the full batch
    o, launches = _tuned(env, 2_000_000, 0.004)
    assert launches == 2 * 8
    assert o.rare_batch == 16


def test_a_shape_no_trace_takes_is_passed_over(env):
    o, launches = _tuned(env, 2000, 1.0, block_size=256, rare_batch=40)
    assert launches == 2 * 8
    assert o.block_size in (64, 128) and o.rare_batch == 12
