"""Device memory after a call: the library keeps at most 4 GiB that nothing
uses, whatever the call and however it ended; it gives all of it back on
request; and it allocates from the program's own pool where the program set
one for the device."""
import ctypes as C

import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu

KEEP = 4 << 30
SLACK = 64 << 20       # kernels loaded meanwhile, the pool's 32 MiB blocks


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_01137_gb300 as m
    from paper_1902_01137_gb300 import build
    build.build()
    yield torch, m
    torch.cuda.empty_cache()


class Held:
    """Device memory that a block of calls took and nothing uses."""

    def __init__(self, env, ctx):
        self.torch, self.m = env
        self.ctx = ctx

    def _now(self):
        used, _ = self.m.mcrt_debug_pool_usage(self.ctx.h)
        return self.torch.cuda.mem_get_info()[0] + used

    def __enter__(self):
        self.before = self._now()
        return self

    def __exit__(self, *a):
        self.unused = self.before - self._now()


def _camera(m, sp, w, h):
    cam, cd = scenes.nadir_camera(sp, w, h), m.CameraDesc()
    for i in range(3):
        cd.pos[i], cd.target[i], cd.up[i] = cam.pos[i], cam.target[i], cam.up[i]
    cd.fov_deg, cd.width, cd.height = cam.fov_deg, w, h
    return cd


def test_wavefront_queues_are_given_back(env):
    torch, m = env
    sp = scenes.homogeneous(8, 8, 8, 0.1, 0.01)
    with m.Context(0) as ctx:
        sc = m.Scene.from_spec(ctx, sp)
        with Held(env, ctx) as held:
            t = m.mcrt_trace_camera(ctx.h, sc.h, _camera(m, sp, 4096, 2048), 4, 1,
                                    m.Scene._opts(schedule=m.MCRT_SCHEDULE_WAVEFRONT, wavefront_slots=1 << 25))
        m.mcrt_tally_destroy(t)
        sc.close()
    assert held.unused <= KEEP + SLACK


def test_a_stopped_learned_trace_gives_its_queues_back(env):
    torch, m = env
    sp = scenes.blobs_small(0)
    flag = torch.ones(1, dtype=torch.int32).pin_memory()
    with m.Context(0) as ctx:
        sc, prop, t = m.Scene.from_spec(ctx, sp), m.Proposal(ctx, seed=1), C.c_void_p()
        with Held(env, ctx) as held:
            o = m.Scene._opts(proposal=prop, cancel_flag=flag.data_ptr())
            cd = _camera(m, sp, 2048, 1024)
            assert m.lib().mcrt_trace_camera(sc.h, C.byref(cd), 16, 1, C.byref(o), C.byref(t)) == m.MCRT_ERR_CANCELLED
        m.mcrt_tally_destroy(t)
        prop.close()
        sc.close()
    assert held.unused <= KEEP + SLACK


def test_network_workspaces_are_given_back(env):
    torch, m = env
    with m.Context(0) as ctx:
        prop = m.Proposal(ctx, seed=1)
        with Held(env, ctx) as held:
            prop.eval(np.zeros((14_000_000, 9), np.float32))          # 388 bytes a row
        prop.close()
    assert held.unused <= KEEP + SLACK


def test_the_staging_copy_of_a_host_field_is_given_back(env):
    torch, m = env
    with m.Context(0) as ctx:
        with Held(env, ctx) as held:
            sc = m.Scene(ctx, np.zeros((640, 1536, 1408), np.float32), 0.1, 0.1, 0.1, storage=m.MCRT_STORAGE_BF16,
                         levels=1)                                    # 5.5 GB staged
        sc.close()
    assert held.unused <= KEEP + SLACK


def test_replaced_heightfields_are_given_back(env):
    torch, m = env
    heights = torch.zeros((16384, 16384), dtype=torch.float32, device="cuda")
    with m.Context(0) as ctx:
        sc = m.Scene.from_spec(ctx, scenes.homogeneous(8, 8, 8, 0.1, 0.01))
        sc.set_heightfield(heights[:4, :4].contiguous(), 0.1)         # (loads the kernels)
        with Held(env, ctx) as held:
            sc.set_heightfield(heights, 0.1)
            sc.set_heightfield(heights, 0.2)
            m.mcrt_scene_set_ground_flat(ctx.h, sc.h, 0.1)
        sc.close()
    assert held.unused <= KEEP + SLACK
