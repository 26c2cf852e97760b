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


class ProgramPool:
    """A memory pool of the program's own, current for device 0 meanwhile."""

    USED_NOW = 7                                    # CU_MEMPOOL_ATTR_USED_MEM_CURRENT

    def __init__(self, max_bytes=0):
        self.cu = C.CDLL("libcuda.so.1")
        self.max_bytes = max_bytes

    def _ok(self, rc):
        assert rc == 0, rc

    def __enter__(self):
        class Props(C.Structure):                   # CUmemPoolProps
            _fields_ = [("alloc_type", C.c_int), ("handle_types", C.c_int), ("loc_type", C.c_int), ("loc_id", C.c_int),
                        ("security", C.c_void_p), ("max_size", C.c_size_t), ("usage", C.c_ushort),
                        ("reserved", C.c_ubyte * 54)]
        p = Props(alloc_type=1, loc_type=1, loc_id=0, max_size=self.max_bytes)      # pinned, on the device
        self.pool, self.default = C.c_void_p(), C.c_void_p()
        self._ok(self.cu.cuDeviceGetDefaultMemPool(C.byref(self.default), 0))
        self._ok(self.cu.cuMemPoolCreate(C.byref(self.pool), C.byref(p)))
        self._ok(self.cu.cuDeviceSetMemPool(0, self.pool))
        return self

    def used(self):
        v = C.c_uint64()
        self._ok(self.cu.cuMemPoolGetAttribute(self.pool, self.USED_NOW, C.byref(v)))
        return v.value

    def __exit__(self, *a):
        self._ok(self.cu.cuDeviceSetMemPool(0, self.default))
        self._ok(self.cu.cuMemPoolDestroy(self.pool))


@pytest.mark.parametrize("first", ["context", "pool"])
def test_the_programs_own_pool_is_used(env, first):
    torch, m = env
    sp = scenes.blobs_small(0)
    cam = scenes.nadir_camera(sp, 16, 16)
    before = m.Context(0) if first == "context" else None
    with ProgramPool() as pool:
        ctx = before or m.Context(0)
        sc = m.Scene.from_spec(ctx, sp)
        assert pool.used() >= sp.k.nbytes
        assert m.mcrt_debug_pool_usage(ctx.h)[0] == pool.used()
        want = sc.trace_camera(cam, 4, seed=1).mean
        sc.close()
        assert pool.used() == 0
    sc = m.Scene.from_spec(ctx, sp)
    np.testing.assert_allclose(sc.trace_camera(cam, 4, seed=1).mean, want, rtol=1e-12, atol=0)
    sc.close()
    ctx.close()


def test_the_programs_bound_holds(env):
    torch, m = env
    with ProgramPool(max_bytes=64 << 20), m.Context(0) as ctx:
        k = torch.ones((128, 512, 512), device="cuda")
        with pytest.raises(m.McrtError) as e:
            m.Scene(ctx, k, 0.1, 0.1, 0.1)
        assert e.value.status == m.MCRT_ERR_OOM
        m.Scene(ctx, k[:8, :64, :64], 0.1, 0.1, 0.1).close()


def test_kept_memory_is_given_back_on_request(env):
    torch, m = env
    with m.Context(0) as ctx:
        sc = m.Scene.from_spec(ctx, scenes.blobs_small(0))
        with Held(env, ctx) as held:
            m.Scene(ctx, torch.zeros((512, 1024, 1024), device="cuda"), 0.1, 0.1, 0.1, levels=1).close()
            torch.cuda.empty_cache()
            kept = torch.cuda.mem_get_info()[0]
            ctx.trim_memory()
            given = torch.cuda.mem_get_info()[0] - kept
        assert given >= 2 << 30
        assert held.unused <= SLACK
        assert sc.trace_flux(1000, seed=1).mean[0] > 0.0      # (what is in use stays)
        sc.close()
