"""Reading a tally into arrays that nothing has touched yet."""
import time

import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("w,h", [(1, 1), (33, 31), (32, 32), (41, 25), (64, 48)])
@pytest.mark.parametrize("want", ["both", "mean", "se"])
def test_mean_and_error_are_those_of_the_sums(w, h, want):
    # 1,023, 1,024 and 1,025 entries: a small tally's one copy and a large one's two
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import ctypes as C
    import paper_1902_01137_gb300 as m
    from paper_1902_01137_gb300 import build
    build.build()
    sp = scenes.blobs_small(0)
    cam, cd = scenes.nadir_camera(sp, w, h), m.CameraDesc()
    for i in range(3):
        cd.pos[i], cd.target[i], cd.up[i] = cam.pos[i], cam.target[i], cam.up[i]
    cd.fov_deg, cd.width, cd.height = cam.fov_deg, w, h
    n = w * h
    with m.Context(0) as ctx:
        sc = m.Scene.from_spec(ctx, sp)
        t = m.mcrt_trace_camera(ctx.h, sc.h, cd, 4, 1, m.mcrt_trace_opts_default())
        s1, s2 = (a.ravel() / 4.0 for a in m.mcrt_tally_read_sums(ctx.h, t))
        mean, se = np.full(n + 1, -7.0), np.full(n + 1, -7.0)       # (nothing behind the last entry is written)
        P = C.POINTER(C.c_double)
        a = mean.ctypes.data_as(P) if want != "se" else None
        b = se.ctypes.data_as(P) if want != "mean" else None
        assert m.lib().mcrt_tally_read(t, a, b, None, n) == 0
        m.mcrt_tally_destroy(t)
        sc.close()
    if a:
        np.testing.assert_array_equal(mean[:n], s1)
    if b:     # the variance cancels s2 / n and mean^2: a few roundings of those
        var = np.maximum(s2 - s1 * s1, 0.0) / 3.0
        np.testing.assert_allclose(se[:n] ** 2, var, rtol=1e-12, atol=1e-15 * max(s2.max(), 1e-300))
    assert mean[n] == -7.0 and se[n] == -7.0 and (a or (mean == -7.0).all()) and (b or (se == -7.0).all())


def test_new_arrays_are_read_as_fast_as_used_ones():
    """Every read makes new arrays of 8 MB, as a program's does.  A copy that
    faults their pages in from the device takes 7 to 14 ms, one to pages that
    are there 0.2 ms, and bringing them in 0.5 ms: three of four reads must stay
    under 5 ms."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_01137_gb300 as m
    from paper_1902_01137_gb300 import build
    build.build()
    sp = scenes.blobs_small(0)
    cam, cd = scenes.nadir_camera(sp, 1024, 1024), m.CameraDesc()
    for i in range(3):
        cd.pos[i], cd.target[i], cd.up[i] = cam.pos[i], cam.target[i], cam.up[i]
    cd.fov_deg, cd.width, cd.height = cam.fov_deg, cam.width, cam.height
    with m.Context(0) as ctx:
        sc = m.Scene.from_spec(ctx, sp)
        t = m.mcrt_trace_camera(ctx.h, sc.h, cd, 1, 1, m.mcrt_trace_opts_default())
        took, first = [], None
        for _ in range(24):
            start = time.perf_counter()
            mean, se, n = m.mcrt_tally_read(ctx.h, t)
            took.append(time.perf_counter() - start)
            first = mean.copy() if first is None else first
            np.testing.assert_array_equal(mean, first)
        s1, _ = m.mcrt_tally_read_sums(ctx.h, t)
        np.testing.assert_array_equal(first.ravel(), s1.ravel())       # (one path a pixel)
        m.mcrt_tally_destroy(t)
        sc.close()
    assert sorted(took)[17] < 5e-3, took
