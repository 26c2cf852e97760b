"""How soon a trace answers its cancel flag and its deadline."""
import ctypes as C

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_every_variant_looks_at_the_flag_after_the_same_steps():
    """A warp looks at the flag every 1024 traversal steps, however many steps
    its variant takes between votes.  One warp crosses a field of voxel leaves
    with next to no extinction (every path: a sun ray and a flight, some 250
    steps, transmissivity 1), the flag raised from the start: the paths ended by
    the first look, sum T_dir, show the steps taken.  Decomposition tracking
    takes one step a vote, the plain variant two; waiting for a pass and odd
    last steps cost at most one step a ray, a tenth is more than both."""
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_01137_gb300 as m
    from paper_1902_01137_gb300 import build
    build.build()
    flag = torch.ones(1, dtype=torch.int32).pin_memory()
    with m.Context(0) as ctx:
        sc = m.Scene(ctx, np.full((64, 32, 32), 1e-7, np.float32), 0.1, 0.1, 0.1, levels=2)
        ended = {}
        for mode in (m.MCRT_SUN_RATIO, m.MCRT_SUN_DECOMP):
            o = m.Scene._opts(sun_mode=mode, tau_merge=0.0, grid_size=1, block_size=32, chunk=1, rare_batch=1,
                              cancel_flag=flag.data_ptr())
            t = C.c_void_p()
            assert m.lib().mcrt_trace_flux(sc.h, 4096, 3, C.byref(o), C.byref(t)) == m.MCRT_ERR_CANCELLED
            ended[mode] = m.mcrt_tally_read_sums(ctx.h, t)[0][0, 0]
            m.mcrt_tally_destroy(t)
        sc.close()
    a, b = ended[m.MCRT_SUN_RATIO], ended[m.MCRT_SUN_DECOMP]
    assert 32 <= b < 4096
    assert 0.9 * b <= a <= 1.1 * b, (a, b)
