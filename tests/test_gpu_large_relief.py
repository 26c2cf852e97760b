"""Reliefs of more than 2^28 cells are kept as plain heights, 4 bytes a cell."""
import numpy as np
import pytest

import scenes

pytestmark = pytest.mark.gpu

NX, NY, L = 16388, 16384, 6.4        # 2^28 + 2^16 cells
SLOPE = 0.15 * 2.0 * np.pi * 3.0 / L * 2.0


@pytest.fixture(scope="module")
def relief():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1902_01137_gb300 as m
    from paper_1902_01137_gb300 import build
    build.build()
    x = torch.arange(NX, device="cuda", dtype=torch.float64) / NX * 6.0 * np.pi
    y = torch.arange(NY, device="cuda", dtype=torch.float64) / NY * 6.0 * np.pi
    h = (0.2 + 0.15 * torch.sin(x)[None, :] * torch.cos(y)[:, None]).to(torch.float32).contiguous()
    ctx = m.Context(0)
    sc = m.Scene.from_spec(ctx, scenes.blobs_small(0))
    used = m.mcrt_debug_pool_usage(ctx.h)[0]
    sc.set_heightfield(h, 0.3)
    yield h, sc, m.mcrt_debug_pool_usage(ctx.h)[0] - used
    sc.close()
    ctx.close()
    del h
    torch.cuda.empty_cache()


def test_memory(relief):
    h, sc, used = relief
    assert 4 * h.numel() <= used <= 4.3 * h.numel() + (1 << 20)      # and 1/16 + 1/256 + ... of maxima


def _surface(h, xy):
    fx, fy = xy[:, 0].astype(np.float64) / L * NX, xy[:, 1].astype(np.float64) / L * NY
    i, j = np.floor(fx).astype(int), np.floor(fy).astype(int)
    u, v = fx - i, fy - j
    at = lambda a, b: h[b % NY, a % NX].double().cpu().numpy()
    h00, h10, h01, h11 = at(i, j), at(i + 1, j), at(i, j + 1), at(i + 1, j + 1)
    return np.where(u >= v, h00 + (h10 - h00) * u + (h11 - h10) * v, h00 + (h11 - h01) * u + (h01 - h00) * v)


def test_heights(relief):
    h, sc, used = relief
    r = np.random.default_rng(1)
    edge = np.nextafter(np.float32(L), np.float32(0))
    xy = np.concatenate([r.uniform(0, L, (2000, 2)), [[0, 0], [edge, 0], [0, edge], [edge, edge]]]).astype(np.float32)
    got = sc.terrain_height(xy)[0]
    # FP32 cell coordinates: 2^-24 of x and of 1 / cell, on the steepest slope; heights to 2^-25
    np.testing.assert_allclose(got, _surface(h, xy), rtol=0, atol=SLOPE * L * 2.0 ** -22 + 2.0 ** -24)


def test_rays(relief):
    # down the vertical, and slanted from above: the hit lies on the surface and nothing before it does
    h, sc, used = relief
    r = np.random.default_rng(2)
    n = 400
    o = np.column_stack([r.uniform(0, L, (n, 2)), np.full(n, 1.0)]).astype(np.float32)
    d = np.column_stack([r.uniform(-2, 2, (n, 2)), np.full(n, -1.0)])
    d[: n // 2, :2] = 0.0
    d = (d / np.linalg.norm(d, axis=1)[:, None]).astype(np.float32)
    t = np.asarray(sc.terrain_hit(o, d), np.float64)
    assert np.isfinite(t).all()
    tol = 4.0 * SLOPE * L * 2.0 ** -22 + 2.0 ** -22          # coordinates up to 2 L, twice over
    for s in np.linspace(0.0, 1.0, 200):
        p = o + (s * t)[:, None] * d
        above = p[:, 2] - _surface(h, np.mod(p[:, :2], L))
        assert (above > -tol).all(), s
    assert (np.abs(above) < tol).all()
