"""A detector whose default tiles make more segments than the allocation-free entry point takes: larger
tiles are built, and where there is no memory to count or to build them the build keeps the default
ones instead of failing."""
import pytest
import torch

from gpu_common import api, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]

NY = NX = 3456
MOST = (8 << 20) // 24


def _build():
    geo = api().Geometry(0.2, 0.47 * NY * 75e-6, 0.52 * NX * 75e-6, 0.01, -0.02, 0.3, 75e-6, 75e-6)
    return api().Integrator.build(geo, (NY, NX), 1950, 0, "q_nm^-1", "full")


def test_larger_tiles_or_the_default_ones():
    g = _build()
    guarded = (g.info["tile_h"], g.info["tile_w"], g.info["n_segments"])
    assert guarded[:2] == (16, 64)
    img = torch.ones((NY, NX), dtype=torch.int32, device="cuda")
    ref = g.integrate(img, precision="fp64")
    g.set_tuning(8, 120)
    assert g.info["n_segments"] > 2 * MOST >= guarded[2]
    kept = failed = 0
    try:
        for after in range(24):
            api().selftest_alloc(after, 1)
            try:
                h = _build()
            except api().AzError as e:
                assert e.code == -3
                failed += 1
                continue
            finally:
                api().selftest_alloc()
            tile = (h.info["tile_h"], h.info["tile_w"])
            assert tile in ((8, 120), (16, 64), (8, 64))
            kept += tile == (8, 120)
            out = h.integrate(img, precision="fp64")
            assert float((out.sum_signal - ref.sum_signal).abs().max() / ref.sum_signal.abs().max()) <= 1e-13
    finally:
        api().selftest_alloc()
    assert kept >= 2 and failed >= 1  # counting or building the larger tiles; the matrix itself
