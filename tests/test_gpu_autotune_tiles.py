"""The tiles that tuning times: the integrator's present one first, the default of its matrix, and the
smaller ones of dense matrices."""
import pytest

from gpu_common import api, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("npt,azim,default", [(300, 0, (8, 120)), (600, 0, (16, 64)), (1700, 0, (16, 40)), (4000, 0, (16, 24)), (90, 60, (48, 40))])
def test_present_and_default_tiles_are_timed(npt, azim, default):
    geo = api().Geometry(0.1, 0.47 * 512 * 75e-6, 0.52 * 512 * 75e-6, 0.01, -0.02, 0.3, 75e-6, 75e-6)
    g = api().Integrator.build(geo, (512, 512), npt, azim, "q_nm^-1", "full")
    assert (g.info["tile_h"], g.info["tile_w"]) == default
    tiles = g.autotune_tiles()
    assert tiles[0] == default and len(set(tiles)) == len(tiles)
    small, wide = {(16, 40), (16, 24), (8, 24), (8, 64)}, {(8, 152), (8, 224), (48, 40)}
    assert (small if npt >= 1700 else wide) <= set(tiles)
    g.set_tuning(20, 28)
    tiles = g.autotune_tiles()
    assert tiles[0] == (20, 28) and default in tiles
    ms = g.autotune(2)
    assert ms > 0 and (g.info["tile_h"], g.info["tile_w"]) in tiles
    assert g.status() == 0
