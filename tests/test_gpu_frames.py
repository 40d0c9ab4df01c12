"""The batched frames kernel: how a launch's frames are cut into stages (every class of frame
numbers, partial and empty stages, two launches), plane blocks of eight, four, two and one frames
(by tile size), long rows cut into pieces, heavy tiles cut into items, word phases.  Against the
cp.async engine's kernel (same entries, another kernel: the same bits) and the oracle."""
import numpy as np
import pytest
import torch

from gpu_common import Case, needs_gpu, rel_err, small_workload, to_dev

pytestmark = [pytest.mark.gpu, needs_gpu]

COUNTS = (1, 2, 3, 4, 5, 7, 9, 17, 24, 33, 37, 63, 64, 67)


def _check(c, tile, counts, frames_per_pass=8, off=0, other_kernel=True):
    g = c.gpu_from_oracle_positions()
    g.set_tuning(tile_h=tile[0], tile_w=tile[1], frames_per_pass=frames_per_pass)
    corr = c.corrections_dev()
    n, ny, nx = max(counts), c.w.ny, c.w.nx
    rng = np.random.default_rng(5)
    fr = rng.integers(0, 5000, size=(n, ny, nx)).astype(np.int32)
    buf = torch.zeros(fr.size + 4, dtype=torch.int32, device="cuda")
    buf[off:off + fr.size] = to_dev(fr).reshape(-1)
    fd = buf[off:off + fr.size].view(n, ny, nx)
    if other_kernel:  # (its stages hold three correction planes: not for the largest tiles)
        g.set_copy_engine("async")
    ref = g.integrate_batch(fd, *corr)
    g.set_copy_engine("tma")
    for k in counts:
        out = g.integrate_batch(fd[:k], *corr)
        assert torch.equal(out.sum_signal, ref.sum_signal[:k]), (tile, k)
        assert torch.equal(out.I, ref.I[:k]) and torch.equal(out.sum_norm, ref.sum_norm), (tile, k)
        assert torch.equal(out.count, ref.count)
    for k in (0, n - 1):
        o = c.oracle(fr[k])
        for name, got, r in zip("ISNC", (out.I[k] if k < out.I.shape[0] else ref.I[k], ref.sum_signal[k], ref.sum_norm,
                                         ref.count), o):
            per, norm = rel_err(got.double().cpu().numpy(), r)
            assert per <= 1e-5 and norm <= 1e-5, (tile, k, name, per, norm)
    assert g.status() == 0


@pytest.mark.parametrize("shape", [(61, 93), (64, 96), (9, 130), (3, 41)])
def test_every_frame_count(shape):
    _check(Case(small_workload(*shape, split=2, npt=40, seed=shape[0])), (16, 64), COUNTS)


# planes per block: 8, 8, 4, 4, 2, 1 by the tile's size
@pytest.mark.parametrize("tile", [(8, 120), (48, 40), (32, 172), (40, 164), (64, 164), (100, 228)])
def test_block_sizes(tile):
    _check(Case(small_workload(151, 240, split=2, npt=70, seed=7)), tile, (1, 2, 5, 8, 21, 66),
           other_kernel=tile[0] < 64)


@pytest.mark.parametrize("off", [1, 2, 3])
@pytest.mark.parametrize("fpp", [2, 4, 8, 16])
def test_phases_and_frames_per_pass(off, fpp):
    _check(Case(small_workload(47, 83, split=1, npt=30, seed=8)), (8, 56), (3, 6, 18), fpp, off)


@pytest.mark.parametrize("npt,azim", [(1, 0), (3, 0), (20, 90)])
def test_long_rows_and_heavy_tiles(npt, azim):
    _check(Case(small_workload(130, 140, split=2, npt=npt, npt_azim=azim, seed=9)), (48, 40), (1, 4, 11))


# entries per pixel from about 1.5 to 25: every default tile
@pytest.mark.parametrize("npt,azim", [(60, 0), (200, 0), (600, 0), (1300, 0), (3500, 0), (20, 30), (150, 300)])
def test_default_tiles_by_density(npt, azim):
    c = Case(small_workload(97, 110, split=1, npt=npt, npt_azim=azim, seed=10))
    i = c.gpu_from_oracle_positions().info
    _check(c, (i["tile_h"], i["tile_w"]), (1, 3, 9))
