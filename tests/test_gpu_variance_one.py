"""One frame's variance (single_kernel) has the bits of the frame in a batch (the frames kernel), over
image types with their extreme values, word phases, tiles (also ones too large for two stages),
1D and 2D, a frame left over after full launches, and one frame a call."""
import numpy as np
import pytest
import torch

from gpu_common import Case, needs_gpu, small_workload, to_dev

pytestmark = [pytest.mark.gpu, needs_gpu]


def _frame(dtype, shape, rng):
    if dtype == "float32":
        f = (rng.uniform(-1, 1, shape) * 10.0 ** rng.uniform(-30, 6, shape)).astype(np.float32)
        f.flat[:6] = [0.0, -0.0, 1e-42, -1e-42, np.nan, -np.inf]
        return f
    info = np.iinfo(dtype)
    f = rng.integers(info.min, info.max, shape, dtype=np.int64, endpoint=True).astype(dtype)
    f.flat[:4] = [0, 1, info.max, info.min]
    return f


@pytest.mark.parametrize("dtype", ["float32", "uint32", "int32"])
@pytest.mark.parametrize("tile", [(8, 120), (8, 152), (16, 64), (48, 40), (100, 228)])
@pytest.mark.parametrize("azim", [0, 20])
def test_one_frame_is_its_batch(dtype, tile, azim):
    ny, nx = 93, 131
    c = Case(small_workload(ny, nx, split=2, npt=40, npt_azim=azim, seed=81, corrections=False))
    g = c.gpu_from_oracle_positions()
    g.set_tuning(*tile)
    rng = np.random.default_rng(9)
    fr = np.stack([_frame(dtype, (ny, nx), rng) for _ in range(3)])
    dev = to_dev(fr)
    ref = g.variance(dev)
    assert bool(torch.isnan(ref).any()) is False
    for k in range(3):  # (odd sizes: another word phase a frame)
        assert torch.equal(g.variance(dev[k]), ref[k])
    assert g.status() == 0


def test_a_frame_left_over():
    c = Case(small_workload(40, 70, split=2, npt=30, seed=82, corrections=False))
    g = c.gpu_from_oracle_positions()
    fr = to_dev(np.random.default_rng(2).integers(0, 9000, (65, 40, 70)).astype(np.int32))
    v = g.variance(fr)  # 64 and 1
    assert torch.equal(v[64:], g.variance(fr[63:])[1:])
