"""az_integrate_noalloc runs the kernels of az_integrate1d / 2d: the same bits for every image type,
precision, copy engine, subset of the corrections and tile (also one too large for them), and in a
fresh process its first calls take no device memory."""
import subprocess
import sys

import numpy as np
import pytest
import torch

from gpu_common import Case, api, needs_gpu, small_workload, to_dev

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("azim", [0, 40])
@pytest.mark.parametrize("dtype", ["float32", "uint32", "int32"])
@pytest.mark.parametrize("tile", [(8, 120), (48, 40), (32, 120), (100, 228)])
def test_bits_of_integrate(dtype, tile, azim):
    c = Case(small_workload(103, 131, split=2, npt=120 if azim else 50, npt_azim=azim, seed=51))
    g = c.gpu_from_oracle_positions()
    g.set_tuning(*tile)
    rng = np.random.default_rng(4)
    img = to_dev(rng.integers(0, 60000, (103, 131)).astype(dtype))
    corr = c.corrections_dev()
    for keep in ((1, 1, 1, 1), (0, 0, 0, 0), (1, 0, 0, 0), (0, 0, 1, 1)):
        x = [a if k else None for a, k in zip(corr, keep)]
        for engine in ("tma", "async"):
            g.set_copy_engine(engine)
            for prec in ("fp64", "fp32"):
                try:
                    got = g.integrate_noalloc(img, *x, precision=prec)
                except api().AzError as e:
                    # the planes of two such tiles exceed the shared memory (integrate has another form)
                    assert tile == (100, 228) and e.code == -6 and "shared memory" in str(e)
                    continue
                for a, b in zip(got, g.integrate(img, *x, precision=prec)):
                    assert torch.equal(a, b), (keep, engine, prec)
    assert g.status() == 0


SCRIPT = r"""
import sys
sys.path[:0] = ["tests", "."]
import torch
from paper_1412_6367_gb300 import api
from gpu_common import Case, small_workload
ig = []
for azim in (0, 70):
    c = Case(small_workload(90, 110, split=2, npt=64, npt_azim=azim, seed=5))
    ig.append(c.gpu_from_oracle_positions())
corr = c.corrections_dev()
imgs = [torch.ones((90, 110), dtype=d, device="cuda") for d in (torch.float32, torch.int32)]
imgs.append(imgs[1].view(torch.uint32))
outs = [[api.Result(*(torch.empty(g.nrows, dtype=d, device="cuda") for _ in range(4))) for d in (torch.float64, torch.float32)] for g in ig]
torch.cuda.synchronize()
free = torch.cuda.mem_get_info()[0]
for g, o in zip(ig, outs):
    for img in imgs:
        for x in (corr, [None] * 4, [corr[0], None, None, None]):
            for prec, out in zip(("fp64", "fp32"), o):
                g.integrate_noalloc(img, *x, precision=prec, out=out)
torch.cuda.synchronize()
assert torch.cuda.mem_get_info()[0] == free, (free, torch.cuda.mem_get_info()[0])
assert all(g.status() == 0 for g in ig)
"""


def test_first_calls_take_no_memory():
    r = subprocess.run([sys.executable, "-c", SCRIPT], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stdout + r.stderr
