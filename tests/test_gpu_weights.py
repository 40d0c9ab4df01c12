"""Weights of an imported matrix at the edges of the number format: negative zeros and subnormals.
The single-frame kernel marks the places past a segment's end in the weights, and no weight of the
matrix may be taken for such a mark.  Against the same sums in numpy and the cp.async engine's
kernel (another kernel: the same bits)."""
import numpy as np
import pytest
import torch

from gpu_common import api, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]

NY, NX = 12, 40
TINY = 4.9406564584124654e-324  # the smallest subnormal

# (weights, pixel values) of the first entries of a row
ROWS = [
    ([-0.0], [np.inf]),                    # NaN
    ([0.0], [np.inf]),                     # NaN
    ([-0.0, 1.0], [7.0, 2.0]),             # 2
    ([1.0, -0.0], [2.0, -np.inf]),         # NaN
    ([-0.0], [np.nan]),                    # NaN
    ([-TINY], [3e38]),
    ([-1e-320, 2e-310], [1e30, -3e38]),
    ([-2.0 ** -1023], [2.0 ** 100]),
    ([1.0, 1.0, 1.0, 1.0, -0.0], [1.0, 2.0, 3.0, 4.0, np.inf]),  # NaN
    ([-1e-310] * 9, [1e38] * 9),
]


def _same(a, b):
    return np.array_equal(np.isnan(a), np.isnan(b)) and np.array_equal(np.nan_to_num(a, nan=1.0), np.nan_to_num(b, nan=1.0))


def test_signed_zeros_and_subnormals_fp64():
    image = np.ones((NY, NX), np.float32)
    indptr, indices, data = [0], [], []
    for r, (ws, vs) in enumerate(ROWS):
        for k, (w, v) in enumerate(zip(ws, vs)):
            p = r * NX + k
            image.flat[p] = v
            indices.append(p)
            data.append(w)
        indptr.append(len(indices))
    ig = api().Integrator.from_csr((NY, NX), indptr, indices, data, len(ROWS))
    img = torch.from_numpy(image).cuda()
    out = ig.integrate(img, precision="fp64")
    ig.set_copy_engine("async")
    other = ig.integrate(img, precision="fp64")
    with np.errstate(invalid="ignore"):
        ref = np.array([np.sum(np.array(ws) * np.array(vs, np.float32).astype(np.float64)) for ws, vs in ROWS])
    got = out.sum_signal.cpu().numpy()
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    fin = ~np.isnan(ref)
    # products of a few terms: each rounded once, their sum at most eight times
    assert np.all(np.abs(got[fin] - ref[fin]) <= 16 * 2.0 ** -52 * np.abs(ref[fin]))
    for a, b in zip(out, other):
        assert _same(a.cpu().numpy(), b.cpu().numpy())
    assert ig.status() == 0
