"""Polarisation of geometries whose squared lengths under- or overflow a double: the correction
depends on directions only, so it is that of the same geometry in other units."""
import numpy as np
import pytest

import oracle as O
from gpu_common import api, needs_gpu

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("scale", [1.0, 1e-140, 1e-200, 1e-300, 1e139, 1e141, 1e200, 1e300])
@pytest.mark.parametrize("factor", [-1.0, 0.0, 0.99])
def test_scaled_geometries(scale, factor):
    ny, nx = 21, 34
    par = [0.1, 0.011, 0.02]
    rot = (0.2, -0.3, 0.7)
    pix = (1e-3, 1.1e-3)
    ref = O.polarization(O.Geometry(*par, *rot, *pix, 1e-10), ny, nx, factor)
    g = api().Geometry(*[p * scale for p in par], *rot, *[p * scale for p in pix], 1e-10)
    got = g.polarization(ny, nx, factor).cpu().numpy().astype(np.float64)
    # a few roundings of doubles on each side, then one to float32 of a value of at most 1
    assert np.max(np.abs(got - ref)) <= 2.0 ** -24 + 1e-12
