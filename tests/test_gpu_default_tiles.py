"""The default tile of every range of the rule (entries per pixel, detector size, 1D or 2D): the tile
that is chosen, and on it one frame, a batch and the variance with the bits of other tiles' sums
within the stated tolerance."""
import pytest
import torch

from gpu_common import api, needs_gpu, rel_err

pytestmark = [pytest.mark.gpu, needs_gpu]

# ny, nx, bins, azimuthal bins, split, distance, entries per pixel (from, to), tile
CASES = [
    (2048, 1700, 700, 0, "full", 0.2, (1.0, 1.75), (8, 152)),   # 3072 tiles
    (1920, 1100, 600, 0, "bbox", 0.2, (1.0, 1.75), (8, 152)),   # 1920
    (1500, 1170, 400, 0, "bbox", 0.2, (1.0, 1.75), (8, 120)),   # 1504: below 12 per SM
    (2048, 1700, 850, 0, "full", 0.2, (1.75, 2.1), (8, 120)),
    (97, 110, 30, 0, "bbox", 0.05, (1.0, 2.1), (8, 120)),
    (512, 512, 600, 0, "full", 0.1, (2.1, 5.0), (16, 64)),
    (512, 512, 1700, 0, "full", 0.1, (5.0, 10.0), (16, 40)),
    (400, 512, 4000, 0, "full", 0.1, (10.0, 20.0), (16, 24)),
    (200, 256, 4000, 0, "full", 0.1, (20.0, 200.0), (8, 24)),
    (700, 800, 120, 60, "full", 0.1, (1.0, 2.4), (48, 40)),
    (300, 300, 180, 300, "full", 0.1, (2.4, 5.0), (16, 64)),
]


@pytest.mark.parametrize("ny,nx,npt,azim,split,dist,density,tile", CASES)
def test_default_tile(ny, nx, npt, azim, split, dist, density, tile):
    geo = api().Geometry(dist, 0.47 * ny * 75e-6, 0.52 * nx * 75e-6, 0.01, -0.02, 0.3, 75e-6, 75e-6)
    g = api().Integrator.build(geo, (ny, nx), npt, azim, "q_nm^-1", split)
    i = g.info
    assert density[0] <= i["nnz"] / i["n_unmasked"] < density[1], i["nnz"] / i["n_unmasked"]
    assert (i["tile_h"], i["tile_w"]) == tile
    gen = torch.Generator(device="cuda").manual_seed(ny + nx)
    fr = torch.randint(0, 5000, (3, ny, nx), generator=gen, device="cuda", dtype=torch.int32)
    dark, flat = (torch.rand((ny, nx), generator=gen, device="cuda") + 0.5 for _ in range(2))

    def calls():
        b = g.integrate_batch(fr, dark, flat)
        return [*g.integrate(fr[0], dark, flat, precision="fp64"), *g.integrate(fr[0], dark, flat), b.I[2], b.sum_signal[1],
                g.variance(fr)[1]]
    got = [t.double().cpu().numpy() for t in calls()]
    g.set_tuning(16, 32)
    for k, (a, b) in enumerate(zip(got, calls())):
        per, norm = rel_err(a, b.double().cpu().numpy())
        tol = 1e-12 if k < 4 else 1e-5
        assert per <= tol and norm <= tol, k
    assert g.status() == 0


@pytest.mark.parametrize("ny,nx,npt,tile", [(2880, 2880, 1000, (8, 120)), (2048, 2048, 600, (8, 152))])
def test_wide_tiles_need_room_for_the_heaviest(ny, nx, npt, tile):
    """Both below 1.75 entries per pixel; around the beam centre of the first a wide tile holds so many
    entries that the kernels' rings would lose stages."""
    geo = api().Geometry(0.1, 0.5 * ny * 100e-6, 0.5 * nx * 100e-6, 0.0, 0.0, 0.0, 100e-6, 100e-6)
    g = api().Integrator.build(geo, (ny, nx), npt, 0, "q_nm^-1", "bbox")
    assert 1.2 < g.info["nnz"] / g.info["n_unmasked"] < 1.75
    assert (g.info["tile_h"], g.info["tile_w"]) == tile
    img = torch.ones((ny, nx), dtype=torch.int32, device="cuda")
    for prec in ("fp64", "fp32"):  # a flat image: S is C in every bin
        r = g.integrate(img, precision=prec)
        assert torch.equal(r.sum_signal, r.count) and torch.equal(r.sum_norm, r.count)
    assert g.status() == 0
