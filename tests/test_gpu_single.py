"""The single-frame kernel (tiles corrected in shared memory, one launch): against the kernel of
the cp.async engine (same entries and order: the same bits) and the oracle, over image types with
their extreme values, every word phase of every array, subsets of the corrections, infinite
pixels, and several detectors with different corrections in one plan."""
import numpy as np
import pytest
import torch

from gpu_common import Case, api, needs_gpu, rel_err, small_workload, to_dev

pytestmark = [pytest.mark.gpu, needs_gpu]


def _shifted(a, words):
    """The array on the device, starting `words` 4-byte words past an allocation's start."""
    if a is None:
        return None
    t = to_dev(a)
    buf = torch.empty(t.numel() + 8, dtype=torch.int32, device="cuda")
    v = buf[words:words + t.numel()]
    v.copy_(t.view(torch.int32).reshape(-1))
    return v.view(t.dtype).view(t.shape)


def _image(dtype, shape, rng):
    if dtype == "float32":
        img = (rng.uniform(-1, 1, shape) * 10.0 ** rng.uniform(-30, 6, shape)).astype(np.float32)
        img.flat[:4] = [0.0, -0.0, np.float32(1e-42), np.float32(3e38)]
        return img
    if dtype == "uint32":
        img = rng.integers(0, 1 << 32, shape, dtype=np.uint32)
        img.flat[:3] = [0, 1, 0xffffffff]
        return img
    img = rng.integers(-(1 << 31), 1 << 31, shape, dtype=np.int64).astype(np.int32)
    img.flat[:3] = [0, -1, -(1 << 31)]
    return img


def _same(a, b):
    return all(torch.equal(torch.nan_to_num(x, nan=12345.0), torch.nan_to_num(y, nan=12345.0)) for x, y in zip(a, b))


@pytest.mark.parametrize("dtype", ["float32", "uint32", "int32"])
@pytest.mark.parametrize("tile", [(8, 120), (16, 64), (48, 40)])
def test_types_and_phases(dtype, tile):
    c = Case(small_workload(93, 131, split=2, npt=50, seed=21, dtype=dtype))
    g = c.gpu_from_oracle_positions()
    g.set_tuning(tile_h=tile[0], tile_w=tile[1])
    rng = np.random.default_rng(3)
    img = _image(dtype, (93, 131), rng)
    full = (c.dark, c.flat, c.sa, c.pol)
    for k, keep in enumerate([(1, 1, 1, 1), (0, 0, 0, 0), (1, 0, 0, 0), (0, 1, 0, 1), (1, 0, 1, 0), (0, 0, 0, 1), (0, 1, 1, 0)]):
        arrs = [a if on else None for a, on in zip(full, keep)]
        dev = [_shifted(a, (k * (i + 2)) % 4) for i, a in enumerate([img] + arrs)]
        for prec, tol in (("fp64", 1e-12), ("fp32", 1e-5)):
            out = g.integrate(*dev, precision=prec)
            g.set_copy_engine("async")
            ref = g.integrate(*dev, precision=prec)
            g.set_copy_engine("tma")
            assert _same(out, ref), (dtype, tile, keep, prec)
            for got, r in list(zip(out, c_oracle(c, img, arrs)))[2:]:  # N and C (no cancellation)
                per, norm = rel_err(got.double().cpu().numpy(), r)
                assert per <= tol and norm <= tol, (dtype, tile, keep, prec)
    assert g.status() == 0


def c_oracle(c, img, arrs):
    import oracle as O
    return O.integrate(c.A, img, *arrs)


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_infinite_pixels(prec):
    c = Case(small_workload(64, 72, split=2, npt=40, seed=22, dtype="float32"))
    g = c.gpu_from_oracle_positions()
    img = c.image.copy()
    img[10:60:7, 5:70:9] = np.inf
    img[11:60:13, 3:70:17] = -np.inf
    corr = c.corrections_dev()
    out = g.integrate(to_dev(img), *corr, precision=prec)
    g.set_copy_engine("async")
    assert _same(out, g.integrate(to_dev(img), *corr, precision=prec))


def test_plan_of_detectors_with_different_corrections():
    cases = [Case(small_workload(40 + 13 * k, 70 + 9 * k, split=2, npt=30 + 10 * k, seed=30 + k)) for k in range(5)]
    igs = [c.gpu_from_oracle_positions() for c in cases]
    for k, g in enumerate(igs):
        g.set_tuning(tile_h=(8, 16, 48)[k % 3], tile_w=(120, 64, 40)[k % 3])
    imgs = [_shifted(c.image, k % 4) for k, c in enumerate(cases)]
    pick = [(1, 1, 1, 1), (0, 0, 0, 0), (1, 0, 0, 0), (0, 1, 0, 0), (0, 0, 1, 1)]
    corr = [[_shifted(a, (i + k) % 4) if on else None for i, (a, on) in enumerate(zip((c.dark, c.flat, c.sa, c.pol), p))]
            for k, (c, p) in enumerate(zip(cases, pick))]
    plan = api().MultiPlan(igs, imgs, *[[x[i] for x in corr] for i in range(4)])
    for use_graph in (False, True, True):
        outs = plan.launch(use_graph=use_graph)
        torch.cuda.synchronize()
        for g, img, x, o in zip(igs, imgs, corr, outs):
            assert _same(o, g.integrate(img, *x, precision="fp32"))
