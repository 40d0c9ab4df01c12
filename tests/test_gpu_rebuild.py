"""A layout whose rebuild fails part way (device memory refused by az_selftest_alloc, an error code on
the host): the integrator is left with the tiles it had, or refuses the calls that need a layout
until one has been built, and never runs on buffers of two layouts."""
import pytest
import torch

from gpu_common import Case, api, needs_gpu, small_workload, to_dev

pytestmark = [pytest.mark.gpu, needs_gpu]

ENOMEM, EINVAL = -3, -1


@pytest.fixture(autouse=True)
def _no_failures_left():
    yield
    api().selftest_alloc()


def _case(azim):
    c = Case(small_workload(83, 121, split=2, npt=30, npt_azim=azim, seed=41))
    return c, c.gpu_from_oracle_positions()


def _all(c, g):
    """Every call that reads the layout or its scratch."""
    img, corr = c.image_dev(), c.corrections_dev()
    fr = torch.stack([img.view(torch.int32)] * 3).view(torch.uint32)
    out = []
    for prec in ("fp64", "fp32"):
        r = g.integrate(img, *corr, precision=prec)
        out += list(r) + list(g.integrate_noalloc(img, *corr, precision=prec))
        out += list(g.backward(torch.ones_like(r.I).reshape(-1), r.I.reshape(-1), r.sum_norm.reshape(-1), precision=prec))
    out += list(g.integrate_batch(fr, *corr))
    g.set_corrections(*corr)
    out += list(g.integrate_batch_bound(fr)) + list(g.integrate_pixelnorm(fr, *corr)) + [g.variance(fr)]
    out += list(g.integrate_batch_host(_host(fr), *corr))
    plan = api().MultiPlan([g], [img])
    out += list(plan.launch()[0])
    torch.cuda.synchronize()
    return [t.cpu().clone() for t in out]


def _host(fr):
    return fr.view(torch.int32).cpu().view(fr.dtype)


def _equal(a, b):
    return all(torch.equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("azim", [0, 24])
def test_one_failed_allocation_keeps_the_tiles(azim):
    c, g = _case(azim)
    g.set_tuning(16, 64)
    ref = _all(c, g)
    failures = 0
    for after in range(16):
        api().selftest_alloc(after, 1)
        try:
            g.set_tuning(8, 40)
        except api().AzError as e:
            assert e.code == ENOMEM and "cudaMalloc" in str(e)
            failures += 1
        api().selftest_alloc()
        if g.refresh_info()["tile_w"] == 64:
            assert _equal(_all(c, g), ref), after
        else:
            assert g.info["tile_w"] == 40
            g.set_tuning(16, 64)
            assert _equal(_all(c, g), ref), after
    assert failures >= 3  # tiles, entries, items or scratch
    assert g.status() == 0


def test_no_memory_left_refuses_until_rebuilt():
    c, g = _case(0)
    g.set_tuning(16, 64)
    ref = _all(c, g)
    img, corr = c.image_dev(), c.corrections_dev()
    fr = to_dev(c.image[None])
    calls = [lambda: g.integrate(img, *corr), lambda: g.integrate(img, precision="fp64"),
             lambda: g.integrate_noalloc(img), lambda: g.integrate_batch(fr), lambda: g.set_corrections(*corr),
             lambda: g.integrate_batch_bound(fr), lambda: g.variance(fr), lambda: g.integrate_pixelnorm(fr),
             lambda: g.integrate_batch_host(_host(fr)), lambda: api().MultiPlan([g], [img])]
    refused = 0
    for after in range(16):
        api().selftest_alloc(after, 10 ** 6)
        try:
            g.set_tuning(8, 40)
            break  # more allocations allowed than it makes
        except api().AzError as e:
            assert e.code == ENOMEM
        finally:
            api().selftest_alloc()
        for call in calls:
            with pytest.raises(api().AzError) as e:
                call()
            assert e.value.code == EINVAL and "no tiled layout" in str(e.value), after
        refused += 1
        g.set_tuning(16, 64)  # the tiles it had: built again, because there is no layout
        assert _equal(_all(c, g), ref)
    assert refused >= 3
    g.autotune(2)  # (may choose the look-up table and another engine)
    g.set_layout("tiled")
    g.set_copy_engine("tma")
    g.set_tuning(16, 64)
    assert _equal(_all(c, g), ref)
    assert g.status() == 0


def test_refused_shapes_leave_everything():
    c, g = _case(0)
    g.set_tuning(16, 64)
    ref = _all(c, g)
    g.set_corrections(*c.corrections_dev())
    fr = to_dev(c.image[None])
    bound = list(g.integrate_batch_bound(fr))
    for th, tw in ((6, 64), (10000, 64)):
        with pytest.raises(api().AzError):
            g.set_tuning(th, tw)
        assert _equal([t.cpu() for t in g.integrate_batch_bound(fr)], [t.cpu() for t in bound])
    assert _equal(_all(c, g), ref)


def test_failed_autotune_keeps_the_tiles():
    c, g = _case(0)
    g.set_tuning(20, 28)  # (none of the tuner's)
    ref = _all(c, g)
    for after, count in ((0, 1), (4, 3), (9, 200)):
        api().selftest_alloc(after, count)
        try:
            g.autotune(2)
        except api().AzError as e:
            assert e.code in (ENOMEM, -6)
        api().selftest_alloc()
        g.set_layout("tiled")
        g.set_copy_engine("tma")
        g.set_tuning(20, 28)
        assert _equal(_all(c, g), ref)
    assert g.status() == 0


def test_a_plan_of_former_tiles_is_refused():
    c, g = _case(0)
    c2, h = _case(24)
    imgs = [c.image_dev(), c2.image_dev()]
    plan = api().MultiPlan([g, h], imgs)
    ref = [t.cpu().clone() for r in plan.launch(use_graph=True) for t in r]
    h.set_tuning(frames_per_pass=4)  # no other tiles
    assert _equal([t.cpu() for r in plan.launch(use_graph=True) for t in r], ref)
    h.set_tuning(8, 40)
    for graph in (False, True):
        with pytest.raises(api().AzError) as e:
            plan.launch(use_graph=graph)
        assert e.value.code == EINVAL and "integrator 1" in str(e.value)
    out = api().MultiPlan([g, h], imgs).launch(use_graph=True)
    assert _equal([t.cpu() for t in out[0]], ref[:4])
    assert g.status() == 0 and h.status() == 0


def test_builds_without_room_for_a_reservation():
    """A build's scratch is reserved in one piece; where that piece does not fit, smaller ones do."""
    c, g = _case(0)
    ref = _all(c, g)
    built = 0
    for after in range(16):
        api().selftest_alloc(after, 1)
        try:
            h = c.gpu_from_oracle_positions()
            built += 1
        except api().AzError as e:
            assert e.code == ENOMEM
            continue
        finally:
            api().selftest_alloc()
        assert (h.info["tile_h"], h.info["tile_w"]) in ((g.info["tile_h"], g.info["tile_w"]), (8, 64))
        if h.info["tile_w"] == g.info["tile_w"]:
            assert _equal(_all(c, h), ref), after
    assert built >= 3  # the two reservations, and more failures allowed than allocations made
