"""One integrator in a plan more than once (the same detector's frames of several exposures): every
instance has partial sums of its own."""
import pytest
import torch

from gpu_common import Case, api, needs_gpu, small_workload, to_dev

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("engine", ["tma", "async"])
def test_repeated_integrators(engine):
    cases = [Case(small_workload(300, 220, split=2, npt=60, seed=61)), Case(small_workload(90, 131, split=2, npt=40, npt_azim=12, seed=62))]
    igs = [c.gpu_from_oracle_positions() for c in cases]
    for g in igs:
        g.set_copy_engine(engine)
    pick = [0, 1, 0, 0, 1]
    imgs = [to_dev((cases[i].image // (k + 1)).astype(cases[i].image.dtype)) for k, i in enumerate(pick)]
    corr = [cases[i].corrections_dev() for i in pick]
    plan = api().MultiPlan([igs[i] for i in pick], imgs, *[[x[j] for x in corr] for j in range(4)])
    refs = [igs[i].integrate(img, *x, precision="fp32") for i, img, x in zip(pick, imgs, corr)]
    for graph in (False, True, True):
        for o, r in zip(plan.launch(use_graph=graph), refs):
            for a, b in zip(o, r):
                assert torch.equal(a.reshape(-1), b.reshape(-1))
    assert all(g.status() == 0 for g in igs)
