"""Phase 2 with a thread per row (patterns of at least 4096 rows with few segments per row): the
four sums of single frames (FP64 and FP32), of batches of 1 to 5 frames and of the allocation-
free entry point against the oracle, for rows of no, one, a few and many segments."""
import numpy as np
import pytest

from gpu_common import Case, needs_gpu, rel_err, small_workload, to_dev

pytestmark = [pytest.mark.gpu, needs_gpu]


@pytest.mark.parametrize("tile", [(32, 64), (4, 8), (4, 4)])
@pytest.mark.parametrize("split", [0, 2])
def test_rows_of_few_segments(tile, split):
    w = small_workload(121, 133, split=split, npt=64, npt_azim=72, seed=91)  # 4608 rows
    c = Case(w)
    g = c.gpu_from_oracle_positions()
    g.set_tuning(tile_h=tile[0], tile_w=tile[1])
    assert g.info["nrows"] >= 4096 and g.info["n_segments"] <= 8 * g.info["nrows"]
    corr = c.corrections_dev()
    ref = c.oracle()
    img = c.image_dev()
    for prec, tol in (("fp64", 1e-12), ("fp32", 1e-5)):
        for res in (g.integrate(img, *corr, precision=prec), g.integrate_noalloc(img, *corr, precision=prec)):
            for name, got, r in zip("ISNC", res, ref):
                per, norm = rel_err(got.double().cpu().numpy(), r)
                assert per <= tol and norm <= tol, (tile, split, prec, name, per, norm)
    one = g.integrate(img, *corr, precision="fp32")
    for n in (1, 4, 5):
        out = g.integrate_batch(to_dev(np.stack([c.image] * n)), *corr)
        for k in range(n):
            assert (out.I[k] == one.I.reshape(-1)).all() and (out.sum_signal[k] == one.sum_signal.reshape(-1)).all()
        assert (out.sum_norm == one.sum_norm.reshape(-1)).all() and (out.count == one.count.reshape(-1)).all()
    assert g.status() == 0
