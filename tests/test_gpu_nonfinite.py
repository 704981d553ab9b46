"""Values that are not finite through the mixed form's set-up and residual: one
NaN or infinity at a corner, inside, at the edge of a tile, in either time level.
The step must end as diverged with the state kept, in every arithmetic of the
residual, and in a batch only that run, the others giving the bits they give
without it."""
import numpy as np
import pytest

from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

H, EPS, GAMMA, DT = 0.05, 0.06, 1.5, 0.005


@pytest.mark.parametrize("shape", [(64, 48), (16, 24, 40), (15, 21)])
@pytest.mark.parametrize("value", [np.nan, np.inf, -np.inf])
def test_one_bad_value(shape, value):
    good = inputs.spinodal(shape, 5, mean=-0.1, amplitude=0.3)
    with chhs.Batch([(shape, H, EPS, GAMMA, DT)]) as b:
        b.runs[0].set_phi(good)
        b.step(1)
        ref = b.runs[0].get_state()
    for place in ((0,) * len(shape), tuple(n - 1 for n in shape), tuple(n // 2 for n in shape), (7,) * len(shape)):
        bad = good.copy()
        bad[place] = value
        for phi, prev in ((bad, bad), (good, bad)):
            for f64, per8 in ((0, 3), (0, 4), (1, 3)):
                opts = chhs.default_opts(precision=1, f64_residual=f64)
                with chhs.Run(shape, H, EPS, GAMMA, DT, opts=opts) as run:
                    run.set_tuning(1024, 8192, 512, 2, 2, norm_f64_per8=per8)
                    run.set_phi(phi, prev)
                    status, v, resid = run.step(1, check=False)
                    assert status == chhs.CHHS_ERR_DIVERGED and v == 0 and not np.isfinite(resid)
                    assert np.array_equal(run.get_state()[0], phi, equal_nan=True)
        with chhs.Batch([(shape, H, EPS, GAMMA, DT)] * 2) as b:
            b.runs[0].set_phi(good)
            b.runs[1].set_phi(bad)
            status, _, _ = b.step(1, check=False)
            assert status == [chhs.CHHS_OK, chhs.CHHS_ERR_DIVERGED]
            for x, y in zip(b.runs[0].get_state(), ref):
                assert np.array_equal(x, y)
