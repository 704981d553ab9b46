"""The marching residual kernel of the mixed form (chhs_norm_df.cuh) at the
edges of its tiles, strips and plane chunks: extents around 32 and 8 cells,
one and several chunks, thin boxes.  For every setting (double-single, tiles
on the FP64 pipe, all in double precision) the reported norm of a step must be
the oracle's residual norm of the same fields within 0.1 % (its single-precision
squares and the double-single residual's 1e-14 are far below that), and the
settings' steps must agree within the mixed form's 1e-8."""
import numpy as np
import pytest

import oracle
from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

H, EPS, GAMMA, DT = 0.05, 0.06, 1.5, 0.005


@pytest.mark.parametrize("shape", [
    (64, 64), (40, 36), (44, 100), (160, 28), (24, 264), (8, 12, 36), (36, 20, 40), (48, 8, 64), (20, 44, 28),
])
def test_norm_of_every_setting_is_the_oracles(shape):
    fields = []
    for per8, f64 in ((0, 0), (3, 0), (8, 0), (0, 1)):
        opts = chhs.default_opts(precision=1, f64_residual=f64)
        with chhs.Run(shape, H, EPS, GAMMA, DT, opts=opts) as run:
            run.set_tuning(256, 8192, 512, 2, 2, norm_f64_per8=per8)
            run.set_phi(inputs.spinodal(shape, 5, mean=-0.1, amplitude=0.4))
            run.step(1)
            before = run.get_state()
            _, _, resid = run.step(1)
            phi, _, mu, p = run.get_state()
        norm = oracle.residual(before[0], before[1], phi, mu, p, oracle.Params(H, EPS, GAMMA, DT))[3]
        assert abs(resid - norm) <= 1e-3 * norm + 1e-14
        assert abs(p.mean()) <= 1e-14 * max(1.0, np.abs(p).max())
        fields.append(phi)
    for phi in fields[1:]:
        assert np.max(np.abs(phi - fields[0])) <= 1e-8
