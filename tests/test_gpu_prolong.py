"""The prolongation's thread per coarse cell on levels of odd half sizes, of
fewer coarse cells than a block and of several blocks, in double precision and
without post-smoothing (where it is a launch of its own in every form); each
step checked with the oracle's residual of the scheme (2e-10)."""
import numpy as np
import pytest

import oracle
from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

H, EPS, GAMMA, DT = 0.05, 0.06, 1.5, 0.005


@pytest.mark.parametrize("shape,nu,precision", [
    ((48, 80), (2, 2), 0), ((6, 10), (2, 2), 0), ((96, 72), (2, 0), 0), ((12, 20, 36), (2, 2), 0),
    ((6, 10, 14), (2, 2), 0), ((48, 16, 32), (2, 0), 0), ((40, 24, 56), (2, 0), 1), ((96, 72), (2, 0), 1),
])
def test_steps_solve_the_scheme(shape, nu, precision):
    opts = chhs.default_opts(precision=precision, nu1=nu[0], nu2=nu[1])
    with chhs.Run(shape, H, EPS, GAMMA, DT, opts=opts) as run:
        run.set_tuning(64, 0, 512, nu[0], nu[1])  # grid-wide levels down to 64 cells
        run.set_phi(inputs.spinodal(shape, 9, mean=-0.1, amplitude=0.4))
        run.step(1)
        before = run.get_state()
        run.step(1)
        phi, _, mu, p = run.get_state()
    norm = oracle.residual(before[0], before[1], phi, mu, p, oracle.Params(H, EPS, GAMMA, DT))[3]
    assert norm <= 2e-10
