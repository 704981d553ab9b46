"""3D mixed-precision tails of more than 1024 cells (chhs_tuning.tail_cells),
which run the general tail code on stored coefficients, the finest level
inside the tail: two and three levels, a box, sweep counts of one, the
double-precision coarsest solve.  The steps must solve the scheme (the
oracle's residual norm of the stored fields at most 2e-10, twice the stopping
norm) in about as many V-cycles as with the default tail, and a batch with the
same setting must give the same fields bit for bit."""
import pytest
import numpy as np

import oracle
from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

H, EPS, GAMMA, DT = 0.05, 0.06, 1.5, 0.005


@pytest.mark.parametrize("shape,nu,f64", [
    ((12, 12, 12), (2, 2), 0), ((12, 12, 12), (1, 1), 1), ((10, 12, 14), (2, 2), 0), ((8, 12, 16), (2, 2), 0),
])
def test_tail_of_more_than_1024_cells_solves(shape, nu, f64):
    opts = chhs.default_opts(precision=1, nu1=nu[0], nu2=nu[1], coarsest_f64=f64)
    phi0 = inputs.spinodal(shape, 9, mean=-0.1, amplitude=0.4)

    def steps(tail_cells):
        with chhs.Run(shape, H, EPS, GAMMA, DT, opts=opts) as run:
            run.set_tuning(tail_cells, 8192, 512, nu[0], nu[1])
            run.set_phi(phi0)
            _, v1, _ = run.step(1)
            before = run.get_state()
            _, v2, _ = run.step(1)
            return v1 + v2, before, run.get_state()

    v, before, (phi, prev, mu, p) = steps(2048)
    assert oracle.residual(before[0], before[1], phi, mu, p, oracle.Params(H, EPS, GAMMA, DT))[3] <= 2e-10
    v_default, _, ref = steps(1024)
    assert abs(v - v_default) <= 2
    assert np.max(np.abs(phi - ref[0])) <= 1e-8
    with chhs.Batch([(shape, H, EPS, GAMMA, DT)], opts=opts) as b:
        b.set_tuning(2048, nu[0], nu[1])
        b.runs[0].set_phi(phi0)
        _, vb, _ = b.step(2)
        assert vb[0] == v
        for x, y in zip(b.runs[0].get_state(), (phi, prev, mu, p)):
            assert np.array_equal(x, y)
