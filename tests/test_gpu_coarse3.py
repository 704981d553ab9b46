"""The 3D mixed form's one-block tail (chhs_tail3.cuh) on shapes at its edges:
the finest level inside it, the most and the fewest cells, a coarsest grid of
one lane per cell, of more than 32 cells (the general solve) and in double
precision, one level above the coarsest, sweep counts of one and zero.  With
the tail from 1024 cells and from its smallest size of two levels the levels
between run in it or as grid-wide passes with the same arithmetic: the fields
must be the same bit for bit, and a batch's too.  Each step is also checked with the oracle's residual of
the scheme (2e-10)."""
import numpy as np
import pytest

import oracle
from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

H, EPS, GAMMA, DT = 0.05, 0.06, 1.5, 0.005


@pytest.mark.parametrize("shape,nu,f64", [
    ((32, 32, 32), (2, 2), 0), ((64, 64, 64), (2, 2), 0), ((24, 40, 48), (2, 2), 0), ((48, 16, 32), (1, 1), 0),
    ((40, 24, 56), (2, 2), 0), ((12, 20, 36), (2, 2), 0), ((20, 28, 36), (2, 2), 0), ((32, 32, 32), (2, 2), 1),
    ((16, 16, 16), (2, 0), 0), ((32, 16, 64), (0, 2), 0), ((8, 8, 8), (2, 2), 0), ((4, 4, 4), (2, 2), 0),
])
def test_tail_is_the_grid_passes(shape, nu, f64):
    opts = chhs.default_opts(precision=1, nu1=nu[0], nu2=nu[1], coarsest_f64=f64)
    phi0 = inputs.spinodal(shape, 9, mean=-0.1, amplitude=0.4)
    results = []
    coarsest = np.array(shape)
    while (coarsest % 2 == 0).all() and (coarsest >= 4).all():
        coarsest = coarsest // 2
    # (a tail of more than 1024 cells, or of one level, is the general code's: other rounding)
    for tail_cells in (1024, min(1024, 8 * int(np.prod(coarsest)))):
        with chhs.Run(shape, H, EPS, GAMMA, DT, opts=opts) as run:
            run.set_tuning(tail_cells, 8192, 512, nu[0], nu[1])
            run.set_phi(phi0)
            _, v1, _ = run.step(1)
            before = run.get_state()
            _, v2, _ = run.step(1)
            results.append((v1 + v2,) + run.get_state())
    with chhs.Batch([(shape, H, EPS, GAMMA, DT)], opts=opts) as b:
        b.runs[0].set_phi(phi0)
        _, v, _ = b.step(2)
        results.append((v[0],) + b.runs[0].get_state())
    # without a pre-smoothing sweep the grid-wide levels take their right-hand
    # side from stored coefficients: other rounding
    same = results[1:] if nu[0] > 0 else results[2:]
    for r in same:
        assert r[0] == results[0][0]
        for x, y in zip(r[1:], results[0][1:]):
            assert np.array_equal(x, y)
    _, phi, _, mu, p = results[0]
    norm = oracle.residual(before[0], before[1], phi, mu, p, oracle.Params(H, EPS, GAMMA, DT))[3]
    assert norm <= 2e-10
