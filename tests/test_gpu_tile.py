"""The 2D mixed form's tile kernel (chhs_tile.cuh, a thread per 2 x 2 cells) at
its edges: grids smaller than, equal to and just past a tile, extents that
leave partial tiles, the tail close to and far below the finest level, sweep
counts that take no pass, one launch, and several launches (more than eight
passes).  Shapes only cut the passes into blocks, so every shape must give the
same fields bit for bit; each step is checked with the oracle's residual of the
scheme (2e-10, twice the stopping norm)."""
import numpy as np
import pytest

import oracle
from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

H, EPS, GAMMA, DT = 0.05, 0.06, 1.5, 0.005


@pytest.mark.parametrize("shape,nu", [
    ((32, 32), (2, 2)), ((36, 68), (2, 2)), ((64, 48), (1, 1)), ((8, 64), (2, 2)), ((64, 8), (2, 1)),
    ((40, 56), (0, 2)), ((56, 40), (2, 0)), ((48, 32), (5, 5)), ((32, 64), (5, 2)), ((64, 32), (2, 6)),
    ((48, 48), (9, 4)),
])
def test_tile_shapes_bitwise_and_step_against_oracle_residual(shape, nu):
    opts = chhs.default_opts(precision=1, nu1=nu[0], nu2=nu[1])
    results = []
    for big, small in (((32, 32), (16, 8)), ((64, 16), (32, 16)), ((2, 2), (32, 32)), ((16, 34), (18, 20))):
        with chhs.Run(shape, H, EPS, GAMMA, DT, opts=opts) as run:
            run.set_tuning(64, 8192, 512, nu[0], nu[1], big[0], big[1], small_tile=(small[0], small[1], 256))
            run.set_phi(inputs.spinodal(shape, 9, mean=-0.1, amplitude=0.4))
            run.step(1)
            before = run.get_state()
            _, v, _ = run.step(1)
            results.append((v,) + run.get_state())
    _, phi, _, mu, p = results[0]
    norm = oracle.residual(before[0], before[1], phi, mu, p, oracle.Params(H, EPS, GAMMA, DT))[3]
    assert norm <= 2e-10
    for r in results[1:]:
        assert r[0] == results[0][0]
        for a, b in zip(r[1:], results[0][1:]):
            assert np.array_equal(a, b)
