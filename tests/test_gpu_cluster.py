"""The double-precision coarse levels in one cluster (k_cluster) on shapes at
the edges of its slabs: rows that do not divide over the blocks, a level with
fewer row pairs than blocks, one row pair, wide and tall levels, the finest
level inside and outside the cluster, sweep counts of zero.  Each step is
checked with the oracle's residual of the scheme (2e-10, twice the stopping
norm; the oracle's own multigrid does not solve the long thin grids here) and
against the run whose coarse passes are grid-wide launches (split_threads 0):
the same solver, so the same V-cycle count and the same step within the parity
bound 1e-9."""
import numpy as np
import pytest

import oracle
from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu


def _step(shape, nu, split):
    h, eps, gamma, dt = 0.05, 0.06, 1.5, 0.005
    opts = chhs.default_opts(nu1=nu[0], nu2=nu[1])
    with chhs.Run(shape, h, eps, gamma, dt, opts=opts) as run:
        run.set_tuning(64, split, 512, nu[0], nu[1])
        run.set_phi(inputs.spinodal(shape, 9, mean=-0.1, amplitude=0.4))
        run.step(1)
        before = run.get_state()
        _, v, _ = run.step(1)
        after = run.get_state()
    return before, after, v


@pytest.mark.parametrize("shape,nu", [
    ((64, 64), (2, 2)), ((128, 128), (2, 2)), ((40, 24), (2, 2)), ((24, 104), (2, 2)), ((36, 36), (1, 1)),
    ((6, 512), (2, 2)), ((512, 6), (2, 2)), ((12, 12), (2, 2)), ((72, 56), (0, 2)), ((56, 72), (2, 0)),
    ((16, 1024), (2, 2)), ((1024, 16), (2, 1)),
])
def test_cluster_levels_against_grid_passes_and_oracle(shape, nu):
    before, got, v = _step(shape, nu, 8192)
    _, grid, v_grid = _step(shape, nu, 0)
    phim, prev, _, _ = before
    norm = oracle.residual(phim, prev, got[0], got[2], got[3], oracle.Params(0.05, 0.06, 1.5, 0.005))[3]
    assert norm <= 2e-10
    assert v == v_grid
    assert np.max(np.abs(got[0] - grid[0])) <= 1e-9
    assert abs(got[0].mean() - phim.mean()) <= 1e-10
