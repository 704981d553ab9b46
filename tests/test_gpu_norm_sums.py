"""The sum of squares of the mixed form's stopping norm.  On a uniform field
phi = c, with mu = p = 0 and a tolerance that accepts the initial guess, every
cell's residual is (0, c^3 - c, 0) and the reported norm |c^3 - c|.  Rounding
the residual and its square to single precision leaves 1.5 2^-24 = 9e-8
relative; the sum over up to 4096 cells of a block (16 rows or planes per
thread) must add nothing to that.  A residual whose square overflows single
precision is reported as infinite, a field that is not a number as such."""
import numpy as np
import pytest

from paper_1611_02967_gb300 import chhs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(640, 2048), (64, 256, 256), (40, 36)])
def test_norm_of_a_uniform_residual(shape):
    opts = chhs.default_opts(precision=1, tol=1e3)
    with chhs.Run(shape, 0.05, 0.06, 1.5, 0.005, opts=opts) as run:
        for c in (0.126, 0.165, 0.191, 0.204, 0.23, 0.282, 0.321, 0.334, 0.399):
            run.set_phi(np.full(shape, c))
            _, v, resid = run.step(1)
            assert v == 0
            assert abs(resid / abs(c**3 - c) - 1.0) <= 1e-7


@pytest.mark.parametrize("shape", [(40, 36), (8, 12, 36)])
def test_norm_beyond_single_precision(shape):
    for value, bad in ((1e9, np.isinf), (np.nan, np.isnan)):
        phi = np.zeros(shape)
        phi[(1,) * len(shape)] = value
        with chhs.Run(shape, 0.05, 0.06, 1.5, 0.005, opts=chhs.default_opts(precision=1)) as run:
            run.set_phi(phi)
            status, _, resid = run.step(1, check=False)
            assert status == chhs.CHHS_ERR_DIVERGED and bad(resid)
