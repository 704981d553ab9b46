"""Grids and settings at the limits of what the mixed form accepts: the largest
2D grids that a block's shared memory holds as one level (2 524 cells) or two
(42 x 48, chhs_tuning.tail_cells 2048), alone and in a batch, and block sizes
of tiles, which matter only where a level of the grid asks for them.  A refused
setting leaves the one before in force, bit for bit."""
import numpy as np
import pytest

import oracle
from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

H, EPS, GAMMA, DT = 0.05, 0.06, 1.5, 0.001


def _steps(shape, n=1, tuning=None, refused=None):
    """The state after n steps of a new handle (a handle keeps its measured
    contraction from step to step) that took one setting or refused one."""
    with chhs.Run(shape, H, EPS, GAMMA, DT, opts=chhs.default_opts(precision=1)) as run:
        if tuning:
            run.set_tuning(*tuning[0], **tuning[1])
        if refused:
            with pytest.raises(chhs.ChhsError):
                run.set_tuning(*refused[0], **refused[1])
        run.set_phi(inputs.spinodal(shape, 3, mean=-0.1, amplitude=0.05))
        run.step(n)
        return run.get_state()


def _same(a, b):
    return all(np.array_equal(x, y) for x, y in zip(a, b))


@pytest.mark.parametrize("shape", [(40, 63), (4, 631)])
def test_largest_one_level_grids(shape):
    """The whole solve is the coarsest-grid one, which is too slow on so many
    cells: it only has to run, to the same residual alone and in a batch."""
    opts = chhs.default_opts(precision=1, max_v=3)
    phi0 = inputs.spinodal(shape, 3, mean=-0.1, amplitude=0.05)
    with chhs.Batch([(shape, H, EPS, GAMMA, DT)], opts=opts) as b:
        b.runs[0].set_phi(phi0)
        status, v, resid = b.step(1, check=False)
    assert status[0] in (chhs.CHHS_OK, chhs.CHHS_ERR_NOT_CONVERGED) and np.isfinite(resid[0])
    with chhs.Run(shape, H, EPS, GAMMA, DT, opts=opts) as run:
        run.set_phi(phi0)
        try:
            assert (chhs.CHHS_OK, run.step(1)[2]) == (status[0], resid[0])
        except chhs.ChhsError as e:
            assert e.status == status[0]


def test_largest_two_level_tail():
    shape = (42, 48)
    phi, prev, mu, p = _steps(shape, tuning=((2048, 8192, 512, 2, 2), {}))
    assert oracle.residual(prev, prev, phi, mu, p, oracle.Params(H, EPS, GAMMA, DT))[3] <= 2e-10


def test_one_more_cell_is_refused():
    for shape in ((5, 505), (42, 50)):  # 2525 cells in one level; 2625 in two
        with pytest.raises(chhs.ChhsError) as e:
            _steps(shape, tuning=((4096, 8192, 512, 2, 2), {}))
        assert e.value.status == chhs.CHHS_ERR_INVALID_ARG


def test_tile_threads_matter_only_to_levels_that_ask_for_them():
    shape = (128, 128)  # every level above the tail is a small one
    ref = _steps(shape)
    assert _same(ref, _steps(shape, tuning=((1024, 8192, 1024, 2, 2), {})))
    assert _same(ref, _steps(shape, refused=((1024, 8192, 512, 2, 2), dict(small_tile=(16, 8, 1024)))))
    shape = (512, 512)  # the finest level is a large one
    assert _same(_steps(shape), _steps(shape, refused=((1024, 8192, 1024, 2, 2), {})))
    opts = chhs.default_opts(precision=1)
    with chhs.Batch([((64, 64), H, EPS, GAMMA, DT)], opts=opts) as b:
        b.set_tuning(1024, 2, 2, tile=(32, 32, 1024))
    with chhs.Batch([(shape, H, EPS, GAMMA, DT)], opts=opts) as b:
        with pytest.raises(chhs.ChhsError):
            b.set_tuning(1024, 2, 2, tile=(32, 32, 1024))
        b.step(1)


def test_refused_tuning_changes_nothing():
    shape = (64, 64)
    ref = _steps(shape, 2)
    # the whole grid in the tail: no room in shared memory
    assert _same(ref, _steps(shape, 2, refused=((4096, 8192, 512, 1, 1), dict(norm_f64_per8=8))))
    # what a setting left behind would have shown
    assert not _same(ref, _steps(shape, 2, tuning=((1024, 8192, 512, 2, 2), dict(norm_f64_per8=8))))
