"""The mixed form's one-block tails (chhs_tail2.cuh, chhs_tail3.cuh) against the
launches that do the same work when the tail starts lower, on shapes whose tail
really starts at another level with the two settings (asserted).

With the coarsest grid and at least one level above it in both tails the
arithmetic is the same: the fields must be equal bit for bit, on non-cubic
grids, ragged ones and with coarsest grids of more than 32 cells.  Against a
tail of the coarsest grid alone (the general code's solve) the rounding differs:
the V-cycle counts must be equal, and after one V-cycle from a solved state the
iterate's change and the residual norm must agree to 1e-3 (single precision,
2^-24, times the V-cycle's condition of at most some thousand; a wrong coarse
correction changes them by more than a hundredth)."""
import numpy as np
import pytest

from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

H, EPS, GAMMA, DT = 0.05, 0.06, 1.5, 0.005


def _levels(shape, coarsest):
    out = [tuple(shape)]
    while all(n % 2 == 0 and n // 2 >= coarsest for n in out[-1]):
        out.append(tuple(n // 2 for n in out[-1]))
    return out


def _tail_start(levels, cells):
    start = len(levels) - 1
    while start > 0 and np.prod(levels[start - 1]) <= cells:
        start -= 1
    return start


def _steps(shape, opts, tail, n=3):
    with chhs.Run(shape, H, EPS, GAMMA, DT, opts=opts) as run:
        run.set_tuning(tail, 8192, 512, opts.nu1, opts.nu2)
        run.set_phi(inputs.spinodal(shape, 9, mean=-0.1, amplitude=0.4))
        _, v, _ = run.step(n)
        return v, run.get_state()


@pytest.mark.parametrize("shape,coarsest,small,nu", [
    ((16, 16, 32), 2, 128, (2, 2)), ((32, 16, 16), 2, 128, (2, 2)), ((16, 32, 16), 2, 128, (1, 2)),
    ((16, 16, 24), 2, 96, (2, 2)), ((16, 24, 16), 2, 96, (2, 1)), ((24, 16, 16), 2, 96, (2, 2)),
    ((32, 64), 2, 32, (2, 2)), ((64, 32), 2, 128, (1, 2)), ((48, 80), 2, 60, (2, 2)), ((80, 48), 2, 240, (2, 1)),
    ((48, 80), 6, 240, (2, 2)), ((80, 48), 6, 240, (1, 1)), ((28, 36), 2, 252, (2, 2)), ((8, 8, 16), 2, 128, (2, 2)),
    ((12, 8, 8), 2, 96, (2, 2)),
])
def test_levels_of_the_tail_are_the_launches(shape, coarsest, small, nu):
    levels = _levels(shape, coarsest)
    a, b = _tail_start(levels, 1024), _tail_start(levels, small)
    assert a < b < len(levels) - 1
    opts = chhs.default_opts(precision=1, nu1=nu[0], nu2=nu[1], coarsest=coarsest)
    va, sa = _steps(shape, opts, 1024)
    vb, sb = _steps(shape, opts, small)
    assert va == vb
    for x, y in zip(sa, sb):
        assert np.array_equal(x, y)


@pytest.mark.parametrize("shape,coarsest", [
    ((16, 32, 48), 2), ((24, 40, 48), 2), ((48, 16, 80), 2), ((16, 16, 16), 4), ((16, 16, 24), 4), ((16, 32, 64), 2),
    ((64, 128), 8), ((48, 80), 6), ((72, 96), 9), ((40, 24), 2),
])
def test_coarsest_solve_against_the_general_one(shape, coarsest):
    levels = _levels(shape, coarsest)
    alone = int(np.prod(levels[-1]))
    assert _tail_start(levels, 1024) < _tail_start(levels, alone) == len(levels) - 1
    opts = chhs.default_opts(precision=1, coarsest=coarsest)
    va, sa = _steps(shape, opts, 1024)
    vb, sb = _steps(shape, opts, alone)
    assert va == vb
    assert np.max(np.abs(sa[0] - sb[0])) <= 1e-8
    one = chhs.default_opts(precision=1, coarsest=coarsest, max_v=1)
    seen = []
    for tail in (1024, alone):
        with chhs.Run(shape, H, EPS, GAMMA, DT, opts=one) as run:
            run.set_tuning(tail, 8192, 512, 2, 2)
            run.set_state(*sa)
            status, v, resid = run.step(1, check=False)
            assert v == 1 and status == chhs.CHHS_ERR_NOT_CONVERGED
            seen.append((resid, run.get_state()))
    (ra, a), (rb, b) = seen
    assert abs(ra - rb) <= 1e-3 * ra
    for q in (2, 3):  # mu and p of the iterate
        assert np.max(np.abs(a[q] - b[q])) <= 1e-3 * np.max(np.abs(a[q] - sa[q]))
