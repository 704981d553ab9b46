"""chhs_tuning.norm_f64_per8: of every 8 blocks of the mixed form's residual
kernel, how many are evaluated with double-precision instructions.  From 4 to 8
they are, whatever the grid, so each setting rounds differently; fewer are none,
the same bits as 0.  With each setting the reported norm of a step is the
oracle's of the same fields within 0.1 % (as for the other settings), alone and
in a batch the same bits."""
import numpy as np
import pytest

import oracle
from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

H, EPS, GAMMA, DT = 0.05, 0.06, 1.5, 0.005


@pytest.mark.parametrize("shape", [(256, 256), (160, 28), (36, 40, 72)])
def test_share_of_double_precision_blocks(shape):
    phi0 = inputs.spinodal(shape, 5, mean=-0.1, amplitude=0.4)
    states = {}
    for per8 in (0, 1, 3, 4, 6, 7, 8):
        with chhs.Run(shape, H, EPS, GAMMA, DT, opts=chhs.default_opts(precision=1)) as run:
            run.set_tuning(256, 8192, 512, 2, 2, norm_f64_per8=per8)
            run.set_phi(phi0)
            run.step(1)
            before = run.get_state()
            _, _, resid = run.step(1)
            states[per8] = run.get_state()
        phi, _, mu, p = states[per8]
        norm = oracle.residual(before[0], before[1], phi, mu, p, oracle.Params(H, EPS, GAMMA, DT))[3]
        assert abs(resid - norm) <= 1e-3 * norm + 1e-14
        if per8 in (0, 6):
            with chhs.Batch([(shape, H, EPS, GAMMA, DT)]) as b:
                b.set_tuning(256, 2, 2, norm_f64_per8=per8)
                b.runs[0].set_phi(phi0)
                b.step(2)
                assert all(np.array_equal(x, y) for x, y in zip(b.runs[0].get_state(), states[per8]))
    for a in states:
        for b in states:
            same = all(np.array_equal(x, y) for x, y in zip(states[a], states[b]))
            assert same == (a == b or max(a, b) < 4), (a, b)
