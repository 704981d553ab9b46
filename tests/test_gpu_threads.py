"""Handles of different sizes created and stepped by several threads at once:
their kernels' opt-ins to shared memory are process-wide and differ from size to
size (the cluster of 2D double precision, the 2D and 3D tails), and no thread
may lower another's.  Every step must give the same bits as alone."""
import threading

import numpy as np
import pytest

from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu

RUNS = [((64, 64), 0), ((32, 48), 0), ((16, 24), 0), ((64, 64), 1), ((40, 24), 1), ((36, 36), 1), ((16, 16, 16), 1),
        ((12, 8, 8), 1)]


def _run(shape, precision):
    with chhs.Run(shape, 0.05, 0.06, 1.5, 0.005, opts=chhs.default_opts(precision=precision)) as run:
        run.set_phi(inputs.spinodal(shape, 5, mean=-0.1, amplitude=0.3))
        run.step(2)
        return run.get_state()


def test_threads_create_and_step():
    got, failed = [], []

    def work(k):
        try:
            for q in range(4):
                r = RUNS[(k + q) % len(RUNS)]
                got.append((r, _run(*r)))
        except Exception as e:
            failed.append((k, e))

    threads = [threading.Thread(target=work, args=(k,)) for k in range(len(RUNS))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not failed
    alone = {r: _run(*r) for r in RUNS}
    for r, state in got:
        assert all(np.array_equal(a, b) for a, b in zip(state, alone[r])), r
