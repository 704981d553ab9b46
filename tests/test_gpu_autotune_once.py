"""The autotuners time settings that give the same launches once: of equal ones
the first of their lists may be chosen, never a later one.  In the 2D mixed form
a block size changes no launch, a run without levels of 512 x 256 cells takes
none of the large levels' tile shapes, and a batch without levels of 65 536
cells neither."""
import pytest

from paper_1611_02967_gb300 import chhs, inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(64, 64), (128, 96)])
def test_run(shape):
    with chhs.Run(shape, 0.05, 0.06, 1.5, 0.005, opts=chhs.default_opts(precision=1)) as run:
        run.set_phi(inputs.spinodal(shape, 41, mean=0.0, amplitude=0.3))
        for _ in range(6):
            t = run.autotune(1)
            tile = (t["tile_w"], t["tile_h"], t["tile_threads"])
            assert tile != (32, 16, 512)
            if t["small_tile"] == (16, 8, 256):
                assert tile == (32, 16, 256)
            else:
                assert t["small_tile"] == tile


def test_batch():
    runs = [((64, 64), 0.05, 0.06, 1.5, 0.005), ((128, 64), 0.05, 0.06, 1.5, 0.005)]
    with chhs.Batch(runs) as b:
        for r in b.runs:
            r.set_phi(inputs.spinodal(r.shape, 41, mean=0.0, amplitude=0.3))
        for _ in range(4):
            assert b.autotune(1)["tile"] == (32, 16, 512)
