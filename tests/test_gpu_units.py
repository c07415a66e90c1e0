"""Work units: a block's particles in parts, whatever the block holds.

The default rule against one unit per block (CKMPM_SPLITS=1) and a fixed count of parts, on a block fuller than its
parts' nominal size, one with a partly filled last chunk, blocks thinner than one part and a body spread over more
blocks than the rule wants units.  The parts of a block round by the same scale and meet in integer sums or float
atomics: positions agree to float32 rounding, velocities to the 64 contributions of a node in each of three steps
(1.2e-5 of the largest; with the kernel gradient, whose strain rates amplify a sparse node's rounding, one step at the
other tests' 2e-5)."""
import os

import numpy as np
import pytest

from gpu_helpers import need_gpu, random_scene, rel
from paper_2412_10399_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _run(ck, sc, B, F, code, splits):
    os.environ.pop("CKMPM_SPLITS", None)
    if splits:
        os.environ["CKMPM_SPLITS"] = str(splits)
    try:
        sim = ck.Simulation(sc, code)
    finally:
        os.environ.pop("CKMPM_SPLITS", None)
    sim.write(ck.FIELD_F, F)
    if not code & ck.TRANSFER_PIC:
        sim.write(ck.FIELD_B, B)
    sim.step(1 if code & 6 else 3)
    out = sim.read(ck.FIELD_X), sim.read(ck.FIELD_V), int(sim.stats().n_particle_blocks)
    sim.sync()
    sim.close()
    return out


@pytest.mark.parametrize("kernel", [S.KERNEL_CK, S.KERNEL_QUADRATIC])
@pytest.mark.parametrize("transfer", [0, 2, 4])
@pytest.mark.parametrize("n,box", [(3001, (9.0, 11.0)), (700, (9.0, 13.5)), (20000, None)])
def test_parts_of_blocks_give_the_step_of_whole_blocks(n, box, transfer, kernel):
    ck = need_gpu()
    sc, B, F = random_scene(n, 64 if box is None else 32, 41, kernel=kernel, f_scale=0.02, box=box, v_scale=0.5)
    code = kernel | transfer
    want = _run(ck, sc, B, F, code, 1)
    for splits in (None, 5):
        got = _run(ck, sc, B, F, code, splits)
        assert np.abs(got[0] - want[0]).max() <= 1e-6 * sc.dx + 2e-7
        assert rel(got[1], want[1]) <= (1.2e-5 if transfer == 0 else 2e-5)
    assert box is not None or want[2] > 2000
