"""P2G of the kernel-gradient transfers in full blocks, against the float64 oracle.

8 particles per cell over cells [8, 24)^3: the 64 inner particle blocks hold about 512 particles each (and those on the
rim fewer than 256), so both roundings of the fixed-point scatter are taken, by every lane rotation.  Tolerance: the
1e-5 of the other grid parity tests, per field and grid."""
import numpy as np
import pytest

from gpu_helpers import need_gpu, oracle_state, random_scene, rel
from oracle import ckmpm_oracle as O
from paper_2412_10399_gb300 import scenes as S

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kernel", [S.KERNEL_CK, S.KERNEL_QUADRATIC])
@pytest.mark.parametrize("transfer", [S.TRANSFER_PIC, S.TRANSFER_APIC_GRAD])
def test_kernel_gradient_p2g_in_full_blocks(kernel, transfer):
    ck = need_gpu()
    sc, B, F = random_scene(32771, 32, 14, model=S.DRUCKER_PRAGER, kernel=kernel, f_scale=0.08, box=(8.0, 24.0))
    sc.transfer = transfer
    if transfer == S.TRANSFER_PIC:
        B = np.zeros_like(B)
    sim = ck.Simulation(sc, ck.kernel_code(sc))
    sim.write(ck.FIELD_F, F)
    if transfer != S.TRANSFER_PIC:
        sim.write(ck.FIELD_B, B)
    sim.probe_grids()
    gm, gp = sim.read(ck.FIELD_GRID_M), sim.read(ck.FIELD_GRID_P)
    sim.close()
    grids = O.p2g(oracle_state(sc, B, F), O.params_from_scene(sc))
    nn = sc.res + 1
    for gi, k in enumerate(O.grid_ids(kernel)):
        assert rel(gm[gi], grids[k][0].numpy().reshape(nn, nn, nn)) <= 1e-5
        assert rel(gp[gi], grids[k][1].numpy().reshape(nn, nn, nn, 3)) <= 1e-5
