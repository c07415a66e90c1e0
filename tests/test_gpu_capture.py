"""Steps recorded by the caller's own stream capture, on key spaces of every scan form.

A recorded step has not run when the call returns, so nothing that it leaves on the device may be counted on by what
the host enqueues before the first replay: here steps on the same context, or a probe and the steps that clear what it
left (a recorded step does not, if it was recorded before).  The recorded pair of steps is then replayed twice, and a
direct step follows.  The run agrees with the same number of direct steps (nine at most) to
the rounding of the float atomics that meet at a node: 64 of them a step in the fused step, whose roundings add up like
a random walk (sqrt(9 * 64) * 2^-24 = 1.4e-6 of a node's sum in each of two runs), so 1e-5 of the largest velocity; and
positions to nine roundings of 2^-30 and the velocities' share (4 * 1e-5 * 9 steps of 1e-5): 1.5e-8.  The probed mass is
the particles' to the roundings of a node's sum: 1e-5."""
import numpy as np
import pytest
import torch

from gpu_helpers import f32, need_gpu, rel
from paper_2412_10399_gb300 import scenes as S

pytestmark = pytest.mark.gpu
DX = 1.0 / 1024


def _scene(res, n=3000):
    g = np.random.default_rng(6)
    x = f32((12.0 + 8.0 * g.random((n, 3))) * DX).astype(np.float64)
    v = f32(g.standard_normal((n, 3))).astype(np.float64)
    return S.Scene("capture", res, DX, 1e-5, x, v, np.zeros(n, np.uint8), [S.ELASTIC], gravity=(0.0, 0.0, 0.0))


@pytest.mark.parametrize("fused,between", [(False, "probe"), (False, "steps"), (False, "nothing"), (True, "steps"),
                                           (True, "nothing")])
@pytest.mark.parametrize("res", [32, 101, 700])  # no tile sums, tile sums a step leaves for the next, sums of its own
def test_recorded_steps_and_what_runs_before_their_replay(res, fused, between):
    ck = need_gpu()
    sc = _scene(res)
    code = ck.KERNEL_CK | (ck.STEP_G2P2G if fused else 0)
    direct = (2 if fused else 0) + (2 if between != "nothing" else 0)
    ref = ck.Simulation(sc, code)
    ref.step(direct + 5)
    want = ref.read(ck.FIELD_X), ref.read(ck.FIELD_V)
    ref.close()
    stream = torch.cuda.Stream()
    sim = ck.Simulation(sc, code, stream=stream.cuda_stream)
    if fused:  # the grid of a fused step comes from the step before
        sim.step(2)
    sim.sync()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph, stream=stream):
        sim.step(2)
    if between == "probe":
        sim.probe_grids()
        m = torch.empty(2, (res + 1) ** 3, device="cuda")
        torch.cuda.synchronize()
        ck.ckmpm_readback(sim.ctx, 0, ck.FIELD_GRID_M, m.data_ptr(), m.numel() * 4, True)
        mass = sc.n * S.ELASTIC.rho * DX ** 3 / sc.ppc
        assert (m.sum(1, dtype=torch.float64) / mass - 1.0).abs().max().item() <= 1e-5
    if between != "nothing":
        sim.step(2)
    with torch.cuda.stream(stream):
        graph.replay()
        graph.replay()
    sim.step(1)
    sim.sync()
    assert np.abs(sim.read(ck.FIELD_X) - want[0]).max() <= 1.5e-8
    assert rel(sim.read(ck.FIELD_V), want[1]) <= 1e-5
    sim.close()
