"""Differentiable stepper on its blocked grids: particles on block edges, scattered over the whole domain and in
warps that share a few blocks, counts that leave a warp partly filled, and the state the grids keep between calls.

Tolerances are those of the one-step parity tests against the float64 oracle (v 2e-5, B 5e-5, F 2e-6 relative to the
field's largest value; adjoints 2e-3); two calls on the same inputs differ by the order of float additions only
(at most 64 contributions a node: 64 * 2^-24 = 4e-6 of the largest value)."""
import numpy as np
import pytest
import torch

from gpu_helpers import f32, need_gpu, rel
from oracle import ckmpm_oracle as O
from paper_2412_10399_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _state(n, res, where, seed=3):
    x, v, B, F = S.random_state(n, res, seed, margin_cells=2.0, f_scale=0.08)
    dx = 1.0 / 32
    x = x * res * dx  # random_state works in a unit domain
    if where == "edges":  # within 1e-3 cells of node multiples of four and of the quarter offsets between grids
        g = np.random.default_rng(seed)
        c = 4.0 * g.integers(1, res // 4, (n, 3)) + g.choice([0.0, 0.25, -0.25, 0.75], (n, 3))
        x = (c + 1e-3 * (2 * g.random((n, 3)) - 1)) * dx
    elif where == "sorted":
        x = x[np.lexsort(x.T)]
    E = 1e5 * (0.5 + np.random.default_rng(seed + 1).random(n))
    sc = S.Scene("blocks", res, dx, 1e-4, f32(x).astype(np.float64), f32(v).astype(np.float64), np.zeros(n, np.uint8),
                 [S.Material(S.FIXED_COROTATED, 1e5, 0.3, 1000.0)])
    return sc, f32(B), f32(F), f32(E)


def _cuda(*arrs):
    return [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in arrs]


@pytest.mark.parametrize("n,res,where", [(1, 16, "scattered"), (33, 17, "edges"), (63, 18, "scattered"),
                                         (64, 19, "sorted"), (700, 31, "edges"), (2000, 32, "scattered")])
def test_step_and_adjoint_match_oracle(n, res, where):
    need_gpu()
    from paper_2412_10399_gb300 import diff
    sc, B, F, E = _state(n, res, where)
    sim = diff.DiffSim(sc)
    st = _cuda(f32(sc.x), f32(sc.v), B, F, E)
    out = sim.step(*st)
    t = [torch.from_numpy(a.astype(np.float64)).requires_grad_(True) for a in (f32(sc.x), f32(sc.v), B, F, E)]
    new = O.step(O.make_state(t[0], t[1], t[2], t[3], E=t[4]), O.params_from_scene(sc), newton=True)
    ref = [a.detach().numpy() for a in (new.x, new.v, new.B, new.F)]
    for got, want, tol in zip(out, ref, (2e-7, 2e-5, 5e-5, 2e-6)):
        assert rel(got.cpu().numpy(), want) <= tol
    g = np.random.default_rng(9)
    adj = [f32(g.standard_normal((n,) + s)) for s in ((3,), (3,), (3, 3), (3, 3))]
    want = torch.autograd.grad((new.x, new.v, new.B, new.F), t, [torch.from_numpy(a.astype(np.float64)) for a in adj])
    for _ in range(2):  # the second call finds the grids as the first left them
        gE = torch.zeros_like(st[4])
        got = sim.step_backward(*st, *_cuda(*adj), gE)
        for a, b in zip(got + (gE,), want):
            assert rel(a.cpu().numpy(), b.numpy()) <= 2e-3
    sim.sync()


def test_grids_are_clean_after_an_out_of_domain_particle_and_on_replay():
    ck = need_gpu()
    from paper_2412_10399_gb300 import diff
    sc, B, F, E = _state(1500, 32, "scattered", seed=8)
    s = torch.cuda.Stream()
    with torch.cuda.stream(s):
        sim = diff.DiffSim(sc)
        st = _cuda(f32(sc.x), f32(sc.v), B, F, E)
        want = [a.cpu().numpy() for a in sim.step(*st)]
        bad = st[0].clone()
        bad[7] = -1.0
        sim.step(bad, *st[1:])
        got = [a.cpu().numpy() for a in sim.step(*st)]
        for a, b in zip(got, want):
            assert rel(a, b) <= 4e-6
        with pytest.raises(ck.CKMPMError):  # the bad particle was reported
            sim.sync()
        graph = torch.cuda.CUDAGraph()
        with torch.cuda.graph(graph, stream=s):
            out = sim.step(*st)
        for _ in range(3):
            graph.replay()
        s.synchronize()
        for a, b in zip(out, want):
            assert rel(a.cpu().numpy(), b) <= 4e-6


@pytest.mark.parametrize("n", [1, 31, 33, 64, 65, 1000])
def test_readback_returns_rows_in_the_callers_order(n):
    """Whatever the binned order, a field written by upload is read back bit for bit."""
    ck = need_gpu()
    x, v, _, _ = S.random_state(n, 16, 5, margin_cells=3.0)
    sc = S.Scene("rows", 16, 1.0 / 16, 1e-4, f32(x).astype(np.float64), f32(v).astype(np.float64),
                 np.zeros(n, np.uint8), [S.ELASTIC])
    sim = ck.Simulation(sc)
    assert np.array_equal(sim.read(ck.FIELD_X), f32(x)) and np.array_equal(sim.read(ck.FIELD_V), f32(v))
    sim.step(3)
    g = np.random.default_rng(1)
    F = f32(np.eye(3) + 0.01 * g.standard_normal((n, 3, 3)))
    w = f32(g.standard_normal((n, 3)))
    sim.write(ck.FIELD_F, F)
    sim.write(ck.FIELD_V, w)
    assert np.array_equal(sim.read(ck.FIELD_F), F) and np.array_equal(sim.read(ck.FIELD_V), w)
    sim.close()
