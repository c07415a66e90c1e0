"""The differentiable step's rotation factor: strains up to 60 per cent, compression to the edge of the iteration's
range and beyond it, and inverted F, each against the float64 oracle.  Tolerances: the one-step parity tests' (v 2e-5,
F 2e-6) and their 2e-3 for adjoints (well-conditioned F, where the oracle's autograd is defined)."""
import numpy as np
import pytest
import torch

from gpu_helpers import f32, need_gpu, rel
from oracle import ckmpm_oracle as O
from paper_2412_10399_gb300 import scenes as S

pytestmark = pytest.mark.gpu


def _stretched(n, sig, seed=2):
    """Random rotations times diag(sig) (jittered) in random axes, spread so that no two particles share a node."""
    g = np.random.default_rng(seed)
    Q = [np.linalg.qr(g.standard_normal((n, 3, 3)))[0] for _ in range(2)]
    Q = [q * np.sign(np.linalg.det(q))[:, None, None] for q in Q]
    s = np.asarray(sig) * (1.0 + 0.02 * g.standard_normal((n, 3)))
    F = np.einsum("nij,nj,nkj->nik", Q[0], s, Q[1])
    i = np.arange(n)
    x = (np.stack([i % 8, (i // 8) % 8, i // 64], 1) * 4.0 + 6.0 + g.random((n, 3))) / 64
    sc = S.Scene("stretch", 40, 1.0 / 64, 1e-4, f32(x).astype(np.float64), f32(g.standard_normal((n, 3))).astype(np.float64),
                 np.zeros(n, np.uint8),
                 [S.Material(S.FIXED_COROTATED, 1e5, 0.3, 1000.0)], gravity=(0.0, 0.0, 0.0))
    return sc, f32(0.1 * sc.dx * g.standard_normal((n, 3, 3))), f32(F), f32(1e5 * (0.5 + g.random(n)))


@pytest.mark.parametrize("sig,adjoint", [((1.6, 1.0, 0.7), True), ((1.0, 1.0, 1.0), True), ((3.0, 2.5, 2.0), True),
                                         ((0.5, 0.45, 0.4), True), ((0.9, 0.4, 0.1), False), ((1.1, 0.9, -0.8), False)])
def test_step_with_stretched_and_inverted_F(sig, adjoint):
    need_gpu()
    from paper_2412_10399_gb300 import diff
    sc, B, F, E = _stretched(100, sig)
    n = sc.n
    sim = diff.DiffSim(sc)
    st = [torch.from_numpy(np.ascontiguousarray(a)).cuda() for a in (f32(sc.x), f32(sc.v), B, F, E)]
    out = sim.step(*st)
    t = [torch.from_numpy(a.astype(np.float64)).requires_grad_(adjoint) for a in (f32(sc.x), f32(sc.v), B, F, E)]
    new = O.step(O.make_state(t[0], t[1], t[2], t[3], E=t[4]), O.params_from_scene(sc), newton=adjoint)
    assert rel(out[1].cpu().numpy(), new.v.detach().numpy()) <= 2e-5
    assert rel(out[3].cpu().numpy(), new.F.detach().numpy()) <= 2e-6
    if not adjoint:
        return
    g = np.random.default_rng(9)
    adj = [f32(g.standard_normal((n,) + s)) for s in ((3,), (3,), (3, 3), (3, 3))]
    want = torch.autograd.grad((new.x, new.v, new.B, new.F), t, [torch.from_numpy(a.astype(np.float64)) for a in adj])
    gE = torch.zeros_like(st[4])
    got = sim.step_backward(*st, *[torch.from_numpy(a).cuda() for a in adj], gE)
    for a, b in zip(got + (gE,), want):
        assert rel(a.cpu().numpy(), b.numpy()) <= 2e-3
