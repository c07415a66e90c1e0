"""Workloads for measuring the framework: what is timed, on which inputs, and what comes out.

Each case is one use of the framework through its public entry points:

  steps    a simulation advanced by a few time steps whose state is then read back (a frame of a
           solver run): ``Simulation.step`` and ``ckmpm_readback`` into device memory
  grids    the allocation-free particle-to-grid transfer (``ckmpm_p2g_grids_static``)
  served   requests of uneven size admitted to a resident context, stepped together, read back and
           released (``ckmpm_admit`` ... ``ckmpm_release``)
  forward  one differentiable step (``DiffSim.step``)
  adjoint  its vector-Jacobian product (``DiffSim.step_backward``)
  rollout  a differentiable rollout with its gradients (``Rollout``)

``exact`` restates the method in float64 torch (weights, transfers, materials) and shares no code
with the framework.
"""
import math

import numpy as np
import torch

from paper_2412_10399_gb300 import ckmpm as ck
from paper_2412_10399_gb300 import scenes as S

ELASTIC, SAND, FLUID, MIXED = "elastic", "sand", "fluid", "mixed"

# (E, nu, rho, friction angle, gamma) of the repository's scenes
_PARAMS = {
    ELASTIC: [S.ELASTIC],
    SAND: [S.SAND],
    FLUID: [S.FLUID],
    MIXED: [S.SAND, S.STIFF_BALL],
}


def listed():
    return [
        # the allocation-free transfer of a small body: the smallest call, bound by launches
        dict(name="grids_small", what="grids", res=32, nx=8, ny=8, nz=8, drop=0, material=ELASTIC, kernel="ck"),
        # the elastic cube on 64^3, ten steps a frame: an interactive soft body, bound by latency
        dict(name="cube", what="steps", shape="box", res=64, grid=64, nx=16, ny=16, nz=16, drop=0, material=ELASTIC,
             kernel="ck", transfer="apic", steps=10, dt=1e-4),
        # the granular column on 128^3 with the compact kernel and with the quadratic B-spline
        dict(name="column", what="steps", shape="box", res=128, grid=128, nx=26, ny=64, nz=26, drop=0, material=SAND,
             kernel="ck", transfer="apic", steps=4, dt=5e-5),
        dict(name="column_quadratic", what="steps", shape="box", res=128, grid=128, nx=26, ny=64, nz=26, drop=0,
             material=SAND, kernel="quadratic", transfer="apic", steps=4, dt=5e-5),
        # the diffusion bar on 256^3 under the two kernel-gradient transfers, ragged counts
        dict(name="bar_pic", what="steps", shape="box", res=256, grid=256, nx=20, ny=10, nz=140, drop=3,
             material=ELASTIC, kernel="ck", transfer="pic", steps=4, dt=2e-5),
        dict(name="bar_apic_grad", what="steps", shape="box", res=256, grid=256, nx=20, ny=10, nz=140, drop=5,
             material=ELASTIC, kernel="ck", transfer="apic_grad", steps=4, dt=2e-5),
        # the dam break on 256^3: fluid particles in no order, filling the domain's corner
        dict(name="dam", what="steps", shape="dam", res=256, grid=256, n=4175808, material=FLUID, kernel="ck",
             transfer="apic", steps=4, dt=1e-4),
        # the large impact on 512^3: a sand castle struck by stiff balls, 16,273,664 particles
        dict(name="impact", what="steps", shape="castle", res=512, grid=512, material=MIXED, kernel="ck",
             transfer="apic", steps=4, dt=2e-5),
        # eight requests of uneven size served together for twenty steps
        dict(name="served", what="served", scenes=8, n_min=10000, n_max=200000, res=64, kernel="ck", steps=20),
        # the differentiable cube on 128^3 (262,144 particles): one step, its adjoint, and a short rollout
        dict(name="diff_forward", what="forward", res=128, grid=128, nx=32, ny=32, nz=32, drop=0, dt=1e-4),
        dict(name="diff_adjoint", what="adjoint", res=128, grid=128, nx=32, ny=32, nz=32, drop=0, dt=1e-4),
        dict(name="rollout", what="rollout", res=64, grid=64, nx=16, ny=16, nz=16, drop=0, dt=1e-4, steps=16, k=8),
    ]


def _draw_box(rng, res, n_lo, n_hi):
    """Cells of a box of about n particles (8 per cell) that fits res^3 with a margin, and how many of its
    particles are left out."""
    top = res - 14
    n = math.exp(rng.uniform(math.log(n_lo), math.log(min(n_hi, 8 * top ** 3))))
    side = (n / 8.0) ** (1.0 / 3.0)
    a, b = rng.uniform(0.6, 1.6), rng.uniform(0.6, 1.6)
    dims = [max(2, min(top, int(round(side * f)))) for f in (a, b, 1.0 / (a * b))]
    return dict(nx=dims[0], ny=dims[1], nz=dims[2], drop=rng.randint(0, 7))


def draw(rng):
    what = rng.choice(["steps", "steps", "steps", "steps", "grids", "served", "forward", "adjoint", "rollout"])
    if what == "grids":
        res = rng.randint(20, 64)
        return dict(what=what, res=res, **_draw_box(rng, res, 500, 40000), material=rng.choice([ELASTIC, SAND]),
                    kernel=rng.choice(["ck", "quadratic"]))
    if what == "served":
        return dict(what=what, scenes=rng.randint(2, 12), n_min=rng.randint(2000, 10000),
                    n_max=rng.randint(50000, 200000), res=rng.choice([48, 64, 72]),
                    kernel=rng.choice(["ck", "ck", "quadratic"]), steps=rng.randint(5, 20))
    if what in ("forward", "adjoint", "rollout"):
        grid = rng.choice([32, 64, 128])
        res = grid if rng.random() < 0.5 else grid - rng.randint(1, 9)
        c = dict(what=what, res=res, grid=grid, **_draw_box(rng, res, 2000, 300000 if what != "rollout" else 60000),
                 dt=1e-4)
        return c if what != "rollout" else dict(c, steps=rng.randint(4, 16), k=rng.randint(2, 8))
    grid = rng.choice([32, 64, 128, 256, 512])
    res = grid if rng.random() < 0.5 else grid - rng.randint(1, grid // 8)
    material = rng.choice([ELASTIC, SAND, SAND, FLUID])
    transfer = rng.choice(["apic", "apic", "apic", "pic", "apic_grad"])
    dt = {ELASTIC: 1e-4, SAND: 5e-5, FLUID: 1e-4}[material] * min(1.0, 128.0 / grid)
    return dict(what="steps", shape="box", res=res, grid=grid, **_draw_box(rng, res, 2000, 8e6), material=material,
                kernel=rng.choice(["ck", "ck", "quadratic"]), transfer=transfer, steps=rng.randint(2, 6), dt=dt)


# ------------------------------------------------------------------------------------ inputs

def _gen(seed, device):
    g = torch.Generator(device=device)
    g.manual_seed(int(seed))
    return g


def _device():
    return "cuda" if torch.cuda.is_available() else "cpu"


def _fill(mask, dx, g):
    """8 stratified particles in every True cell of mask [z, y, x], cells in scan order."""
    cells = mask.nonzero()  # (m, 3): z, y, x
    m = cells.shape[0]
    sub = torch.arange(8, device=mask.device)
    off = torch.stack([sub & 1, (sub >> 1) & 1, (sub >> 2) & 1], -1).double() * 0.5
    u = torch.rand(m, 8, 3, generator=g, device=mask.device, dtype=torch.float64) * 0.5
    x = (cells.flip(1).double()[:, None, :] + off[None] + u) * dx
    return x.reshape(-1, 3)


def _box_mask(case, device):
    res = case["res"]
    d = [case["nx"], case["ny"], case["nz"]]
    lo = [(res - k) // 2 for k in d]
    mask = torch.zeros(res, res, res, dtype=torch.bool, device=device)
    mask[lo[2]:lo[2] + d[2], lo[1]:lo[1] + d[1], lo[0]:lo[0] + d[0]] = True
    return mask


def _castle(device):
    """Sand cells of the large-impact scene and its four balls with their directions."""
    r = torch.arange(512, device=device, dtype=torch.float32) + 0.5
    cx, cy, cz = r[None, None, :], r[None, :, None], r[:, None, None]

    def box(lo, hi):
        return ((cx >= lo[0]) & (cx < hi[0]) & (cy >= lo[1]) & (cy < hi[1]) & (cz >= lo[2]) & (cz < hi[2]))

    sand = box((154, 4, 154), (358, 36, 358)) | box((226, 36, 226), (286, 86, 286))
    for tx in (174, 338):
        for tz in (174, 338):
            sand |= ((cx - tx) ** 2 + (cz - tz) ** 2 < 400.0) & (cy >= 36) & (cy < 136)
    balls = []
    for c in ((201, 60, 256), (311, 60, 256), (256, 60, 201), (256, 60, 311)):
        m = (cx - c[0]) ** 2 + (cy - c[1]) ** 2 + (cz - c[2]) ** 2 < 100.0
        d = np.array([256.0 - c[0], 0.0, 256.0 - c[2]])
        balls.append((m, d / np.linalg.norm(d)))
    return sand, balls


def _particles(case, seed):
    """Positions, velocities, deformation gradients (float32) and material indices of a case."""
    dev = _device()
    g = _gen(seed, dev)
    shape = case.get("shape", "box")
    dx = 1.0 / case.get("grid", case["res"])

    def rand(*s):
        return torch.rand(*s, generator=g, device=dev, dtype=torch.float64)

    def randn(*s):
        return torch.randn(*s, generator=g, device=dev, dtype=torch.float64)

    mat = None
    if shape == "castle":
        sand, balls = _castle(dev)
        xs, vs = [_fill(sand, dx, g)], []
        vs.append(0.01 * randn(xs[0].shape[0], 3))
        for m, d in balls:
            xs.append(_fill(m, dx, g))
            vs.append(torch.tensor(20.0 * d, device=dev).expand(xs[-1].shape[0], 3))
        mat = torch.cat([torch.full((x.shape[0],), int(i > 0), dtype=torch.uint8, device=dev)
                         for i, x in enumerate(xs)])
        x, v = torch.cat(xs), torch.cat(vs)
    else:
        if shape == "dam":
            n, w = case["n"], 96.0
            x = (4.0 + rand(n, 3) * torch.tensor([w, n / 8.0 / (w * w), w], device=dev, dtype=torch.float64)) * dx
        else:
            x = _fill(_box_mask(case, dev), dx, g)
            x = x[:x.shape[0] - case["drop"]].contiguous()
        # a body in flight: a common velocity, a linear field (spin and strain) and a little noise
        base = torch.nn.functional.normalize(randn(1, 3), dim=1)
        lin = 2.0 * randn(3, 3)
        v = base + (x - x.mean(0)) @ lin.T + 0.05 * randn(x.shape[0], 3)
    n = x.shape[0]
    eye = torch.eye(3, device=dev, dtype=torch.float64)
    amount = {ELASTIC: 0.02, SAND: 0.003, MIXED: 0.001, FLUID: 0.005}[case.get("material", ELASTIC)]
    if case.get("material") == FLUID:  # the fluid keeps only its volume ratio
        F = eye * (1.0 + amount * (2.0 * rand(n, 1, 1) - 1.0))
    else:
        F = eye * (1.0 - 0.5 * amount) + amount * (2.0 * rand(n, 3, 3) - 1.0)
    return x.float().contiguous(), v.float().contiguous(), F.float().contiguous(), mat


def _diff_inputs(case, seed):
    """A state of the differentiable cube in motion, per-particle stiffness and adjoints of the outputs."""
    x, _, _, _ = _particles(dict(case, material=ELASTIC), seed)
    g = _gen(seed + 1000003, x.device)
    n = x.shape[0]

    def randn(*s):
        return torch.randn(*s, generator=g, device=x.device, dtype=torch.float32)

    v = 0.5 * randn(n, 3)
    v[:, 0] += 0.5
    dx = 1.0 / case["grid"]
    eye = torch.eye(3, device=x.device)
    F = (eye + 0.05 * (2.0 * torch.rand(n, 3, 3, generator=g, device=x.device) - 1.0)).contiguous()
    B = dx * 0.2 * randn(n, 3, 3)
    E = 1e5 * (0.75 + 0.5 * torch.rand(n, generator=g, device=x.device))
    adj = (randn(n, 3), randn(n, 3), 10.0 * randn(n, 3, 3), randn(n, 3, 3))
    return x, v, B, F, E, adj


def _requests(case, seed):
    """The scenes of a served case: boxes of log-uniform size, elastic or sand, falling."""
    g = np.random.default_rng(seed)
    out = []
    for s in range(case["scenes"]):
        # sizes belong to the case, not to the seed: passes on other inputs have the same work
        h = np.random.default_rng(7 * s + case["scenes"])
        n = math.exp(h.uniform(math.log(case["n_min"]), math.log(case["n_max"])))
        a = max(2, int(round((n / 8.0) ** (1.0 / 3.0))))
        c = dict(res=case["res"], nx=a, ny=min(case["res"] - 14, a + s % 3), nz=max(2, a - s % 2), drop=s % 8,
                 material=SAND if s % 2 else ELASTIC, dt=5e-5 if s % 2 else 1e-4, kernel=case["kernel"],
                 grid=64 if case["res"] <= 64 else 128, transfer="apic")
        x, v, _, _ = _particles(c, int(g.integers(1 << 30)))
        out.append((c, x, (2.0 * v).contiguous()))
    return out


def _scene(case, x, v, mat=None):
    gravity = (0.0, 0.0, 0.0) if case["material"] == ELASTIC and case.get("dt") == 2e-5 else (0.0, -9.8, 0.0)
    grid = case.get("grid", case["res"])
    return S.Scene("case", case["res"], 1.0 / grid, case.get("dt", 1e-4), x, v, mat, _PARAMS[case["material"]],
                   gravity=gravity, kernel=S.KERNEL_CK if case["kernel"] == "ck" else S.KERNEL_QUADRATIC,
                   transfer={"apic": 0, "pic": 1, "apic_grad": 2}[case.get("transfer", "apic")])


# ------------------------------------------------------------------------------------ the passes

class _Server:
    """A resident context sized for a case's requests."""

    def __init__(self, reqs, kernel):
        cfg = ck.ckmpm_config()
        cfg.kernel = kernel
        npb = [-(-c["res"] // 4) for c, _, _ in reqs]
        # room for a second generation: a released request's particles leave at the next step
        cfg.max_particles = 2 * sum(x.shape[0] for _, x, _ in reqs)
        cfg.max_keys = sum(k ** 3 for k in npb)
        cfg.max_virtual_blocks = sum((k + 1) ** 3 for k in npb)
        cfg.max_grid_blocks = sum(min((k + 1) ** 3, x.shape[0] // 64 + 64) for k, (_, x, _) in zip(npb, reqs))
        cfg.max_scenes = len(reqs)
        cfg.max_materials = 4 * len(reqs)
        self.ctx = ck.ckmpm_create_server(cfg)

    def __del__(self):
        ck.ckmpm_destroy(self.ctx)


def prepare(case, seed):
    what = case["what"]
    st = {"case": case}
    if what == "steps":
        x, v, F, mat = _particles(case, seed)
        scene = _scene(case, x, v, mat)
        torch.cuda.synchronize()
        st["sim"] = ck.Simulation(scene, x=x, v=v)
        ck.ckmpm_upload(st["sim"].ctx, 0, ck.FIELD_F, F.data_ptr(), F.numel() * 4, True)
        st["out"] = {"x": torch.empty_like(x), "v": torch.empty_like(v), "F": torch.empty_like(F)}
    elif what == "grids":
        x, v, F, _ = _particles(case, seed)
        B = (0.2 / case["res"]) * torch.randn(F.shape, generator=_gen(seed + 17, F.device), device=F.device)
        sc, keep = ck.scene_struct(_scene(dict(case, transfer="apic"), x, v), x=x, v=v)
        ng, nn = (2 if case["kernel"] == "ck" else 1), case["res"] + 1
        st.update(scene=sc, keep=keep, B=B, F=F, kernel=ck.KERNEL_CK if case["kernel"] == "ck" else ck.KERNEL_QUADRATIC)
        st["out"] = {"m": torch.empty(ng, nn, nn, nn, device=x.device), "p": torch.empty(ng, nn, nn, nn, 3, device=x.device)}
    elif what == "served":
        reqs = _requests(case, seed)
        st["reqs"] = [(_scene(c, x, v), x, v) for c, x, v in reqs]
        st["server"] = _Server(reqs, ck.KERNEL_CK if case["kernel"] == "ck" else ck.KERNEL_QUADRATIC)
        st["out"] = [{"x": torch.empty_like(x), "v": torch.empty_like(v)} for _, x, v in reqs]
    else:
        from paper_2412_10399_gb300 import diff
        x, v, B, F, E, adj = _diff_inputs(case, seed)
        scene = S.Scene("case", case["res"], 1.0 / case["grid"], case["dt"], np.zeros((x.shape[0], 3)),
                        np.zeros((1, 3)), None, [S.ELASTIC])
        st.update(sim=diff.DiffSim(scene), state=(x, v, B, F, E), adj=adj, rollout=diff.Rollout)
    torch.cuda.synchronize()
    return st


def run(st):
    case = st["case"]
    what = case["what"]
    if what == "steps":
        sim, out = st["sim"], st["out"]
        sim.step(case["steps"])
        for field, t in ((ck.FIELD_X, out["x"]), (ck.FIELD_V, out["v"]), (ck.FIELD_F, out["F"])):
            ck.ckmpm_readback(sim.ctx, 0, field, t.data_ptr(), t.numel() * 4, True)
        return out
    if what == "grids":
        out = st["out"]
        ck.ckmpm_p2g_grids_static(st["scene"], st["kernel"], st["B"].data_ptr(), st["F"].data_ptr(),
                                  out["m"].data_ptr(), out["p"].data_ptr())
        return out
    if what == "served":
        ctx = st["server"].ctx
        ids = []
        for scene, x, v in st["reqs"]:
            sc, keep = ck.scene_struct(scene, x=x, v=v)
            ids.append(ck.ckmpm_admit(ctx, sc))
        ck.ckmpm_step(ctx, case["steps"])
        for sid, out in zip(ids, st["out"]):
            ck.ckmpm_readback(ctx, sid, ck.FIELD_X, out["x"].data_ptr(), out["x"].numel() * 4, True)
            ck.ckmpm_readback(ctx, sid, ck.FIELD_V, out["v"].data_ptr(), out["v"].numel() * 4, True)
            ck.ckmpm_release(ctx, sid)
        return st["out"]
    sim, (x, v, B, F, E) = st["sim"], st["state"]
    if what == "forward":
        return dict(zip(("x", "v", "B", "F"), sim.step(x, v, B, F, E)))
    if what == "adjoint":
        gE = torch.zeros_like(E)
        got = sim.step_backward(x, v, B, F, E, *st["adj"], gE)
        return dict(zip(("gx", "gv", "gB", "gF", "gE"), got + (gE,)))
    leaf = [t.detach().requires_grad_(True) for t in (x, v, E)]
    xT, vT = st["rollout"].apply(*leaf, sim, case["steps"], case["k"])
    grads = torch.autograd.grad((xT, vT), leaf, st["adj"][:2])
    return dict(zip(("x", "v", "gx", "gv", "gE"), (xT, vT) + tuple(grads)))


# ------------------------------------------------------------------------------------ the work

def _count(case):
    if case.get("shape") == "castle":
        return 16273664
    if case.get("shape") == "dam":
        return case["n"]
    return 8 * case["nx"] * case["ny"] * case["nz"] - case["drop"]


def work(case):
    what = case["what"]
    ng, stencil = (2, 16) if case.get("kernel", "ck") == "ck" else (1, 27)
    flops = 420 + 62 * stencil  # of one particle's step: stencil, transfers both ways, update
    # a step reads and writes x, v, F (and B) once; at 8 per cell a particle has ng / 8 nodes, whose four
    # sums are written and read once and whose three velocities are written and read once
    nodes = ng / 8.0 * (2 * 16 + 2 * 12)
    if what == "grids":
        nn = (case["res"] + 1) ** 3
        return {"bytes": _count(case) * 96.0 + 16.0 * ng * nn, "flops": _count(case) * (200.0 + 20 * stencil)}
    if what == "served":
        n = 0
        for s in range(case["scenes"]):
            h = np.random.default_rng(7 * s + case["scenes"])
            n += math.exp(h.uniform(math.log(case["n_min"]), math.log(case["n_max"])))
        return {"bytes": n * (case["steps"] * (192 + nodes) + 48), "flops": n * case["steps"] * flops}
    n = _count(case)
    if what == "steps":
        b = 120 if case["transfer"] == "pic" else 192
        return {"bytes": n * (case["steps"] * (b + nodes) + 60.0), "flops": n * case["steps"] * flops}
    fwd, bwd = 100 + 96 + nodes, 100 + 96 + 96 + 8 + 2 * nodes
    if what == "forward":
        return {"bytes": n * fwd, "flops": n * flops}
    if what == "adjoint":
        return {"bytes": n * bwd, "flops": n * 3.0 * flops}
    return {"bytes": n * case["steps"] * (2 * fwd + bwd), "flops": n * case["steps"] * 5.0 * flops}


# ------------------------------------------------------------------------------------ in 64 bits

def _mm(a, b):
    return (a[:, :, :, None] * b[:, None, :, :]).sum(2)


def _cof(a):
    r = [a[:, i] for i in range(3)]
    return torch.stack([torch.linalg.cross(r[1], r[2]), torch.linalg.cross(r[2], r[0]),
                        torch.linalg.cross(r[0], r[1])], 1)


def _det(a):
    return (a[:, 0] * torch.linalg.cross(a[:, 1], a[:, 2])).sum(-1)


def _polar(F):
    """Rotation of the polar decomposition by Newton's iteration R <- (R + R^-T) / 2."""
    R = F
    for _ in range(9):
        C = _cof(R)
        R = 0.5 * (R + C / (R[:, 0] * C[:, 0]).sum(-1)[:, None, None])
    return R


def _eig3(S):
    """Eigenvalues and vectors of symmetric 3x3 matrices by cyclic Jacobi rotations."""
    S = S.clone()
    U = torch.eye(3, dtype=S.dtype, device=S.device).expand(S.shape[0], 3, 3).clone()
    for _ in range(6):
        for p, q in ((0, 1), (0, 2), (1, 2)):
            apq = S[:, p, q]
            th = (S[:, q, q] - S[:, p, p]) / (2.0 * torch.where(apq == 0, torch.ones_like(apq), apq))
            t = torch.where(th >= 0, 1.0, -1.0) / (th.abs() + (th * th + 1.0).sqrt())
            t = torch.where(apq == 0, torch.zeros_like(t), t)
            c = (1.0 / (t * t + 1.0).sqrt())[:, None]
            s = t[:, None] * c
            for M, rows in ((S, True), (S, False), (U, False)):
                a, b = (M[:, p, :].clone(), M[:, q, :].clone()) if rows else (M[:, :, p].clone(), M[:, :, q].clone())
                if rows:
                    M[:, p, :], M[:, q, :] = c * a - s * b, s * a + c * b
                else:
                    M[:, :, p], M[:, :, q] = c * a - s * b, s * a + c * b
    return torch.diagonal(S, dim1=1, dim2=2).clone(), U


def _log_strain(F):
    e, U = _eig3(_mm(F, F.transpose(1, 2)))
    return 0.5 * e.log(), U


def _from(U, d):
    return _mm(U * d[:, None, :], U.transpose(1, 2))


def _lame(m, E=None):
    E = m.E if E is None else E
    return E / (2.0 * (1.0 + m.nu)), E * m.nu / ((1.0 + m.nu) * (1.0 - 2.0 * m.nu))


def _stress(m, F, E=None):
    eye = torch.eye(3, dtype=F.dtype, device=F.device)
    mu, lam = _lame(m, E)
    if torch.is_tensor(mu):
        mu, lam = mu[:, None, None], lam[:, None, None]
    if m.model == S.J_FLUID:
        J = _det(F)
        return (-J * m.E * (J ** -m.gamma - 1.0))[:, None, None] * eye
    if m.model == S.DRUCKER_PRAGER:
        eps, U = _log_strain(F)
        return _from(U, 2.0 * mu * eps + lam * eps.sum(1, keepdim=True))
    J = _det(F)[:, None, None]
    return 2.0 * mu * _mm(F - _polar(F), F.transpose(1, 2)) + lam * J * (J - 1.0) * eye


def _plastic(m, F):
    if m.model == S.J_FLUID:
        return _det(F).pow(1.0 / 3.0)[:, None, None] * torch.eye(3, dtype=F.dtype, device=F.device)
    if m.model == S.FIXED_COROTATED:
        return F
    mu, lam = _lame(m)
    eps, U = _log_strain(F)
    tr = eps.sum(1, keepdim=True)
    dev = eps - tr / 3.0
    nrm = dev.norm(dim=1, keepdim=True)
    s = math.sin(math.radians(m.friction_deg))
    alpha = math.sqrt(2.0 / 3.0) * 2.0 * s / (3.0 - s)
    dg = nrm + (3.0 * lam + 2.0 * mu) / (2.0 * mu) * tr * alpha
    new = torch.where(tr >= 0, torch.zeros_like(eps),
                      torch.where((dg > 0) & (nrm > 0), eps - dg * dev / nrm.clamp_min(1e-300), eps))
    return _mm(_from(U, (new - eps).exp()), F)


def _per_material(fn, mats, mat, F):
    if len(mats) == 1:
        return fn(mats[0], F)
    out = torch.empty_like(F)
    for i, m in enumerate(mats):
        at = (mat == i).nonzero()[:, 0]
        out[at] = fn(m, F[at])
    return out


class _Stencil:
    """Nodes, weights, offsets (cells) and weight gradients of one grid; node i sits at i + shift cells."""

    def __init__(self, u, quadratic, shift):
        base = torch.floor(u - (0.5 if quadratic else shift))
        f = u - shift - base
        self.base, self.N = base.long(), 3 if quadratic else 2
        if quadratic:
            self.w = [0.5 * (1.5 - f) ** 2, 0.75 - (f - 1.0) ** 2, 0.5 * (f - 0.5) ** 2]
            self.k = [f - 1.5, -2.0 * (f - 1.0), f - 0.5]  # d w / d u
        else:
            s = torch.sin(2.0 * math.pi * f) / (2.0 * math.pi)
            c = torch.cos(2.0 * math.pi * f)
            self.w = [1.0 - f + s, f - s]
            self.k = [c - 1.0, 1.0 - c]
        self.d = [j - f for j in range(self.N)]

    def nodes(self, nn):
        for kz in range(self.N):
            for ky in range(self.N):
                for kx in range(self.N):
                    j = (kx, ky, kz)
                    idx = ((self.base[:, 2] + kz) * nn + self.base[:, 1] + ky) * nn + self.base[:, 0] + kx
                    w = [self.w[j[a]][:, a] for a in range(3)]
                    k = [self.k[j[a]][:, a] for a in range(3)]
                    d = torch.stack([self.d[j[a]][:, a] for a in range(3)], 1)
                    g = torch.stack([k[0] * w[1] * w[2], w[0] * k[1] * w[2], w[0] * w[1] * k[2]], 1)
                    yield idx, w[0] * w[1] * w[2], d, g


def _dinv(stens, quadratic):
    if quadratic:
        return 4.0 * torch.eye(3, dtype=torch.float64, device=stens[0].base.device)[None]
    D = 0.0
    for s in stens:
        m1 = sum(w * d for w, d in zip(s.w, s.d))
        m2 = sum(w * d * d for w, d in zip(s.w, s.d))
        D = D + 0.5 * (m1[:, :, None] * m1[:, None, :] + torch.diag_embed(m2 - m1 * m1))
    return _cof(D).transpose(1, 2) / _det(D)[:, None, None]


class _Exact:
    """The method's step in float64 on dense grids."""

    def __init__(self, scene, quadratic=False, transfer="apic"):
        self.sc, self.q, self.tr = scene, quadratic, transfer
        self.V0 = scene.dx ** 3 / scene.ppc
        self.nn = scene.res + 1

    def mass(self, mat, n, dev):
        m = torch.tensor([k.rho * self.V0 for k in self.sc.materials], dtype=torch.float64, device=dev)
        return m[mat.long()] if mat is not None else m[0].expand(n)

    def stencils(self, x):
        u = x / self.sc.dx
        return [_Stencil(u, True, 0.0)] if self.q else [_Stencil(u, False, 0.25), _Stencil(u, False, -0.25)]

    def p2g(self, stens, x, v, B, F, mat, E=None):
        sc, n = self.sc, x.shape[0]
        m = self.mass(mat, n, x.device)
        tau = _stress(sc.materials[0], F, E) if E is not None else _per_material(_stress, sc.materials, mat, F)
        f = -sc.dt * self.V0 * tau
        Di = _dinv(stens, self.q) / sc.dx  # times an offset in cells
        apic = _mm(m[:, None, None] * B, Di.expand(n, 3, 3)) if self.tr != "pic" else torch.zeros_like(F)
        if self.tr == "apic":
            apic = apic + _mm(f, Di.expand(n, 3, 3))
        out = []
        for s in stens:
            G = torch.zeros(self.nn ** 3, 4, dtype=torch.float64, device=x.device)
            for idx, w, d, g in s.nodes(self.nn):
                p = w[:, None] * (m[:, None] * v + (apic * d[:, None, :]).sum(2))
                if self.tr != "apic":
                    p = p + (f * (g / sc.dx)[:, None, :]).sum(2)
                G = G.index_add(0, idx, torch.cat([(w * m)[:, None], p], 1)) if G.requires_grad or p.requires_grad \
                    else G.index_add_(0, idx, torch.cat([(w * m)[:, None], p], 1))
            out.append(G)
        return out

    def update(self, G, shift):
        sc = self.sc
        m = G[:, :1]
        grav = sc.dt * torch.tensor(sc.gravity, dtype=torch.float64, device=G.device)
        i = torch.arange(self.nn, device=G.device) + shift
        wall1 = (i < sc.bc_cells) | (i > sc.res - sc.bc_cells)
        wall = (wall1[:, None, None] | wall1[None, :, None] | wall1[None, None, :]).reshape(-1, 1)
        keep = (m > 0) & ~wall
        return torch.where(keep, G[:, 1:] / torch.where(m > 0, m, torch.ones_like(m)) + grav, torch.zeros_like(G[:, 1:]))

    def step(self, x, v, B, F, mat=None, E=None):
        sc, n = self.sc, x.shape[0]
        stens = self.stencils(x)
        shifts = [0.0] if self.q else [0.25, -0.25]
        vel = [self.update(G, h) for G, h in zip(self.p2g(stens, x, v, B, F, mat, E), shifts)]
        v1, B1, L = 0.0, 0.0, 0.0
        for s, gv in zip(stens, vel):
            for idx, w, d, g in s.nodes(self.nn):
                a = gv[idx] / len(stens)
                v1 = v1 + w[:, None] * a
                if self.tr != "pic":
                    B1 = B1 + (w[:, None] * a)[:, :, None] * (sc.dx * d)[:, None, :]
                if self.tr != "apic":
                    L = L + a[:, :, None] * (g / sc.dx)[:, None, :]
        if self.tr == "apic":
            L = _mm(B1, (_dinv(stens, self.q) / sc.dx ** 2).expand(n, 3, 3))
        F1 = F + sc.dt * _mm(L, F)
        if E is None:
            F1 = _per_material(_plastic, sc.materials, mat, F1)
        return x + sc.dt * v1, v1, (B1 if self.tr != "pic" else torch.zeros_like(F)), F1


def exact(case, seed):
    what = case["what"]
    quadratic = case.get("kernel", "ck") != "ck"
    if what == "steps":
        x, v, F, mat = _particles(case, seed)
        ex = _Exact(_scene(case, x, v, mat), quadratic, case["transfer"])
        s = (x.double(), v.double(), torch.zeros_like(F).double(), F.double())
        for _ in range(case["steps"]):
            s = ex.step(*s, mat)
        return {"x": s[0], "v": s[1], "F": s[3]}
    if what == "grids":
        x, v, F, _ = _particles(case, seed)
        B = (0.2 / case["res"]) * torch.randn(F.shape, generator=_gen(seed + 17, F.device), device=F.device)
        ex = _Exact(_scene(dict(case, transfer="apic"), x, v), quadratic)
        G = torch.stack(ex.p2g(ex.stencils(x.double()), x.double(), v.double(), B.double(), F.double(), None))
        G = G.reshape(G.shape[0], ex.nn, ex.nn, ex.nn, 4)
        return {"m": G[..., 0].contiguous(), "p": G[..., 1:].contiguous()}
    if what == "served":
        out = []
        for c, x, v in _requests(case, seed):
            ex = _Exact(_scene(c, x, v), quadratic)
            F = torch.eye(3, dtype=torch.float64, device=x.device).expand(x.shape[0], 3, 3)
            s = (x.double(), v.double(), torch.zeros_like(F), F)
            for _ in range(case["steps"]):
                s = ex.step(*s)
            out.append({"x": s[0], "v": s[1]})
        return out
    x, v, B, F, E, adj = _diff_inputs(case, seed)
    scene = S.Scene("case", case["res"], 1.0 / case["grid"], case["dt"], x, v, None, [S.ELASTIC])
    ex = _Exact(scene)
    state = [t.double() for t in (x, v, B, F, E)]
    if what == "forward":
        with torch.no_grad():
            return dict(zip(("x", "v", "B", "F"), ex.step(*state[:4], None, state[4])))
    if what == "adjoint":
        leaf = [t.requires_grad_(True) for t in state]
        got = torch.autograd.grad(ex.step(*leaf[:4], None, leaf[4]), leaf, [a.double() for a in adj])
        return dict(zip(("gx", "gv", "gB", "gF", "gE"), got))
    if x.shape[0] * case["steps"] > 1_500_000:
        return None  # the recorded graph of a longer rollout takes too long
    lx, lv, lE = (t.requires_grad_(True) for t in (state[0], state[1], state[4]))
    F0 = torch.eye(3, dtype=torch.float64, device=x.device).expand(x.shape[0], 3, 3)
    s = (lx, lv, torch.zeros_like(F0), F0)
    for _ in range(case["steps"]):
        s = ex.step(*s, None, lE)
    got = torch.autograd.grad(s[:2], (lx, lv, lE), [a.double() for a in adj[:2]])
    return dict(zip(("x", "v", "gx", "gv", "gE"), (s[0].detach(), s[1].detach()) + got))
