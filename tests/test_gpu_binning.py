"""Binning at the sizes where its scan changes form.

The same few particles, in the same cells, are stepped on key spaces of 8^3 to 175^3 particle blocks: up to 8192 keys
(the scan counts the keys before a tile itself), up to 4096 tiles of 1024 keys (it sums tile sums) and beyond (one CTA
scans the tile sums first).  Walls are far from the particles and gravity is off, so every run computes the same step:
results agree to the rounding of the float atomics that meet between blocks (64 contributions a node: 4e-6 of the
largest velocity).  An upload, a second scene and a release in between check the sums a step leaves for the next."""
import numpy as np
import pytest

from gpu_helpers import f32, need_gpu, rel
from paper_2412_10399_gb300 import scenes as S

pytestmark = pytest.mark.gpu
DX = 1.0 / 1024


def _scene(res, n=3000, kernel=S.KERNEL_CK, seed=4):
    g = np.random.default_rng(seed)
    x = f32((12.0 + 8.0 * g.random((n, 3))) * DX).astype(np.float64)
    v = f32(g.standard_normal((n, 3))).astype(np.float64)
    return S.Scene("bins", res, DX, 1e-5, x, v, np.zeros(n, np.uint8), [S.ELASTIC], gravity=(0.0, 0.0, 0.0),
                   kernel=kernel)


def _run(ck, sc, steps=3):
    sim = ck.Simulation(sc)
    sim.step(steps)
    sim.write(ck.FIELD_V, sim.read(ck.FIELD_V))
    sim.step(steps)
    out = sim.read(ck.FIELD_X), sim.read(ck.FIELD_V)
    sim.close()
    return out


@pytest.mark.parametrize("kernel", [S.KERNEL_CK, S.KERNEL_QUADRATIC])
@pytest.mark.parametrize("res", [80, 84, 101, 260, 700])
def test_key_spaces_of_every_scan_form_give_the_same_step(res, kernel):
    ck = need_gpu()
    want = _run(ck, _scene(32, kernel=kernel))
    got = _run(ck, _scene(res, kernel=kernel))
    assert np.abs(got[0] - want[0]).max() <= 1e-6 * DX + 2e-9
    assert rel(got[1], want[1]) <= 4e-6


@pytest.mark.parametrize("res", [32, 101])
def test_tile_sums_follow_admission_and_release(res):
    ck = need_gpu()
    a, b = _scene(res), _scene(res, n=500, seed=9)
    cfg = ck.ckmpm_config()
    nb = -(-res // 4)
    cfg.kernel, cfg.max_particles, cfg.max_keys = 0, 8000, 2 * nb ** 3
    cfg.max_virtual_blocks, cfg.max_grid_blocks, cfg.max_scenes, cfg.max_materials = 2 * (nb + 1) ** 3, 4096, 2, 4
    ctx = ck.ckmpm_create_server(cfg)
    keep = [ck.scene_struct(s) for s in (a, b)]

    def read(sid, n):
        out = np.empty((n, 3), np.float32)
        ck.ckmpm_readback(ctx, sid, ck.FIELD_X, out.ctypes.data, out.nbytes, False)
        return out

    ia = ck.ckmpm_admit(ctx, keep[0][0])
    ck.ckmpm_step(ctx, 2)
    ib = ck.ckmpm_admit(ctx, keep[1][0])
    ck.ckmpm_step(ctx, 3)
    xb = read(ib, b.n)
    ck.ckmpm_release(ctx, ib)
    ck.ckmpm_step(ctx, 2)
    xa = read(ia, a.n)
    ck.ckmpm_destroy(ctx)
    for sc, steps, got in ((a, 7, xa), (b, 3, xb)):
        sim = ck.Simulation(sc)
        sim.step(steps)
        assert np.abs(got - sim.read(ck.FIELD_X)).max() <= 1e-6 * DX + 2e-9
        sim.close()
