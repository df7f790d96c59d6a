"""The shape that a step takes: by the lattice's size, or the one set where it
fills the GPU; every shape that is reached gives the same bits."""
import os
import re
import subprocess
import sys

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

TRACED = """
import torch, sys
import paper_2405_14551_gb300.lbcg as L
for nx, ny, nz, tile, model in {cases}:
    s = L.Sim(nx, ny, nz, **(dict(model=1, G=2.0) if model else dict(A_h=0.1)))
    s.init_droplets([[nx / 2, ny / 2, nz / 2]], [6.0], 1.3)
    if tile >= 0:
        L.lb_set_tile(s.h, tile)
    s.step(1)
    torch.cuda.synchronize()
    print("CASE", file=sys.stderr, flush=True)
    s.step(1)
    torch.cuda.synchronize()
    s.close()
"""

# (nx, ny, nz), tile set (-1: none), Shan-Chen -> nodes in y and z of the tile on 152 SMs
CHOICE = [
    ((32, 32, 32), -1, 0, (8, 1)), ((48, 48, 48), -1, 0, (8, 2)), ((64, 64, 64), -1, 0, (8, 4)),
    ((33, 74, 86), -1, 0, (8, 2)), ((96, 80, 112), -1, 0, (8, 4)), ((64, 64, 128), -1, 0, (8, 8)),
    ((128, 128, 256), -1, 0, (8, 8)), ((24, 24, 24), 1, 0, (8, 1)), ((24, 24, 24), 0, 0, (8, 1)),
    ((48, 48, 48), 4, 0, (8, 2)), ((96, 80, 112), 1, 0, (8, 8)), ((96, 80, 112), 5, 0, (8, 8)), ((96, 80, 112), 4, 0, (4, 4)),
    ((96, 80, 112), 3, 0, (8, 4)), ((128, 128, 256), 2, 0, (8, 8)), ((48, 48, 48), -1, 1, (8, 2)), ((128, 128, 256), -1, 1, (8, 4)),
]


def test_shape_by_size_and_by_setting():
    import torch
    if torch.cuda.get_device_properties(0).multi_processor_count != 152:
        pytest.skip("the expected shapes are those of 152 SMs")
    cases = [shape + (tile, model) for shape, tile, model, _ in CHOICE]
    r = subprocess.run([sys.executable, "-c", TRACED.format(cases=cases)], cwd=ROOT, capture_output=True, text=True,
                       env=dict(os.environ, LBCG_TRACE="1"), timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    traced = [re.search(r"k_step grid=\((\d+),(\d+),(\d+)\)", part) for part in r.stderr.split("CASE")[1:]]
    assert len(traced) == len(CHOICE)
    for (shape, tile, model, (ty, tz)), m in zip(CHOICE, traced):
        grid = tuple(int(v) for v in m.groups())
        want = (-(-shape[0] // 32), -(-shape[1] // ty), -(-shape[2] // tz))
        assert grid == want, (shape, tile, model)


def _phi(shape, seed):
    nx, ny, nz = shape
    r = np.random.default_rng(seed)
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    d = np.full((nz, ny, nx), 1e9)
    for _ in range(40):
        c = r.uniform(0, 1, 3) * np.array(shape)
        e = [(v - o + n / 2) % n - n / 2 for v, o, n in zip((x, y, z), c, shape)]
        d = np.minimum(d, np.sqrt(sum(v * v for v in e)))
    return np.tanh((9.0 - d) / 1.3).astype(np.float32)


# sizes whose own choice is 32x8x2, x4 and x8, each large enough for every shape that can
# be set (the first has 396 CTAs of 32x8x8)
@pytest.mark.parametrize("shape", [(65, 88, 90), (70, 100, 60), (64, 64, 128)])
@pytest.mark.parametrize("storage,walls,p", [
    ("twoset_f32", 0b011, dict(A_h=0.1)), ("twoset_f32", 0b010, dict()), ("reduced_f32", 0b110, dict(A_h=0.1)),
    ("reduced_f16", 0b001, dict()), ("reduced_f16", 0b010, dict(A_h=0.1, collision=1)),
    ("moment_f32", 0b101, dict(A_h=0.1, collision=1)), ("twoset_f32", 0b111, dict(A_h=0.1, h_min=2.0, h_max=5.0)),
    ("twoset_f32", 0b011, dict(model=1, G=2.0))])
def test_every_shape_gives_the_same_bits(shape, storage, walls, p):
    import paper_2405_14551_gb300.lbcg as L
    phi, ref = _phi(shape, 7), None
    for tile in (-1, 0, 1, 2, 4):
        s = L.Sim(*shape, walls=walls, storage=storage, g=(1e-5, 0.0, 1e-5), g_mode=1, tau_a=0.8, tau_b=1.0, **p)
        s.init_fields(phi)
        if tile >= 0:
            L.lb_set_tile(s.h, tile)
        s.step(15)
        s.check()
        f = s.fields(("phi", "rho", "ux", "uz", "h"))
        s.close()
        ref = ref or f
        for k in f:
            np.testing.assert_array_equal(f[k], ref[k], err_msg=f"tile {tile} field {k}")
