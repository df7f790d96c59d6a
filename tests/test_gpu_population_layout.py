"""Memory and addressing of the population blocks at extents that are not a
multiple of a block: thin boxes cost no more than their nodes, and planes beyond
32-bit byte offsets give the bits of a small box."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


# bytes a node of both lattices, the three accumulators and the initial phi; beyond
# them a handle holds the padded phase field and scratch that does not grow with nx
@pytest.mark.parametrize("storage,pop", [("twoset_f32", 432), ("reduced_f32", 248), ("reduced_f16", 140), ("twoset_f64", 864)])
@pytest.mark.parametrize("shape", [(33, 96, 64), (57, 64, 64), (1, 256, 256), (9, 128, 96), (145, 33, 64)])
def test_a_box_costs_its_nodes(storage, pop, shape):
    import paper_2405_14551_gb300.lbcg as L
    nx, ny, nz = shape
    s = L.Sim(nx, ny, nz, storage=storage)
    f64 = storage == "twoset_f64"
    n = nx * ny * nz
    rows = n * (pop + (48 if f64 else 24) + 4)
    padded = ((nx + 31) // 32 * 32 + 8) * (ny + 9) * (nz + 9) * (8 if f64 else 4)
    # rows on whole sectors: at most a sixteenth; the last block of a plane: 31 nodes
    limit = rows * 17 / 16 + 2 * 31 * nz * pop + padded + (1 << 20)
    got = L.lb_device_bytes(s.h)
    s.close()
    assert got <= limit, (got / n, limit / n)


def test_planes_beyond_32_bit_offsets_equal_a_small_box():
    """A plane of 4.5 GB holding copies of a periodic 256 x 128 pattern moves as the
    pattern alone: the same operations on the same values at every node."""
    import torch

    import paper_2405_14551_gb300.lbcg as L
    if torch.cuda.mem_get_info()[0] < 30 << 30:
        pytest.skip("needs 30 GB")
    kx, ky = 32, 20
    r = np.random.default_rng(4)
    x, y = np.meshgrid(np.arange(256), np.arange(128))
    d = np.full((128, 256), 1e9)
    for cx, cy in r.uniform(0, 1, (14, 2)) * (256, 128):
        ex, ey = (x - cx + 128) % 256 - 128, (y - cy + 64) % 128 - 64
        d = np.minimum(d, np.hypot(ex, ey))
    phi = np.tanh((14.0 - d) / 1.3).astype(np.float32)[None]
    p = dict(A_h=0.1, g=(1e-5, 0.0, 0.0), g_mode=1)
    small, big = L.Sim(256, 128, 1, **p), L.Sim(256 * kx, 128 * ky, 1, **p)
    small.init_fields(phi)
    big.init_fields(np.tile(phi, (1, ky, kx)))
    for s in (small, big):
        s.step(14)
    mask = sum(L.FIELD_BIT[k] for k in ("phi", "rho", "ux", "uy", "uz", "h"))
    a, b = small.fields_device(mask), big.fields_device(mask)
    for f in range(a.shape[0]):
        tiles = b[f].reshape(ky, 128, kx, 256)
        assert torch.equal(tiles, a[f].reshape(1, 128, 1, 256).expand_as(tiles)), f
    small.close()
    big.close()
