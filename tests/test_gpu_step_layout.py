"""Layout and dispatch of the step: the tile picked by size, the population
blocks behind a checkpoint's plain order, packed field masks, and the batch's
work list, at the sizes where they can go wrong (ragged rows, one block and
just over one, tiny periodic boxes)."""
import struct

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

C27 = [(i % 3 - 1, i // 3 % 3 - 1, i // 9 - 1) for i in range(27)]


def _phi(shape, seed):
    nz, ny, nx = shape[::-1]
    r = np.random.default_rng(seed)
    z, y, x = np.meshgrid(np.arange(nz), np.arange(ny), np.arange(nx), indexing="ij")
    d = np.full((nz, ny, nx), 1e9)
    for _ in range(3):
        c = r.uniform(0, 1, 3) * np.array(shape)
        e = [(v - o + n / 2) % n - n / 2 for v, o, n in zip((x, y, z), c, shape)]
        d = np.minimum(d, np.sqrt(sum(v * v for v in e)))
    return np.tanh((0.25 * min(shape) - d) / 1.3).astype(np.float32)


def _sim(shape, walls, storage, seed=3, **p):
    import paper_2405_14551_gb300.lbcg as L
    s = L.Sim(*shape, walls=walls, storage=storage, **p)
    s.init_fields(_phi(shape, seed))
    return s


@pytest.mark.parametrize("shape,walls", [((31, 9, 8), 0), ((33, 17, 9), 0b010), ((64, 40, 48), 0), ((96, 96, 66), 0b100)])
@pytest.mark.parametrize("storage,ah", [("twoset_f32", 0.1), ("reduced_f16", 0.1), ("reduced_f32", 0.0)])
def test_tile_picked_by_size_gives_the_same_bits(shape, walls, storage, ah):
    import paper_2405_14551_gb300.lbcg as L
    ref = None
    for tile in (None, 0, 1, 2, 3, 4, 5):
        s = _sim(shape, walls, storage, A_h=ah, g=(0.0, 0.0, 1e-5), g_mode=1)
        if tile is not None:
            L.lb_set_tile(s.h, tile)
        assert L.lb_get_tile(s.h) == (tile or 0)
        s.step(15)  # single steps and one graph replay
        f = s.fields()
        s.check()
        s.close()
        ref = ref or f
        for k in f:
            np.testing.assert_array_equal(f[k], ref[k], err_msg=f"tile {tile} field {k}")


@pytest.mark.parametrize("shape", [(1, 2, 3), (31, 5, 4), (32, 6, 5), (33, 4, 7), (70, 3, 4)])
@pytest.mark.parametrize("storage,dtype", [("twoset_f32", np.float32), ("twoset_f64", np.float64)])
def test_checkpoint_holds_plain_arrays_per_direction(tmp_path, shape, storage, dtype):
    """The file's [component][direction][z][y][x] order does not follow the
    device's blocks: the stored post-collision value of direction i at x is
    what the node x + c_i pulls."""
    import paper_2405_14551_gb300.lbcg as L
    s = _sim(shape, 0, storage)
    s.step(3)
    path = str(tmp_path / "c.bin")
    s.save(path)
    fa, fb = s.populations()
    n = shape[0] * shape[1] * shape[2]
    raw = open(path, "rb").read()
    head = 16 + struct.calcsize("<3iI") + len(bytes(L.make_params())) + 8
    assert len(raw) == head + 2 * 27 * n * np.dtype(dtype).itemsize
    f = np.frombuffer(raw[head:], dtype=dtype).reshape(2, 27, shape[2], shape[1], shape[0])
    for comp, pulled in ((0, fa), (1, fb)):
        for i, c in enumerate(C27):
            want = np.roll(f[comp, i].astype(np.float64), (c[2], c[1], c[0]), (0, 1, 2))
            np.testing.assert_array_equal(pulled[i], want, err_msg=f"component {comp} direction {i}")
    t = _sim(shape, 0, storage, seed=9)
    t.step(2)
    t.load(path)
    s.step(5)
    t.step(5)
    for a, b in zip(s.fields().values(), t.fields().values()):
        np.testing.assert_array_equal(a, b)


@pytest.mark.parametrize("storage", ["twoset_f32", "reduced_f16", "moment_f32", "twoset_f64"])
@pytest.mark.parametrize("names", [("phi",), ("rho", "uz"), ("phi", "rho", "ux", "uy", "uz"), ("h", "gz")])
def test_packed_fields_on_the_device_equal_the_host_copy(storage, names):
    import torch

    import paper_2405_14551_gb300.lbcg as L
    s = _sim((33, 12, 10), 0b010, storage, A_h=0.1, collision=int(storage == "moment_f32"))
    mask = sum(L.FIELD_BIT[k] for k in names)
    for steps in (0, 4):
        s.step(steps)
        dev = s.fields_device(mask).cpu().numpy()
        host = s.fields(names)
        full = s.fields()
        for j, k in enumerate(n for n in L.FIELD_NAMES if n in names):
            np.testing.assert_array_equal(dev[j], host[k])
            np.testing.assert_array_equal(full[k], host[k])
        assert torch.isfinite(torch.from_numpy(dev)).all()


def test_field_tensors_outlive_their_handle():
    """Device tensors filled by a handle may be freed after the handle is gone."""
    import gc

    import torch
    kept = []
    for k in range(6):
        s = _sim((32, 16, 16), 0, "twoset_f32", seed=k)
        s.step(2)
        kept.append(s.fields_device(0b11111))
        s.close()
        if k % 2:
            kept.clear()
            gc.collect()
    torch.cuda.synchronize()
    assert all(torch.isfinite(t).all() for t in kept)


def test_batch_of_uneven_runs_follows_its_work_list():
    """More runs than one of each kind, sizes around a block of 32, retiled
    between steps (the work list is rebuilt)."""
    import paper_2405_14551_gb300.lbcg as L
    from paper_2405_14551_gb300 import workloads as W
    shapes = [(31, 9, 5), (64, 8, 8), (33, 20, 9), (8, 8, 40), (32, 32, 32)]
    runs = [W.Workload(f"r{k}", s, 0b010 if k == 2 else 0, dict(W.BASE, A_h=0.1 if k % 2 else 0.0), 9, phi=_phi(s, k))
            for k, s in enumerate(shapes)]
    b = L.Batch(runs)
    for tile, bps in ((0, 1), (5, 2), (2, 3)):
        L.lb_batch_set_tile(b.b, tile, bps)
        b.step(13)
    b.check()
    for r, w in enumerate(runs):
        s = L.Sim(*w.shape, walls=w.walls, **w.params)
        s.init_fields(w.phi)
        s.step(39)
        fb, fs = b.fields(r), s.fields()
        for k in fs:
            np.testing.assert_array_equal(fb[k], fs[k], err_msg=f"run {r} field {k}")


@pytest.mark.parametrize("h_max", [4.5, 5.9, 6.0])
def test_batch_with_wide_scan_steps_every_node(h_max):
    """Scan lengths beyond 3 have one tile shape, whatever the batch's setting."""
    import paper_2405_14551_gb300.lbcg as L
    from paper_2405_14551_gb300 import workloads as W
    p = dict(W.BASE, A_h=0.1, h_min=2.0, h_max=h_max)
    runs = [W.Workload(f"r{k}", s, 0b010 * k, p, 5, phi=_phi(s, k)) for k, s in enumerate([(40, 24, 20), (33, 17, 21)])]
    b = L.Batch(runs)
    L.lb_batch_set_tile(b.b, 5, 2)
    b.step(6)
    for r, w in enumerate(runs):
        for tile in (None, 0, 5):
            s = L.Sim(*w.shape, walls=w.walls, **w.params)
            s.init_fields(w.phi)
            if tile is not None:
                L.lb_set_tile(s.h, tile)
            s.step(6)
            fb, fs = b.fields(r), s.fields()
            for k in fs:
                np.testing.assert_array_equal(fb[k], fs[k], err_msg=f"run {r} tile {tile} field {k}")
