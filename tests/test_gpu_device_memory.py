"""What calls need beyond the memory of the handle: nothing for a checkpoint or a
batch's steps; and the destinations that a field readout takes."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STORAGES = ["twoset_f32", "reduced_f32", "reduced_f16", "twoset_f64", "moment_f32"]


def _phi(shape, seed=1):
    r = np.random.default_rng(seed)
    return np.clip(r.standard_normal(shape[::-1]), -1, 1).astype(np.float32)


class _Budget:
    """Memory from PyTorch until `full` is set."""

    def __new__(cls, device=0):
        import paper_2405_14551_gb300.lbcg as L

        class A(L.TorchAllocator):
            full = False

            def _alloc(self, ctx, nbytes):
                return None if self.full else super()._alloc(ctx, nbytes)
        return A(device)


def _handle(shape, storage, seed=1):
    import ctypes

    import paper_2405_14551_gb300.lbcg as L
    a = _Budget()
    h = L.lb_create(L.make_grid(*shape), L.make_params(storage=storage, collision=int(storage == "moment_f32")), a)
    L.lb_init_fields(h, _phi(shape, seed))
    return h, a


def _populations(h, shape):
    import paper_2405_14551_gb300.lbcg as L
    return L.lb_get_populations(h, (0, 0, 0) + shape)


@pytest.mark.parametrize("storage", STORAGES)
def test_checkpoints_need_no_device_memory(tmp_path, storage):
    import paper_2405_14551_gb300.lbcg as L
    shape, path = (37, 6, 5), str(tmp_path / "c.bin")
    h, a = _handle(shape, storage)
    k, b = _handle(shape, storage, 2)
    for steps in (3, 4):  # both lattices of the pair as the current one
        L.lb_step(h, steps)
        a.full = b.full = True
        L.lb_save(h, path)
        L.lb_load(k, path)
        L.lb_step(h, 2)
        L.lb_step(k, 2)
        a.full = b.full = False
        for p, q in zip(_populations(h, shape), _populations(k, shape)):
            np.testing.assert_array_equal(p, q)
    L.lb_destroy(h)
    L.lb_destroy(k)


def test_batched_steps_need_no_device_memory():
    import paper_2405_14551_gb300.lbcg as L
    shapes = [(33, 17, 9), (8, 40, 3), (64, 4, 4)]
    a = _Budget()
    b = L.lb_batch_create([L.make_grid(*s) for s in shapes], [L.make_params(A_h=0.1 * (k % 2)) for k in range(3)], a)
    for k, s in enumerate(shapes):
        L.lb_init_fields(L.lb_batch_run(b, k), _phi(s, k))
    a.full = True
    for tile in range(L.NUM_TILES):
        L.lb_batch_set_tile(b, tile, 2)
        L.lb_batch_step(b, 13)
    L.lb_batch_check(b)
    a.full = False
    L.lb_batch_destroy(b)


@pytest.mark.parametrize("storage,mask", [("twoset_f32", 0b1), ("reduced_f16", 0b10011), ("twoset_f64", 0b101)])
def test_device_destination_that_is_not_this_gpus_memory(storage, mask):
    """Pinned host memory, as a tensor and as a bare pointer, passed as a device
    destination."""
    import torch

    import paper_2405_14551_gb300.lbcg as L
    shape = (37, 6, 5)
    s = L.Sim(*shape, storage=storage)
    s.init_fields(_phi(shape))
    s.step(4)
    n = bin(mask).count("1")
    for f64 in (False, True):
        dt = torch.float64 if f64 else torch.float32
        want = torch.empty((n,) + shape[::-1], dtype=dt, device="cuda")
        L.lb_fields(s.h, mask, want, True, f64=f64)
        pinned = torch.zeros(want.shape, dtype=dt, pin_memory=True)

        class Bare:
            def data_ptr(self):
                return pinned.data_ptr()
        for dst in (pinned, Bare()):
            pinned.zero_()
            L.lb_fields(s.h, mask, dst, True, f64=f64)
            torch.cuda.synchronize()
            assert torch.equal(pinned, want.cpu())
    s.close()
