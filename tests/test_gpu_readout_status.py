"""Readouts of phi alone (the droplet count, lb_fields of phi to the device)
test the level's density as a pass over the populations does, and give the
values that every other mask gives."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

STORAGES = ["twoset_f32", "reduced_f32", "reduced_f16", "twoset_f64", "moment_f32"]
SHAPE = (40, 10, 12)


def _sim(storage, walls=0, model=0):
    import paper_2405_14551_gb300.lbcg as L
    p = dict(model=1, G=2.0, psi0=1.0) if model else dict(A_h=0.1)
    return L.Sim(*SHAPE, walls=walls, storage=storage, collision=int(storage == "moment_f32"), **p)


def _phi():
    x = np.arange(SHAPE[0])
    return np.broadcast_to(np.tanh((8.0 - np.abs(x - 19.5)) / 1.5), SHAPE[::-1]).astype(np.float32).copy()


def _readouts():
    import torch

    import paper_2405_14551_gb300.lbcg as L

    def fields(s):
        f64 = s.storage == L.STORAGE["twoset_f64"]
        out = torch.empty((1,) + SHAPE[::-1], dtype=torch.float64 if f64 else torch.float32, device="cuda")
        L.lb_fields(s.h, 1, out, True, f64=f64)
    return {"count": lambda s: s.droplet_count(), "phi": fields}


def _unstable(s):
    import paper_2405_14551_gb300.lbcg as L
    try:
        s.check()
    except L.LBError as e:
        assert e.code == L.LB_EUNSTABLE
        return True
    return False


@pytest.mark.parametrize("storage", STORAGES)
@pytest.mark.parametrize("how", ["count", "phi"])
def test_bad_initial_density_is_reported(storage, how):
    read = _readouts()[how]
    limit = 64.0 if storage == "twoset_f64" else 4.0
    for value, which, bad in [(1.0, "rho", False), (0.0, "rho", True), (-1.0, "rho", True), (np.nan, "rho", True),
                              (limit, "rho", True), (0.99 * limit, "rho", False),
                              (np.nan, "phi", True), (np.inf, "phi", True), (1e30, "phi", True)]:
        for walls, node, solid in [(0, (3, 4, 5), False), (0b010, (3, 0, 5), True)]:  # (z, y, x)
            rho, phi = np.ones(SHAPE[::-1], np.float32), _phi()
            (rho if which == "rho" else phi)[node] = value
            s = _sim(storage, walls)
            s.init_fields(phi, rho, np.zeros((3,) + SHAPE[::-1], np.float32))
            assert not _unstable(s)
            read(s)
            assert _unstable(s) == (bad and not solid), (value, which, walls)
            s.close()


@pytest.mark.parametrize("storage,model", [(s, 0) for s in STORAGES] + [("twoset_f32", 1), ("twoset_f64", 1)])
@pytest.mark.parametrize("how", ["count", "phi"])
def test_density_of_a_stepped_level_is_reported(storage, model, how):
    """Two streams that meet: the density passes the limit at the first level that
    no step has tested yet."""
    read = _readouts()[how]
    limit = 64.0 if storage == "twoset_f64" else 4.0
    for scale, bad in [(0.25, False), (0.9, True)]:
        rho = np.full(SHAPE[::-1], scale * limit, np.float32)
        u = np.zeros((3,) + SHAPE[::-1], np.float32)
        u[0] = np.where(np.arange(SHAPE[0]) < SHAPE[0] // 2, 0.25, -0.25)
        s = _sim(storage, 0, model)
        s.init_fields(_phi(), rho, u)
        s.step(1)
        assert not _unstable(s)
        read(s)
        assert _unstable(s) == bad, scale
        s.close()


@pytest.mark.parametrize("storage", STORAGES)
def test_phi_alone_equals_phi_among_others(storage):
    """Also where phi is infinite, not a number or as large as the marker of
    solid nodes."""
    import torch

    import paper_2405_14551_gb300.lbcg as L
    f64 = storage == "twoset_f64"
    for steps in (0, 3):
        phi = _phi()
        if steps == 0:
            phi[2, 3, 4], phi[2, 3, 6], phi[5, 5, 5], phi[6, 5, 5] = np.inf, np.nan, 1e30, -np.inf
        s = _sim(storage, 0b010)
        s.init_fields(phi)
        s.step(steps)
        n = SHAPE[::-1]
        one = torch.empty((1,) + n, dtype=torch.float64 if f64 else torch.float32, device="cuda")
        two = torch.empty((2,) + n, dtype=one.dtype, device="cuda")
        L.lb_fields(s.h, 0b1, one, True, f64=f64)
        L.lb_fields(s.h, 0b11, two, True, f64=f64)
        np.testing.assert_array_equal(one[0].cpu().numpy(), two[0].cpu().numpy())
        assert not one[0, :, 0].any() and not one[0, :, -1].any()  # solid layers
        s.close()
