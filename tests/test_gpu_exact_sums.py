"""The FP64 readouts that sum FP32 terms: single terms at FP64's precision, sums
that cancel, and shares whose terms leave FP32's range, against exact rational
sums."""
from fractions import Fraction as Fr

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PHI, RHO, UX, UY, UZ, RHOA, RHOB, H = 0, 1, 2, 3, 4, 5, 6, 10


def _reduce(f, shape):
    """lb_reduce_fields_f64_static of the FP32 field array f [14][N]."""
    import torch

    import paper_2405_14551_gb300.lbcg as L
    d = torch.from_numpy(np.ascontiguousarray(f, np.float32)).cuda()
    out = torch.zeros(8, dtype=torch.float64, device="cuda")
    L.lb_reduce_fields_f64_static(d.data_ptr(), False, *shape, 0, out.data_ptr(), torch.cuda.current_stream().cuda_stream)
    torch.cuda.synchronize()
    return out.cpu().numpy()


def _exact(f):
    fl = [[Fr(float(v)) for v in row] for row in np.asarray(f, np.float32)]
    n = len(fl[0])
    mom = [sum(fl[RHO][i] * fl[UX + k][i] for i in range(n)) for k in range(3)]
    vol = sum(1 + fl[PHI][i] for i in range(n)) / 2
    ke = sum(fl[RHO][i] * sum(fl[UX + k][i] ** 2 for k in range(3)) for i in range(n)) / 2
    return [sum(fl[RHOA]), sum(fl[RHOB]), *mom, vol, Fr(int((np.asarray(f)[H] > 0).sum())), ke]


def _fields(n, seed, scale=0.05):
    r = np.random.default_rng(seed)
    f = np.zeros((14, n), np.float32)
    f[PHI], f[RHO] = r.uniform(-1, 1, n), r.uniform(0.9, 1.1, n)
    f[UX:UZ + 1] = scale * r.standard_normal((3, n))
    f[RHOA], f[RHOB] = r.uniform(0, 1, n), r.uniform(0, 1, n)
    return f


def test_single_nodes_keep_fp64_precision():
    """One node, so nothing hides a term's own rounding: the three-term sum is
    rounded to FP64 once and scaled by powers of two (2^-53), twice as much allowed."""
    for seed in range(48):
        f = _fields(1, seed)
        got, ref = _reduce(f, (1, 1, 1)), _exact(f)
        for k in range(8):
            assert abs(Fr(float(got[k])) - ref[k]) <= abs(ref[k]) * Fr(1, 2**52), (seed, k)


# a thread's share is at most 12 nodes here; summed in FP64 a node rounds 6 times, and
# the trees over 256 threads and over the blocks add at most 8 levels each
@pytest.mark.parametrize("kind", ["plain", "cancelling", "beyond", "beyond_phi", "tiny", "far"])
def test_sums_cancelling_and_out_of_range(kind):
    shape = (16, 16, 12)
    n = 16 * 16 * 12
    f = _fields(n, 5)
    if kind == "cancelling":  # volume of a phase that is almost absent, momenta that cancel
        f[PHI] = -1.0 + 2.0**-24 * np.random.default_rng(1).integers(0, 3, n)
        f[UX:UZ + 1, 1::2] = -f[UX:UZ + 1, ::2]
        f[RHO, 1::2] = f[RHO, ::2]
    elif kind == "beyond":  # squares above FP32's range: the share is summed in FP64
        f[UX, 7] = 3e25
    elif kind == "beyond_phi":  # two values of one share whose FP32 sum overflows
        f[PHI, [5, 261]] = 3e38
    elif kind == "tiny":  # all squares below it
        f[UX:UZ + 1] *= np.float32(1e-24)
    elif kind == "far":  # a large term beside the round-off of the others
        f[UX, 11] = 1e6
    got, ref = _reduce(f, shape), _exact(f)
    mag = _exact(np.abs(f))
    mag[5] = ref[5]  # a sum of non-negative terms 1 + phi
    for k in range(8):
        assert abs(Fr(float(got[k])) - ref[k]) <= (12 + 6 + 16) * mag[k] * Fr(1, 2**53), k


@pytest.mark.parametrize("big", [1.0, 3e38])
def test_volume_of_a_phase_field(big):
    """lb_phi_monitor's volume, also where a share overflows FP32: the sum that
    lb_reduce_f64 gives, bit for bit."""
    import torch

    import paper_2405_14551_gb300.lbcg as L
    shape = (16, 16, 12)
    f = _fields(16 * 16 * 12, 9)
    f[PHI, [5, 261]] = big
    s = L.Sim(*shape)
    d = torch.from_numpy(f[PHI].copy()).cuda()
    torch.cuda.synchronize()
    _, volume = L.lb_phi_monitor(s.h, d)
    s.close()
    assert volume == _reduce(f, shape)[5]
    ref = _exact(f)[5]
    assert abs(Fr(volume) - ref) <= (12 + 6 + 16) * ref * Fr(1, 2**53)


@pytest.mark.parametrize("c,nch", [(4, 1), (4, 3), (8, 5)])
@pytest.mark.parametrize("scale", [1.0, 1e-3, 1e-22])
def test_single_loss_terms_keep_fp64_precision(c, nch, scale):
    """One voxel: 2^-53 each for the sum's value, the tree's one addition, the
    FP64 shares at the smallest scale (two products, up to three additions) and
    the product with 1/count."""
    import torch

    import paper_2405_14551_gb300.lbcg as L
    lib = L.load_library()
    for seed in range(24):
        r = np.random.default_rng(100 * c + 10 * nch + seed)
        p, t = (scale * r.standard_normal((1, c))).astype(np.float32), (scale * r.standard_normal((1, c))).astype(np.float32)
        w = r.uniform(0.5, 4.0, nch).astype(np.float32)
        dp, dt, dw = (torch.from_numpy(a).cuda() for a in (p, t, w))
        grad, loss = torch.zeros((1, c), device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
        assert lib.lbnn_mse(dp.data_ptr(), dt.data_ptr(), 1, c, nch, dw.data_ptr(), grad.data_ptr(), loss.data_ptr(), None) == 0
        torch.cuda.synchronize()
        d = p[0] - t[0]  # FP32, as in the kernel
        ref = sum(Fr(float(w[k])) * Fr(float(d[k])) ** 2 for k in range(nch)) * Fr(float(np.float32(1.0) / np.float32(nch)))
        assert abs(Fr(float(loss)) - ref) <= (8 if scale == 1e-22 else 4) * ref * Fr(1, 2**53), seed
