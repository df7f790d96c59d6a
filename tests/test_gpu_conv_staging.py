"""Staging and work split of the convolutions at the edges of their ranges,
against the FP64 reference."""
import numpy as np
import pytest

from oracle import unet_ref as U

pytestmark = pytest.mark.gpu

PER = (True, False, True)


def _setup():
    import torch
    import paper_2405_14551_gb300.lbcg as L
    return torch, L, L.load_library()


def _bf(torch, a):
    return torch.from_numpy(np.asarray(a, np.float32)).to(torch.bfloat16).cuda()


# chunks of 16, 32, 48 and 64 channels; 96 to 1024 weight pieces a step; blocks
# of 1, 2, 4 and 8 planes; one work item, and more items than the chip has SMs
@pytest.mark.parametrize("dims,cin,cout", [
    ((8, 16, 8, 1), 16, 16), ((8, 16, 4, 1), 48, 32), ((16, 16, 2, 1), 144, 48), ((8, 16, 6, 2), 64, 80),
    ((8, 16, 1, 1), 64, 128), ((16, 16, 3, 1), 192, 256), ((64, 64, 40, 1), 32, 16), ((64, 64, 5, 1), 64, 96)])
def test_tiled_convolution(dims, cin, cout):
    torch, L, lib = _setup()
    nx, ny, nz, nb = dims
    r = np.random.default_rng(cin + cout + nz)
    x = _bf(torch, r.standard_normal((nb, nz, ny, nx, cin)))
    w = _bf(torch, r.standard_normal((cout, 27, cin)) / np.sqrt(27 * cin))
    y = torch.zeros((nb, nz, ny, nx, cout), device="cuda")
    st = torch.zeros(4, dtype=torch.int32, device="cuda")
    rc = lib.lbnn_conv3d_fwd(x.data_ptr(), cin, w.data_ptr(), 27, None, None, y.data_ptr(), cout, 0, nx, ny, nz, nb, 5, 0,
                             st.data_ptr(), None)
    assert rc == 0, lib.lb_last_error()
    torch.cuda.synchronize()
    f8 = lambda t: t.float().cpu().numpy().astype(np.float64)
    ref = U.conv3d(f8(x), f8(w), np.zeros(cout), PER, 27)
    # 27 cin exact products in FP32 sums: at worst 27 cin 2^-24 of the summed magnitudes, here random walks
    assert int(st[0]) == 0
    assert np.abs(y.cpu().numpy() - ref).max() <= 1e-5 * max(1.0, np.abs(ref).max())


# both halo operands, both parities at a block's first group, one to many P slices
@pytest.mark.parametrize("dims,cin,cout", [
    ((8, 16, 1, 1), 16, 16), ((8, 16, 5, 1), 48, 80), ((16, 16, 3, 1), 192, 64), ((8, 32, 3, 2), 32, 96),
    ((16, 16, 2, 1), 384, 128), ((8, 16, 2, 1), 256, 256), ((64, 64, 12, 1), 16, 32)])
def test_tiled_weight_gradient(dims, cin, cout):
    torch, L, lib = _setup()
    nx, ny, nz, nb = dims
    r = np.random.default_rng(cin * 3 + cout + nz)
    x = _bf(torch, r.standard_normal((nb, nz, ny, nx, cin)))
    g = _bf(torch, r.standard_normal((nb, nz, ny, nx, cout)))
    dw = torch.zeros((cout, 27, cin), device="cuda")
    st = torch.zeros(4, dtype=torch.int32, device="cuda")
    rc = lib.lbnn_conv3d_wgrad(g.data_ptr(), cout, x.data_ptr(), cin, 27, dw.data_ptr(), nx, ny, nz, nb, 5, 64, st.data_ptr(),
                               None)
    assert rc == 0, lib.lb_last_error()
    torch.cuda.synchronize()
    f8 = lambda t: t.float().cpu().numpy().astype(np.float64)
    _, ref, _ = U.conv3d_backward(f8(x), np.zeros((cout, 27, cin)), f8(g), PER, 27)
    assert int(st[0]) == 0
    assert np.abs(dw.cpu().numpy() - ref).max() <= 1e-5 * max(1.0, np.abs(ref).max())


# one voxel, a remainder of every kind, a run of full groups; 1x1x1 taps
@pytest.mark.parametrize("nvox", [1, 63, 64, 65, 4096 + 17])
@pytest.mark.parametrize("cin,cout", [(16, 16), (48, 16), (32, 64)])
def test_pointwise_weight_gradient(nvox, cin, cout):
    torch, L, lib = _setup()
    r = np.random.default_rng(nvox + cin)
    x, g = _bf(torch, r.standard_normal((nvox, cin))), _bf(torch, r.standard_normal((nvox, cout)))
    dw = torch.zeros((cout, cin), device="cuda")
    st = torch.zeros(4, dtype=torch.int32, device="cuda")
    for vpc in (64, 256):
        dw.zero_()
        assert lib.lbnn_conv3d_wgrad(g.data_ptr(), cout, x.data_ptr(), cin, 1, dw.data_ptr(), nvox, 1, 1, 1, 7, vpc,
                                     st.data_ptr(), None) == 0, lib.lb_last_error()
        torch.cuda.synchronize()
        ref = g.double().T @ x.double()
        assert int(st[0]) == 0
        assert float((dw.double() - ref).abs().max()) <= 1e-5 * max(1.0, float(ref.abs().max()))
