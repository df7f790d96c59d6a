"""The vector forms of the surrogate's glue kernels, against the scalar forms or
FP64 sums."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _setup():
    import torch
    import paper_2405_14551_gb300.lbcg as L
    return torch, L, L.load_library()


@pytest.mark.parametrize("nvox,c", [(1, 4), (1021, 16), (70001, 32), (513, 128), (130, 256)])
@pytest.mark.parametrize("relu", [0, 1])
def test_relu_bias_bwd(nvox, c, relu):
    """One pass equals the two entry points it stands for: the same BF16 gradient
    and, up to the order of nvox FP32 additions, the same sums."""
    torch, L, lib = _setup()
    r = torch.Generator(device="cuda").manual_seed(nvox + c)
    g = torch.randn((nvox, c), generator=r, device="cuda")
    y = torch.randn((nvox, c), generator=r, device="cuda").to(torch.bfloat16)
    y[0, 0] = float("nan")  # not > 0
    gb, gb2 = (torch.empty((nvox, c), dtype=torch.bfloat16, device="cuda") for _ in range(2))
    gf, db = torch.empty_like(g), torch.ones(c, device="cuda")
    assert lib.lbnn_relu_bias_bwd(g.data_ptr(), y.data_ptr() if relu else None, nvox, c, relu, gb.data_ptr(), db.data_ptr(),
                                  None) == 0, lib.lb_last_error()
    assert lib.lbnn_relu_bwd(g.data_ptr(), y.data_ptr() if relu else None, nvox * c, relu, gb2.data_ptr(), gf.data_ptr(),
                             None) == 0
    torch.cuda.synchronize()
    assert torch.equal(gb, gb2)
    ref, mag = 1 + gf.double().sum(0), 1 + gf.double().abs().sum(0)
    # at most nvox / 1 + 460 additions in a chain, each 2^-24 of a partial sum; random signs
    assert bool(((db.double() - ref).abs() <= mag * 2.0**-24 * (8 + nvox**0.5)).all())
    for bad in (3, 12, 512):
        assert lib.lbnn_relu_bias_bwd(g.data_ptr(), None, 1, bad, 0, gb.data_ptr(), db.data_ptr(), None) != 0
    assert lib.lbnn_relu_bias_bwd(g.data_ptr() + 4, None, 1, 4, 0, gb.data_ptr(), db.data_ptr(), None) != 0


# an aligned and a misaligned copy of the same tensors take the vector and the scalar form
@pytest.mark.parametrize("cs,cl", [(4, 8), (32, 64), (16, 20)])
def test_vector_glue_equals_scalar(cs, cl):
    torch, L, lib = _setup()
    nx, ny, nz, nb = 6, 4, 2, 2
    r = torch.Generator(device="cuda").manual_seed(cs + cl)

    def two(*shape):
        a = torch.randn(shape, generator=r, device="cuda")
        flat = torch.empty(a.numel() + 1, device="cuda")
        flat[1:] = a.flatten()
        return a, flat[1:].view(shape)  # 4 bytes off

    nv, nl = nb * nz * ny * nx, nb * nz * ny * nx // 8
    dout, skip, low = two(nv, cs + cl), two(nv, cs), two(nl, cl)
    dy, dx = two(nl, cs), two(nv, cs)
    for k in range(2):
        assert lib.lbnn_up_concat_bwd(dout[k].data_ptr(), cs, cl, nx, ny, nz, nb, skip[k].data_ptr(), low[k].data_ptr(), None) == 0
        assert lib.lbnn_avgpool2_bwd(dy[k].data_ptr(), cs, nx, ny, nz, nb, dx[k].data_ptr(), None) == 0
    torch.cuda.synchronize()
    for a, b in (skip, low, dx):
        assert torch.equal(a, b)


@pytest.mark.parametrize("c,nch", [(16, 5), (8, 8), (4, 1), (6, 5)])
@pytest.mark.parametrize("big", [1.0, 1e19, float("inf")])
def test_mse_sums(c, nch, big):
    """The loss to 1e-12 of its FP64 value (about 2^-45 a term), also where the
    squares leave FP32, and infinite where a term is."""
    torch, L, lib = _setup()
    n = 3001
    r = torch.Generator(device="cuda").manual_seed(c + nch)
    p, t = (torch.randn((n, c), generator=r, device="cuda") for _ in range(2))
    w = torch.rand(nch, generator=r, device="cuda") + 0.5
    p[7, 0] = big
    grad, loss = torch.full((n, c), 9.0, device="cuda"), torch.zeros(1, dtype=torch.float64, device="cuda")
    assert lib.lbnn_mse(p.data_ptr(), t.data_ptr(), n, c, nch, w.data_ptr(), grad.data_ptr(), loss.data_ptr(), None) == 0, \
        lib.lb_last_error()
    torch.cuda.synchronize()
    d = (p - t)[:, :nch].double()
    ref = float((w.double() * d * d).sum()) * float(np.float32(1.0) / np.float32(n * nch))
    got = float(loss)
    assert got == ref if np.isinf(ref) else abs(got - ref) <= 1e-12 * ref
    assert bool((grad[:, nch:] == 0).all())
