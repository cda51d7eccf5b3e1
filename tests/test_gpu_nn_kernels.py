"""Kernels of the learned operator one by one, against FP64 on the same FP32 inputs.

Tolerance: a sum of n products in FP32 is off by at most n half-ulps of the sum
of magnitudes, (n + 2) 2^-24 sum |a b|; the FP64 reductions round once, 2^-24 of
the result (2^-23 asked).
"""
import ctypes

import pytest
import torch

pytestmark = pytest.mark.gpu
EPS = 2.0 ** -24


def lib():
    from paper_2005_00322_gb300 import _abi
    return _abi.load(), _abi


def rnd(*shape, seed=0):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn(*shape, generator=g, device="cuda")


def ptr(t):
    return None if t is None else ctypes.c_void_p(t.data_ptr())


def stream():
    return ctypes.c_void_p(torch.cuda.current_stream().cuda_stream)


@pytest.mark.parametrize("M", [304 * 128, 304 * 128 + 1, 304 * 128 + 127, 100])
@pytest.mark.parametrize("N,K", [(16, 127), (9, 17), (16, 256), (12, 128), (16, 16), (16, 257)])
@pytest.mark.parametrize("beta", [0.0, 0.5])
def test_tall_products(M, N, K, beta):
    """Many rows onto few columns, at the edges of the tiles."""
    L, abi = lib()
    A, B, C = rnd(M, K, seed=1), rnd(N, K, seed=2), rnd(M, N, seed=3)
    want = 2.0 * (A.double() @ B.double().T) + beta * C.double()
    mag = 2.0 * (A.double().abs() @ B.double().abs().T) + beta * C.double().abs()
    d = abi.PstdGemmDesc(1, M, N, K, A.data_ptr(), 0, K, 1, B.data_ptr(), 0, 1, K, C.data_ptr(), 0, N, 1, 2.0, beta,
                         1, 0, 0, 0, K)
    assert L.pstd_nn_gemm(ctypes.byref(d), stream()) == 0
    assert ((C.double() - want).abs() <= (K + 4) * EPS * mag).all()


@pytest.mark.parametrize("C,K,X,Y", [(32, 16, 9, 127), (1, 1, 1, 1), (8, 32, 17, 129), (31, 5, 8, 300), (32, 32, 3, 128)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_mix(C, K, X, Y, adjoint):
    """The one-pass layer half: forward (bias, relu) and adjoint (transposed
    weights, basis by mode, mask)."""
    L, _ = lib()
    B = 3
    W, v, A = rnd(C, C, seed=1), rnd(B, C, X, Y, seed=2), rnd(B, C, X, K, seed=3)
    T = rnd(K, Y, seed=4) if adjoint else rnd(Y, K, seed=4)
    bias = None if adjoint else rnd(C, seed=5)
    mask = rnd(B, C, X, Y, seed=6) if adjoint else None
    out = torch.full_like(v, 7.0)
    assert L.pstd_nn_mix(ptr(W), int(adjoint), ptr(v), ptr(A), ptr(T), int(adjoint), ptr(bias), ptr(mask), ptr(out),
                         B, C, X, Y, K, 0 if adjoint else 1, stream()) == 0
    Wm = (W.T if adjoint else W).double()
    Tm = (T if adjoint else T.T).double()
    z = torch.einsum("oi,bixy->boxy", Wm, v.double()) + torch.einsum("boxk,ky->boxy", A.double(), Tm)
    mag = (torch.einsum("oi,bixy->boxy", Wm.abs(), v.double().abs())
           + torch.einsum("boxk,ky->boxy", A.double().abs(), Tm.abs()))
    if bias is not None:
        z = torch.relu(z + bias.double()[None, :, None, None])
        mag = mag + bias.double().abs()[None, :, None, None]
    if mask is not None:
        z = torch.where(mask > 0, z, torch.zeros_like(z))
    assert ((out.double() - z).abs() <= (C + K + 4) * EPS * mag).all()


def test_mix_limits():
    L, abi = lib()
    t = rnd(4)
    args = (ptr(t), 0, ptr(t), ptr(t), ptr(t), 0, None, None, ptr(t))
    assert L.pstd_nn_mix(*args, 1, 33, 1, 1, 1, 0, stream()) == -6
    assert L.pstd_nn_mix(*args, 1, 1, 1, 1, 33, 0, stream()) == -6
    assert L.pstd_nn_mix(*args, 1, 0, 1, 1, 1, 0, stream()) == -1
    assert L.pstd_nn_mix(None, *args[1:], 1, 1, 1, 1, 1, 0, stream()) == -1
    assert L.pstd_nn_mix(*args, 0, 1, 1, 1, 1, 0, stream()) == 0


@pytest.mark.parametrize("B,C,P", [(1, 1, 1), (3, 2, 255), (2, 5, 2048), (2, 3, 8193), (4, 32, 16383), (2, 1, 0)])
def test_reductions(B, C, P):
    """Channel dots, leading sums and the loss: fewer values than threads,
    tails of every unrolled block, empty rows."""
    L, _ = lib()
    x, y = rnd(B, C, max(P, 1), seed=1)[..., :P].contiguous(), rnd(B, C, max(P, 1), seed=2)[..., :P].contiguous()
    if P == 0:      # an empty tensor has no address; nothing of it is read
        x = y = rnd(1)
    g = torch.full((C,), 7.0, device="cuda")
    cases = [(None, 0), (y, 1)] if P else [(None, 0)]
    for yy, ch in cases:
        assert L.pstd_nn_chan_dot(ptr(x), ptr(yy), ch, ptr(g), B, C, P, stream()) == 0
        prod = (x.double() if yy is None else x.double() * yy.double()) if P else torch.zeros(B, C, 1).cuda().double()
        want, mag = prod.sum(dim=(0, 2)), prod.abs().sum(dim=(0, 2))
        assert ((g.double() - want).abs() <= 2 * EPS * want.abs() + 1e-14 * mag).all()
    if P == 0:
        return
    out = torch.empty(C * P, device="cuda")
    assert L.pstd_nn_sum_lead(ptr(x), ptr(out), B, C * P, stream()) == 0
    want = x.double().reshape(B, -1).sum(0)
    assert ((out.double() - want).abs() <= 2 * EPS * want.abs() + 1e-14 * x.double().abs().reshape(B, -1).sum(0)).all()
    loss, dout = torch.empty(1, device="cuda"), torch.empty_like(x)
    n = x.numel()
    assert L.pstd_nn_mse(ptr(x), ptr(y), ptr(dout), ptr(loss), n, stream()) == 0
    df = (x - y).double()
    want = df.square().mean()
    assert abs(loss.double().item() - want.item()) <= 2 * EPS * want.item()
    assert ((dout.double() - 2.0 / n * df).abs() <= 3 * EPS * (2.0 / n * df).abs()).all()
