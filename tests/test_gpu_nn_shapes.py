"""Kernels of the learned operator over the shapes where their launch rules
change, against FP64 on the same FP32 inputs.

Tolerances: a fused multiply-add rounds once, 2^-24 of its result (2^-23 asked).
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


# all channels in a thread, groups with and without a remainder, one channel each; fewer points than threads
@pytest.mark.parametrize("B,C,P", [(32, 32, 16383), (3, 7, 5000), (1, 32, 70000), (1, 20000, 16), (2, 1000, 257),
                                   (1, 1, 400001), (65535, 1, 3), (1, 65535, 1)])
def test_lift_and_its_adjoint(B, C, P):
    L, _ = lib()
    x, w, b = rnd(B, P, seed=1), rnd(C, seed=2), rnd(C, seed=3)
    v = torch.full((B, C, P), 7.0, device="cuda")
    assert L.pstd_nn_lift(ptr(x), ptr(w), ptr(b), ptr(v), B, C, P, stream()) == 0
    want = w.double()[None, :, None] * x.double()[:, None, :] + b.double()[None, :, None]
    assert ((v.double() - want).abs() <= 2 * EPS * want.abs()).all()
    v.fill_(7.0)
    assert L.pstd_nn_proj_bwd(ptr(x), ptr(w), ptr(v), B, C, P, stream()) == 0
    want = w.double()[None, :, None] * x.double()[:, None, :]
    assert ((v.double() - want).abs() <= 2 * EPS * want.abs()).all()


# one CTA a channel (few values, many channels), eight with whole samples or points shared out, tails of each
@pytest.mark.parametrize("B,C,P", [(1, 4096, 64), (1, 304, 8192), (1, 305, 8192), (8, 3, 1024), (9, 2, 8191), (8, 2, 8192),
                                   (7, 2, 2000), (100, 1, 83), (8191, 5, 1)])
def test_channel_dots(B, C, P):
    """The FP64 sums round once (2^-24 of the result, twice that asked)."""
    L, _ = lib()
    x, y = rnd(B, C, P, seed=1), rnd(B, C, P, seed=2)
    g = torch.full((C,), 7.0, device="cuda")
    for yy, ch in ((None, 0), (y, 1), (y[:, 0].contiguous(), 0)):
        assert L.pstd_nn_chan_dot(ptr(x), ptr(yy), ch, ptr(g), B, C, P, stream()) == 0
        prod = x.double() if yy is None else x.double() * (yy if ch else yy[:, None]).double()
        want, mag = prod.sum(dim=(0, 2)), prod.abs().sum(dim=(0, 2))
        assert ((g.double() - want).abs() <= 2 * EPS * want.abs() + 1e-14 * mag).all()


# either side of the rule (256 columns a row), rows and columns that fill no group
@pytest.mark.parametrize("B,n", [(1, 255), (1, 256), (4, 1023), (4, 1024), (33, 7), (100, 25600), (100, 25599), (3, 400001)])
def test_leading_sums(B, n):
    """The FP64 sums round once (2^-24 of the result, twice that asked)."""
    L, _ = lib()
    x, out = rnd(B, n, seed=1), torch.full((n,), 7.0, device="cuda")
    assert L.pstd_nn_sum_lead(ptr(x), ptr(out), B, n, stream()) == 0
    want, mag = x.double().sum(0), x.double().abs().sum(0)
    assert ((out.double() - want).abs() <= 2 * EPS * want.abs() + 1e-14 * mag).all()


# 64 x 64 against 32 x 32 tiles (ragged by up to half a tile), few and many small products
@pytest.mark.parametrize("batch,M,N,K", [(1, 1056, 1056, 40), (1, 1031, 64, 33), (1, 96, 96, 17), (40, 96, 96, 17),
                                         (151, 32, 32, 50), (152, 32, 32, 50), (38, 33, 40, 7), (1, 32, 32, 1024)])
def test_product_tiles(batch, M, N, K):
    """A sum of n products in FP32 is off by at most n half-ulps of the sum of
    magnitudes, (n + 2) 2^-24 sum |a b|."""
    L, abi = lib()
    A, B, C = rnd(batch, M, K, seed=1), rnd(batch, K, N, seed=2), torch.full((batch, M, N), 7.0, device="cuda")
    d = abi.PstdGemmDesc(batch, M, N, K, A.data_ptr(), M * K, K, 1, B.data_ptr(), K * N, N, 1, C.data_ptr(), M * N, N, 1,
                         1.0, 0.0, 1, 0, 0, 0, K)
    assert L.pstd_nn_gemm(ctypes.byref(d), stream()) == 0
    want, mag = A.double() @ B.double(), A.double().abs() @ B.double().abs()
    assert ((C.double() - want).abs() <= (K + 2) * EPS * mag).all()


# 1, 2 and 4 points a lane, in the last and in the only tile; channels that leave warps idle; 8, 4 and 1 rows a CTA
@pytest.mark.parametrize("B,C,X,Y", [(3, 32, 17, 32), (3, 9, 17, 33), (2, 8, 9, 64), (2, 16, 9, 65), (1, 5, 5, 160),
                                     (1, 24, 5, 192), (1, 4, 5, 193), (304, 2, 9, 10), (40, 3, 37, 20), (1, 32, 129, 127)])
@pytest.mark.parametrize("adjoint", [False, True])
def test_mix_rows(B, C, X, Y, adjoint):
    """A layer's second half, bit for bit the separate products (sums in index
    order, added last) followed by bias and relu, or by the mask."""
    L, abi = lib()
    K, P = 7, X * Y
    W, v, A, T = rnd(C, C, seed=1), rnd(B, C, X, Y, seed=2), rnd(B, C, X, K, seed=3), rnd(K, Y, seed=4)
    bias, mask = (None, rnd(B, C, X, Y, seed=5)) if adjoint else (rnd(C, seed=5), None)
    out = torch.full_like(v, 7.0)
    assert L.pstd_nn_mix(ptr(W), int(adjoint), ptr(v), ptr(A), ptr(T), 1, ptr(bias), ptr(mask), ptr(out), B, C, X, Y, K,
                         0 if adjoint else 1, stream()) == 0

    def product(batch, M, N, K, A, sA, Bm, sB):
        o = torch.empty(batch * M * N, device="cuda")
        d = abi.PstdGemmDesc(batch, M, N, K, A.data_ptr(), *sA, Bm.data_ptr(), *sB, o.data_ptr(), M * N, N, 1, 1.0, 0.0, 1,
                             0, 0, 0, K)
        assert L.pstd_nn_gemm(ctypes.byref(d), stream()) == 0
        return o.view(B, C, X, Y)
    z = (product(B, C, P, C, W, (0, 1, C) if adjoint else (0, C, 1), v, (C * P, P, 1))
         + product(1, B * C * X, Y, K, A, (0, K, 1), T, (0, Y, 1)))
    want = torch.where(mask > 0, z, torch.zeros_like(z)) if adjoint else torch.relu(z + bias[None, :, None, None])
    assert torch.equal(out, want)
