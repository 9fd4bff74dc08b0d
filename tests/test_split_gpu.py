"""Layers with few tiles and long reductions: the reduction of a tile split over a
cluster of 2, 4 or 8 CTAs, the parts' sums exchanged through distributed shared
memory.  Products and convolutions of every activation source, both N tiles, ragged
rows, channels and shares, the output stage; every output against the fp64 oracle."""
import numpy as np
import pytest
import torch

import oracle
import paper_1910_11971_gb300 as cci
from paper_1910_11971_gb300 import workloads as wl
from parity_util import TOL, assert_within_tol, f64, oracle_reference

pytestmark = pytest.mark.gpu
BF16 = torch.bfloat16


@pytest.fixture(scope="module")
def dev():
    return torch.device("cuda:0")


# (N, Cin, Cout, G, K, dtype): 8, 4 and 2 parts; N past one M tile (narrower bf16
# products take another kernel); shares of unequal length; a ragged N tile
PRODUCTS = [(130, 4096, 64, 8, 2, "bf16"), (200, 4000, 1000, 8, 2, "bf16"), (513, 1096, 488, 8, 4, "bf16"),
            (300, 2056, 72, 4, 1, "bf16"), (104, 1968, 64, 16, 8, "f32"), (33, 1100, 200, 8, 2, "f32"),
            (700, 2048, 260, 4, 2, "f32")]


@pytest.mark.parametrize("N,Cin,Cout,G,K,dtype", PRODUCTS)
def test_split_product(dev, N, Cin, Cout, G, K, dtype):
    X, W = wl.random_small(N + Cin, dtype, N, Cin, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    st = cci.new_status(dev)
    Y = cci.linear(X.to(dev), v, i, Cout, G, K, status=st)
    assert cci.read_status(st) == 0
    _, _, Wd, mask = oracle_reference(W, G, K)
    Yo, S = oracle.linear(f64(X), Wd, mask)
    assert_within_tol(f64(Y), Yo, S, f"split product {N} x {Cin} -> {Cout}")


# (B, H, W, Cin, Cout, k, stride, pad, G, K, dtype): boxes (also in the place of halo
# copies), ragged channels, the gather (stride 3; fp32 channels off the stage depth)
CONVS = [(2, 7, 7, 512, 512, 3, 1, 1, 8, 2, "bf16"), (3, 9, 9, 256, 72, 3, 2, 1, 8, 2, "bf16"),
         (1, 14, 14, 320, 32, 3, 1, 1, 16, 4, "bf16"), (2, 11, 13, 104, 96, 3, 1, 1, 8, 2, "bf16"),
         (1, 20, 20, 64, 64, 5, 3, 2, 8, 2, "bf16"), (2, 8, 8, 64, 128, 3, 1, 1, 8, 2, "f32"),
         (1, 13, 9, 100, 40, 3, 1, 1, 4, 1, "f32")]


@pytest.mark.parametrize("bf16_out", [False, True])
@pytest.mark.parametrize("B,H,Wi,Cin,Cout,k,stride,pad,G,K,dtype", CONVS)
def test_split_conv(dev, B, H, Wi, Cin, Cout, k, stride, pad, G, K, dtype, bf16_out):
    g = torch.Generator().manual_seed(B + H + Cin + Cout)
    dt = BF16 if dtype == "bf16" else torch.float32
    X = torch.randn((B, H, Wi, Cin), generator=g).clamp_min(0).to(dt)
    W = torch.randn((Cout, k * k * Cin), generator=g).to(dt)
    bias = torch.linspace(-3.0, 3.0, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    st = cci.new_status(dev)
    Y = cci.conv2d_fused(X.to(dev), v, i, Cout, G, K, k, k, (stride, stride), (pad, pad), bias=bias.to(dev), relu=True,
                         out_dtype=BF16 if bf16_out else torch.float32, status=st)
    assert cci.read_status(st) == 0
    _, _, Wd, mask = oracle_reference(W, G, K)
    Yo, S = oracle.conv2d(f64(X), Wd, mask, k, k, (stride, stride), (pad, pad))
    b = f64(bias)
    ref = np.maximum(Yo + b, 0.0)
    lim = TOL * (S + np.abs(b)) + (2.0 ** -8 * np.abs(ref) if bf16_out else 0.0)
    assert (np.abs(f64(Y).reshape(-1, Cout) - ref) <= lim).all()


@pytest.mark.parametrize("N,chunk", [(300, 128), (5000, 200)])
def test_host_chunks_keep_the_bits_of_a_split_product(dev, N, chunk):
    """The split is chosen for the whole call: chunks of a split and of an unsplit
    product give its bits."""
    Cin, Cout, G, K = 2048, 256, 8, 2
    X, W = wl.random_small(12, "bf16", N, Cin, Cout)
    v, i = cci.pack(W.to(dev), G, K)
    Y = cci.linear(X.to(dev), v, i, Cout, G, K).cpu()
    Yh = cci.linear_host(X.pin_memory(), v, i, Cout, G, K, chunk=chunk)
    torch.cuda.synchronize()
    assert torch.equal(Y.view(torch.int32), Yh.view(torch.int32))
