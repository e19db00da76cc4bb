"""The GEMM kernel that keeps its weights in shared memory (K <= 384), where its order of tiles and its weight reloads can go wrong: a
single N tile (CTAs stride over the rows), CTAs on one group each with and without left-over row tiles, contiguous shares that cross one and
several N tiles, one to three k-blocks with ragged K, ragged N, asymmetric layers, layers with a bias, one tile per CTA and fewer.  Oracle:
the integer accumulators computed on the host from the codes and weights, every element, and the scaled output within the repository's
bound max(2^-10 |y|, 1e-3)."""
import numpy as np
import pytest

from paper_2412_20386_b200 import workloads as wl
from parity_util import assert_y_close, layer_inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__ as entry
    entry.build()
    import paper_2412_20386_b200 as ptq
    torch.cuda.set_device(0)
    return ptq, torch


@pytest.mark.parametrize("K,N,T,B,bias,asym", [
    (96, 96, 784, 80, False, False),       # one N tile, strided
    (384, 200, 197, 300, True, True),      # one N tile, three k-blocks
    (200, 600, 197, 110, True, False),     # K and N ragged, CTAs on one N tile each
    (384, 1792, 128, 148, True, False),    # seven N tiles on 148 row tiles: contiguous shares, which cross one N tile
    (40, 60000, 67, 3, False, False),      # two row tiles: a share crosses several N tiles
    (384, 58000, 64, 4, False, True),
    (256, 16, 7, 8121, False, False),      # a single 16-column step per tile
    (16, 64, 37, 1800, True, False),       # two stages of codes: four tiles per CTA
    (13, 8, 64, 900, False, True),
    # the weights of all N tiles at once, row panels as units: two and three N tiles (of a panel's odd number each team has the other half of
    # the tiles in the next panel), last tiles and panels that are not full, two k-blocks
    (96, 384, 784, 48, False, False),
    (128, 488, 37, 1024, True, False),
    (33, 648, 197, 192, False, True),
    (40, 512, 128, 103, False, False),     # code rows of 48 bytes, weights read in lines of 128
    (80, 528, 128, 115, True, False),
    (200, 264, 50, 740, True, False),
    (64, 1536, 197, 128, False, False),    # six N tiles: 24 CTAs on each, and four that share the row tiles that are left
    (104, 1000, 70, 301, True, False),     # four N tiles, every CTA on one: 37 CTAs each, rows of 2000 bytes
    (300, 600, 64, 150, True, False),      # few tiles: one and two per CTA
    (96, 48, 197, 60, False, False),       # fewer tiles than SMs
    (384, 40, 128, 149, False, False),     # one tile more than CTAs
])
def test_resident_weights(env, K, N, T, B, bias, asym):
    ptq, torch = env
    spec = wl.LinearSpec(13, K % 89, N % 7, "resident", B, T, K, N, bias=bias)
    x, wq, dw, b, s, dx = layer_inputs(spec, B=1)
    z = (np.arange(T) * 37 % 256).astype(np.int32) if asym else None
    layer = ptq.PtqLinear(wq, dw, s, dx, b, act_zero=z) if asym else ptq.PtqLinear(wq, dw, s, dx, b)
    assert layer.gemm_variant(B) == 1
    g = torch.Generator(device="cuda").manual_seed(K + N)
    xd = torch.randn(B, T, K, device="cuda", generator=g).half() * torch.from_numpy(s).cuda().half()
    y, codes, acc = layer.forward_debug(xd)
    y2 = layer.forward(xd)
    torch.cuda.synchronize()
    layer.device_status()
    assert torch.equal(y, y2)
    M = B * T
    c = codes.reshape(M, K).double()
    if asym:
        c = c - torch.from_numpy(z).cuda().double().repeat(B)[:, None]
    w = torch.from_numpy(wq).cuda().double()
    acc, y = acc.reshape(M, N), y.reshape(M, N)
    dxr = torch.from_numpy(dx).cuda().double().repeat(B)[:, None]
    for m0 in range(0, M, 8192):                                     # |acc| < 2^53: the products and sums are exact in binary64
        ref = c[m0:m0 + 8192] @ w.T
        assert torch.equal(acc[m0:m0 + 8192].double(), ref), "accumulators differ in rows from %d" % m0
        ref = ref * dxr[m0:m0 + 8192] * torch.from_numpy(dw).cuda().double()
        if b is not None:
            ref = ref + torch.from_numpy(b).cuda().double()
        assert_y_close(y[m0:m0 + 8192].cpu().numpy(), ref.cpu().numpy(), "rows from %d" % m0)
    layer.close()


@pytest.mark.parametrize("K,N,rows,variant", [
    (384, 192, 74, 1), (384, 192, 73, 0), (384, 200, 99, 0), (206, 208, 140, 0),      # one tile per CTA: layers that narrow by half, behind
    (256, 128, 75, 1), (256, 128, 74, 0), (128, 64, 148, 0),                          # a four times wider one with more tiles than SMs,
    (96, 48, 98, 1), (96, 48, 99, 0),                                                 # or up to 48 columns on less than two thirds of the SMs
    (128, 512, 74, 0), (128, 512, 75, 1),                                                              # 148 and 150 tiles
])
def test_which_short_layers_keep_their_weights(env, K, N, rows, variant):
    ptq, torch = env
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("row counts for 148 SMs")
    layer = ptq.PtqLinear(np.ones((N, K), np.int8), np.ones(N, np.float32), np.ones(K, np.float32), np.ones(1, np.float32))
    assert layer.gemm_variant(128 * rows) == variant
    layer.close()
