"""Sizes that fill no chunk, no vector store and no tile: the quantize kernel's partial chunks at every load width (row
alignment 16, 8, 4 and 2 bytes; dense and padded code rows) and the GEMM's row copies at every store width (N a multiple
of 4, of 2, odd; y offset by 1, 2 and 4 elements), against the oracle.  The sizes come with few rows, which one kernel takes, and
with rows for the quantize and the GEMM kernel; the number of launches tells which ran."""
import numpy as np
import pytest

import oracle
from paper_2412_20386_b200 import workloads as wl
from parity_util import assert_y_close, check_layer, launches, layer_inputs

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


@pytest.mark.parametrize("K,N,T,B", [(1, 1, 1, 1), (7, 9, 3, 200), (9, 65, 5, 31), (12, 44, 197, 9), (129, 257, 5, 30),
                                     (250, 130, 13, 70), (520, 601, 197, 30), (31, 1028, 1, 300)])
def test_ragged_layers_match_oracle(env, K, N, T, B):
    ptq, torch = env
    check_layer(ptq, torch, wl.LinearSpec(11, K % 89, N % 7, "ragged", B, T, K, N, bias=bool(K & 1)), flags_list=(0,))


# as above, with rows beyond the one-kernel path
@pytest.mark.parametrize("K,N,T,B", [(1, 1, 1, 9500), (7, 9, 3, 3200), (9, 65, 5, 1901), (12, 44, 197, 49), (129, 257, 5, 640),
                                     (250, 130, 13, 365), (31, 1028, 1, 1100), (33, 1026, 1, 1100)])
def test_ragged_layers_in_two_kernels_match_oracle(env, K, N, T, B):
    ptq, torch = env
    check_layer(ptq, torch, wl.LinearSpec(11, K % 89, N % 7, "ragged", B, T, K, N, bias=bool(K & 1)), flags_list=(0,))
    layer = ptq.PtqLinear(np.ones((N, K), np.int8), np.ones(N, np.float32), np.ones(K, np.float32), np.ones(T, np.float32))
    assert launches(ptq, lambda: layer.forward(torch.zeros((B, T, K), dtype=torch.float16, device="cuda"))) == 2
    layer.close()


@pytest.mark.parametrize("K", [4, 6, 13, 24, 520])
@pytest.mark.parametrize("x_off,y_off", [(0, 0), (1, 1), (2, 2), (4, 4)])
@pytest.mark.parametrize("B", [37, 870])
def test_ragged_alignments(env, K, x_off, y_off, B):
    ptq, torch = env
    spec = wl.LinearSpec(12, K, 1, "align", B, 11, K, 40, bias=False)
    x, wq, dw, bias, s, dx = layer_inputs(spec)
    M = spec.M
    layer = ptq.PtqLinear(wq, dw, s, dx, bias)
    xb = torch.zeros(x.size + 8, dtype=torch.float16, device="cuda")
    xv = xb[x_off:x_off + x.size].view(x.shape)
    xv.copy_(torch.from_numpy(x).cuda())
    yb = torch.full((M * spec.N + 8,), -7.0, dtype=torch.float16, device="cuda")
    yv = yb[y_off:y_off + M * spec.N].view(spec.B, spec.T, spec.N)
    y_ref, q_ref, _ = oracle.linear_forward(x.reshape(M, K), spec.T, wq, dw, s, dx, bias, taps=True)
    qb = torch.full((M * K + 8,), 99, dtype=torch.int8, device="cuda")
    layer.quantize(xv, q=qb[x_off:x_off + M * K])
    one_kernel = B == 37 or (K == 4 and y_off == 0)          # few rows; few channels, for which y has to be aligned
    assert launches(ptq, lambda: layer.forward(xv, y=yv)) == (1 if one_kernel else 2)
    torch.cuda.synchronize()
    layer.device_status()
    q = qb.cpu().numpy()
    assert np.array_equal(q[x_off:x_off + M * K].reshape(M, K), q_ref)
    assert (q[:x_off] == 99).all() and (q[x_off + M * K:] == 99).all()
    assert_y_close(yv.cpu().numpy().reshape(M, spec.N), y_ref, "offsets")
    assert bool((yb[:y_off] == -7).all()) and bool((yb[y_off + M * spec.N:] == -7).all())
    layer.close()
