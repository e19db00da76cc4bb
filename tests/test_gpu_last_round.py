"""Layers whose last round of GEMM tiles is cut into narrower pieces: one row tile too many for the SMs, the largest numbers of tiles
that pieces of 64 and of 128 columns can serve and one more of each, outputs that end inside a piece or before it (pieces beyond N),
outputs without TMA stores (odd N), zero offsets, a bias, per-token dynamic steps.  Every case asserts how it is cut: the sizes are
those of 148 SMs.  Codes and accumulators bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2412_20386_b200 import workloads as wl
from parity_util import assert_y_close, check_layer, layer_inputs, row_blocks

pytestmark = pytest.mark.gpu

T = 67


@pytest.fixture(scope="module")
def env():
    import torch
    assert torch.cuda.is_available(), "GPU tests need a CUDA device"
    import __graft_entry__ as entry
    entry.build()
    import paper_2412_20386_b200 as ptq
    torch.cuda.set_device(0)
    if torch.cuda.get_device_properties(0).multi_processor_count != 148:
        pytest.skip("the sizes below are cut as they say on 148 SMs")
    return ptq, torch


def spec_of(K, N, m_tiles, bias=False):
    """Images of T = 67 rows that fill m_tiles row tiles, the last one not quite (67 < 128)."""
    spec = wl.LinearSpec(21, K % 83, N % 7, "cut", m_tiles * 128 // T, T, K, N, bias=bias)
    assert (spec.M + 127) // 128 == m_tiles
    return spec


CUT = [  # K, N, row tiles, tile and piece columns, bias
    (1536, 768, 50, 256, 64, False),     # 150 tiles
    (900, 256, 185, 256, 64, True),      # 37 tiles x 4 pieces: as many as there are SMs
    (900, 256, 186, 256, 128, False),    # one tile more
    (416, 512, 111, 256, 128, False),    # 74 tiles x 2 pieces: as many as there are SMs
    (416, 512, 112, 256, 0, False),      # one tile more: whole
    (416, 768, 50, 192, 128, False),     # a piece of 128 and one of 64 columns per tile
    (900, 200, 151, 208, 64, False),     # the last piece of a tile has 16 columns, of which 8 lie below N
    (900, 392, 75, 256, 64, False),      # the second N tile ends in its third piece: the fourth lies beyond N
    (900, 385, 75, 256, 64, True),       # the same, one column into it, no TMA stores
    (900, 761, 50, 256, 64, False),      # no TMA stores
    (416, 523, 60, 192, 64, False),      # no TMA stores, the third N tile ends in its third piece
]


@pytest.mark.parametrize("K,N,m_tiles,tile,piece,bias", CUT)
def test_cut_last_round_matches_oracle(env, K, N, m_tiles, tile, piece, bias):
    ptq, torch = env
    spec = spec_of(K, N, m_tiles, bias)
    _, wq, dw, b, s, dx = layer_inputs(spec, B=1)
    layer = ptq.PtqLinear(wq, dw, s, dx, b)
    assert layer.gemm_tiling(spec.B) == (0, tile, piece)
    layer.close()
    check_layer(ptq, torch, spec, flags_list=(0,))


@pytest.mark.parametrize("N", [760, 761])                  # with and without TMA stores
def test_cut_last_round_with_zero_offsets(env, N):
    ptq, torch = env
    spec = spec_of(900, N, 50, bias=True)
    K = spec.K
    x = wl.activations(spec)
    x[:, ::3] = np.abs(x[:, ::3])
    wq, dw, bias = wl.weights(spec)
    s, dx, z = oracle.calibrate_asym(wl.activations(spec, wl.ROLE_CALIB), wq, dw)
    layer = ptq.PtqLinear(wq, dw, s, dx, bias, act_zero=z)
    assert layer.gemm_tiling(spec.B) == (0, 256, 64)
    xd = torch.from_numpy(x).cuda()
    y, q, acc = layer.forward_debug(xd)
    torch.cuda.synchronize()
    layer.device_status()
    y_ref, q_ref, acc_ref = oracle.linear_forward_asym(x.reshape(-1, K), spec.T, wq, dw, s, dx, z, bias, taps=True)
    assert np.array_equal(q.cpu().numpy().reshape(-1, K), q_ref)
    assert np.array_equal(acc.cpu().numpy().reshape(-1, N), acc_ref)
    assert_y_close(y.cpu().numpy().reshape(-1, N), y_ref, "zero offsets")
    assert torch.equal(layer.forward(xd), y)
    layer.close()


@pytest.mark.parametrize("N", [768, 761])
def test_cut_last_round_with_dynamic_steps(env, N):
    ptq, torch = env
    spec = spec_of(1536, N, 50)
    x, wq, dw, bias, s, dx = layer_inputs(spec)
    layer = ptq.PtqLinear(wq, dw, s, dx, bias)
    assert layer.gemm_tiling(spec.B) == (0, 256, 64)
    xd = torch.from_numpy(x).cuda()
    y, q, acc, step = layer.forward_dynamic_debug(xd)
    y2 = layer.forward_dynamic(xd)
    torch.cuda.synchronize()
    layer.device_status()
    assert torch.equal(y, y2)
    x = x.reshape(spec.M, spec.K)
    q_ref, step_ref = oracle.quantize_dynamic(x, s)
    assert np.array_equal(step.cpu().numpy().view(np.uint32), step_ref.view(np.uint32))
    assert np.array_equal(q.cpu().numpy().reshape(spec.M, spec.K), q_ref)
    acc, y = acc.cpu().numpy().reshape(spec.M, N), y.cpu().numpy().reshape(spec.M, N)
    for m0, m1 in row_blocks(spec.M):
        acc_ref = oracle.int_matmul(q_ref[m0:m1], wq)
        assert np.array_equal(acc[m0:m1], acc_ref), "accumulators differ in rows from %d" % m0
        assert_y_close(y[m0:m1], oracle.dequant(acc_ref, m1 - m0, step_ref[m0:m1], dw, bias), "rows from %d" % m0)
    layer.close()
