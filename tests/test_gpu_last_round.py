"""Layers whose last round of GEMM tiles is cut into narrower ones: one tile too many for the SMs, the largest numbers that pieces
of 64 and of 128 columns can serve and one more, outputs that end inside a piece or before it, outputs without TMA stores, zero
offsets.  Rows come from the SM count of the device.  Codes and accumulators bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2412_20386_b200 import workloads as wl
from parity_util import assert_y_close, check_layer

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


T = 67


def images_for(torch, n_tiles, last):
    """Images of T rows whose 128-row tiles times n_tiles make one round of tiles and `last` more (or the next number that can be made)."""
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    m_tiles = (sms + last(sms) + n_tiles - 1) // n_tiles
    return m_tiles * 128 // T


@pytest.mark.parametrize("K,N,n_tiles,last", [(416, 768, 3, lambda sms: 1), (416, 760, 3, lambda sms: sms // 4),
                                              (450, 768, 3, lambda sms: sms // 4 + 1), (416, 512, 2, lambda sms: sms // 2),
                                              (416, 512, 2, lambda sms: sms // 2 + 1), (900, 523, 3, lambda sms: 2),
                                              (900, 200, 1, lambda sms: 3)])
def test_cut_last_round_matches_oracle(env, K, N, n_tiles, last):
    ptq, torch = env
    check_layer(ptq, torch, wl.LinearSpec(21, K % 83, N % 7, "cut", images_for(torch, n_tiles, last), T, K, N, bias=bool(K & 2)), flags_list=(0,))


def test_cut_last_round_with_zero_offsets(env):
    ptq, torch = env
    K, N = 900, 760
    spec = wl.LinearSpec(22, 1, 1, "cut", images_for(torch, 3, lambda sms: 1), T, K, N, bias=True)
    x = wl.activations(spec)
    x[:, ::3] = np.abs(x[:, ::3])
    wq, dw, bias = wl.weights(spec)
    s, dx, z = oracle.calibrate_asym(wl.activations(spec, wl.ROLE_CALIB), wq, dw)
    layer = ptq.PtqLinear(wq, dw, s, dx, bias, act_zero=z)
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
