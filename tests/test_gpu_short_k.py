"""The one-kernel path for layers of a few channels at the sizes where it can go wrong: K around a chunk of 8 and at the largest,
row tiles and shares that end raggedly, more units per CTA than are prefetched, one to seven N tiles (units of one, two and three tiles, the last group smaller), CTAs
that change their weights (RELOADS), rows of x at every alignment, saturating, infinite and NaN inputs, 4-bit codes, and the sizes on either
side of its rule.  Codes and accumulators bit for bit."""
import numpy as np
import pytest

import oracle
from paper_2412_20386_b200 import workloads as wl
from parity_util import assert_y_close, launches, layer_inputs

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


# Layers of which some CTA takes units of several groups on 148 SMs: left-over row tiles of one-tile and of two-tile groups, and contiguous
# shares.  That they do is checked on the host with the order's own functions, beside its other tests.
RELOADS = [(16, 1280, 64, 7552, False, 0), (24, 768, 197, 25216, True, 0), (8, 1536, 197, 25216, False, 0), (5, 1600, 128, 18944, True, 1)]


@pytest.mark.parametrize("K,N,T,M,bias,off", RELOADS + [
    (1, 8, 7, 9800, False, 0), (8, 64, 19, 19000, True, 0), (9, 72, 197, 10047, False, 1), (12, 384, 197, 4925, True, 0),
    (12, 384, 197, 25216, False, 4), (16, 1280, 64, 6400, False, 0), (24, 768, 49, 10045, True, 2), (31, 1000, 3, 3999, False, 0),
    (32, 256, 1, 20001, True, 0), (5, 1600, 128, 12800, False, 0), (3, 24, 7, 329287, True, 1)])
def test_few_channels_match_oracle(env, K, N, T, M, bias, off):
    ptq, torch = env
    spec = wl.LinearSpec(16, K % 83, N % 7, "short_k", M // T, T, K, N, bias=bias)
    x, wq, dw, b, s, dx = layer_inputs(spec)
    M = spec.M
    x = x.reshape(M, K)
    x[M // 3, 0], x[M // 2, K - 1], x[M - 1, K // 2], x[M // 5] = np.inf, np.nan, -np.inf, 60000.0
    layer = ptq.PtqLinear(wq, dw, s, dx, b)
    xb = torch.zeros(x.size + 8, dtype=torch.float16, device="cuda")
    xd = xb[off:off + x.size].view(spec.B, T, K)
    xd.copy_(torch.from_numpy(x.reshape(spec.B, T, K)).cuda())
    assert launches(ptq, lambda: layer.forward(xd)) == 1
    y, q, acc = layer.forward_debug(xd)
    y2 = layer.forward(xd)
    torch.cuda.synchronize()
    layer.device_status()
    y_ref, q_ref, acc_ref = oracle.linear_forward(x, T, wq, dw, s, dx, b, taps=True)
    assert np.array_equal(q.cpu().numpy().reshape(M, K), q_ref)
    assert np.array_equal(acc.cpu().numpy().reshape(M, N), acc_ref)
    assert torch.equal(y, y2)
    assert_y_close(y.cpu().numpy().reshape(M, N), y_ref, "short_k")
    layer.close()


def test_few_channels_4bit(env):
    ptq, torch = env
    K, N, T, B = 12, 384, 197, 25
    spec = wl.LinearSpec(17, 1, 1, "short_k", B, T, K, N, bias=True)
    x, xcal = wl.activations(spec), wl.activations(spec, wl.ROLE_CALIB)
    wq, dw, bias = wl.weights(spec)
    w4 = np.clip(np.rint(wq.astype(np.float32) / 18.0), -8, 7).astype(np.int8)
    s, dx = oracle.calibrate4(xcal, w4, dw)
    layer = ptq.PtqLinear(oracle.pack_int4(w4), dw, s, dx, bias, packed4_K=K)
    xd = torch.from_numpy(x).cuda()
    assert launches(ptq, lambda: layer.forward(xd)) == 1
    y, _, acc = layer.forward_debug(xd, want_q=False)
    torch.cuda.synchronize()
    layer.device_status()
    y_ref, _, acc_ref = oracle.linear_forward4(x.reshape(-1, K), T, w4, dw, s, dx, bias, taps=True)
    assert np.array_equal(acc.cpu().numpy().reshape(-1, N), acc_ref)
    assert_y_close(y.cpu().numpy().reshape(-1, N), y_ref, "short_k 4-bit")
    layer.close()


def test_which_layers_take_one_kernel(env):
    ptq, torch = env
    for K, N, want in ((32, 256, 1), (33, 264, 2), (32, 248, 2), (12, 388, 2)):
        layer = ptq.PtqLinear(np.ones((N, K), np.int8), np.ones(N, np.float32), np.ones(K, np.float32), np.ones(9, np.float32))
        x = torch.zeros((1200, 9, K), dtype=torch.float16, device="cuda")
        assert launches(ptq, lambda: layer.forward(x)) == want, (K, N)
        layer.close()
