"""The one-kernel path for few rows at the sizes where it can go wrong: rows around its 16- and 32-token tiles, output
channels around its 128-channel tiles, K around a k-block, an MMA step and its largest, grids on either side of one and
two CTAs per SM, rows of x at every alignment; the three code formats.  Codes and accumulators bit for bit."""
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


@pytest.mark.parametrize("K,N,T,B", [(1, 1, 1, 1), (8, 127, 15, 1), (31, 128, 16, 1), (33, 129, 17, 1), (128, 8, 31, 1),
                                     (136, 300, 33, 2), (384, 192, 197, 1), (1536, 768, 49, 1), (1530, 16, 3, 7),
                                     (192, 130, 148 * 8, 1), (192, 130, 148 * 8 + 1, 1), (96, 100, 148 * 32, 1),
                                     (96, 100, 148 * 32 + 1, 2), (770, 1000, 7, 5)])
def test_few_rows_match_oracle(env, K, N, T, B):
    ptq, torch = env
    check_layer(ptq, torch, wl.LinearSpec(13, K % 83, N % 7, "small", B, T, K, N, bias=bool(N & 1)), flags_list=(0,))


def test_which_sizes_take_one_kernel(env):
    ptq, torch = env
    for K, N, T, want in ((384, 192, 197, 1), (1536, 768, 49, 1), (1544, 64, 16, 2), (192, 768, 12608, 2)):
        layer = ptq.PtqLinear(np.ones((N, K), np.int8), np.ones(N, np.float32), np.ones(K, np.float32), np.ones(T, np.float32))
        x = torch.zeros((1, T, K), dtype=torch.float16, device="cuda")
        assert launches(ptq, lambda: layer.forward(x)) == want, (K, N, T)
        layer.close()


@pytest.mark.parametrize("K,N,T,B", [(384, 192, 197, 1), (129, 257, 9, 3), (12, 100, 40, 5)])
def test_few_rows_asymmetric_and_4bit(env, K, N, T, B):
    ptq, torch = env
    spec = wl.LinearSpec(14, K % 83, 1, "small", B, T, K, N, bias=True)
    x = wl.activations(spec)
    x[:, ::3] = np.abs(x[:, ::3])
    xcal = wl.activations(spec, wl.ROLE_CALIB)
    wq, dw, bias = wl.weights(spec)
    w4 = np.clip(np.rint(wq.astype(np.float32) / 18.0), -8, 7).astype(np.int8)
    xd, x2 = torch.from_numpy(x).cuda(), x.reshape(-1, K)
    s, dx, z = oracle.calibrate_asym(xcal, wq, dw)
    s4, dx4 = oracle.calibrate4(xcal, w4, dw)
    for layer, ref in ((ptq.PtqLinear(wq, dw, s, dx, bias, act_zero=z),
                        oracle.linear_forward_asym(x2, T, wq, dw, s, dx, z, bias, taps=True)),
                       (ptq.PtqLinear(oracle.pack_int4(w4), dw, s4, dx4, bias, packed4_K=K),
                        oracle.linear_forward4(x2, T, w4, dw, s4, dx4, bias, taps=True))):
        assert launches(ptq, lambda: layer.forward(xd)) == 1
        y, _, acc = layer.forward_debug(xd, want_q=False)
        torch.cuda.synchronize()
        layer.device_status()
        assert np.array_equal(acc.cpu().numpy().reshape(-1, N), ref[2])
        assert_y_close(y.cpu().numpy().reshape(-1, N), ref[0], "small")
        assert torch.equal(layer.forward(xd), y)
        layer.close()


@pytest.mark.parametrize("K", [40, 44, 46, 45])
@pytest.mark.parametrize("off", [0, 1, 2, 4])
def test_few_rows_alignments_and_scales_outside_the_reciprocal_range(env, K, off):
    ptq, torch = env
    spec = wl.LinearSpec(15, K, 1, "small", 3, 11, K, 72)
    x, wq, dw, bias, s, dx = layer_inputs(spec)
    x[0, 0, 0], x[1, 2, 3], x[2, 1, 5] = np.inf, -np.inf, np.nan
    buf = torch.zeros(x.size + 8, dtype=torch.float16, device="cuda")
    xv = buf[off:off + x.size].view(x.shape)
    xv.copy_(torch.from_numpy(x).cuda())
    for scale in (1.0, 1e13):
        s2, dx2 = (s * np.float32(scale)).astype(np.float32), (dx / np.float32(scale)).astype(np.float32)
        layer = ptq.PtqLinear(wq, dw, s2, dx2, bias)
        assert launches(ptq, lambda: layer.forward(xv)) == 1
        y, q, acc = layer.forward_debug(xv)
        torch.cuda.synchronize()
        layer.device_status()
        y_ref, q_ref, acc_ref = oracle.linear_forward(x.reshape(-1, K), spec.T, wq, dw, s2, dx2, bias, taps=True)
        assert np.array_equal(q.cpu().numpy().reshape(-1, K), q_ref)
        assert np.array_equal(acc.cpu().numpy().reshape(-1, spec.N), acc_ref)
        assert_y_close(y.cpu().numpy().reshape(-1, spec.N), y_ref, "scale %g" % scale)
        layer.close()
