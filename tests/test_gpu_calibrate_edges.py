"""Calibration kernels at the sizes where their splits change: channel counts around one thread's chunk, one block's row
lanes and one block's width, few positions with many images, weights that are not a multiple of a row block; aligned and
unaligned inputs; NaN and infinite activations.  The result is unique, so it is compared bit for bit."""
import numpy as np
import pytest

import oracle

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


@pytest.mark.parametrize("K,N,T,Bc", [(1, 1, 1, 1), (7, 33, 3, 5), (8, 31, 2, 700), (257, 32, 4, 9), (264, 65, 1, 300),
                                      (2056, 5, 2, 3), (1032, 40, 150, 17)])
@pytest.mark.parametrize("offset", [0, 1])
def test_calibration_edges_all_schemes(env, K, N, T, Bc, offset):
    ptq, torch = env
    rng = np.random.default_rng(K * 1000 + N)
    x = (rng.standard_t(3, (Bc, T, K)) * np.exp(rng.normal(0, 1, (1, T, 1)))).astype(np.float16)
    x[0, 0, 0] = np.nan
    x[-1, -1, -1] = 0.0
    wq = rng.integers(-127, 128, (N, K)).astype(np.int8)
    dw = rng.uniform(1e-3, 1e-2, N).astype(np.float32)
    buf = torch.zeros(x.size + 8, dtype=torch.float16, device="cuda")
    xd = buf[offset:offset + x.size].view(Bc, T, K)
    xd.copy_(torch.from_numpy(x).cuda())
    w4 = rng.integers(-8, 8, (N, K)).astype(np.int8)
    pairs = [(ptq.calibrate(xd, wq, dw), oracle.calibrate(x, wq, dw)),
             (ptq.calibrate_asym(xd, wq, dw), oracle.calibrate_asym(x, wq, dw)),
             (ptq.calibrate_w4a4(xd, oracle.pack_int4(w4), K, dw), oracle.calibrate4(x, w4, dw))]
    s, dx = ptq.calibrate(xd, wq, dw, per_tensor=True)
    s_ref, step_ref = oracle.calibrate_per_tensor(x, wq, dw)
    pairs.append(((s, dx), (s_ref, np.full(T, step_ref, np.float32))))
    for got, want in pairs:
        for a, b in zip(got, want):
            assert np.array_equal(a, np.asarray(b).reshape(a.shape))


def test_infinite_activations_reach_the_maxima(env):
    ptq, torch = env
    x = np.ones((2, 3, 16), np.float16)
    x[1, 2, 5] = np.inf
    x[0, 1, 3] = -np.inf
    wq = np.ones((4, 16), np.int8)
    dw = np.full(4, 0.01, np.float32)
    for got, want in ((ptq.calibrate(torch.from_numpy(x).cuda(), wq, dw), oracle.calibrate(x, wq, dw)),):
        for a, b in zip(got, want):
            assert np.array_equal(a, b, equal_nan=True)
