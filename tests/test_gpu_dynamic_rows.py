"""The row kernel of the per-token dynamic quantizer around its switches: 8, 16 and 32 lanes per row, one to six chunks per
lane, the largest K it takes and the first it does not; row counts around a block; rows whose maximum is shared by several
near-equal quotients (decided by the exact divisions), dead rows and rows of inf / NaN."""
import numpy as np
import pytest

import oracle
from paper_2412_20386_b200 import workloads as wl

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


@pytest.mark.parametrize("K", [8, 64, 72, 128, 136, 256, 264, 520, 768, 776, 1024, 1032, 1288, 1536, 1544])
@pytest.mark.parametrize("M", [1, 31, 33, 1031])
def test_row_steps_and_codes_match_oracle(env, K, M):
    ptq, torch = env
    rng = np.random.default_rng(K * 7 + M)
    x = (rng.standard_t(3, (M, K)) * np.exp(rng.normal(0, 2, (M, 1)))).astype(np.float16)
    s = np.exp(rng.uniform(-3, 3, K)).astype(np.float32)
    # quotients within a few binary32 ulps of each other: x = fp16, s a little off a common ratio
    if M > 4:
        x[1] = np.float16(3.0)
        s[: K // 2] = np.nextafter(np.float32(0.37), np.float32(1))
        s[K // 2:] = np.float32(0.37)
        x[2], x[3, K // 3], x[4, -1] = 0.0, np.inf, np.nan
    layer = ptq.PtqLinear(np.ones((8, K), np.int8), np.ones(8, np.float32), s, np.ones(1, np.float32))
    _, q, _, step = layer.forward_dynamic_debug(torch.from_numpy(x.reshape(M, 1, K)).cuda())
    torch.cuda.synchronize()
    layer.device_status()
    q_ref, step_ref = oracle.quantize_dynamic(x, s)
    assert np.array_equal(step.cpu().numpy().view(np.uint32), step_ref.view(np.uint32))
    assert np.array_equal(q.cpu().numpy().reshape(M, K), q_ref)
    layer.close()


@pytest.mark.parametrize("K,M", [(8, 47000), (128, 23003), (264, 12001), (768, 11003), (1536, 9007)])
def test_rows_of_later_rounds(env, K, M):
    """More rows than the chip takes at once: a warp's second and third row come from the copies it made ahead, with rows
    missing in the last round and an infinite and an all-zero row among them."""
    ptq, torch = env
    rng = np.random.default_rng(K)
    x = (rng.standard_normal((M, K)) * np.exp(rng.normal(0, 2, (M, 1)))).astype(np.float16)
    x[M // 2, K // 2], x[M - 2] = np.inf, 0.0
    s = np.exp(rng.uniform(-3, 3, K)).astype(np.float32)
    layer = ptq.PtqLinear(np.ones((8, K), np.int8), np.ones(8, np.float32), s, np.ones(1, np.float32))
    _, q, _, step = layer.forward_dynamic_debug(torch.from_numpy(x.reshape(M, 1, K)).cuda())
    torch.cuda.synchronize()
    layer.device_status()
    q_ref, step_ref = oracle.quantize_dynamic(x, s)
    assert np.array_equal(step.cpu().numpy().view(np.uint32), step_ref.view(np.uint32))
    assert np.array_equal(q.cpu().numpy().reshape(M, K), q_ref)
    layer.close()
