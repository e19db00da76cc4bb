"""Calls on a stream that is not the current one: their temporary buffers must not be blocks that work queued on the current
stream still uses."""
import contextlib

import numpy as np
import pytest

import oracle
from paper_2412_20386_b200 import binding
from parity_util import assert_y_close


def test_scratch_is_allocated_on_the_stream_that_uses_it(monkeypatch):
    import torch
    current, seen = ["current"], []

    @contextlib.contextmanager
    def on(stream):
        before = current[0]
        current[0] = before if stream is None else stream
        yield
        current[0] = before

    real_empty = torch.empty
    monkeypatch.setattr(torch.cuda, "stream", on)
    monkeypatch.setattr(torch, "empty", lambda *a, **k: (seen.append(current[0]), real_empty(*a, **k))[1])

    class Stream:
        pass
    side = Stream()
    monkeypatch.setattr(torch.Tensor, "record_stream", lambda self, s: None)
    assert binding._scratch(100, "cpu", side).numel() == 100 and binding._scratch(1, "cpu", None).numel() == 16
    assert seen == [side, "current"]


@pytest.mark.gpu
def test_offline_steps_on_another_stream_while_freed_memory_is_still_written():
    import torch
    import __graft_entry__ as entry
    entry.build()
    import paper_2412_20386_b200 as ptq
    torch.cuda.set_device(0)
    rng = np.random.default_rng(5)
    K, N, T, Bc = 256, 512, 197, 8
    x = rng.standard_normal((Bc, T, K)).astype(np.float16)
    wq, dw = rng.integers(-127, 128, (N, K)).astype(np.int8), rng.uniform(1e-3, 1e-2, N).astype(np.float32)
    s, dx = oracle.calibrate(x, wq, dw)
    want = [(s, dx), oracle.calibrate_asym(x, wq, dw), oracle.search_act_step(x, s, dx, 20, 11)[:2]]
    xd = torch.from_numpy(x).cuda()
    side = torch.cuda.Stream()
    L = ptq.load_library()
    sizes = [L.ptq_calibrate_workspace_bytes(K, N, T)] * 2 + [L.ptq_search_workspace_bytes(K, T, 20, 11)]
    calls = [lambda: ptq.calibrate(xd, wq, dw, stream=side), lambda: ptq.calibrate_asym(xd, wq, dw, stream=side),
             lambda: ptq.search_act_step(xd, s, dx, 20, 11, stream=side)[:2]]
    a = torch.randn(8192, 8192, device="cuda", dtype=torch.bfloat16)
    for call, nbytes, ref in zip(calls, sizes, want):
        call()
        torch.cuda.synchronize()
        block = torch.empty(nbytes, dtype=torch.uint8, device="cuda")
        for _ in range(8):                                   # some milliseconds of work, then writes to the freed block
            a @ a
            block.fill_(255)
        del block
        got = call()
        torch.cuda.synchronize()
        for g, r in zip(got, ref):
            assert np.array_equal(g, np.asarray(r))


@pytest.mark.gpu
def test_a_new_layer_can_be_used_at_once_on_any_stream():
    """Create returns with the parameters on the device: a call on a stream that is not ordered behind the upload sees them all."""
    import torch
    import __graft_entry__ as entry
    entry.build()
    import paper_2412_20386_b200 as ptq
    torch.cuda.set_device(0)
    rng = np.random.default_rng(6)
    K, N, T = 8192, 2048, 16
    wq, dw = rng.integers(-127, 128, (N, K)).astype(np.int8), rng.uniform(1e-3, 1e-2, N).astype(np.float32)
    s, dx = np.ones(K, np.float32), np.full(T, 0.05, np.float32)
    x = rng.standard_normal((1, T, K)).astype(np.float16)
    y_ref = oracle.linear_forward(x.reshape(T, K), T, wq, dw, s, dx)
    xd, y = torch.from_numpy(x).cuda(), torch.empty((1, T, N), dtype=torch.float16, device="cuda")
    ws = torch.empty(T * K, dtype=torch.uint8, device="cuda")
    side = torch.cuda.Stream()
    torch.cuda.synchronize()
    for _ in range(5):
        layer = ptq.PtqLinear(wq, dw, s, dx)
        layer.forward(xd, y=y, workspace=ws, stream=side)
        side.synchronize()
        assert_y_close(y.cpu().numpy().reshape(T, N), y_ref, "new layer")
        layer.device_status()
        layer.close()
