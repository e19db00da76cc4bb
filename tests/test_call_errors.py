"""Error classes of the forward calls: what the extension module refuses by itself (no GPU needed), and a failed allocation,
which raises the class that torch's own allocations raise, so that a caller can catch it and shrink its batch."""
import numpy as np
import pytest

import __graft_entry__ as entry


@pytest.fixture(scope="module")
def native():
    entry.build()
    from paper_2412_20386_b200 import binding
    return binding._load_native()


@pytest.mark.parametrize("call", ["forward", "forward_static", "forward_dynamic"])
def test_bad_arguments_are_refused_before_the_library_is_called(native, call):
    import torch
    f = getattr(native, call)
    with pytest.raises(TypeError):
        f(0, 1, 1, 1)
    with pytest.raises(TypeError):
        f(0, 1, 1, 1, np.zeros((1, 1, 1), np.float16), None, None)
    for x in (torch.zeros(1, 1, 1), torch.zeros(1, 1, 1, dtype=torch.float16)):      # wrong type, not on the device
        with pytest.raises(ValueError):
            f(0, 1, 1, 1, x, None, None)


@pytest.mark.parametrize("call", ["calibrate", "search"])
def test_bad_arguments_of_the_offline_steps_are_refused_before_the_library_is_called(native, call):
    import torch
    f, t, a = getattr(native, call), torch.zeros(1), np.ones(1, np.float32)
    fixed = a.copy()
    fixed.flags.writeable = False
    with pytest.raises(TypeError):
        f(0, 1, 1, 1, 1, t, t, a, a)
    with pytest.raises(TypeError):
        f(0, 1, 1, 1, 1, a, t, a, a, a, a, a)                                        # no tensor
    with pytest.raises(TypeError):
        f(0, 1, 1, 1, 1, t, t, 1.0, a, a, a, a)                                      # no array
    with pytest.raises((BufferError, ValueError)):
        f(0, 1, 1, 1, 1, t, t, a, a, fixed, a, a)                                    # an output that cannot be written
    with pytest.raises((BufferError, ValueError)):
        f(0, 1, 1, 1, 1, t, t, np.ones((4, 4), np.int8)[:, ::2], a, a, a, a)         # not contiguous


def test_offline_steps_report_a_failed_allocation_as_the_librarys_error(native, monkeypatch):
    import torch
    import paper_2412_20386_b200 as ptq

    class DeviceTensor:                                      # as far as the offline calls look before they allocate
        dtype, is_cuda, shape, device = torch.float16, True, (2, 3, 8), "cuda"
        is_contiguous, dim, data_ptr = (lambda self: True), (lambda self: 3), (lambda self: 16)

    def no_memory(*args, **kwargs):
        raise torch.OutOfMemoryError("no memory")
    monkeypatch.setattr(ptq.binding, "_scratch", no_memory)
    x, w, dw = DeviceTensor(), np.ones((4, 8), np.int8), np.ones(4, np.float32)
    for call in (lambda: ptq.calibrate(x, w, dw), lambda: ptq.calibrate(x, w, dw, per_tensor=True), lambda: ptq.calibrate_asym(x, w, dw),
                 lambda: ptq.calibrate_w4a4(x, np.ones((4, 4), np.uint8), 8, dw),
                 lambda: ptq.search_act_step(x, np.ones(8, np.float32), np.ones(3, np.float32))):
        with pytest.raises(ptq.PtqError) as e:
            call()
        assert e.value.status == 7                           # PTQ_ERR_NOMEM


@pytest.mark.gpu
@pytest.mark.parametrize("call", ["forward", "forward_dynamic"])
def test_an_output_that_does_not_fit_raises_torchs_out_of_memory(call):
    import torch
    entry.build()
    import paper_2412_20386_b200 as ptq
    torch.cuda.set_device(0)
    N = 65536
    layer = ptq.PtqLinear(np.ones((N, 1), np.int8), np.ones(N, np.float32), np.ones(1, np.float32), np.ones(1, np.float32))
    x = torch.zeros((1 << 21, 1, 1), dtype=torch.float16, device="cuda")             # 4 MB in, 256 GiB out
    with pytest.raises(torch.OutOfMemoryError):
        getattr(layer, call)(x)
    y = getattr(layer, call)(x[:3])                                                  # a smaller batch goes on
    torch.cuda.synchronize()
    layer.device_status()
    assert tuple(y.shape) == (3, 1, N) and float(y.float().abs().max()) == 0.0
    layer.close()
