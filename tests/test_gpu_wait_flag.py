"""A device wait that ran out is reported by every call that waits for the stream to give a result.

The transform kernels report such a wait in an int on the device (the handle's only 4-byte allocation).
Here no wait runs out: the test sets the int as a kernel would, through the allocator that it gave the
grid, and looks at what each call answers; ch_device_status clears it."""
import ctypes

import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2406_01322_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

SIZE = dict(nx=64, ny=64, nz=17)   # 34816 modes: the physical fields and x, y on the tensor cores
TIMEOUT = -6


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_01322_gb300 import build
    build.build_library()
    from paper_2406_01322_gb300 import binding as b
    b.lib()
    return b


def initial(seed):
    f = inputs.initial_fields(*SIZE.values(), 150.0, 0.05, 1, 0.4, seed)
    return [torch.from_numpy(np.ascontiguousarray(a)) for a in f]


def set_flag(alloc):
    flags = [t for t in alloc.live.values() if t.numel() == 4]
    assert flags
    for t in flags:
        t.copy_(torch.tensor([1, 0, 0, 0], dtype=torch.uint8))
    torch.cuda.synchronize()


def test_waiting_calls_report_it_until_the_status_is_read(binding):
    alloc = binding.TorchAllocator(torch.device("cuda:0"))
    g = binding.Grid(**SIZE, allocator=alloc)
    g.set_fields(*initial(1))
    state = g.get_state()
    copy = state.clone()
    g.step(1)
    L = binding.lib()
    host = [np.empty(g.shape) for _ in range(4)]
    ptr = [ctypes.c_void_p(a.ctypes.data) for a in host]
    J, ms = ctypes.c_double(), (ctypes.c_double * 16)()
    st = ctypes.c_void_p(state.data_ptr())
    waiting = {
        "diagnostics": lambda: L.ch_diagnostics(g.h, ctypes.byref(binding.Diag())),
        "get_fields_host": lambda: L.ch_get_fields_host(g.h, *ptr),
        "get_state": lambda: L.ch_get_state(g.h, ctypes.c_void_p(copy.data_ptr())),
        "step_timed": lambda: L.ch_step_timed(g.h, 1, ms, ctypes.byref(J)),
        "objective": lambda: L.ch_objective(g.h, ctypes.byref(J)),
        "adjoint_begin": lambda: L.ch_adjoint_begin(g.h, ctypes.byref(J)),
    }
    for name, call in waiting.items():
        assert call() == 0, name
        g.adjoint_end()
        set_flag(alloc)
        assert call() == TIMEOUT, name
        with pytest.raises(binding.ChError) as e:
            g.device_status()
        assert e.value.code == TIMEOUT
        g.device_status()
    reverse = {
        "adjoint_step": lambda: L.ch_adjoint_step(g.h, st),
        "adjoint_step_timed": lambda: L.ch_adjoint_step_timed(g.h, st, ms),
        "adjoint_segment": lambda: L.ch_adjoint_segment(g.h, st, 1),
        "adjoint_end": lambda: L.ch_adjoint_end(g.h),
    }
    for name, call in reverse.items():
        g.set_state(state)
        g.adjoint_begin()
        set_flag(alloc)
        assert call() == TIMEOUT, name
        with pytest.raises(binding.ChError):
            g.device_status()
        g.adjoint_end()
    g.close()


def test_objective_and_gradient_raise(binding):
    alloc = binding.TorchAllocator(torch.device("cuda:0"))
    g = binding.Grid(**SIZE, allocator=alloc)
    ts = [t.cuda().requires_grad_(True) for t in initial(2)]
    J = binding.objective_after(g, *ts, 2)
    set_flag(alloc)
    with pytest.raises(binding.ChError) as e:
        J.backward()
    assert e.value.code == TIMEOUT
    with pytest.raises(binding.ChError):
        binding.objective_after(g, *ts, 2)
    with pytest.raises(binding.ChError):
        g.device_status()
    binding.objective_after(g, *ts, 2).backward()   # usable again
    assert all(bool(torch.isfinite(t.grad).all()) for t in ts)
    g.close()


def test_ensemble_calls_report_any_member(binding):
    ens = binding.Ensemble([SIZE, SIZE])
    for i, g in enumerate(ens.grids):
        g.set_fields(*initial(3 + i))
    ens.step_timed(1)
    flag = [t for t in ens._alloc.live.values() if t.numel() == 4][-1]
    flag.copy_(torch.tensor([1, 0, 0, 0], dtype=torch.uint8))
    for call in (lambda: ens.step_timed(1), lambda: ens.autotune(1)):
        with pytest.raises(binding.ChError) as e:
            call()
        assert e.value.code == TIMEOUT
    ens.grids[0].device_status()
    with pytest.raises(binding.ChError):
        ens.grids[1].device_status()
    ens.autotune(1)
    ens.close()
