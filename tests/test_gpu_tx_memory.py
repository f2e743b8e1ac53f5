"""Scratch of the float64 x/y transforms on the tensor cores: the step's padded physical fields lie in
buffers that the calls between steps use too, so those calls must leave a trajectory bit for bit as it
is, and a grid holds no padded physical field of its own."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2406_01322_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

# 2^15 modes and more, float64 throughout; the second with odd padded lengths (81, 243), the third from
# 2^18 modes on (Chebyshev coefficients in the same buffers)
SIZES = [(64, 64, 17), (54, 162, 17), (64, 64, 129)]


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_01322_gb300 import build
    build.build_library()
    from paper_2406_01322_gb300 import binding as b
    b.lib()
    return b


def initial(n, seed):
    f = inputs.initial_fields(*n, 150.0, 0.05, 1, 0.4, seed)
    return [torch.from_numpy(np.ascontiguousarray(a)) for a in f]


@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
def test_calls_between_steps_leave_the_trajectory(binding, n):
    out = []
    for busy in (False, True):
        g = binding.Grid(*n)
        g.set_fields(*initial(n, 5))
        for _ in range(4):
            g.step(1)
            if busy:
                f = g.get_fields()
                g.diagnostics()
                g.transform_backward(g.transform_forward(f[0]))
                g.objective()
                g.nonlinear()
                g.get_fields_host()
        out.append(g.get_state())
        g.close()
    assert torch.equal(*out)


@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
def test_nine_padded_fields_only_during_a_sweep(binding, n):
    nine = 9 * (3 * n[0] // 2) * (3 * n[1] // 2) * n[2] * 8
    alloc = binding.TorchAllocator(torch.device("cuda:0"))

    def held():
        return sorted(t.numel() for t in alloc.live.values())

    g = binding.Grid(*n, allocator=alloc)
    g.set_fields(*initial(n, 6))
    g.step(1)
    before = held()
    assert nine not in before
    g.adjoint_begin()
    assert nine in held()
    g.adjoint_end()
    # the sweep's own plans (digits) stay with the grid, the fields do not
    assert nine not in held()
    g.adjoint_begin()
    g.adjoint_end()
    assert nine not in held() and len(held()) == len(before) + 2
    g.close()
    assert not alloc.live
