"""What runs when the memory for the tensor-core transforms is not to be had: the FFT kernels, with the same
results, and everything given back.

An allocator that refuses one request (the k-th of ch_init_grid) stands in for a full device.  64 x 64 x 129
(2^18 modes) asks last, in order, for: the Chebyshev matrices and scratch (digits, scratch, flag, digits), the
digits of four unpadded and four padded x/y plans, and their scratch.  Refused the first four, a grid
has no tensor-core transforms at all; refused one of the nine others, none in x and y (and no Chebyshev
ones unless selected).  Bounds: the float64 bar of the step, 1e-10, fields and gradients (2 (128 / 32)^2 1e-10 for
gradients, as in tests/test_gpu_z_method.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from paper_2406_01322_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

N = (64, 64, 129)
PHYS = dict(re_tau=150.0, we=1.0, ch=0.05, pe=20.0, dt=1e-4)


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_01322_gb300 import build
    build.build_library()
    from paper_2406_01322_gb300 import binding as b
    b.lib()
    return b


def allocator(binding, refuse=()):
    class Refusing(binding.TorchAllocator):
        n, sizes = 0, []

        def _alloc(self, nbytes, ctx):
            self.n += 1
            self.sizes = self.sizes + [int(nbytes)]
            return None if self.n in refuse else super()._alloc(nbytes, ctx)
    return Refusing(torch.device("cuda:0"))


def grid(binding, alloc, **kw):
    return binding.Grid(*N, allocator=alloc, **PHYS, **kw)


def fields(seed=4):
    return [torch.from_numpy(np.ascontiguousarray(a))
            for a in inputs.initial_fields(*N, 150.0, 0.05, 1, 0.4, seed)]


def rel(a, b):
    return float((a - b).abs().max() / b.abs().max())


def run(g):
    g.set_fields(*fields())
    state = g.get_state()
    g.step(3)
    out = g.get_fields()
    g.diagnostics()
    g.set_state(state)
    g.step(1)
    g.adjoint_begin()
    g.adjoint_step(state)
    grads = g.adjoint_gradient()
    g.adjoint_end()
    g.device_status()
    return out, grads


def test_each_refusal_leaves_the_fft_kernels(binding):
    full = allocator(binding)
    g = grid(binding, full)
    assert g.launches_per_step() == 11
    total = full.n
    ref, gref = run(g)
    g.close()
    assert not full.live
    for back in range(13):   # the last thirteen requests, newest first
        a = allocator(binding, refuse=(total - back,))
        g = grid(binding, a)
        # nothing is kept of what was asked for together with the refused piece: the flag and tables of the
        # Chebyshev transforms (four pieces) stay when an x/y piece was refused
        assert g.launches_per_step() == 6
        assert len(a.live) == total - 13 + (4 if back < 9 else 0)
        out, grads = run(g)
        for x, y in zip(out, ref):
            assert rel(x, y) <= 1e-10
        for x, y in zip(grads, gref):
            assert rel(x, y) <= 3.2e-9
        if back in (0, 12):   # the method can still be selected
            g.set_chebyshev(binding.CHEB_TC)
            assert g.launches_per_step() == 8
            g.set_fields(*fields())
            g.step(3)
            for x, y in zip(g.get_fields(), ref):
                assert rel(x, y) <= 1e-10
        g.close()
        assert not a.live


@pytest.mark.parametrize("refused", ["plan", "plans", "fields"])
def test_reverse_sweep_without_room(binding, refused):
    """ch_adjoint_begin asks for two plans' digits, the workspace and nine padded fields; without a plan or
    the fields the FFT kernels run, and the gradient is the same to rounding."""
    full = allocator(binding)
    g = grid(binding, full)
    _, gref = run(g)
    first = full.n   # requests up to the end of the first sweep
    g.close()
    probe = allocator(binding)
    g = grid(binding, probe)
    init = probe.n
    g.close()
    assert first == init + 4
    which = {"plan": (init + 1,), "plans": (init + 1, init + 2), "fields": (init + 4,)}[refused]
    a = allocator(binding, refuse=which)
    g = grid(binding, a)
    _, grads = run(g)
    for x, y in zip(grads, gref):
        assert rel(x, y) <= 3.2e-9
    g.close()
    assert not a.live


@pytest.mark.parametrize("precision", [0, 2])
def test_lengths_beyond_the_tensor_core_transforms(binding, precision):
    """ny = 768: the padded length 1152 is beyond them (the unpadded one is not), so the step's x and y
    stages run by FFT at 2^16 modes; pruned schedules apply there and agree to the float64 bar, and
    the fields come back through the tensor-core transforms of the unpadded grid."""
    n = (12, 768, 17)
    f = [torch.from_numpy(np.ascontiguousarray(a)) for a in inputs.initial_fields(*n, 150.0, 0.05, 1, 0.4, 5)]
    out = []
    for prune in (0, 1):
        g = binding.Grid(*n, precision=precision, **PHYS)
        assert g.launches_per_step() == 6
        g.set_fft_pruning(prune)
        g.set_fields(*f)
        g.step(5)
        g.device_status()
        out.append(g.get_fields())
        g.close()
    for a, b in zip(*out):
        assert rel(a, b) <= 1e-10
