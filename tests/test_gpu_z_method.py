"""Chebyshev transforms of grids whose method was not selected: on the tensor cores from 2^18 modes
on, with either explicit choice still honoured, in single steps, reverse steps and ensembles.

Bounds.  Fields: the float64 bar of the step, 1e-10.  Gradients: the bar against the oracle is 1e-10
at N = 32; rounding in the highest coefficients grows with N^2, and two such results are compared:
2 (128 / 32)^2 1e-10 = 3.2e-9."""
import pytest

torch = pytest.importorskip("torch")

from paper_2406_01322_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

PHYS = dict(re_tau=150.0, we=1.0, ch=0.05, pe=20.0, dt=1e-4)
BIG, SMALL = dict(nx=64, ny=64, nz=129), dict(nx=64, ny=64, nz=65)   # 264192 and 133120 modes


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_01322_gb300 import build
    build.build_library()
    from paper_2406_01322_gb300 import binding as b
    b.lib()
    return b


def fields(m, seed):
    f = inputs.initial_fields(m["nx"], m["ny"], m["nz"], PHYS["re_tau"], PHYS["ch"], 1, 0.4, seed)
    return [torch.from_numpy(a) for a in f]


def rel(a, b):
    return float((a - b).abs().max() / b.abs().max())


@pytest.mark.parametrize("precision,small,big", [(0, 9, 11), (2, 6, 8)])
def test_large_grids_use_the_tensor_cores_until_a_method_is_selected(binding, precision, small, big):
    g, f = (binding.Grid(precision=precision, **BIG, **PHYS) for _ in range(2))
    f.set_chebyshev(binding.CHEB_FFT)
    assert g.launches_per_step() == big and g.chebyshev() == binding.CHEB_FFT
    assert f.launches_per_step() == small
    assert binding.Grid(precision=precision, **SMALL, **PHYS).launches_per_step() == small
    for x in (g, f):
        x.set_fields(*fields(BIG, 7))
        x.step(3)
        x.device_status()
    for a, b in zip(g.get_fields(), f.get_fields()):
        assert rel(a, b) <= 1e-10


def test_reverse_step_agrees_with_the_fft_transforms(binding):
    grads = []
    for method in (None, binding.CHEB_FFT):
        g = binding.Grid(**BIG, **PHYS)
        if method is not None:
            g.set_chebyshev(method)
        g.set_fields(*fields(BIG, 8))
        state = g.get_state()
        g.step(1)
        g.adjoint_begin()
        g.adjoint_step(state)
        grads.append([t.clone() for t in g.adjoint_gradient()])
        g.adjoint_end()
        g.device_status()
    for a, b in zip(*grads):
        assert rel(a, b) <= 3.2e-9


@pytest.mark.parametrize("precision", [0, 1])
def test_ensemble_members_keep_their_own_method(binding, precision):
    """Members of both kinds in one ensemble (two work lists for zrhs and zbwd) evolve bit for bit as
    in ensembles of their own."""
    ms = [dict(SMALL, **PHYS), dict(BIG, **PHYS), dict(nx=32, ny=32, nz=33, **PHYS)]
    ens = binding.Ensemble(ms, precision=precision)
    own = [binding.Ensemble([m], precision=precision) for m in ms]
    for i, (g, e, m) in enumerate(zip(ens.grids, own, ms)):
        for x in (g, e.grids[0]):
            x.set_fields(*fields(m, 20 + i))
        e.step(3)
    ens.step(3)
    for g, e in zip(ens.grids, own):
        for a, b in zip(g.get_fields(), e.grids[0].get_fields()):
            assert torch.equal(a, b)
        e.close()
    ens.close()
