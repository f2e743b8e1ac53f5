"""Reverse steps whose x and y transforms run on the tensor cores (grids from 2^15 modes on) against the
oracle's reverse-mode gradient, and the two ways to reverse a segment against each other bit for bit.

Sizes: whole tiles (64 x 64 x 17); odd padded lengths (54 x 162 x 17: 81 and 243, no middle sample, ragged
tiles); several K groups and shared output slices in the transposed x transforms (384 x 24 x 17: 576 points);
y passes by FFT beside them (8 x 512 x 17).  Tolerances: those of tests/test_gpu_adjoint.py, J to 1e-12,
gradients to 1e-10 of each field's largest oracle value."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle import adjoint  # noqa: E402
from oracle.channel import Params  # noqa: E402
from paper_2406_01322_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

PHYS = dict(re_tau=50.0, ch=0.15, pe=10.0, we=1.0, dt=2e-3)
SIZES = [(64, 64, 17), (54, 162, 17), (384, 24, 17), (8, 512, 17)]
STEPS = 2


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_01322_gb300 import build
    build.build_library()
    from paper_2406_01322_gb300 import binding as b
    b.lib()
    return b


def fields(n, seed=3):
    return [np.ascontiguousarray(a)
            for a in inputs.initial_fields(*n, PHYS["re_tau"], PHYS["ch"], 1, 0.6, seed, amp=0.5)]


@pytest.mark.parametrize("n", SIZES, ids=lambda n: "x".join(map(str, n)))
def test_gradient_matches_oracle_adjoint(binding, n):
    f = fields(n)
    g = binding.Grid(*n, **PHYS)
    assert g.launches_per_step() > 6
    ts = [torch.from_numpy(a).cuda().requires_grad_(True) for a in f]
    J = binding.objective_after(g, *ts, STEPS, checkpoint_every=2)
    J.backward()
    g.device_status()
    Jr, gr = adjoint.gradient(Params(nx=n[0], ny=n[1], nz=n[2], **PHYS), f, STEPS)
    assert abs(float(J.detach()) - Jr) <= 1e-12 * abs(Jr)
    for name, t, b in zip("uvwp", ts, gr):
        err = np.max(np.abs(t.grad.cpu().numpy() - b))
        assert err <= 1e-10 * np.max(np.abs(b)), (name, err)
    g.close()


@pytest.mark.parametrize("n", SIZES[1:2], ids=lambda n: "x".join(map(str, n)))
def test_segments_and_checkpoints_are_bitwise_neutral(binding, n):
    f = fields(n, seed=9)
    grads = []
    for mode in ("segment", "steps"):
        g = binding.Grid(*n, **PHYS)
        g.set_fields(*[torch.from_numpy(a) for a in f])
        states = []
        for _ in range(4):
            states.append(g.get_state())
            g.step(1)
        g.adjoint_begin()
        if mode == "segment":
            g.adjoint_segment(states[2], 2)
            g.adjoint_segment(states[0], 2)
        else:
            for st in reversed(states):
                g.adjoint_step(st)
        grads.append(g.adjoint_gradient())
        g.adjoint_end()
        g.close()
    for every in (1, 3):
        g = binding.Grid(*n, **PHYS)
        ts = [torch.from_numpy(a).cuda().requires_grad_(True) for a in f]
        binding.objective_after(g, *ts, 4, checkpoint_every=every).backward()
        grads.append([t.grad for t in ts])
        g.close()
    for other in grads[1:]:
        for a, b in zip(grads[0], other):
            assert torch.equal(a, b)
