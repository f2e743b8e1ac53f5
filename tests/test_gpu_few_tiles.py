"""Tensor-core x and y transforms of few tiles: several CTAs share a tile's output slices, so that long
transforms of few lines do not leave the chip idle.  Every output is the same sum whoever forms it.

Sizes: (384, 24, 17): x backward 35 tiles, four CTAs for five slices; (512, 24, 9): 21 tiles, a CTA for
each of six slices, and 27 x forward tiles with four; (32, 384, 33): y backward 54 tiles, two CTAs for five
slices; (16, 512, 33): y forward 45 tiles, three CTAs for four slices, and y backward by FFT;
(8, 512, 17): both y passes by FFT, the x line on the tensor cores.  Bound against the oracle: 1e-12 of each
field's largest value, that of the products everywhere (tests/test_gpu_txy.py)."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.channel import Channel, Params  # noqa: E402
from paper_2406_01322_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_01322_gb300 import build
    build.build_library()
    from paper_2406_01322_gb300 import binding as b
    b.lib()
    return b


def initial(n, seed=1):
    return [np.ascontiguousarray(a) for a in inputs.initial_fields(*n, 150.0, 0.05, 1, 0.4, seed)]


@pytest.mark.parametrize("n,launches", [((384, 24, 17), 9), ((512, 24, 9), 9), ((32, 384, 33), 9),
                                        ((16, 512, 33), 9), ((8, 512, 17), 8)])
def test_products_match_oracle(binding, n, launches):
    kw = dict(re_tau=150.0, we=1.0, ch=0.05, pe=20.0, dt=1e-4)
    f = initial(n)
    o = Channel(Params(nx=n[0], ny=n[1], nz=n[2], **kw))
    o.set_fields(*f)
    g = binding.Grid(*n, **kw)
    g.set_fields(*[torch.from_numpy(a) for a in f])
    assert g.launches_per_step() == launches   # the forward y pass by FFT is one launch fewer
    r = o.nonlinear_spectral()
    ref = [r[0] - r[2], r[1] - r[2], r[3], r[4], r[5], r[6], r[7], r[8], r[9]]
    for k, a in enumerate(g.nonlinear()):
        d = np.abs(a.cpu().numpy().transpose(2, 1, 0) - ref[k])
        assert np.max(d) < 1e-12 * np.max(np.abs(ref[k])), k
    g.device_status()
    g.close()


@pytest.mark.parametrize("n", [(64, 256, 65), (24, 768, 65), (256, 256, 17)],
                         ids=lambda n: "x".join(map(str, n)))
def test_one_field_equals_the_same_field_among_four(binding, n):
    """phi alone (one field's tiles, more CTAs a tile) and in get_fields (four fields' tiles)."""
    g = binding.Grid(*n)
    g.set_fields(*[torch.from_numpy(a) for a in initial(n, 2)])
    g.step(1)
    phi = g.get_fields()[3]
    assert torch.equal(g.transform_backward(g.get_spectral()[2]), phi)
    g.close()


@pytest.mark.parametrize("n", [(512, 6, 33), (72, 72, 49), (256, 16, 17), (8, 648, 17), (96, 96, 65),
                               (24, 1024, 33)],
                         ids=lambda n: "x".join(map(str, n)))
def test_routes_of_one_and_four_fields_agree(binding, n):
    """A field that the grid holds exactly (three x, three y and five z modes): set_fields and get_fields (one
    by FFT, the other on the tensor cores for the first and third size), and the transforms of one field
    (forward by FFT and backward on the tensor cores for the second, both by FFT for the fourth, both on the
    tensor cores for the last two, in four K groups at 1024 points) give it back.  Bound: 1e-12 of the largest value, as above."""
    nx, ny, nz = n
    x = np.arange(nx) * (2 * np.pi / nx)
    y = (np.arange(ny) * (2 * np.pi / ny))[:, None]
    z = np.cos(np.pi * np.arange(nz) / (nz - 1))[:, None, None]
    phi = np.cos(x) * np.sin(2 * y) * (1 - z ** 4) + 0.3 * np.cos(2 * x + y) * z ** 3 + 0.1 * z ** 2
    phi = torch.from_numpy(np.array(np.broadcast_to(phi, (nz, ny, nx)))).cuda()
    zero = torch.zeros_like(phi)
    g = binding.Grid(*n)
    g.set_fields(zero, zero, zero, phi)
    scale = float(phi.abs().max())
    assert float((g.get_fields()[3] - phi).abs().max()) < 1e-12 * scale
    spec = g.transform_forward(phi)
    assert float((spec - g.get_spectral()[2]).abs().max()) < 1e-12 * scale
    assert float((g.transform_backward(spec) - phi).abs().max()) < 1e-12 * scale
    g.device_status()
    g.close()
