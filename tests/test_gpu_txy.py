"""Float64 y and x transforms of the step on the tensor cores (grids from 2^15 modes on) at the
sizes where their tiles, slices and K groups can go wrong, against the oracle: the nine non-linear
fields (backward y and x, products, forward x and y).  The bound is that of the float64 path
everywhere else (1e-12 of each field's maximum): a row's quantisation is 2^-54 of its largest
element, far below it."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

from oracle.channel import Channel, Params  # noqa: E402
from paper_2406_01322_gb300 import inputs  # noqa: E402

pytestmark = pytest.mark.gpu

# (nx, ny, nz): whole and ragged tiles of 64 and 128 lines, odd padded lengths (81, 243: no middle
# sample), one and several output slices (16 to 64 columns), one to three K groups (Px = 768: three)
SIZES = [(64, 64, 17), (54, 162, 33), (216, 24, 17), (24, 216, 17), (512, 16, 9), (128, 128, 5)]


@pytest.fixture(scope="module")
def binding():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2406_01322_gb300 import build
    build.build_library()
    from paper_2406_01322_gb300 import binding as b
    b.lib()
    return b


def rel(a, b):
    return float(np.max(np.abs(a - b)) / max(np.max(np.abs(b)), 1e-300))


def to_oracle(t):
    return t.cpu().numpy().transpose(2, 1, 0)


@pytest.mark.parametrize("nx,ny,nz", SIZES)
def test_products_match_oracle(binding, nx, ny, nz):
    w = dict(inputs.WORKLOADS["channel_128x128x129"], nx=nx, ny=ny, nz=nz, ch=0.05, pe=20.0)
    fields = inputs.initial_fields(**w)
    kw = dict(re_tau=w["re_tau"], we=w["we"], ch=w["ch"], pe=w["pe"], dt=w["dt"])
    o = Channel(Params(nx=nx, ny=ny, nz=nz, **kw))
    o.set_fields(*fields)
    g = binding.Grid(nx, ny, nz, **kw)
    g.set_fields(*[torch.from_numpy(f) for f in fields])
    # the x line is three launches on this path and the forward y pass two
    assert g.launches_per_step() == 9
    r = o.nonlinear_spectral()
    ref = [r[0] - r[2], r[1] - r[2], r[3], r[4], r[5], r[6], r[7], r[8], r[9]]
    for k, a in enumerate(g.nonlinear()):
        assert rel(to_oracle(a), ref[k]) < 1e-12, k
    g.device_status()


def test_small_grids_keep_the_fft_kernels(binding):
    assert binding.Grid(32, 32, 33).launches_per_step() == 6


def test_nan_reaches_the_diagnostics(binding):
    nx, ny, nz = 64, 64, 17
    w = dict(inputs.WORKLOADS["channel_128x128x129"], nx=nx, ny=ny, nz=nz)
    f = [torch.from_numpy(x.copy()) for x in inputs.initial_fields(**w)]
    f[0][3, 5, 7] = float("nan")
    g = binding.Grid(nx, ny, nz)
    g.set_fields(*f)
    g.step(2)
    assert g.diagnostics()["nan"] == 1
