"""Weights of the tensor-core y transforms at long lengths: as many fractional bits as the recombined sums
leave room for.

One mode pair, c_k = c_{-k} = 0.45 on the line kx = 0, n = 0, so that the samples are 0.9 cos(2 pi k j / Ny).  z
carries 0.45 over exactly; x does so for values whose mantissa is at most 0.95 of a power of two (one
term of weight 1, 2^53 steps a unit), and only those are compared.  What is left is the y transform: its weight's
rounding, 0.9 2^-(q+1), its recombined sum's, 2^-(q+2) (the row's scale is 2^-1), and the result's, 2^-54.  The
scale q that the sums allow (2^-62 of 2 0.976 2^62 (sum |cos| + sum |sin|) 2^q below 2^63, at most 54; the sums
are at most 1.28 Ny / 2) is 54 for 288 points, 53 for 512 and 52 for 1024."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

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


@pytest.mark.parametrize("n,q", [((96, 288, 65), 54), ((64, 512, 17), 53), ((24, 1024, 33), 52)],
                         ids=["288", "512", "1024"])
def test_single_modes_have_the_weights_rounding(binding, n, q):
    nx, ny, nz = n
    g = binding.Grid(*n)
    ld = np.longdouble
    pi = np.arccos(ld(-1))
    for k in (1, 5, 37, ny // 2 - 1):
        spec = torch.zeros((nx // 2, ny, nz), dtype=torch.complex128, device="cuda")
        spec[0, k, 0] = spec[0, ny - k, 0] = 0.45
        got = g.transform_backward(spec)[0, :, 0].cpu().numpy()
        ref = 2 * ld(0.45) * np.cos((k * np.arange(ny) % ny).astype(ld) * (2 * pi / ld(ny)))
        exact = np.abs(np.frexp(got)[0]) <= 0.95
        err = float(np.max(np.abs(got.astype(ld) - ref)[exact]))
        assert err <= 0.9 * 2.0 ** -(q + 1) + 2.0 ** -(q + 2) + 2.0 ** -54 + 1e-18, (k, err)
    g.device_status()
    g.close()
