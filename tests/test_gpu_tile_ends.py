"""Tensor-core transforms at the ends: of a tile, of a CTA.

The last tile may end inside a warp: some lanes of an epilogue warp have a row and others have none, and
all of them go on to the next tensor-memory load together.

Chebyshev lines: 64 lines a tile, 16 a warp.  Fields of 8, 36, 72 and 162 lines leave 8, 4, 8 and 2 lines
in the last warp, for one, two and three output slices (nz = 5 to 17, 193, 385; four columns at a time, so
every slice of more than four has later loads after the first stores).  Bound: that of the transform
everywhere, 1e-15 max|x| max_n sum_k |B_nk| per line (tests/test_gpu_chebyshev_tc.py)."""
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


def matrices(N):
    ld = np.longdouble
    n = np.arange(N + 1)
    B = np.cos(((n[:, None] * n[None, :]) % (2 * N)).astype(ld) * (np.arccos(ld(-1)) / ld(N)))
    cb = np.ones(N + 1, dtype=ld)
    cb[0] = cb[N] = 2
    return 2 / (cb[:, None] * N) * B / cb[None, :], B


@pytest.mark.parametrize("nx,ny", [(4, 4), (12, 6), (18, 8), (54, 6)])
@pytest.mark.parametrize("nz", [5, 9, 17, 193, 385])
def test_lines_of_a_ragged_last_warp(binding, nx, ny, nz):
    rng = np.random.Generator(np.random.PCG64(nx * 1000 + nz))
    shape = (2 if nz <= 17 else 1, nx // 2, ny, nz)
    x = rng.standard_normal(shape) + 1j * rng.standard_normal(shape)
    g = binding.Grid(nx, ny, nz)
    g.set_chebyshev(binding.CHEB_TC)
    flat = x.reshape(-1, nz)
    for direction, M in enumerate(matrices(nz - 1)):
        got = g.chebyshev_lines(torch.from_numpy(x).cuda(), direction).cpu().numpy().reshape(-1, nz)
        g.device_status()
        rowsum = float(np.max(np.sum(np.abs(M), axis=1)))
        for part in (np.real, np.imag):
            xr = part(flat).astype(np.longdouble)
            err = np.abs(part(got).astype(np.longdouble) - xr @ M.T)
            assert np.all(err <= 1e-15 * rowsum * np.max(np.abs(xr), axis=1)[:, None])
    g.close()


@pytest.mark.parametrize("nz", [17, 385])
def test_back_to_back_launches_leave_nothing_in_flight(binding, nz):
    """A CTA ends after its last copies and MMAs, whichever warp finishes first: 200 transforms in a row
    without a wait between them (each CTA's tensor memory and shared memory go straight to the next
    launch) give the first one's bits, and no wait runs out."""
    nx, ny = 18, 8
    g = binding.Grid(nx, ny, nz)
    g.set_chebyshev(binding.CHEB_TC)
    rng = np.random.Generator(np.random.PCG64(nz))
    x = torch.from_numpy(rng.standard_normal((5, nx // 2, ny, nz, 2))).cuda()
    x = torch.view_as_complex(x)
    first = [g.chebyshev_lines(x, d) for d in (0, 1)]
    for _ in range(100):
        last = [g.chebyshev_lines(x, d) for d in (0, 1)]
    g.device_status()
    for a, b in zip(first, last):
        assert torch.equal(a, b)
    g.close()


@pytest.mark.parametrize("nz", [17, 129, 385])
def test_last_output_is_rounded_once(binding, nz):
    """The output n = N, an alternating sum formed apart from the products, of rows whose terms cancel to a
    thousandth: off by the rounding of the row's elements to 2^-63 of the power of two above the
    largest (at most 2.11 of it) and by the roundings of the result, not of the row's scale."""
    N = nz - 1
    rng = np.random.Generator(np.random.PCG64(nz))
    nx, ny = 12, 6
    x = rng.standard_normal((1, nx // 2, ny, nz)) + 1j * rng.standard_normal((1, nx // 2, ny, nz))
    x[..., 1::2] = x[..., 0:-1:2] * (1.0 + 1e-3 * rng.random((1, nx // 2, ny, N // 2)))
    x[..., N] *= 1e-3
    g = binding.Grid(nx, ny, nz)
    g.set_chebyshev(binding.CHEB_TC)
    F, B = matrices(N)
    flat = x.reshape(-1, nz)
    for direction, row in enumerate((F[N], B[N])):
        got = g.chebyshev_lines(torch.from_numpy(x).cuda(), direction).cpu().numpy().reshape(-1, nz)[:, N]
        for part in (np.real, np.imag):
            xr = part(flat).astype(np.longdouble)
            ref = xr @ row
            bound = (2.0 ** -52 * np.abs(ref) + 1e-30
                     + 2.0 ** -63 * 2.11 * np.max(np.abs(xr), axis=1) * float(np.sum(np.abs(row))))
            assert np.all(np.abs(part(got).astype(np.longdouble) - ref) <= bound), direction
    g.close()
