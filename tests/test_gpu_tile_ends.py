"""Tensor-core transforms at the ends: of a tile, of a CTA.

The last tile may end inside a warp: some lanes of an epilogue warp have a row and others have none, and
all of them go on to the next tensor-memory load together.

Chebyshev lines: 64 lines a tile, 16 a warp.  Fields of 8, 36, 72 and 162 lines leave 8, 4, 8 and 2 lines
in the last warp, for one, two and three output slices (nz = 17, 193, 385; four columns at a time, so
every slice has later loads after the first stores).  Bound: that of the transform
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
@pytest.mark.parametrize("nz", [17, 193, 385])
def test_lines_of_a_ragged_last_warp(binding, nx, ny, nz):
    rng = np.random.Generator(np.random.PCG64(nx * 1000 + nz))
    shape = (2 if nz == 17 else 1, nx // 2, ny, nz)
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
