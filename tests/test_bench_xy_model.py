"""bench.py's count of the tensor-core flops of the float64 x and y stages (no GPU), against an enumeration of
the kernel's MMAs."""
import bench


def mma_flops(lines, rows, nf, nk, nout):
    """Per field and tile, per slice of at most 64 output columns (widths rounded up to 16, equal), cosine
    and sine, per 16 inputs: digit planes i < 8 against 7 matrix planes, diagonals i + j < 8, 128 rows."""
    nsl = (nout + 63) // 64
    width = (nout + nsl - 1) // nsl
    width = (width + 15) // 16 * 16
    total = 0
    for _ in range(nf):
        for _ in range(0, lines, rows):
            for _ in range(nsl):
                for _ in ("cos", "sin"):
                    for _ in range(0, nk, 16):
                        products = sum(1 for i in range(8) for j in range(7) if i + j < 8)
                        total += products * 2 * 128 * width * 16
    return total


def test_xy_flops_match_an_enumeration_of_the_mmas():
    for nx, ny, nz in ((128, 128, 129), (54, 162, 33), (512, 16, 9)):
        w = dict(nx=nx, ny=ny, nz=nz)
        Mx, Px, Py = nx // 2, 3 * nx // 2, 3 * ny // 2
        hx, hy, Q = (Px + 1) // 2, (Py + 1) // 2, Py * nz
        xb = mma_flops(Q, 128, 1, Mx, hx)
        xf = mma_flops(Q, 128, 1, hx, Mx)
        yb = mma_flops(Mx * nz, 64, 1, ny // 2, hy)
        yf = mma_flops(Mx * nz, 64, 1, hy, ny // 2)
        ref = {"ybwd": 6 * yb, "xline": 7 * xb + 9 * xf, "yfwd": 9 * yf, "adj_ybwd": 9 * yb,
               "adj_xline": 16 * xb + 7 * xf, "adj_yfwd": 6 * yf}
        for k, v in ref.items():
            assert bench.xy_issued_flops(w, k) == v
    assert bench.xy_issued_flops(w, "zsolve") is None
