"""Memory that is counted before it is used (CPU only): aim_footprint's padding."""

import pytest

from aim_inputs import rect_plate_mesh

@pytest.fixture(scope="module")
def lib():
    from paper_1010_1456_gb300 import build

    build.build()


def test_footprint_counts_padded_rows_and_right_hand_sides(lib):
    """A 6.25 x 0.5 x 0 plate: rows of 66 nodes are held as 68; an odd number of
    right-hand sides from 17 on is held as the next even one in the RHS-minor copies."""
    import paper_1010_1456_gb300 as g

    v, t = rect_plate_mesh(6.25, 0.5, 56, 4)

    def fp(nrhs):
        return g.aim_footprint(v, t, 0.1, 2, 0.3, nrhs, precision=g.AIM_C64)

    n, L, px = (66, 8, 3), (135, 15, 5), 68
    N = int(1.5 * len(t))
    nc = n[0] * n[1] * n[2]
    grids = 4 * 24 * (nc + px * L[2] * (n[1] + L[1]))  # complex64 and float-float grids of a right-hand side
    solver = N * (16 * 53 + 48)
    assert fp(2) - fp(1) == grids + solver
    assert fp(18) - fp(17) == grids + solver  # 18 columns either way
    assert fp(19) - fp(18) == grids + solver + 2 * 16 * (4 * nc + N)
