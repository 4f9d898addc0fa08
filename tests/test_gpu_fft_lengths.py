"""Four-step against Stockham at every padded length a grid can have, on each axis.

A padded length is the smallest 2,3,5-smooth integer >= 2 n - 1 for the grid
extent n of that axis.  A strip two cells wide, meshed at lambda / 9, is laid
along x, y or z and cut so that its long axis has the wanted length, at the
smallest or the largest extent n with that length (odd and even lengths,
ragged numbers of grids).  Each of the two kernel families is within 1e-12
(complex128 vectors) and 1e-5 (complex64) of the FP64 oracle, relative L2, by
the product's own bounds, so they are within twice that of one another.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from aim_inputs import random_complex, rect_plate_mesh  # noqa: E402
from oracle import aim as oaim  # noqa: E402

import paper_1010_1456_gb300 as g  # noqa: E402

K0 = 2 * np.pi
H = 0.1


def reachable(top):
    """Padded lengths up to `top`: the smallest smooth L >= 2 n - 1 for some n."""
    return sorted({oaim.smooth_length(2 * n - 1) for n in range(4, top) if oaim.smooth_length(2 * n - 1) <= top})


def strip(L, along, wide):
    """A strip along axis `along` (0: x, 1: y, 2: z) whose padded length there is L, or None."""
    ns = [n for n in range(4, (L + 1) // 2 + 1) if oaim.smooth_length(2 * n - 1) == L]
    want = ns[-1] if wide else ns[0]
    for shift in (0.0, 0.05):  # centred on a node: odd extents; between two: even ones
        for side in np.arange(max(0.1, 0.1 * want - 0.6), 0.1 * want + 0.2, 0.01):
            cells = max(1, int(round(9 * side)))
            # the outermost basis functions sit at cell centres (diagonals) and edges inside the strip
            c = np.concatenate([(np.arange(cells) + 0.5), np.arange(1, cells)]) * (side / cells) - 0.5 * side + shift
            a = np.floor(c / H - 0.5)
            if a.max() - a.min() + 3 == want:
                v0, t = rect_plate_mesh(side, 0.2, cells, 2)
                v = np.empty_like(v0)
                long_, short, flat = {0: (0, 1, 2), 1: (1, 0, 2), 2: (2, 0, 1)}[along]
                v[:, long_], v[:, short], v[:, flat] = v0[:, 0] + shift, v0[:, 1], 0.013
                return v, t
    return None


@pytest.mark.parametrize("along", [0, 1, 2])
@pytest.mark.parametrize("L", reachable(900))
def test_four_step_equals_stockham(L, along):
    found = strip(L, along, wide=L % 2 == 0)
    assert found is not None
    nrhs = 1 + L % 3
    ctx = g.aim_setup(*found, K0, H, M=2, max_rhs=nrhs)
    assert g.aim_grid_info(ctx)[1][along] == L
    x = torch.from_numpy(random_complex((nrhs, ctx.N), L)).cuda()
    for prec, bound in ((g.AIM_C128, 2e-12), (g.AIM_C128_F64, 2e-12), (g.AIM_C64, 2e-5)):
        xp = x.to(torch.complex64) if prec == g.AIM_C64 else x
        y = g.aim_matvec(ctx, xp, precision=prec)
        g.aim_fft_config(ctx, prec, [g.AIM_FFT_STOCKHAM] * 5)
        ref = g.aim_matvec(ctx, xp, precision=prec)
        assert float(torch.linalg.norm(y - ref) / torch.linalg.norm(ref)) <= bound, prec
    ctx.close()
