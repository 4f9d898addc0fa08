"""Bodies large enough for the half-warp layouts of the many-RHS kernels.

From 4,864 unknowns (eight row groups of four for each of 152 SMs) 16 to 32
right-hand sides share half a warp: one a lane for 16 (and, with a memory
budget, for odd counts), two a lane in rows padded to an even length for 17
to 32.  The interpolation then stages 64 rows a block, so the bodies' numbers of
unknowns (5,985 and 5,070) leave a ragged last block.  Compared eight right-hand
sides at a time: both paths are within 1e-12 (complex128 vectors) and 1e-5
(complex64) of the FP64 oracle by the product's own bounds, relative L2.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from aim_inputs import icosphere_mesh, plate_mesh, random_complex  # noqa: E402

import paper_1010_1456_gb300 as g  # noqa: E402

K0 = 2 * np.pi
H = 0.1


@pytest.mark.parametrize("budget", [0, 16 << 30])
@pytest.mark.parametrize("nrhs", [16, 17, 31, 32, 33])
@pytest.mark.parametrize("body", ["plate", "cfie_sphere"])
def test_half_warp_layouts_equal_eight_at_a_time(body, nrhs, budget):
    mesh, alpha = (plate_mesh(5.0, 45), 1.0) if body == "plate" else (icosphere_mesh(1.2, 13), 0.6)
    ctx = g.aim_setup(*mesh, K0, H, M=2, max_rhs=nrhs, cfie_alpha=alpha, mem_budget=budget)
    assert ctx.N >= 152 * 8 * 4 and ctx.N % 64
    x = torch.from_numpy(random_complex((nrhs, ctx.N), nrhs)).cuda()
    for prec, bound in ((g.AIM_C64, 2e-5), (g.AIM_C128_F64, 2e-12)):
        xp = x.to(torch.complex64) if prec == g.AIM_C64 else x
        y = g.aim_matvec(ctx, xp, precision=prec)
        for b in range(0, nrhs, 8):
            part = g.aim_matvec(ctx, xp[b:b + 8].contiguous(), precision=prec)
            assert float(torch.linalg.norm(y[b:b + 8] - part) / torch.linalg.norm(part)) <= bound, (prec, b)
    ctx.close()


@pytest.mark.parametrize("nrhs", [16, 17, 32, 33, 64])
@pytest.mark.parametrize("body", ["plate", "cfie_sphere"])
def test_larger_bodies_equal_eight_at_a_time(body, nrhs):
    mesh, alpha = (plate_mesh(9.45, 85), 1.0) if body == "plate" else (icosphere_mesh(2.4, 26), 0.6)
    ctx = g.aim_setup(*mesh, K0, H, M=2, max_rhs=nrhs, cfie_alpha=alpha, precision=g.AIM_C64)
    assert ctx.N > 2 * 152 * 64 and ctx.N % 64
    x = torch.from_numpy(random_complex((nrhs, ctx.N), nrhs).astype(np.complex64)).cuda()
    y = g.aim_matvec(ctx, x, precision=g.AIM_C64)
    for b in range(0, nrhs, 8):
        part = g.aim_matvec(ctx, x[b:b + 8].contiguous(), precision=g.AIM_C64)
        assert float(torch.linalg.norm(y[b:b + 8] - part) / torch.linalg.norm(part)) <= 2e-5, b
    ctx.close()
