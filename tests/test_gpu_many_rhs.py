"""Products of 16 and more right-hand sides against the same vectors eight at a time.

The many-RHS kernels lay right-hand sides over half a warp or a whole one, one
or two a lane, in rows padded to an even length; the counts below sit at the
edges of these choices.  Both paths are within 1e-12 (complex128 vectors) and
1e-5 (complex64) of the FP64 oracle by the product's own bounds, relative L2,
so they are within twice that of one another.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from aim_inputs import icosphere_frequency, icosphere_mesh, plate_mesh, random_complex  # noqa: E402

import paper_1010_1456_gb300 as g  # noqa: E402

K0 = 2 * np.pi
H = 0.1


@pytest.mark.parametrize("budget", [0, 8 << 30])
@pytest.mark.parametrize("nrhs", [16, 17, 31, 32, 33, 47, 63, 64, 65, 96, 129])
@pytest.mark.parametrize("body", ["plate", "sphere"])
def test_many_rhs_equals_eight_at_a_time(body, nrhs, budget):
    mesh = plate_mesh(1.0, 9) if body == "plate" else icosphere_mesh(0.4, icosphere_frequency(0.4))
    ctx = g.aim_setup(*mesh, K0, H, M=2, max_rhs=nrhs, cfie_alpha=1.0 if body == "plate" else 0.6, mem_budget=budget)
    x = torch.from_numpy(random_complex((nrhs, ctx.N), nrhs)).cuda()
    for prec, bound in ((g.AIM_C64, 2e-5), (g.AIM_C128_F64, 2e-12)):
        xp = x.to(torch.complex64) if prec == g.AIM_C64 else x
        y = g.aim_matvec(ctx, xp, precision=prec)
        for b in range(0, nrhs, 8):
            part = g.aim_matvec(ctx, xp[b:b + 8].contiguous(), precision=prec)
            assert float(torch.linalg.norm(y[b:b + 8] - part) / torch.linalg.norm(part)) <= bound, (prec, b)
    ctx.close()
