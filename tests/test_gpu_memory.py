"""Device memory of a context: what a solve allocates, and an allocation that fails.

Free memory is read from the driver (torch.cuda.mem_get_info) around the call
that allocates; torch's own tensors exist before the first reading.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from aim_inputs import icosphere_frequency, icosphere_mesh, plate_mesh, random_complex  # noqa: E402

import paper_1010_1456_gb300 as g  # noqa: E402

K0 = 2 * np.pi
H = 0.1


@pytest.mark.parametrize("budget", [0, 60 << 30])
def test_solver_storage_is_its_vectors(budget):
    """GMRES(200) for 64 right-hand sides holds the basis, two work vectors and
    the Hessenberg columns; the partial sums of its reductions are a few blocks a
    right-hand side (10 here: 2 MB), however many blocks update the vector.  Each
    of about fifteen allocations is rounded up to 2 MB."""
    v, t = plate_mesh(16.0, 144)
    nrhs, m = 64, 200
    ctx = g.aim_setup(v, t, K0, H, M=2, precision=g.AIM_C64, restart=m, maxit=1, max_rhs=nrhs, mem_budget=budget)
    V = torch.from_numpy(random_complex((nrhs, ctx.N), 1)).cuda()
    X = torch.empty_like(V)
    g.aim_matvec(ctx, V.to(torch.complex64), precision=g.AIM_C64)
    g.aim_matvec(ctx, V, X, precision=g.AIM_C128)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    g.aim_solve(ctx, V, 1e-6, X=X, raise_on_noconv=False)
    used = before - torch.cuda.mem_get_info()[0]
    held = 16 * nrhs * (ctx.N * (m + 1 + 2) + (m + 1) * m)
    assert held <= used <= held + (48 << 20), (used, held)
    ctx.close()
