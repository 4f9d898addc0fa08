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


def test_an_allocation_that_fails_leaves_nothing_behind():
    """Two small plates at opposite corners of a 20 lambda box: 203^3 nodes (padded
    405^3), whose complex64 grids for 256 right-hand sides hold 68 + 137 + 273 GB.
    The first two fit the GPU and the third does not; a second call fails as the
    first did (it must not take the two for the whole), and the memory is free."""
    v0, t0 = plate_mesh(0.2, 2)
    shift = np.array([19.9, 19.9, 19.9])
    v, t = np.concatenate([v0, v0 + shift]), np.concatenate([t0, t0 + len(v0)])
    ctx = g.aim_setup(v, t, K0, H, M=2, precision=g.AIM_C64, max_rhs=256)
    n, L, _ = g.aim_grid_info(ctx)
    need = [32.0 * 256 * a for a in (n[0] * n[1] * n[2], L[2] * n[1] * n[0], L[2] * L[1] * n[0])]
    total = torch.cuda.mem_get_info()[1]
    assert need[0] + need[1] < 0.75 * total and sum(need) > 1.5 * total  # sizes of this GPU's memory
    x = torch.from_numpy(random_complex((1, ctx.N), 2).astype(np.complex64)).cuda()
    y = torch.empty_like(x)
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    for _ in range(2):
        with pytest.raises(g.AIMError, match="out of memory"):
            g.aim_matvec(ctx, x, y, precision=g.AIM_C64)
        assert free - torch.cuda.mem_get_info()[0] < 1 << 30
    V = x.to(torch.complex128)
    for _ in range(2):  # the solver's own storage fits, the grids do not
        with pytest.raises(g.AIMError, match="out of memory"):
            g.aim_solve(ctx, V, 1e-6)
    ctx.close()
    small = g.aim_setup(v0, t0, K0, H, M=2)  # the failures do not reach another context
    xs = torch.from_numpy(random_complex((1, small.N), 3)).cuda()
    assert torch.isfinite(torch.view_as_real(g.aim_matvec(small, xs, precision=g.AIM_C128))).all()
    small.close()
