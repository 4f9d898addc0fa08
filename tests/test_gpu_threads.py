"""Solves in one thread while others build and free contexts.

A solve captures its step as a CUDA graph.  A wait for the whole device while any
stream captures fails and spoils the capture, and freeing a context makes one.  The
solves alternate between one and two right-hand sides, which captures anew each
time.
"""

import threading

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from aim_inputs import plate_mesh, random_incidence  # noqa: E402

import paper_1010_1456_gb300 as g  # noqa: E402

K0 = 2 * np.pi
H = 0.1


def churn(stop, errors):
    """Build and free small contexts until told to stop."""
    v, t = plate_mesh(0.5, 4)
    s = torch.cuda.Stream()
    while not stop.is_set():
        try:
            g.aim_setup(v, t, K0, H, M=2, stream=s.cuda_stream).close()
        except Exception as e:  # reported by the test
            errors.append(repr(e))


@pytest.mark.parametrize("krylov", ["gmres", "tfqmr"])
def test_solves_beside_other_threads(krylov):
    v, t = plate_mesh(1.0, 9)
    kind = g.AIM_GMRES if krylov == "gmres" else g.AIM_TFQMR
    stream = torch.cuda.Stream()
    errors, stop = [], threading.Event()
    with torch.cuda.stream(stream):
        ctx = g.aim_setup(v, t, K0, H, M=2, max_rhs=2, precision=g.AIM_C64, stream=stream.cuda_stream, krylov=kind)
        kh, po = random_incidence(1, rng=np.random.default_rng(1))
        V = g.aim_rhs_planewave(ctx, kh, po)
        alone = [g.aim_solve(ctx, V[:n].contiguous(), 1e-6)[0].cpu() for n in (1, 2)]
        threads = [threading.Thread(target=churn, args=(stop, errors)) for _ in range(2)]
        for th in threads:
            th.start()
        try:
            for i in range(60):
                X, info = g.aim_solve(ctx, V[: 1 + i % 2].contiguous(), 1e-6)
                assert info["converged"].all()
                assert torch.equal(X.cpu(), alone[i % 2]), i
        finally:
            stop.set()
            for th in threads:
                th.join()
    assert not errors, errors[:3]
    ctx.close()
