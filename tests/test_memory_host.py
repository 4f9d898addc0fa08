"""Memory that is counted before it is used (CPU only): aim_footprint's padding,
and the server's claim for the workspace a context keeps after a pattern."""

import numpy as np
import pytest

from aim_inputs import rect_plate_mesh
from paper_1010_1456_gb300 import serve
from test_serve_host import FakeMergingServer, _FakeCtx, mesh_reqs

WS = serve.RCS_WORKSPACE


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


def with_patterns(reqs, which):
    for i in which:
        reqs[i].rcs_dirs = (np.zeros(1), np.zeros(1))
    return reqs


class PatternServer(FakeMergingServer):
    """The real footprint of a request on fake base footprints."""

    def _footprint(self, req):
        return self.fps[req.rid] + (WS if req.rcs_dirs is not None else 0)


def test_a_resident_context_is_charged_for_its_pattern_workspace_once():
    reqs = with_patterns(mesh_reqs(["a", "a", "a", "a"], nrhs=2), [1, 3])
    s = PatternServer([40] * 4, slots=1, mem_budget=40 + 2 * WS, merge_rhs=2)
    res, _ = s.run(reqs, realtime=False)
    assert all(r.error is None for r in res)
    assert s.setups == 1 and s.claimed == 40 + WS == s.peak_claimed
    s.close()
    assert s.claimed == 0


def test_a_pattern_evicts_idle_contexts_but_not_its_own():
    _FakeCtx.closed = 0
    reqs = with_patterns(mesh_reqs(["a", "b", "a"]), [2])
    s = PatternServer([40] * 3, slots=1, mem_budget=60 + WS, merge_rhs=1)
    res, _ = s.run(reqs, realtime=False)
    assert all(r.error is None for r in res)
    assert s.solves[2] == ([2], False)  # a's context served it; b's made room
    assert _FakeCtx.closed == 1 and s.claimed == 40 + WS


def test_a_pattern_beyond_the_budget_still_runs_alone():
    reqs = with_patterns(mesh_reqs(["a", "a", "b"]), [1])
    s = PatternServer([40] * 3, slots=2, mem_budget=50, merge_rhs=1)
    res, _ = s.run(reqs, realtime=False)
    assert all(r.error is None for r in res)


def test_a_real_request_for_a_pattern_claims_the_workspace(lib):
    s = serve.Server(slots=1, mem_budget=1 << 30)
    plain = mesh_reqs(["a"])[0]
    plain.verts, plain.tris = rect_plate_mesh(0.5, 0.5, 4, 4)
    fp = s._footprint(plain)
    with_patterns([plain], [0])
    assert s._footprint(plain) == fp + WS
