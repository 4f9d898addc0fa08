"""Which FFT kernel runs: explicit choices, the built-in rule, what is reported.

Every product is deterministic, so two products are the same bits exactly when
the same kernels ran, and a four-step and a Stockham x pass of 125 and more
points round differently.  Both kernel families are within 1e-12 (complex128
vectors) and 1e-5 (complex64) of the FP64 oracle, relative L2, by the product's
own bounds, so they are within twice that of one another.
"""

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

from aim_inputs import plate_mesh, random_complex  # noqa: E402
from oracle import aim as oaim  # noqa: E402
from oracle.rwg import RWG  # noqa: E402
from test_gpu_fft_lengths import H, K0, reachable, strip  # noqa: E402

import paper_1010_1456_gb300 as g  # noqa: E402

BOUND = {g.AIM_C128: 1e-12, g.AIM_C128_F64: 1e-12, g.AIM_C64: 1e-5}
# the lengths whose four-step split has a DFT of 24 or more, which few pencils of a 16-byte type leave to Stockham
LONG = [L for L in reachable(900) if L in (125, 243, 250, 375) or (L >= 384 and L != 400)] + [1296]


def x_choice(k):
    return [g.AIM_FFT_AUTO, g.AIM_FFT_AUTO, k, g.AIM_FFT_AUTO, g.AIM_FFT_AUTO]


def product(ctx, x, prec, k):
    g.aim_fft_config(ctx, prec, x_choice(k))
    return g.aim_matvec(ctx, x.to(torch.complex64) if prec == g.AIM_C64 else x, precision=prec)


def rel(a, b):
    return float(torch.linalg.norm(a - b) / torch.linalg.norm(b))


@pytest.mark.parametrize("L", LONG)
def test_an_explicit_four_step_x_pass_runs(L):
    """At every length the rule keeps from a thin strip, in every precision: the
    four-step kernels that are asked for run and agree with Stockham, and the
    rule's own choice is the one reported."""
    found = strip(L, 0, wide=L % 2 == 0)
    assert found is not None
    nrhs = 1 + L % 3
    ctx = g.aim_setup(*found, K0, H, M=2, max_rhs=nrhs)
    assert g.aim_grid_info(ctx)[1][0] == L
    x = torch.from_numpy(random_complex((nrhs, ctx.N), L)).cuda()
    for prec, bound in BOUND.items():
        ref = product(ctx, x, prec, g.AIM_FFT_STOCKHAM)
        for k in (g.AIM_FFT_FOURSTEP, g.AIM_FFT_FOURSTEP_SMALL):
            y = product(ctx, x, prec, k)
            assert not torch.equal(y, ref), (prec, k)
            assert rel(y, ref) <= 2 * bound, (prec, k)
        y = product(ctx, x, prec, g.AIM_FFT_AUTO)
        ran = g.aim_fft_config(ctx, prec)[2]
        assert ran == (g.AIM_FFT_FOURSTEP if prec == g.AIM_C64 else g.AIM_FFT_STOCKHAM)
        assert torch.equal(y, product(ctx, x, prec, ran)), prec
    ctx.close()


@pytest.mark.parametrize("side, L", [(0.9, 24), (3.2, 72), (6.5, 135), (16.0, 324), (19.2, 400)])
def test_x_pass_shapes_on_a_plane(side, L):
    """Planar grids of 1 to 5 right-hand sides: few rows, which the x pass lays over
    blocks by the number of grids, down to one row and one grid a block."""
    ctx = g.aim_setup(*plate_mesh(side, int(round(9 * side))), K0, H, M=2, max_rhs=5)
    assert g.aim_grid_info(ctx)[1] == [L, L, 1]
    x = torch.from_numpy(random_complex((5, ctx.N), L)).cuda()
    for nrhs in (1, 2, 5):
        xs = x[:nrhs].contiguous()
        for prec, bound in BOUND.items():
            ref = product(ctx, xs, prec, g.AIM_FFT_STOCKHAM)
            assert rel(product(ctx, xs, prec, g.AIM_FFT_FOURSTEP), ref) <= 2 * bound, (nrhs, prec)
    ctx.close()


@pytest.mark.parametrize("prec, nrhs", [(g.AIM_C128, 76), (g.AIM_C128_F64, 17)])
def test_the_rule_on_both_sides_of_its_line(prec, nrhs):
    """125 = 5 x 25 points, 8 x 5 rows: 1,000 units a grid, 4 grids a right-hand
    side; the line is at 304,000 units (float-float DFTs of 25) and 65,664 (FP64)."""
    v, t = strip(125, 0, wide=False)
    ctx = g.aim_setup(v, t, K0, H, M=2, max_rhs=nrhs)
    assert g.aim_grid_info(ctx)[1] == [125, 8, 5]
    assert g.aim_fft_config(ctx, prec)[2] == g.AIM_FFT_FOURSTEP  # resolved for max_rhs
    x = torch.from_numpy(random_complex((nrhs, ctx.N), 3)).cuda()
    for n, k in ((nrhs, g.AIM_FFT_FOURSTEP), (nrhs - 1, g.AIM_FFT_STOCKHAM)):
        xs = x[:n].contiguous()
        assert torch.equal(product(ctx, xs, prec, g.AIM_FFT_AUTO), product(ctx, xs, prec, k)), n
    ctx.close()


@pytest.mark.parametrize("along, passes", [(1, (1, 3)), (2, (0, 4))])
def test_the_rule_of_the_strided_passes(along, passes):
    """125 points along y or z of a strip: Stockham in the 16-byte types' passes of
    that axis, four-step in complex64's, and what is reported is what runs."""
    ctx = g.aim_setup(*strip(125, along, wide=False), K0, H, M=2, max_rhs=2)
    assert g.aim_grid_info(ctx)[1][along] == 125
    x = torch.from_numpy(random_complex((2, ctx.N), 4)).cuda()
    for prec in BOUND:
        xp = x.to(torch.complex64) if prec == g.AIM_C64 else x
        y = g.aim_matvec(ctx, xp, precision=prec)
        ran = g.aim_fft_config(ctx, prec)
        assert ran == [1 if prec != g.AIM_C64 and p in passes else 2 for p in range(5)]
        g.aim_fft_config(ctx, prec, ran)
        assert torch.equal(y, g.aim_matvec(ctx, xp, precision=prec))
        g.aim_fft_config(ctx, prec, [g.AIM_FFT_FOURSTEP] * 5)
        assert rel(g.aim_matvec(ctx, xp, precision=prec), y) <= 2 * BOUND[prec]
    ctx.close()


def test_an_x_axis_without_a_four_step_kernel():
    """960 points: the rule and an explicit four-step choice run Stockham, the
    rule says so, and the autotuner does not time the same kernel again."""
    v, t = strip(960, 0, wide=True)
    ctx = g.aim_setup(v, t, K0, H, M=2, max_rhs=2)
    assert g.aim_grid_info(ctx)[1][0] == 960
    op = oaim.AIMOperator(RWG(v, t), K0, H, 2, near_radius=3 * H)
    xh = random_complex((2, ctx.N), 960)
    x = torch.from_numpy(xh).cuda()
    for prec, bound in BOUND.items():
        y = product(ctx, x, prec, g.AIM_FFT_AUTO)
        assert g.aim_fft_config(ctx, prec) == [2, 2, 1, 2, 2]
        assert torch.equal(y, product(ctx, x, prec, g.AIM_FFT_FOURSTEP))
        xr = xh.astype(np.complex64).astype(np.complex128) if prec == g.AIM_C64 else xh
        ref = op.matvec(xr)
        assert np.linalg.norm(y.cpu().numpy() - ref) <= bound * np.linalg.norm(ref), prec
        kernels, ms = g.aim_autotune(ctx, prec, nrhs=2, reps=1)
        assert kernels[2] == g.AIM_FFT_STOCKHAM and ms[2, 1] > 0 and (ms[2, 2:] == -1).all()
    ctx.close()

def test_autotune_times_a_kernel_once():
    """Small blocks are a kernel of their own in the 16-byte types only: complex64
    x passes run in them anyway."""
    ctx = g.aim_setup(*plate_mesh(1.0, 9), K0, H, M=2, max_rhs=1, planar=False)
    for prec in BOUND:
        kernels, ms = g.aim_autotune(ctx, prec, nrhs=1, reps=1)
        tried = [1, 2] if prec == g.AIM_C64 else [1, 2, 3]
        assert [k for k in range(g.AIM_FFT_KERNELS) if ms[2, k] > 0] == tried, prec
        assert kernels[2] in tried
    ctx.close()
