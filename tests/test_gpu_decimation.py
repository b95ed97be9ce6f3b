"""Decimated rows of the FP32 form (k_dec) at the sizes where they can go wrong:
grid sizes on either side of the rule's lines (none, 16 and 32 columns to a grid
point), odd row counts and single rows, the diagonal and the axis in one chunk,
one transform and several per row, folded and not, and every transmission rule.

Fields are compared with the FP64 form's.  Tolerance, relative: hardware sine and
cosine 4e-7, phase walk 1e-7, interpolation 1.2e-7 and a few hundred roundings of
2^-24 over a row's transforms and sums -- 1e-5 bounds them all."""
import pytest

from gpu_util import rel_l2, run_plan

pytestmark = pytest.mark.gpu
LAM = 632.8e-9
TOL = 1e-5
RIDGES = ((1e-4, -2e-4, 0.4, 6e-8, 3e-4), (0.0, 1e-4, 2.0, 5e-8, 4e-4), (2e-4, 0.0, 1.1, 3e-8, 5e-4))


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2609_01978_gb300 as fzp
    return fzp, torch


def _compare(fzp, torch, N, M, ranges, shift=0.0, levels=0, **kw):
    D = (N - 0.5) * LAM * 5 / (2 * max(levels, 2))
    p = LAM * 5 / 8
    geom = dict(D=D, f=5 * D, lam=LAM, M=M, pitch=p, N=N, levels=levels, **kw)
    if shift:
        geom["x0"] = -(M / 2 - shift) * p
    with fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32, **geom) as plan, \
            fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP64, **geom) as exact:
        c = plan.info["N"] // 2
        for a, b in ranges(N, c):
            U, _ = run_plan(fzp, torch, plan, M, a, b)
            R, _ = run_plan(fzp, torch, exact, M, a, b)
            assert rel_l2(U, R) <= TOL, (a, b)


def _ranges(N, c):
    return [(0, N), (c, c + 1), (c + 1, c + 4), (c - 20, c + 45), (7, 90), (N - 33, N)]


@pytest.mark.parametrize("N", [2899, 2921, 5811, 5831, 6001])
@pytest.mark.parametrize("levels", [0, 3, 16])
@pytest.mark.parametrize("shift", [0.0, 7.25])
def test_lines_of_the_rule(env, N, levels, shift):
    _compare(*env, N, 64, _ranges, shift, levels)


@pytest.mark.parametrize("N", [2921, 5831])
@pytest.mark.parametrize("ridges", [0, 1, 2, 3])
def test_membranes(env, N, ridges):
    fzp, torch = env
    d = fzp.make_deform(amp=1.2e-7, period=1.1e-3, theta=0.7, taper=0.4, ridges=RIDGES[:ridges])
    _compare(fzp, torch, N, 64, _ranges, deform=d)


@pytest.mark.parametrize("N,M,shift,levels", [(40001, 512, 3.5, 0), (62463, 64, 7.25, 0), (62599, 64, 7.25, 3), (126001, 64, 0.0, 0),
                                              (126001, 64, 0.0, 4)])
def test_several_transforms_per_row(env, N, M, shift, levels):
    _compare(*env, N, M, lambda N, c: [(c - 4, c + 5), (c // 2, c // 2 + 7), (3, 40)], shift, levels)


@pytest.mark.parametrize("N", [3, 31, 33, 35, 37])
@pytest.mark.parametrize("shift", [0.0, 7.25])
def test_smallest_grids(env, N, shift):
    """Grids of fewer columns than one block has grid points: the centre of a large
    plate (open there), and a whole small plate under a fine ROI pitch."""
    fzp, torch = env
    for D, M, p, opened in [(5e-3, 64, 1e-8, 1), ((N - 0.5) * LAM * 5 / 4, 64, 1e-9, 0)]:
        geom = dict(D=D, f=5 * D, lam=LAM, M=M, pitch=p, N=N, centre_open=opened)
        if shift:
            geom["x0"] = -(M / 2 - shift) * p
        with fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32, **geom) as plan, \
                fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP64, **geom) as exact:
            for a, b in [(0, N), (N // 2, N // 2 + 1), (0, N // 2), (N // 2 - 1, N)]:
                U, _ = run_plan(fzp, torch, plan, M, a, b)
                R, _ = run_plan(fzp, torch, exact, M, a, b)
                if abs(R).max() == 0:
                    assert abs(U).max() == 0, (a, b)
                else:
                    assert rel_l2(U, R) <= TOL, (D, a, b)


def test_chirp_at_the_largest_grids(env):
    """N = 16,000,241 (its chirp rate has 0.996 of a unit below 2^-64 turns per
    squared column): three rows about the axis.  Left out, that part would turn the
    rim by 2e-5 rad and move the row's field by a third of it.  Tolerance: sine and
    cosine 4e-7, three tables 6e-8 each, interpolation 1.2e-7, 24 butterfly stages
    of 3e-8 each: 1.4e-6, so 2e-6."""
    fzp, torch = env
    N = 16000241
    D = (N - 0.5) * LAM * 5 / 4
    geom = dict(D=D, f=5 * D, lam=LAM, M=64, pitch=LAM * 5 / 8, N=N, stripe_rows=256, form=fzp.FORM_BLUESTEIN)
    c = N // 2
    with fzp.Plan(precision=fzp.PREC_FP32, **geom) as plan, fzp.Plan(precision=fzp.PREC_FP64, **geom) as exact:
        U, _ = run_plan(fzp, torch, plan, 64, c - 1, c + 2)
        R, _ = run_plan(fzp, torch, exact, 64, c - 1, c + 2)
    assert rel_l2(U, R) <= 2e-6
