"""The rule that takes small grids with large ROIs past the interpolation nodes
(nodes.cu, nodes_pay): plans on both sides of it, in every form that has nodes,
flat and deformed, on the axis and off it, whole and in part, against the FP64
form.  Tolerances as of the forms: FP32 1e-5, dense 3e-5."""
import pytest

from gpu_util import rel_l2, run_plan

pytestmark = pytest.mark.gpu
LAM = 632.8e-9


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2609_01978_gb300 as fzp
    return fzp, torch


@pytest.mark.parametrize("N", [41, 301, 1401, 2001])
@pytest.mark.parametrize("M,scale", [(64, 1.0), (256, 2.0), (512, 1.0), (1024, 0.5)])
@pytest.mark.parametrize("kind", ["axis", "off", "membrane", "L4"])
def test_both_sides(env, N, M, scale, kind):
    fzp, torch = env
    levels = 4 if kind == "L4" else 0
    D, p = (N - 0.5) * LAM * 5 / (2 * max(levels, 2)), scale * LAM * 5 / 8
    kw = dict(D=D, f=5 * D, lam=LAM, M=M, pitch=p, N=N, levels=levels)
    if kind in ("off", "L4"):
        kw["x0"] = -(M / 2 - 9.5) * p
    if kind == "membrane":
        kw["deform"] = fzp.make_deform(amp=1.2e-7, period=D / 4, theta=0.7, taper=0.4, ridges=[(D / 10, -D / 5, 0.4, 6e-8, D / 8)])
    c = N // 2
    ranges = [(0, N), (c - N // 8, c + N // 5)]
    with fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP64, **kw) as exact:
        ref = [run_plan(fzp, torch, exact, M, a, b)[0] for a, b in ranges]
    for form, prec, tol in ((fzp.FORM_BLUESTEIN, fzp.PREC_FP32, 1e-5), (fzp.FORM_DENSE, fzp.PREC_SPLIT_BF16, 3e-5)):
        with fzp.Plan(form=form, precision=prec, **kw) as plan:
            for (a, b), R in zip(ranges, ref):
                U, _ = run_plan(fzp, torch, plan, M, a, b)
                assert rel_l2(U, R) <= tol, (form, a, b)
