"""FP32 row ranges about the axis that are not their own mirror image: where the rows
one by one take no more waves of CTAs than the folded and the one-sided part, they
run in one launch each of the row and the column pass (plan.cu, propagate_rows).
Ranges on both sides of that rule against the FP64 form, relative, 1e-5 (a few
hundred roundings of 2^-24 over a row's transforms and sums)."""
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


def _geom(N, M, shift=0.0, levels=0, scale=1.0):
    D, p = (N - 0.5) * LAM * 5 / (2 * max(levels, 2)), scale * LAM * 5 / 8
    kw = dict(D=D, f=5 * D, lam=LAM, M=M, pitch=p, N=N, levels=levels)
    if shift:
        kw["x0"] = -(M / 2 - shift) * p
    return kw


@pytest.mark.parametrize("N", [2001, 5831])
def test_launches(env, N):
    """32 rows about the axis take the launches of 32 rows on one side of it."""
    fzp, torch = env
    c, U = N // 2, torch.empty((64, 64), dtype=torch.complex128, device="cuda")
    with fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32, **_geom(N, 64)) as plan:
        plan.profile(True)
        n = []
        for a, b in [(c + 4, c + 36), (c - 16, c + 16)]:
            plan.profile_read()
            plan.propagate_roi(a, b, U)
            torch.cuda.synchronize()
            n.append(plan.profile_read()["kernel_launches"])
    assert n[0] == n[1]


@pytest.mark.parametrize("N,M,scale", [(1501, 64, 1.0), (2001, 256, 1.0), (5831, 64, 1.0), (1501, 512, 4.0)])
@pytest.mark.parametrize("shift", [0.0, 7.25])
@pytest.mark.parametrize("levels", [0, 3])
def test_ranges(env, N, M, scale, shift, levels):
    fzp, torch = env
    kw, c = _geom(N, M, shift, levels, scale), N // 2
    with fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32, **kw) as plan, \
            fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP64, **kw) as exact:
        for a, b in [(c - 16, c + 16), (c - 1, c + 1), (c - 7, c + 250), (c - 151, c + 152), (c - 152, c + 152), (c - 153, c + 152),
                     (c - 303, c + 305), (c - 305, c + 304), (c - 10, c + 700), (1, N), (0, N - 1), (N // 3, N)]:
            U, _ = run_plan(fzp, torch, plan, M, a, b)
            R, _ = run_plan(fzp, torch, exact, M, a, b)
            assert rel_l2(U, R) <= 1e-5, (a, b)
