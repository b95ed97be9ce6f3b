"""Column pass of the FP32 form on ROI samples: few rows in one block a tile, and the
kernel that runs three blocks to an SM, from more than two waves of blocks on,
against the FP64 form.  Relative, 1e-5 (a few hundred roundings of 2^-24)."""
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


@pytest.mark.parametrize("N,M,scale,kind", [(101, 1024, 1.0, "mem"), (2001, 1024, 1.0, "mem"), (4097, 1024, 1.0, "mem"), (4201, 1024, 1.0, "mem"),
                                            (9001, 1024, 4.0, "flat"), (9001, 1024, 4.0, "off"), (20001, 512, 2.0, "mem"),
                                            (8191, 1024, 1.0, "single")])
def test_against_fp64(env, N, M, scale, kind):
    fzp, torch = env
    D, p, c = (N - 0.5) * LAM * 5 / 4, scale * LAM * 5 / 8, N // 2
    kw = dict(D=D, f=5 * D, lam=LAM, M=M, pitch=p, N=N)
    if kind == "off":
        kw["x0"] = -(M / 2 - 9.25) * p
    if kind == "mem":
        kw["deform"] = fzp.make_deform(amp=1.2e-7, period=D / 4, theta=0.7, taper=0.4, ridges=[(D / 10, -D / 5, 0.4, 6e-8, D / 8)])
    conv = dict(conv=fzp.CONV_SINGLE) if kind == "single" else {}
    with fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32, **kw, **conv) as plan, \
            fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP64, **kw) as exact:
        for a, b in [(0, N), (0, c)]:
            U, _ = run_plan(fzp, torch, plan, M, a, b)
            R, _ = run_plan(fzp, torch, exact, M, a, b)
            assert rel_l2(U, R) <= 1e-5, (a, b)
