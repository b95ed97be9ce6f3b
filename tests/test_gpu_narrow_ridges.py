"""Membranes whose ridges are a few columns wide, in every form that takes a
membrane: rows of the FP32 form without decimation, with 16 and with 32 columns
to a grid point, the dense form on nodes and in clusters.  Widths on both sides
of the generators' rule (every column evaluated below 64 columns along the row,
in the dense form below 12; walked above); a ridge across the rows, one at an
angle, one nearly along them.

Fields are compared with the FP64 form's.  Tolerance as for smooth membranes: FP32
1e-5 (hardware sine and cosine 4e-7, a few hundred roundings of 2^-24); dense 3e-5
(kernel and mask values to 2^-17).  A ridge of w columns and 0.2 turns that was
left out would move the field by about w / N, 3e-4 and more here."""
import math

import pytest

from gpu_util import rel_l2, run_plan

pytestmark = pytest.mark.gpu
LAM = 632.8e-9
DX = LAM * 5 / 4


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2609_01978_gb300 as fzp
    return fzp, torch


@pytest.mark.parametrize("form,N,cluster", [("fp32", 1501, 0), ("fp32", 2921, 0), ("fp32", 5831, 0), ("dense", 1501, 0),
                                            ("dense", 1501, 1), ("dense", 1501, 2)])
@pytest.mark.parametrize("width", [1, 2, 5, 8, 11.5, 12, 40, 63.5, 64.5])
def test_ridge_widths(env, form, N, cluster, width):
    fzp, torch = env
    D, M = (N - 0.5) * DX, 64 if form == "fp32" else 128
    ridges = [(3e-5, -2e-5, math.pi / 2, 6e-8, width * DX), (-4e-5, 1e-5, 0.4, 5e-8, width * DX), (0.0, 6e-5, 0.02, 4e-8, width * DX)]
    geom = dict(D=D, f=5 * D, lam=LAM, M=M, pitch=LAM * 5 / 8, N=N,
                deform=fzp.make_deform(amp=1.2e-7, period=1.1e-3, theta=0.7, taper=0.4, ridges=ridges))
    how = dict(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32) if form == "fp32" else \
        dict(form=fzp.FORM_DENSE, precision=fzp.PREC_SPLIT_BF16, cluster=cluster)
    with fzp.Plan(**geom, **how) as plan, fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP64, **geom) as exact:
        U, _ = run_plan(fzp, torch, plan, M, 0, N)
        R, _ = run_plan(fzp, torch, exact, M, 0, N)
    assert rel_l2(U, R) <= (1e-5 if form == "fp32" else 3e-5)
