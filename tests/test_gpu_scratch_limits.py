"""Plans whose row intermediate cannot be allocated whole: a small membrane gives up
the images that only make its sums reproducible before it halves its rows, and
needs no more memory than a flat plate of its size then (256 rows x 2 M x 4 B)."""
import numpy as np
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


@pytest.mark.parametrize("form", ["dense", "fp32"])
@pytest.mark.parametrize("limit,rows", [(None, 2816), (8_000_000, 2816), (3_000_000, 768), (600_000, 256)])
def test_membranes_under_an_allocation_limit(env, monkeypatch, form, limit, rows):
    fzp, torch = env
    N, M = 2801, 256
    D = (N - 0.5) * LAM * 5 / 4
    kw = dict(D=D, f=5 * D, lam=LAM, M=M, pitch=LAM * 5 / 8, N=N,
              deform=fzp.make_deform(amp=1.2e-7, period=1.1e-3, theta=0.7, taper=0.4, ridges=[]))
    how = dict(form=fzp.FORM_DENSE, precision=fzp.PREC_SPLIT_BF16) if form == "dense" else \
        dict(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32)
    with fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP64, **kw) as exact:
        _, R = run_plan(fzp, torch, exact, M, 0, N)
    if limit:
        monkeypatch.setenv("FZP_FAULT_ALLOC_LIMIT", str(limit))
    with fzp.Plan(**kw, **how) as plan:
        assert plan.info["chunk_rows"] == rows
        _, I = run_plan(fzp, torch, plan, M, 0, N)
    assert rel_l2(I, R) <= 1e-4
