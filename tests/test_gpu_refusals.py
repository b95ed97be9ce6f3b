"""What the library refuses, it refuses at every entry point: a transform above 2^24
points, by fzp_plan_query as by fzp_plan, also where the plan itself would run
half the length (FP64, ROI on the axis)."""
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import __graft_entry__
    __graft_entry__.build()
    import paper_2609_01978_gb300 as fzp
    return fzp, torch


@pytest.mark.parametrize("how", ["fp64", "fp64 off the axis", "fp32 single", "fp32 partitioned"])
def test_transforms_above_the_limit(env, how):
    fzp, torch = env
    kw = dict(D=4e-3, f=20e-3, lam=632.8e-9, M=64, pitch=0.4e-6, stripe_rows=256, form=fzp.FORM_BLUESTEIN,
              precision=fzp.PREC_FP64 if how.startswith("fp64") else fzp.PREC_FP32,
              conv=fzp.CONV_SINGLE if how == "fp32 single" else 0)
    if how.endswith("axis"):
        kw["x0"] = -10e-6
    most = (1 << 24) - 63  # N + M - 1 = 2^24
    assert fzp.plan_query(N=most, **kw)["fft_length"] == 1 << 24
    for call in (fzp.plan_query, fzp.Plan):
        with pytest.raises(fzp.FzpError) as ei:
            call(N=most + 2, **kw)
        assert ei.value.status == fzp.FZP_E_UNSUPPORTED
    fzp.Plan(N=most, **kw).close()
