"""What a plan reports about itself is what it runs: CTAs and the name of the
dominant kernel."""
import pytest

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


def _geom(N, M, scale=1.0):
    D = (N - 0.5) * LAM * 5 / 4
    return dict(D=D, f=5 * D, lam=LAM, M=M, pitch=scale * LAM * 5 / 8, N=N)


@pytest.mark.parametrize("M,scale,nodes", [(64, 1.0, True), (256, 1.0, True), (512, 1.0, True), (1024, 4.0, False)])
def test_ctas(env, M, scale, nodes):
    """On nodes a CTA on every SM, whatever the ROI; k_dense's clusters of four
    leave some SMs without one."""
    fzp, torch = env
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    with fzp.Plan(form=fzp.FORM_DENSE, precision=fzp.PREC_SPLIT_BF16, **_geom(1501, M, scale)) as plan:
        assert plan.info["ctas"] == sms if nodes else plan.info["ctas"] % 4 == 0


@pytest.mark.parametrize("N,kw,name", [(1501, {}, "k_seg"), (5831, {}, "k_dec"), (5831, dict(conv=1), "bluestein_f2<float>")])
def test_dominant_kernel_of_the_fp32_form(env, N, kw, name):
    fzp, torch = env
    with fzp.Plan(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32, **_geom(N, 64), **kw) as plan:
        plan.profile(True)
        plan.propagate_roi(0, 8, torch.empty((64, 64), dtype=torch.complex128, device="cuda"))
        plan.propagate_roi(N // 2, N // 2 + 2, torch.empty((64, 64), dtype=torch.complex128, device="cuda"))
        assert plan.profile_read()["dominant_name"].startswith(name)
