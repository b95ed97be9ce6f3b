"""The FP32 form's mask generators (the zone phase walked along 16 columns, with the
threshold search or the zone rule near a zone's end), bit for bit through the
export against the oracle's masks: every rule, row passes with and without
decimated rows, from the axis on and over all columns, and plates whose zones end
on samples (kappa = 1 / (4 N): a tie at every multiple of 4 N)."""
import numpy as np
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
    import oracle
    import paper_2609_01978_gb300 as fzp
    return fzp, torch, oracle


@pytest.mark.parametrize("kind", ["negative", "positive", "membrane", "L2", "L3", "L4", "L16", "L64"])
@pytest.mark.parametrize("N", [63, 1501, 5831])
@pytest.mark.parametrize("shift,tie", [(0.0, False), (7.25, False), (0.0, True)])
def test_masks_bit_for_bit(env, kind, N, shift, tie):
    fzp, torch, O = env
    levels = int(kind[1:]) if kind[0] == "L" else 0
    S = max(levels, 2)
    D = (N - (0.0 if tie else 0.5)) * LAM * 5 / (2 * S)
    p = LAM * 5 / 8
    x0 = dict(x0=-(32 - shift) * p) if shift else {}
    okw = dict(kind=O.FZP_PHASE, levels=levels) if levels else dict(kind=O.FZP_POSITIVE) if kind == "positive" else {}
    g = O.Geometry(D=D, f=5 * D, lam=LAM, M=64, p=p, dx=LAM * 5 * D / (2 * S * D), N=N, **okw, **x0)
    kw = dict(x0)
    if kind == "membrane":
        kw["deform"] = fzp.make_deform(amp=1e-7, period=1e-3, theta=0.3, taper=0.2, ridges=[])
    with fzp.Plan(D=D, f=5 * D, lam=LAM, M=64, pitch=p, dx=g.dx, N=N, levels=levels, centre_open=int(kind == "positive"),
                  form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32, **kw) as plan:
        for a, b in [(0, min(N, 70)), (g.c - 20, g.c + 21), (N - 9, N)] + ([(0, N)] if N < 2000 else []):
            out = torch.full((b - a, N), 255, dtype=torch.uint8, device="cuda")
            plan.aperture_mask(a, b, out)
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), O.mask_rows(g, a, b)), (a, b)
