"""The FP64 form's folded rows and symmetric column pass where they can go wrong:
every inner FFT split (one 4096-point transform, several, shorter ones), output
counts on either side of a column tile, centred and off the axis, whole
apertures (their own transpose) and ranges that are not.

Fields are compared with the oracle's, and the single convolution in FP32 with
them.  Tolerances, relative: FP64, 1e-10 as elsewhere (phases reduced from 1e5
turns); FP32, a few hundred roundings of 2^-24 over a row's transforms: 1e-5."""
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
    import oracle
    import paper_2609_01978_gb300 as fzp
    return fzp, torch, oracle


def _check(env, N, M, shift, levels, precision, conv, tol, ranges=None):
    fzp, torch, O = env
    D = (N - 0.5) * LAM * 5 / (2 * max(levels, 2))
    p = LAM * 5 / 8
    kw = dict(x0=-(M / 2 - shift) * p) if shift else {}
    okw = dict(kind=O.FZP_PHASE, levels=levels) if levels else {}
    g = O.Geometry(D=D, f=5 * D, lam=LAM, M=M, p=p, dx=LAM * 5 / (2 * max(levels, 2)), N=N, **kw, **okw)
    with fzp.Plan(D=D, f=5 * D, lam=LAM, M=M, pitch=p, dx=g.dx, N=N, levels=levels, form=fzp.FORM_BLUESTEIN,
                  precision=getattr(fzp, precision), conv=conv, **kw) as plan:
        for a, b in ranges or [(0, N), (g.c - 30, g.c + 31), (g.c + 5, N - 20), (11, g.c + 8)]:
            U, _ = run_plan(fzp, torch, plan, M, a, b)
            assert rel_l2(U, O.field_czt(g, a, b)) <= tol, (a, b)


@pytest.mark.parametrize("N,M,shift,levels", [(301, 64, 0.0, 0), (1501, 128, 0.0, 0), (1501, 128, 5.25, 3), (2047, 512, 0.0, 0),
                                              (3585, 512, 0.0, 4), (4097, 256, 0.0, 0), (7001, 64, 3.5, 0)])
def test_fp64(env, N, M, shift, levels):
    _check(env, N, M, shift, levels, "PREC_FP64", 0, 1e-10)


@pytest.mark.parametrize("N,M,shift", [(301, 64, 0.0), (1501, 128, 4.25), (2047, 512, 0.0)])
def test_single_convolution_fp32(env, N, M, shift):
    _check(env, N, M, shift, 0, "PREC_FP32", 1, 1e-5)
