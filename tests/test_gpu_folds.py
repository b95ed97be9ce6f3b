"""The SA-CZT's folded route and the surrogate's fused products at the sizes where
they can go wrong: grids just under and over a padded size, ROIs on either side
of a node tile, on and off the axis, and batches and layers that are no multiple
of a tile.

Tolerances: the SA-CZT's intensity against the oracle's FP64 evaluation, 1e-4 as
the form's other tests; gradients against the oracle with its BF16 operands, 2e-3
per tensor, and the loss 1e-5, as the surrogate's."""
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
    import oracle
    from oracle import saczt, surrogate
    import paper_2609_01978_gb300 as fzp
    return fzp, torch, oracle, saczt, surrogate


@pytest.mark.parametrize("N", [301, 681, 683, 1365, 2731])
@pytest.mark.parametrize("M,shift", [(64, 0.0), (128, 0.0), (256, 11.25)])
def test_saczt_whole_apertures(env, N, M, shift):
    fzp, torch, O, SA, _ = env
    D = (N - 0.5) * LAM * 5 / 4
    p = LAM * 5 / 8
    kw = dict(x0=-(M / 2 - shift) * p) if shift else {}
    g = O.Geometry(D=D, f=5 * D, lam=LAM, M=M, p=p, dx=LAM * 5 / 4, N=N, kind=O.FZP_EXACT, **kw)
    with fzp.Plan(D=D, f=g.f, lam=LAM, M=M, pitch=p, dx=g.dx, N=N, form=fzp.FORM_SACZT, precision=fzp.PREC_FP32,
                  exact_radii=1, **kw) as plan:
        _, I = run_plan(fzp, torch, plan, M, 0, N)
        assert rel_l2(I, np.abs(SA.field_saczt(g)) ** 2) <= 1e-4


@pytest.mark.parametrize("sizes,B", [((8, 64, 40), 8), ((8, 64, 64, 72), 24), ((8, 128, 128, 128, 200), 136), ((8, 512, 512, 1048), 264)])
def test_surrogate_gradients(env, sizes, B):
    fzp, torch, _, _, S = env
    net = fzp.SurrogateNet(n_in=sizes[0], hidden=sizes[1], layers=len(sizes) - 2, n_out=sizes[-1], max_batch=B, seed=3)
    rng = np.random.default_rng(2)
    X = rng.normal(size=(B, sizes[0])).astype(np.float32)
    Y = rng.normal(size=(B, sizes[-1])).astype(np.float32)
    g = torch.empty(net.param_count, dtype=torch.float32, device="cuda")
    loss = torch.empty(1, dtype=torch.float32, device="cuda")
    net.grad(torch.from_numpy(X).cuda(), torch.from_numpy(Y).cuda(), g, loss)
    torch.cuda.synchronize()
    params = S.unflatten(net.get_params().astype(np.float64), list(sizes))
    lref, gref = S.loss_and_grads(params, X.astype(np.float64), Y.astype(np.float64), rnd=True)
    assert abs(loss.item() / lref - 1) < 1e-5
    got = g.cpu().numpy().astype(np.float64)
    k = 0
    for ref in (r.ravel() for pair in gref for r in pair):
        assert np.linalg.norm(got[k:k + ref.size] - ref) / np.linalg.norm(ref) < 2e-3
        k += ref.size
    net.close()
