"""The dense form on interpolation nodes (nodes.cu) at the sizes where it can go
wrong: grids smaller than a stripe, a K block or a unit and around them, ROI
sides and pitches on either side of every node count, row ranges with and
without their mirror image, and the general kernels (k_dense) where the pitch
is too coarse for nodes.

Fields are compared with the oracle's.  Tolerance: a kernel value is stored to
2^-17 of itself (BF16 hi + lo), so the field is within 2^-17 of the sum of the
moduli that make it up; near the focus that is the field itself, and I moves
by twice that, 1.5e-5 -- 3e-5 leaves room for the FP32 sums."""
import numpy as np
import pytest

from gpu_util import rel_l2, run_plan

pytestmark = pytest.mark.gpu
LAM = 632.8e-9
TOL = 3e-5


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


def _geom(O, N, M, pitch=None, **kw):
    """A plate of N samples at f/5 (four per outermost zone)."""
    L = max(kw.get("levels", 0), 2)
    D = (N - 0.5) * LAM * 5 / (2 * L)
    return O.Geometry(D=D, f=5 * D, lam=LAM, M=M, p=pitch or LAM * 5 / 8, dx=LAM * 5 * D / (2 * L * D), N=N, **kw)


def _plan(fzp, g, form="dense", **kw):
    f, p = {"dense": (fzp.FORM_DENSE, fzp.PREC_SPLIT_BF16), "fp32": (fzp.FORM_BLUESTEIN, fzp.PREC_FP32),
            "fp64": (fzp.FORM_BLUESTEIN, fzp.PREC_FP64)}[form]
    return fzp.Plan(D=g.D, f=g.f, lam=g.lam, M=g.M, pitch=g.p, dx=g.dx, N=g.N, form=f, precision=p, **kw)


@pytest.mark.parametrize("N", [41, 63, 65, 1021, 1027, 2049])
def test_small_grids(env, N):
    """Half grids of 21 to 1,025 rows: inside one K block, one stripe (512 rows)
    and at their ends."""
    fzp, torch, O = env
    g = _geom(O, N, 128)
    with _plan(fzp, g) as plan:
        _, I = run_plan(fzp, torch, plan, g.M, 0, N)
        assert rel_l2(I, np.abs(O.field_czt(g)) ** 2) <= TOL


@pytest.mark.parametrize("M,scale", [(64, 1.0), (64, 4.0), (128, 1.0), (256, 1.0), (512, 1.0), (512, 1.13), (512, 1.17),
                                     (1024, 1.0), (1024, 1.3)])
@pytest.mark.parametrize("shift", [0.0, 37.25])
@pytest.mark.parametrize("form", ["dense", "fp32"])
def test_node_counts_and_row_ranges(env, M, scale, shift, form):
    """ROI pitches on both sides of the limits of 64, 128 and 256 nodes, centred
    (even field) and off the axis; row ranges: whole, one side of the axis,
    straddling it unevenly, one row, and their sum."""
    fzp, torch, O = env
    p = LAM * 5 / 8 * scale
    kw = dict(x0=-(M / 2 - shift) * p) if shift else {}
    g = _geom(O, 1501, M, pitch=p, **kw)
    # FP32: a few hundred roundings of 2^-24 over a row's transforms and sums
    tol = TOL if form == "dense" else 1e-5
    with _plan(fzp, g, form, **kw) as plan:
        for a, b in [(0, g.N), (g.c + 3, g.N - 100), (120, g.c), (g.c - 200, g.c + 431), (g.c, g.c + 1)]:
            U, _ = run_plan(fzp, torch, plan, M, a, b)
            ref = O.field_czt(g, a, b)
            assert rel_l2(U, ref) <= tol, (a, b)
        parts = torch.zeros((M, M), dtype=torch.complex128, device="cuda")
        for a, b in [(0, 333), (333, g.c + 8), (g.c + 8, g.N)]:
            plan.propagate_roi(a, b, parts, accumulate=True)
        torch.cuda.synchronize()
        assert rel_l2(parts.cpu().numpy(), O.field_czt(g)) <= tol


@pytest.mark.parametrize("form,levels,N", [("fp32", 0, 301), ("fp32", 3, 9001), ("fp32", 16, 15001), ("fp64", 0, 1501),
                                           ("fp64", 3, 301)])
def test_folded_rows_of_the_fft_forms(env, form, levels, N):
    """Flat plates run each distance from the axis once; FP32 on nodes also stops
    at the diagonal: chunked rows, whole and one-sided ranges, one block and
    several per row."""
    fzp, torch, O = env
    g = _geom(O, N, 128, **(dict(kind=O.FZP_PHASE, levels=levels) if levels else {}))
    with _plan(fzp, g, form, levels=levels, stripe_rows=512) as plan:
        for a, b in [(0, N), (g.c + 5, N - 20), (10, g.c - 1), (g.c - 30, g.c + 99)]:
            U, _ = run_plan(fzp, torch, plan, g.M, a, b)
            assert rel_l2(U, O.field_czt(g, a, b)) <= (1e-5 if form == "fp32" else 1e-10), (a, b)


@pytest.mark.parametrize("kind", ["negative", "positive", "L2", "L4"])
@pytest.mark.parametrize("N", [63, 2047, 9001])
def test_masks_and_fields_of_every_rule(env, kind, N):
    """Every mask rule of the generators, bit for bit through the export, and
    the whole field, chunked rows included (N = 9001 in chunks of 1024)."""
    fzp, torch, O = env
    levels = {"L2": 2, "L4": 4}.get(kind, 0)
    okw = dict(kind=O.FZP_PHASE, levels=levels) if levels else dict(kind=O.FZP_POSITIVE) if kind == "positive" else {}
    g = _geom(O, N, 128, **okw)
    with _plan(fzp, g, levels=levels, centre_open=int(kind == "positive"), stripe_rows=1024) as plan:
        for a, b in [(0, min(N, 70)), (g.c - 20, g.c + 21), (N - 9, N)]:
            out = torch.empty((b - a, N), dtype=torch.uint8, device="cuda")
            plan.aperture_mask(a, b, out)
            torch.cuda.synchronize()
            assert np.array_equal(out.cpu().numpy(), O.mask_rows(g, a, b)), (a, b)
        _, I = run_plan(fzp, torch, plan, g.M, 0, N)
        assert rel_l2(I, np.abs(O.field_czt(g)) ** 2) <= TOL


@pytest.mark.parametrize("cluster", [0, 1])
def test_coarse_pitch_keeps_the_general_kernel(env, cluster):
    """Sixteen times the usual pitch on a 1024^2 ROI: no node count holds the
    band, so the cluster kernels and, with one CTA, the row walker run."""
    fzp, torch, O = env
    g = _geom(O, 1501, 1024, pitch=LAM * 5 / 2)
    with _plan(fzp, g, cluster=cluster) as plan:
        assert plan.info["cluster"] == (cluster or 4)
        out = torch.empty((g.N, g.N), dtype=torch.uint8, device="cuda")
        plan.aperture_mask(0, g.N, out)
        torch.cuda.synchronize()
        assert np.array_equal(out.cpu().numpy(), O.mask_rows(g, 0, g.N))
        _, I = run_plan(fzp, torch, plan, g.M, 0, g.N)
        assert rel_l2(I, np.abs(O.field_czt(g)) ** 2) <= TOL


@pytest.mark.parametrize("M,N", [(64, 301), (128, 2001), (256, 2047), (256, 9001)])
def test_membranes_in_one_pass(env, M, N):
    """Deformed membranes: both masks of a pass, 0 and 3 ridges, uneven rows."""
    fzp, torch, O = env
    for ridges in ((), ((1e-4, -2e-4, 0.4, 6e-8, 3e-4), (0.0, 1e-4, 2.0, 5e-8, 4e-4), (2e-4, 0.0, 1.1, 3e-8, 5e-4))):
        d = dict(amp=1.2e-7, period=1.1e-3, theta=0.7, taper=0.4, ridges=ridges)
        g = _geom(O, N, M, deform=O.Deform(**d))
        with _plan(fzp, g, deform=fzp.make_deform(**d)) as plan:
            for a, b in [(0, N), (g.c - 40, N - 30)]:
                U, _ = run_plan(fzp, torch, plan, M, a, b)
                assert rel_l2(U, O.field_czt(g, a, b)) <= TOL, (len(ridges), a, b)
