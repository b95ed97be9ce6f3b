"""Performance cases of the library: what its users run, through its public entry points.

A case is a plain dict; ``prepare`` makes the plan and the device buffers that a user's program holds
(the plate's parameters come from the seed), ``run`` is one call, ``work`` counts what the call cannot do
without, and ``exact`` evaluates the same outputs in 64 bits from the method's equations, with torch alone.

Fields come back from the library as complex128.  Those of the FP32 and split-BF16 forms are kept as
complex64, the precision their row transform has (the stored fields of this repository are complex64 too);
those of the FP64 form are kept as they are.

Cases are named after the plate's diameter at f/5 and 550 nm; the seed draws the wavelength, the focal ratio
and the ROI pitch around those values and the grid stays the case's N.
"""
import math
import random

import torch

import fzp_inputs
import paper_2609_01978_gb300 as fzp
from paper_2609_01978_gb300 import shard

#: FP64 operations that an exact value may take (about 1 TFLOP/s, at most 20 s)
EXACT_FLOPS = 1.3e13


def listed():
    return [
        # the parity configuration, a whole engine call in FP64: propagate a 4 mm plate, extract the metrics
        dict(name="fp64-4mm", kind="flat", form="fp64", N=5057, M=256, levels=0, shift=0.0),
        # the smallest plates, as the surrogate's test set has them: launches and latency
        dict(name="dense-2mm", kind="flat", form="dense", N=2529, M=128, levels=0, shift=0.0),
        # an ordinary plate, the ROI off the axis (side lobes)
        dict(name="dense-30mm-offaxis", kind="flat", form="dense", N=37929, M=256, levels=0, shift=37.25),
        # the 0.25 m plate on its 512^2 ROI, the whole aperture
        dict(name="dense-250mm", kind="flat", form="dense", N=316057, M=512, levels=0, shift=0.0),
        # the headline plate's share of one of 8 processes (or one row group of a resumable run)
        dict(name="dense-1m-shard", kind="flat", form="dense", N=1264223, M=512, levels=0, shift=0.0, shard=3, shards=8),
        # a 4-level phase plate (Tables 3 and 4) on the dense form: two signed-mask passes
        dict(name="dense-L4", kind="flat", form="dense", N=60001, M=512, levels=4, shift=0.0),
        # the plain FP32 form on the 5 cm plate
        dict(name="fp32-50mm", kind="flat", form="fp32", N=63213, M=512, levels=0, shift=0.0),
        # a 16-level phase plate (Table 1), which the plain FP32 form runs in one pass
        dict(name="fp32-L16", kind="flat", form="fp32", N=50001, M=512, levels=16, shift=0.0),
        # deformed membranes, several apertures in one graph, on the FP32 form ...
        dict(name="membranes-fp32", kind="membranes", form="fp32", N=34567, M=256, count=4),
        # ... and on the dense form, as the surrogate's training set is generated
        dict(name="membranes-dense", kind="membranes", form="dense", N=36363, M=128, count=4),
        # the SA-CZT with the exact zone radii, 8 mm
        dict(name="saczt-8mm", kind="saczt", N=10115, M=512),
        # one batch of the surrogate's training: loss and gradients
        dict(name="surrogate-grad", kind="surrogate", what="grad", batch=256, hidden=512, layers=3, n_out=4114),
    ]


def _odd(rng, lo, hi):
    return 2 * int(math.exp(rng.uniform(math.log(lo), math.log(hi))) / 2) + 1


def draw(rng):
    kind = rng.choice(["fp64", "dense", "dense", "dense", "fp32", "fp32", "membranes", "membranes", "shard", "saczt", "surrogate"])
    shift = rng.choice([0.0, 0.0, 0.0, round(rng.uniform(-120, 120), 2)])
    if kind == "fp64":
        return dict(kind="flat", form="fp64", N=_odd(rng, 1001, 12001), M=rng.choice([64, 128, 256]), levels=0, shift=0.0)
    if kind == "dense":
        levels = rng.choice([0, 0, 0, 2, 4])
        return dict(kind="flat", form="dense", N=_odd(rng, 2001, 220001 if levels > 2 else 316001),
                    M=rng.choice([128, 256, 512, 512]), levels=levels, shift=shift)
    if kind == "fp32":
        return dict(kind="flat", form="fp32", N=_odd(rng, 2001, 120001), M=rng.choice([64, 128, 256, 512, 512]),
                    levels=rng.choice([0, 0, 0, 3, 4, 16]), shift=shift)
    if kind == "membranes":
        form = rng.choice(["fp32", "dense"])
        return dict(kind="membranes", form=form, N=_odd(rng, 3001, 60001), M=rng.choice([128, 256]), count=rng.randint(1, 4))
    if kind == "shard":
        shards = rng.choice([4, 8, 16])
        return dict(kind="flat", form="dense", N=_odd(rng, 300001, 900001), M=512, levels=0, shift=0.0,
                    shard=rng.randrange(shards), shards=shards)
    if kind == "saczt":
        return dict(kind="saczt", N=_odd(rng, 1001, 10921), M=rng.choice([128, 256, 512]))
    return dict(kind="surrogate", what=rng.choice(["grad", "infer"]), batch=8 * rng.randint(1, 64), hidden=512, layers=3, n_out=4114)


# ------------------------------------------------------------------------------------------- plates
def _plate(case, seed):
    """A flat plate's parameters: f/# about 5, the visible range, ROI pitch about lambda f/# / 8, N as given."""
    rng = random.Random(seed)
    lam, fnum = rng.uniform(450e-9, 650e-9), rng.uniform(4.5, 5.5)
    pitch = lam * fnum / 8 * rng.uniform(0.9, 1.1)
    D = (case["N"] - 0.5) * lam * fnum / (2 * max(case.get("levels", 0), 2))  # N = ceil(D / dx) at the default dx
    p = dict(D=D, f=fnum * D, lam=lam, M=case["M"], pitch=pitch)
    if case.get("shift"):
        p["x0"] = -(case["M"] / 2 - case["shift"]) * pitch
    return p


_FORMS = {
    "fp64": dict(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP64),
    "fp32": dict(form=fzp.FORM_BLUESTEIN, precision=fzp.PREC_FP32),
    "dense": dict(form=fzp.FORM_DENSE, precision=fzp.PREC_SPLIT_BF16),
}


def _membranes(case, seed):
    """Seeded deformed membranes (fzp_inputs.batch_draws) on grids up to the case's N."""
    rng = random.Random(seed)
    probs = []
    for k, m in enumerate(fzp_inputs.batch_draws(case["count"], seed)):
        N = 2 * int(case["N"] * (1 - 0.1 * k) / 2) + 1
        fnum = 5.0
        D = (N - 0.5) * m.lam * fnum / 4
        s = D / m.D  # the draw's geometry scaled to the plate
        ridges = [(px * s, py * s, al, h, max(w, 200 * D / N)) for px, py, al, h, w in m.ridges]
        probs.append(dict(D=D, f=fnum * D, lam=m.lam, M=case["M"], pitch=m.lam * fnum / 8 * rng.uniform(0.95, 1.05),
                          deform=dict(amp=m.amp, period=m.period, theta=m.theta, taper=m.taper, ridges=ridges)))
    return probs


def _sizes(case):
    return [8] + [case["hidden"]] * case["layers"] + [case["n_out"]]


def _weights(case, seed):
    """The network's parameters as a user loads them: per layer W (n_out x n_in), then b."""
    g = torch.Generator().manual_seed(seed)
    parts = []
    for a, b in zip(_sizes(case), _sizes(case)[1:]):
        parts += [(torch.rand(a * b, generator=g) * 2 - 1) * math.sqrt(3 / a), torch.rand(b, generator=g) * 0.2 - 0.1]
    return torch.cat(parts)


def _samples(case, seed):
    """Encoded inputs in [-1, 1] and standardised targets."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    x = torch.rand((case["batch"], 8), generator=g, device="cuda") * 2 - 1
    return x, torch.randn((case["batch"], case["n_out"]), generator=g, device="cuda")


def _rows(case, info):
    if "shard" not in case:
        return 0, info["N"]
    # equal shares of the disc's area, as shard.chord_weights gives them, on a coarse grid of rows
    N, coarse = info["N"], 4096
    w = shard.chord_weights(coarse, coarse // 2, (coarse // 2) ** 2)
    a, b = shard.row_ranges(coarse, case["shards"], w)[case["shard"]]
    return N * a // coarse, N * b // coarse


def prepare(case, seed):
    dev = torch.device("cuda")
    if case["kind"] == "surrogate":
        net = fzp.SurrogateNet(n_in=8, hidden=case["hidden"], layers=case["layers"], n_out=case["n_out"], max_batch=case["batch"], seed=seed)
        net.set_params(_weights(case, seed).numpy())
        x, y = _samples(case, seed)
        return dict(case=case, net=net, x=x, y=y, out=torch.empty_like(y), loss=torch.empty(1, device=dev),
                    grad=torch.empty(net.param_count, device=dev))
    if case["kind"] == "membranes":
        probs = [dict(p, deform=fzp.make_deform(**p["deform"])) for p in _membranes(case, seed)]
        form = dict(_FORMS[case["form"]], **({"cluster": 1} if case["form"] == "dense" and case["M"] == 128 else {}))
        batch = fzp.Batch([dict(p, **form) for p in probs])
        return dict(case=case, batch=batch, fields=[torch.empty((case["M"], case["M"]), dtype=torch.complex128, device=dev) for _ in probs])
    if case["kind"] == "saczt":
        plan = fzp.Plan(form=fzp.FORM_SACZT, precision=fzp.PREC_FP32, exact_radii=1, **_plate(case, seed))
    else:
        plan = fzp.Plan(levels=case["levels"], **_FORMS[case["form"]], **_plate(case, seed))
    info = plan.info
    return dict(case=case, plan=plan, rows=_rows(case, info), field=torch.empty((case["M"], case["M"]), dtype=torch.complex128, device=dev))


def run(state):
    case = state["case"]
    if case["kind"] == "surrogate":
        if case["what"] == "infer":
            state["net"].infer(state["x"], state["out"])
            return state["out"]
        state["net"].grad(state["x"], state["y"], grad_out=state["grad"], loss_out=state["loss"])
        return dict(grad=state["grad"], loss=state["loss"])
    if case["kind"] == "membranes":
        state["batch"].propagate(state["fields"])
        return [f.to(torch.complex64) for f in state["fields"]]
    state["plan"].propagate_roi(*state["rows"], state["field"])
    if case.get("form") == "fp64":
        return dict(field=state["field"], metrics=state["plan"].metrics(state["field"]))
    return state["field"].to(torch.complex64)


def work(case):
    """Each sample of the aperture disc enters the sum at least once (a complex multiply-add, 8 operations); what comes
    back is written once.  The SA-CZT also transforms its padded grid forth and back; the surrogate reads its weights."""
    if case["kind"] == "surrogate":
        sizes = _sizes(case)
        params = sum((a + 1) * b for a, b in zip(sizes, sizes[1:]))
        mults = sum(a * b for a, b in zip(sizes, sizes[1:])) * case["batch"]
        io = case["batch"] * (8 + case["n_out"]) * 4
        if case["what"] == "infer":
            return dict(bytes=2 * params + io, flops=2 * mults)
        return dict(bytes=2 * params + 4 * params + io, flops=6 * mults - 2 * 8 * case["hidden"] * case["batch"])
    out = case["M"] ** 2 * 8
    disc = math.pi / 4 * case["N"] ** 2
    if case["kind"] == "membranes":
        share = sum((1 - 0.1 * k) ** 2 for k in range(case["count"]))
        return dict(bytes=out * case["count"], flops=8 * disc * share)
    if case["kind"] == "saczt":
        P = 1 << math.ceil(math.log2(1.5 * case["N"]))
        return dict(bytes=out, flops=8 * disc + 20 * P * P * math.log2(P))
    if case["form"] == "fp64":
        out *= 2
    return dict(bytes=out, flops=8 * disc / case.get("shards", 1))


# ------------------------------------------------------------------------------- 64-bit evaluation
def _cis(turns):
    t = (turns - torch.round(turns)) * (2 * math.pi)
    return torch.complex(torch.cos(t), torch.sin(t))


def _grid(p, levels):
    lf = p["lam"] * p["f"]
    dx = lf / (2.0 * (levels if levels > 2 else 2) * p["D"])
    N = math.ceil(p["D"] / dx)
    N += 1 - N % 2
    R = min(p["D"] / 2, lf / (2 * dx))
    return lf, dx, N, R * R


def _deform_turns(d, u, v, R, lam):
    """2 w / lambda of the membrane, in turns (u, v: columns and rows in metres)."""
    w = d["amp"] * torch.sin(2 * math.pi * (u * math.cos(d["theta"]) + v * math.sin(d["theta"])) / d["period"])
    w = w * (1 - d["taper"] * (u * u + v * v) / (R * R))
    for px, py, al, h, width in d["ridges"]:
        sig = width / (2 * math.sqrt(2 * math.log(2)))
        dist = -(u - px) * math.sin(al) + (v - py) * math.cos(al)
        w = w + h * torch.exp(-dist * dist / (2 * sig * sig))
    return 2 * w / lam


def _exact_field(p, levels, deform=None):
    """Eq. 2 as the separable double sum over the aperture grid (rows in chunks); a flat plate's rows j and 2c - j are equal."""
    dev = torch.device("cuda")
    lf, dx, N, R2 = _grid(p, levels)
    c, M = (N - 1) // 2, p["M"]
    if (2 if deform is None else 4) * (2 if levels or deform else 1) * M * N * N > EXACT_FLOPS:
        return None
    dx2 = dx * dx
    kappa = dx2 / lf
    step = kappa * (0.5 * levels) if levels >= 2 else kappa
    x0 = p.get("x0", -(M // 2) * p["pitch"])
    x = x0 + torch.arange(M, dtype=torch.float64, device=dev) * p["pitch"]
    i = torch.arange(N, dtype=torch.float64, device=dev) - c

    def kern(d):  # e^{i pi u^2 / (lambda f)} e^{-2 pi i x u / (lambda f)}, rows over d
        return _cis((d * d * (0.5 * kappa))[:, None] - (d * (dx / lf))[:, None] * x[None, :])

    K = kern(i)
    Kr, Ki = K.real.contiguous(), K.imag.contiguous()
    U = torch.zeros((M, M), dtype=torch.complex128, device=dev)
    first = c if deform is None else 0
    chunk = max(1, min(2048, int(1e8 / N)))
    for j0 in range(first, N, chunk):
        dj = i[j0:min(N, j0 + chunk)]
        s = dj[:, None] ** 2 + i[None, :] ** 2
        inside = s * dx2 <= R2
        zone = torch.floor(s * step)
        if levels >= 2:
            T = torch.where(inside, _cis(-torch.remainder(zone, levels) / levels), 0)
        else:
            T = (inside & (torch.remainder(zone, 2) == 1)).to(torch.float64)
        if deform is not None:
            T = T * _cis(_deform_turns(deform, i[None, :] * dx, dj[:, None] * dx, math.sqrt(R2), p["lam"]))
        if T.is_complex():
            Tr, Ti = T.real.contiguous(), T.imag.contiguous()
            C = torch.complex(Tr @ Kr - Ti @ Ki, Tr @ Ki + Ti @ Kr)
        else:
            C = torch.complex(T @ Kr, T @ Ki)
        W = kern(dj)
        if deform is None:
            W = torch.where((dj != 0)[:, None], W + kern(-dj), W)
        U += W.T @ C
    return U * _post(p, x, lf, p["f"], dx2 / lf)


def _post(p, x, lz, f, amp):
    q = x * x / (2 * lz)
    return amp * _cis(math.fmod(f / p["lam"], 1.0) - 0.25 + q[:, None] + q[None, :])


def _exact_saczt(p):
    """The angular spectrum on the padded grid, its quadratic part as a Fresnel integral zoomed onto the ROI."""
    dev = torch.device("cuda")
    lf, dx, N, R2 = _grid(p, 0)
    c, M, lam, f = (N - 1) // 2, p["M"], p["lam"], p["f"]
    P = 1
    while P < 1.5 * N:
        P *= 2
    i = torch.arange(N, dtype=torch.float64, device=dev) - c
    s = i[:, None] ** 2 + i[None, :] ** 2
    r2 = s * (dx * dx)
    zone = torch.floor(2 * r2 / (lam * (torch.sqrt(f * f + r2) + f)))
    T = ((r2 <= R2) & (torch.remainder(zone, 2) == 1)).to(torch.complex128)
    del s, r2, zone
    G = torch.zeros((P, P), dtype=torch.complex128, device=dev)
    o = P // 2 - c
    G[o:o + N, o:o + N] = T
    del T
    G = torch.fft.fft2(G)
    k0 = 2 * math.pi / lam
    kmax = 2 * k0 / 3
    d = (math.sqrt(k0 * k0 - kmax * kmax) - k0) / kmax
    kf = 2 * math.pi * torch.fft.fftfreq(P, d=dx, dtype=torch.float64, device=dev)
    for a in range(0, P, 1024):  # in bands of rows: the phase h f / (2 pi) in turns
        K2 = kf[a:a + 1024, None] ** 2 + kf[None, :] ** 2
        kz = torch.sqrt(torch.clamp(k0 * k0 - K2, min=0.0))
        h = -K2 / (k0 + kz) - d * K2 / kmax
        G[a:a + 1024] *= torch.where(K2 < k0 * k0, _cis(h * (f / (2 * math.pi))), 0)
    G = torch.fft.ifft2(G)
    zF = -2 * k0 * d * f / kmax
    lz = lam * zF
    u = (torch.arange(P, dtype=torch.float64, device=dev) - P // 2) * dx
    x = -(M // 2) * p["pitch"] + torch.arange(M, dtype=torch.float64, device=dev) * p["pitch"]
    E = _cis((u * u / (2 * lz))[None, :] - x[:, None] * u[None, :] / lz)
    return (E @ G @ E.T) * _post(p, x, lz, f, dx * dx / lz)


def _exact_surrogate(case, seed):
    vec = _weights(case, seed).to("cuda").double().requires_grad_(True)
    x, y = (t.double() for t in _samples(case, seed))
    sizes, at, h = _sizes(case), 0, x
    for k, (a, b) in enumerate(zip(sizes, sizes[1:])):
        W = vec[at:at + a * b].view(b, a)
        bias = vec[at + a * b:at + a * b + b]
        at += a * b + b
        h = h @ W.T + bias
        if k + 2 < len(sizes):
            h = h * torch.sigmoid(h)
    if case["what"] == "infer":
        return h.detach()
    loss = ((h - y) ** 2).mean()
    loss.backward()
    return dict(grad=vec.grad, loss=loss.detach().reshape(1))


def exact(case, seed):
    if case["kind"] == "surrogate":
        return _exact_surrogate(case, seed)
    if case["kind"] == "membranes":
        return [_exact_field(dict(p), 0, p["deform"]) for p in _membranes(case, seed)]
    p = _plate(case, seed)
    if case["kind"] == "saczt":
        return _exact_saczt(p)
    if "shard" in case:
        return None
    U = _exact_field(p, case["levels"])
    if case["form"] != "fp64" or U is None:
        return U
    # the metrics that are plain sums of I; the widths and the MTF read a spline and radial bins
    lf, dx, N, R2 = _grid(p, 0)
    c, M = (N - 1) // 2, case["M"]
    inten = U.abs() ** 2
    s = (torch.arange(N, dtype=torch.float64, device="cuda") - c) ** 2
    count = sum(int(((s[a:a + 1024, None] + s[None, :]) * (dx * dx) <= R2).sum()) for a in range(0, N, 1024))
    peak = inten[M // 2, M // 2].item()
    disc = math.pi * R2
    metrics = dict(fwhm_x=None, fwhm_y=None, de_lobe=None, de_roi=(inten.sum() * p["pitch"] ** 2 / (count * dx * dx)).item(),
                   p_in=count * dx * dx, p_in_disc=disc, peak=peak, strehl=peak / (disc / lf) ** 2, mtf_half_cut=None,
                   mtf16=None, aperture_count=count)
    return dict(field=U, metrics=metrics)
