"""The fixed-point zone phase of the node form's mask generators, emulated on
the CPU in the kernel's integer steps: along 32-column blocks carried from
block to block, a sample whose 32-bit phase keeps its distance E from the zone
boundaries has exactly the zone parity (or level) of the threshold table."""
import math

import numpy as np
import pytest

import paper_2609_01978_gb300 as fzp

M64 = (1 << 64) - 1
LAM = 632.8e-9


def _walk(K, dj, di0, blocks):
    """(column, 32-bit phase) of `blocks` blocks from di0 (block_words)."""
    phase, step = ((dj * dj + di0 * di0) * K) & M64, ((2 * di0 + 1) * K) & M64
    c2 = ((K >> 32) * 2 + ((K >> 31) & 1)) & 0xFFFFFFFF
    out = []
    for b in range(blocks):
        f, d = phase >> 32, step >> 32
        for k in range(32):
            out.append((di0 + 32 * b + k, f))
            f, d = (f + d) & 0xFFFFFFFF, (d + c2) & 0xFFFFFFFF
        phase, step = (phase + 32 * step + 992 * K) & M64, (step + 64 * K) & M64
    return out


@pytest.mark.parametrize("D,levels", [(4e-3, 0), (0.25, 0), (5.0, 0), (5.0, 2), (0.05, 4), (3.0, 4)])
def test_walk_agrees_with_the_threshold_table(D, levels):
    kw = dict(D=D, f=5 * D, lam=LAM, M=64, pitch=LAM * 5 / 8, levels=levels)
    info = fzp.plan_query(**kw)
    S = fzp.zone_thresholds(**kw)
    c, sR = info["c"], info["s_R"]
    lev = levels if levels > 2 else 2
    kappa = info["kappa"] * (0.5 * levels if levels >= 2 else 1.0)
    K = math.floor(math.ldexp(kappa / levels, 64)) if levels > 2 else math.floor(math.ldexp(kappa, 63))
    E = 640 + (sR >> 32)
    rng = np.random.default_rng(7)
    sampled = near = 0
    for _ in range(60):
        dj = int(rng.integers(0, c + 1))
        chord = math.isqrt(max(sR - dj * dj, 0))
        di0 = int(rng.integers(-chord, chord + 1))
        for di, f in _walk(K, dj, di0, 6):
            s = dj * dj + di * di
            if s > sR:
                continue
            zone = int(np.searchsorted(S, s, side="right"))  # #{m : S_m <= s}
            p = f * lev
            frac = p & 0xFFFFFFFF
            sampled += 1
            if (frac + E * lev) & 0xFFFFFFFF < 2 * E * lev:
                near += 1
                continue
            assert p >> 32 == zone % lev, (dj, di, zone)
    assert sampled > 5000 and near < sampled / 100
