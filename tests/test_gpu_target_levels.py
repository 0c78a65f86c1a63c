"""Levels of the surrogate's targets relative to their own size: taps next to 0 dB (one
strong path among weak ones), at both ends of the range and around the factors of
sqrt 2 at which the logarithm's reduction changes, against numpy on the same gains in
FP64.

Tolerance: the rounding to FP32 (6e-8), the double-float logarithm (2^-36) and the
FP64 rounding of the sum of powers, 2^-53 over the part that the tap lacks of it
(1e-6 at least: 1.2e-10): 6.1e-8 of the value.
"""
import numpy as np
import pytest
import torch

import scenes

pytestmark = pytest.mark.gpu
C0 = 299792458.0


@pytest.mark.parametrize("level", [1e-6, 1e-4, 1e-2, 0.3, 0.41421, 0.41422, 1.0, 2.4142, 30.0])
@pytest.mark.parametrize("scale", [1.0, 1e-6, 1e-18])
def test_levels_relative_to_their_size(level, scale):
    import paper_2208_10006_gb300 as sbr
    sc = scenes.shoebox(N=60, K=2, n_rx=4)
    r = sbr.run_scene(sc)
    ex = {k: v.cpu().numpy() for k, v in r["export"].items()}
    n, F, taps, tap_s, floor = r["paths"].n, 5, 32, 1.5e-9, -90.0
    rng = np.random.default_rng(int(1e7 * level))
    g = np.empty((n, F), np.complex64)
    for q in range(4):
        on = np.flatnonzero(ex["rx"] == q)
        # the first path against all others together: 1 to `level` in power
        p = rng.uniform(0.5, 1.0, (len(on), F))
        p[1:] *= level / p[1:].sum(0)
        p[0] = 1.0
        g[on] = scale * np.sqrt(p) * np.exp(2j * np.pi * rng.uniform(size=p.shape))
    t = sbr.surrogate_targets(r["paths"], torch.as_tensor(g, device="cuda"), F, taps, tap_s, floor).cpu().numpy().astype(np.float64)
    for q in range(4):
        on = ex["rx"] == q
        pw = g[on].real.astype(np.float64) ** 2 + g[on].imag.astype(np.float64) ** 2
        tau = ex["L"][on] / C0
        b = np.floor((tau - tau.min()) / tap_s)
        tot = pw.sum(0)
        want = np.full((F, 2 + taps), floor)
        want[:, 0] = -10 * np.log10(tot)
        for k in range(taps):
            v = pw[b == k].sum(0)
            if v.any():
                # log1p of what the tap lacks: exact next to 0 dB
                want[:, 2 + k] = np.maximum(10 / np.log(10) * np.log1p(-(pw[b != k].sum(0) / tot)) if (v > 0.5 * tot).all()
                                            else 10 * np.log10(v / tot), floor)
        off = np.abs(t[q][:, 2:] - want[:, 2:])
        assert (off <= 6.1e-8 * np.abs(want[:, 2:])).all(), (q, (off / np.abs(want[:, 2:])).max())
        if scale != 1.0:   # (at 1 the total itself is next to 0 dB, where a sum in another order differs)
            assert (np.abs(t[q][:, 0] - want[:, 0]) <= 6.1e-8 * np.abs(want[:, 0])).all()
