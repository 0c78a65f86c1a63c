"""Path gains over the range of materials and the surrogate's targets over
ragged frequency and tap counts.

Gains, against the oracle (FP64): the result is rounded to FP32 (6e-8); the
double-float arithmetic (2^-44, 6e-14) can be amplified by the cancellation of
the co-polar projection, to 1e-5 of the field at most: 6e-9. Bound: 1e-6 of each
gain, plus one unit of the smallest FP32 number. Targets, against numpy on the
same gains in FP64: FP32 rounding of the results (6e-8) and at most 1e-8 dB from
the logarithms; bound 1e-6 of the value plus 1e-6.
"""
import numpy as np
import pytest
import torch

import oracle
import scenes

pytestmark = pytest.mark.gpu
C0 = 299792458.0


@pytest.fixture(scope="module")
def sbr():
    import paper_2208_10006_gb300 as m
    return m


@pytest.mark.parametrize("sigma", [0.0, 0.01, 1e4, 1e10, 1e17])   # 1e17 S/m: |eta| beyond 1e15, the FP64 form
@pytest.mark.parametrize("rough", [0.0, 1e-4, 1e-3, 0.05])          # 0.05 m: the roughness factor underflows
def test_gains_over_materials(sbr, sigma, rough):
    sc = scenes.shoebox(N=60, K=3)
    sc["materials"] = np.array([[5.31, sigma, rough], [1.0, sigma, rough], [3.0, 10 * sigma, rough]] * 2)
    sc["freqs"] = np.array([1e9, 60e9, 300e9])
    sc["gamma_db_km"] = np.array([0.0, 15.0, 5.0], np.float32)
    sc["disp_deg_km"] = np.array([0.0, 1e3, -1e6], np.float32)
    r = sbr.run_scene(sc)
    ex = {k: v.cpu().numpy() for k, v in r["export"].items()}
    o = oracle.run(sc)
    key = lambda p, i: (int(p["rx"][i]), tuple(p["seq"][i][: p["nb"][i]]))
    at = {key(o["paths"], i): i for i in range(len(o["paths"]["rx"]))}
    g = r["g"].cpu().numpy()
    assert len(at) == len(g) > 60
    go = o["g"][[at[key(ex, i)] for i in range(len(g))]]
    if sigma == 0.0:   # surfaces 1 and 4 are those of a vacuum: they reflect exactly nothing, where the oracle leaves FP64 rounding
        go[[any(s in (1, 4) for s in ex["seq"][i][: ex["nb"][i]]) for i in range(len(g))]] = 0.0
    assert (np.abs(g - go) <= 1e-6 * np.abs(go) + 2e-45).all(), np.nanmax(np.abs(g - go) / np.abs(go))


@pytest.mark.parametrize("gamma", [0.0, 3e2, 3e4])   # dB/km: absorption exponents to 0, 0.1 and 10 a path
@pytest.mark.parametrize("rough", [0.0, 2e-4])
def test_gains_round_as_in_fp64(sbr, gamma, rough):
    """The delay and angle statistics are FP64 sums over the gains, so the gains have to
    be the FP32 rounding of the exact value: double-float errors (2^-42 with the
    cancellations of most paths) move 2^-17 of the parts to the neighbouring number.
    Bound: 1e-3 of them (an exponential in FP32 terms moves several in a hundred)."""
    sc = scenes.shoebox(N=60, K=3)
    sc["materials"] = np.array([[5.31, 0.1, rough], [2.0, 0.01, rough], [3.0, 1.0, rough]] * 2)
    sc["freqs"] = np.geomspace(1e9, 300e9, 64)
    sc["gamma_db_km"] = np.full(64, gamma, np.float32)
    sc["disp_deg_km"] = np.zeros(64, np.float32)
    r = sbr.run_scene(sc)
    ex = {k: v.cpu().numpy() for k, v in r["export"].items()}
    o = oracle.run(sc)
    key = lambda p, i: (int(p["rx"][i]), tuple(p["seq"][i][: p["nb"][i]]))
    at = {key(o["paths"], i): i for i in range(len(o["paths"]["rx"]))}
    g = r["g"].cpu().numpy()
    go = o["g"][[at[key(ex, i)] for i in range(len(g))]].astype(np.complex64)
    parts, want = g.view(np.float32), go.view(np.float32)
    assert parts.size > 2 * 60 * 64
    assert (parts != want).mean() <= 1e-3, (parts != want).mean()


@pytest.mark.parametrize("F", [1, 2, 5, 8, 31, 33])
@pytest.mark.parametrize("n_taps", [1, 7, 32])
def test_targets_over_ragged_sizes(sbr, F, n_taps):
    sc = scenes.shoebox(N=60, K=3, n_rx=5)   # 63 paths a receiver: two chunks of 32
    r = sbr.run_scene(sc)
    pl, ex = r["paths"], {k: v.cpu().numpy() for k, v in r["export"].items()}
    rng = np.random.default_rng(F)
    g = (rng.normal(size=(pl.n, F)) + 1j * rng.normal(size=(pl.n, F))) * 10.0 ** rng.uniform(-25, -3, (pl.n, 1))
    g = g.astype(np.complex64)
    tap_s, floor = 3e-9, -40.0
    t = sbr.surrogate_targets(pl, torch.as_tensor(g, device="cuda"), F, n_taps, tap_s, floor).cpu().numpy()
    for q in range(5):
        on = ex["rx"] == q
        assert on.sum() > 32
        pw = np.abs(g[on].astype(np.complex128)) ** 2
        tau = ex["L"][on] / C0
        tau = tau - tau.min()
        tot = pw.sum(0)
        mean = (pw * tau[:, None]).sum(0) / tot
        want = np.full((F, 2 + n_taps), floor)
        want[:, 0] = -10 * np.log10(tot)
        want[:, 1] = np.sqrt(np.maximum((pw * (tau ** 2)[:, None]).sum(0) / tot - mean ** 2, 0)) * 1e9
        for k in range(n_taps):
            v = pw[np.floor(tau / tap_s) == k].sum(0)
            with np.errstate(divide="ignore"):
                want[:, 2 + k] = np.maximum(10 * np.log10(v / tot), floor)
        got = t[q].astype(np.float64)
        got[:, 1] *= 1e9
        # the spread is a difference of moments: its FP64 error is 1e-16 tau^2 before the root
        assert np.abs(got - want).max() <= 1e-6 * np.abs(want).max() + 1e-6, (q, np.abs(got - want).max())
