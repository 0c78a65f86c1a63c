"""CUDA-core synthesis with elements far from their array's reference: delays of 2^18
to 2^25 turns, on both sides of the 2^19 at which the phase is reduced in another
way, against the oracle's FP64 sum over the same path list.

Tolerance, of the sum of the path magnitudes: an element delay to 2^-46 of the
distance and its product with f / c to 2^-45 (d, f, at 2^25 turns: 2e-6 of a turn,
1e-5 rad), the FP32 phase, sine and cosine 4e-7 and the FP32 sum. The
FP64 form is below the same bound.
"""
import numpy as np
import pytest

import oracle
import scenes
from parity import to_numpy

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("metres", [260.0, 520.0, 530.0, 1e3, 5e3, 3e4])   # 300 GHz: 1000 turns a metre
@pytest.mark.parametrize("form", ["reference", "elements"])
def test_far_elements(form, metres):
    import paper_2208_10006_gb300 as sbr
    rng = np.random.default_rng(int(metres))
    sc = scenes.shoebox(N=60, K=2, n_rx=2)
    r = sbr.run_scene(sc)
    ex = to_numpy(r["export"])
    f = 300e9 + np.arange(3) * 1.37e9
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    te = np.asarray(sc["tx"], np.float64) + metres * rng.uniform(0.98, 1.02, (5, 1)) * np.array([0.6, 0.0, 0.8])
    n = r["paths"].n
    g = ((rng.normal(size=(n, 3)) + 1j * rng.normal(size=(n, 3))) * 1e-4).astype(np.complex64)
    turns = 1.03 * metres * f.max() / 299792458.0
    tol = 2 * np.pi * turns * 2.0 ** -44 + 2e-6
    G = torch.as_tensor(g, device="cuda")
    for p in (sbr.SYNTH_FP32, sbr.SYNTH_FP64):
        if form == "elements":
            H = sbr.synthesize_H_elements(r["paths"], G, dev(f), dev(te), p).cpu().numpy()
            Ho = oracle.synth_H_elements(ex, g.astype(np.complex128), f, sc["tx"], te, sc["rx"])
        else:
            on = ex["rx"] == 1
            re = np.asarray(sc["rx"], np.float64)[1] + np.array([[0, 0, 0], [0, 2.5e-3, 0]])
            H = sbr.synthesize_H(r["paths"], G, dev(f), dev(te), dev(re), 1, p).cpu().numpy()
            Ho = oracle.synth_H({k: v[on] for k, v in ex.items()}, g[on].astype(np.complex128), f, sc["tx"], sc["rx"][1], te, re, rx_index=1)
        scale = np.abs(g).sum(0).max()
        assert np.abs(H - Ho).max() < tol * scale, (p, np.abs(H - Ho).max() / scale, tol)
