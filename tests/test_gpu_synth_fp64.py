"""The FP64 form of H(f) entry by entry, where the paths cancel to 1e-7 of their sum
of magnitudes and where gains are near the lower end of the FP32 range, against the
oracle's FP64 sum over the same path list.

Tolerance of an entry: its rounding to FP32 (6e-8, or half of the smallest FP32
number) and the FP64 rounding of phases of at most `turns` turns in either sum (2 pi
turns 2^-51) of the paths' magnitudes.
"""
import numpy as np
import pytest

import oracle
import scenes
from parity import to_numpy

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("scale", [1e-4, 1e-30, 1e-36])
@pytest.mark.parametrize("Nr,Nt,F", [(1, 1, 1), (3, 70, 2), (9, 5, 40), (17, 64, 3)])
def test_entries_that_cancel(scale, Nr, Nt, F):
    import paper_2208_10006_gb300 as sbr
    rng = np.random.default_rng([Nr, Nt, F])
    sc = scenes.shoebox(N=60, K=3, n_rx=2)
    r = sbr.run_scene(sc)
    ex = to_numpy(r["export"])
    f = 60e9 + np.arange(F) * 20e6
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    te, re = scenes.upa_yz(sc["tx"], Nt, 1, 2.5e-3), scenes.ula_y(sc["rx"][1], Nr, 2.5e-3)
    n, on = r["paths"].n, ex["rx"] == 1
    g = ((rng.normal(size=(n, F)) + 1j * rng.normal(size=(n, F))) * scale).astype(np.complex64)
    paths = {k: v[on] for k, v in ex.items()}
    last = np.flatnonzero(on)[-1]
    H = lambda x: oracle.synth_H(paths, x[on].astype(np.complex128), f, sc["tx"], sc["rx"][1], te, re, rx_index=1)
    # the last path takes the sum of the others away at the last receive and the first transmit element
    one, rest = np.zeros_like(g), g.copy()
    one[last], rest[last] = 1.0, 0.0
    g[last] = (-H(rest)[:, -1, 0] / H(one)[:, -1, 0]).astype(np.complex64)
    Ho = H(g)
    mag = np.abs(g[on].astype(np.complex128)).sum(0)[:, None, None]
    assert (np.abs(Ho[:, -1, 0]) < 1e-6 * mag[:, 0, 0]).all()
    got = sbr.synthesize_H(r["paths"], torch.as_tensor(g, device="cuda"), dev(f), dev(te), dev(re), 1, sbr.SYNTH_FP64).cpu().numpy()
    turns = ex["L"][on].max() * f.max() / 299792458.0
    tol = 9e-8 * np.abs(Ho) + 2e-45 + 2 * np.pi * turns * 2.0 ** -51 * mag
    assert (np.abs(got - Ho) <= tol).all(), (np.abs(got - Ho) / tol).max()
