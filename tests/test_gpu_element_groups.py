"""Per-element synthesis of few elements: blocks whose groups of threads share the
paths of an element (8, 4 and 2 groups by the number of elements and frequencies,
none above), with receivers of no path, of fewer paths than groups and of more than
one chunk of 64, against the oracle's FP64 sum over the same path list.

Tolerance, of max |H|: 2e-6, as for the other FP32 forms (phases in double-float,
their sine and cosine and the sum of up to some 130 terms in FP32).
"""
import numpy as np
import pytest

import oracle
import scenes
from parity import to_numpy

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K,n_rx,F,Nt", [(1, 3, 8, 1), (4, 3, 17, 65), (1, 200, 20, 3), (4, 200, 50, 2), (4, 200, 100, 2), (4, 200, 200, 2)])
def test_groups_of_paths(K, n_rx, F, Nt):
    import paper_2208_10006_gb300 as sbr
    rng = np.random.default_rng([K, F])
    sc = scenes.shoebox(N=60, K=K, n_rx=n_rx)
    sc["rx"] = np.asarray(sc["rx"], np.float64).copy()
    sc["rx"][0] = (500.0, 500.0, 500.0)   # outside the room: no path
    r = sbr.run_scene(sc)
    f = 60e9 + (np.arange(F) - F // 2) * 20e6
    te = scenes.upa_yz(sc["tx"], Nt, 1, 2.5e-3)
    n = r["paths"].n
    g = ((rng.normal(size=(n, F)) + 1j * rng.normal(size=(n, F))) * 1e-4).astype(np.complex64)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    Ho = oracle.synth_H_elements(to_numpy(r["export"]), g.astype(np.complex128), f, sc["tx"], te, sc["rx"])
    H = sbr.synthesize_H_elements(r["paths"], torch.as_tensor(g, device="cuda"), dev(f), dev(te), sbr.SYNTH_FP32).cpu().numpy()
    assert (H[:, 0] == 0).all()
    assert np.abs(H - Ho).max() < 2e-6 * np.abs(Ho).max(), np.abs(H - Ho).max() / np.abs(Ho).max()


@pytest.mark.parametrize("F,Nt", [(64, 7), (220, 7), (128, 40)])
def test_error_of_few_paths(F, Nt):
    """Per-element FP32 synthesis of 7 paths against FP64, 2-norm. Per term, rms: weight 2e-8,
    the middle frequency's phasor 5e-8, 1.6 rotations on average of 4e-8 each, product and
    sum 4e-8: 8.5e-8 together; bound 1e-7 (as with a sine and a cosine per term)."""
    import paper_2208_10006_gb300 as sbr
    rng = np.random.default_rng([F, Nt])
    sc = scenes.shoebox(N=60, K=1, n_rx=40)
    r = sbr.run_scene(sc)
    f = 100e9 + (np.arange(F) - F // 2) * (10e9 / F)
    te = scenes.upa_yz(sc["tx"], Nt, 1, 1.5e-3)
    n = r["paths"].n
    g = ((rng.normal(size=(n, F)) + 1j * rng.normal(size=(n, F))) * 1e-4).astype(np.complex64)
    dev = lambda a: torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")
    Ho = oracle.synth_H_elements(to_numpy(r["export"]), g.astype(np.complex128), f, sc["tx"], te, sc["rx"])
    H = sbr.synthesize_H_elements(r["paths"], torch.as_tensor(g, device="cuda"), dev(f), dev(te), sbr.SYNTH_FP32).cpu().numpy()
    err = np.linalg.norm(H - Ho) / np.linalg.norm(Ho)
    assert err < 1e-7, err
