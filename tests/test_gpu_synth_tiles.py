"""CUDA-core synthesis at the edges of its tiles (8, 16, 32 and 64 receive rows,
64 transmit columns, 16 paths, 16 frequencies), on equally spaced and irregular
frequency grids, against the oracle's FP64 sum over the same path list.

Tolerances, of max |H|: FP32 2e-6 (phases in double-float, their sine and
cosine and the sum of some 60 terms in FP32); FP64 form 1e-7, the rounding of H to
FP32 (6e-8) and of its gains.
"""
import numpy as np
import pytest

import oracle
import scenes
from parity import to_numpy

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbr():
    import paper_2208_10006_gb300 as m
    return m


@pytest.fixture(scope="module")
def room(sbr):
    sc = scenes.shoebox(N=60, K=3, n_rx=3)   # 60-odd paths per receiver
    return sc, sbr.run_scene(sc)


def dev(a):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=torch.float64, device="cuda")


def grid(F, spacing):
    if spacing == "even":
        return 60e9 + (np.arange(F) - F // 2) * 20e6
    return np.sort(np.random.default_rng(F).uniform(55e9, 65e9, F))


def gains(n, F):
    rng = np.random.default_rng(n * F)
    return ((rng.normal(size=(n, F)) + 1j * rng.normal(size=(n, F))) * 1e-4).astype(np.complex64)


@pytest.mark.parametrize("Nr", [1, 8, 9, 16, 17, 33, 64, 65])
@pytest.mark.parametrize("Nt,F,spacing", [(1, 1, "even"), (63, 3, "odd"), (65, 2, "even"), (200, 1, "odd")])
def test_reference_point_tiles(sbr, room, Nr, Nt, F, spacing):
    sc, r = room
    f = grid(F, spacing)
    te, re = scenes.upa_yz(sc["tx"], Nt, 1, 2.5e-3), scenes.ula_y(sc["rx"][1], Nr, 2.5e-3)
    g = gains(r["paths"].n, F)
    ex = to_numpy(r["export"])
    on = ex["rx"] == 1
    paths = {k: v[on] for k, v in ex.items()}
    Ho = oracle.synth_H(paths, g[on].astype(np.complex128), f, sc["tx"], sc["rx"][1], te, re, rx_index=1)
    for precision, tol in ((sbr.SYNTH_FP32, 2e-6), (sbr.SYNTH_FP64, 1e-7)):
        H = sbr.synthesize_H(r["paths"], torch.as_tensor(g, device="cuda"), dev(f), dev(te), dev(re), 1, precision).cpu().numpy()
        assert np.abs(H - Ho).max() < tol * np.abs(Ho).max(), (precision, np.abs(H - Ho).max() / np.abs(Ho).max())


@pytest.mark.parametrize("F", [1, 7, 8, 9, 15, 16, 17, 33])
@pytest.mark.parametrize("Nt", [1, 33, 257])
@pytest.mark.parametrize("spacing", ["even", "odd"])
def test_per_element_tiles(sbr, room, F, Nt, spacing):
    sc, r = room
    f = grid(F, spacing)
    te = scenes.upa_yz(sc["tx"], Nt, 1, 2.5e-3)
    g = gains(r["paths"].n, F)
    Ho = oracle.synth_H_elements(to_numpy(r["export"]), g.astype(np.complex128), f, sc["tx"], te, sc["rx"])
    for precision, tol in ((sbr.SYNTH_FP32, 2e-6), (sbr.SYNTH_FP64, 1e-7)):
        H = sbr.synthesize_H_elements(r["paths"], torch.as_tensor(g, device="cuda"), dev(f), dev(te), precision).cpu().numpy()
        assert np.abs(H - Ho).max() < tol * np.abs(Ho).max(), (precision, np.abs(H - Ho).max() / np.abs(Ho).max())


def test_per_element_steps_of_many_turns(sbr, room):
    # equally spaced, but a step turns the phase by more than 1/16 cycle at the far elements
    sc, r = room
    f = 60e9 + np.arange(20) * 1.7e9
    te = scenes.upa_yz(sc["tx"], 40, 1, 2.5e-2)
    g = gains(r["paths"].n, 20)
    Ho = oracle.synth_H_elements(to_numpy(r["export"]), g.astype(np.complex128), f, sc["tx"], te, sc["rx"])
    H = sbr.synthesize_H_elements(r["paths"], torch.as_tensor(g, device="cuda"), dev(f), dev(te), sbr.SYNTH_FP32).cpu().numpy()
    assert np.abs(H - Ho).max() < 2e-5 * np.abs(Ho).max()   # an aperture of 1 m: phases of 60 cycles in FP32
