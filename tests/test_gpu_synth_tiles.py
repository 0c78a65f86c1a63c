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


@pytest.mark.parametrize("K", [0, 1, 2, 3])   # paths: LoS alone, one K-step, one chunk and more than a chunk of 32
@pytest.mark.parametrize("Nr,Nt,F", [(1, 1, 1), (7, 15, 3), (8, 17, 2), (63, 255, 2), (64, 256, 3), (65, 257, 2), (64, 514, 160), (130, 30, 200)])
def test_tensor_core_tiles(sbr, K, Nr, Nt, F):
    """Both tensor-core forms against the oracle. Per term: three FP32 roundings of a
    phase of at most `cycles` (delay, f / c, product), the hardware sine and cosine
    (1e-6 each) and the dropped lo-lo products (2^-22 FP16, 2^-16 BF16); bound: that,
    times the sum of the path magnitudes."""
    sc = scenes.shoebox(N=60, K=K, n_rx=2)
    r = sbr.run_scene(sc)
    f = grid(F, "odd")
    te, re = scenes.upa_yz(sc["tx"], Nt, 1, 2.5e-3), scenes.ula_y(sc["rx"][1], Nr, 2.5e-3)
    g = gains(r["paths"].n, F)
    ex = to_numpy(r["export"])
    on = ex["rx"] == 1
    paths = {k: v[on] for k, v in ex.items()}
    Ho = oracle.synth_H(paths, g[on].astype(np.complex128), f, sc["tx"], sc["rx"][1], te, re, rx_index=1)
    aperture = np.linalg.norm(te - sc["tx"], axis=1).max() + np.linalg.norm(re - sc["rx"][1], axis=1).max()
    phase = 3 * 2 * np.pi * aperture * f.max() / 299792458.0 * 2.0 ** -24
    scale = np.abs(g[on]).sum(0).max()
    for precision, split in ((sbr.SYNTH_FP16X3, 2.0 ** -20), (sbr.SYNTH_BF16X3, 2.0 ** -14)):
        H = sbr.synthesize_H(r["paths"], torch.as_tensor(g, device="cuda"), dev(f), dev(te), dev(re), 1, precision).cpu().numpy()
        assert np.abs(H - Ho).max() < (phase + 4e-6 + split) * scale, (precision, np.abs(H - Ho).max() / scale)


@pytest.mark.parametrize("form,Nt", [("reference", 65535 * 64 + 100), ("elements", 65535 * 256 + 100)])
def test_more_columns_than_one_grid(sbr, form, Nt):
    """Arrays past the 65,535 column blocks of one launch: the last elements and those
    around the seam against a call with these alone (the same terms, summed in another
    order of path groups: 1e-6 of max |H|)."""
    sc = scenes.shoebox(N=40, K=1, n_rx=1)
    r = sbr.run_scene(sc)
    n = r["paths"].n
    assert 1 <= n <= 7
    f = grid(1, "even")
    g = torch.as_tensor(gains(n, 1), device="cuda")
    te = torch.zeros((Nt, 3), dtype=torch.float64, device="cuda") + torch.as_tensor(np.asarray(sc["tx"], np.float64), device="cuda")
    te[:, 1] += torch.linspace(-0.2, 0.2, Nt, dtype=torch.float64, device="cuda")
    seam = Nt - 100
    pick = torch.cat([torch.arange(0, 64), torch.arange(seam - 64, Nt)]).cuda()
    if form == "reference":
        call = lambda t: sbr.synthesize_H(r["paths"], g, dev(f), t, dev(np.asarray(sc["rx"])[:1]), 0, sbr.SYNTH_FP32)
    else:
        call = lambda t: sbr.synthesize_H_elements(r["paths"], g, dev(f), t, sbr.SYNTH_FP32)
    big, small = call(te.contiguous()), call(te[pick].contiguous())
    assert (big[..., pick] - small).abs().max() <= 1e-6 * small.abs().max() and small.abs().max() > 0
