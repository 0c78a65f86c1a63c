"""Squares below the normal FP32 range in double-float arithmetic: grazing incidence
on a surface like air, and array elements closer to each other than 1e-19 m.
"""
import numpy as np
import pytest

import oracle

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbr():
    import paper_2208_10006_gb300 as m
    return m


def dev(a, dtype=torch.float64):
    return torch.as_tensor(np.ascontiguousarray(a), dtype=dtype, device="cuda")


def floor_paths(sbr, tx, rx, nb):
    """Paths of one receiver over a floor: line of sight (nb 0) or its reflection (nb 1)."""
    tri = np.array([[-50, -50, 0, 50, -50, 0, 50, 50, 0], [-50, -50, 0, 50, 50, 0, -50, 50, 0]], np.float32)
    bvh = sbr.build_bvh(dev(tri, torch.float32), dev([0, 0], torch.int32), 1)
    keys = np.full((1, 10), -1, np.int64)
    keys[0, :2] = 0, nb
    if nb:
        keys[0, 2] = 0
    tr = sbr.trace_merge(list(tx), dev([rx]), 60, 1, dev(keys, torch.int32), dev([0], torch.int64))
    return bvh, sbr.paths(tr, bvh)


@pytest.mark.parametrize("h", [1e-11, 1e-10, 2e-10])   # cos of incidence h / 1.8
def test_grazing_incidence_on_air(sbr, h):
    """eps_r = 1, no loss, cos^2 far below FP64's resolution of 1: the FP64 formula has
    sin^2 = 1, a zero root and both coefficients 1, which the gain is expected to be."""
    tx, rx = (1.0, 7.0, h), (2.0, 10.5, h)
    bvh, pl = floor_paths(sbr, tx, rx, 1)
    assert pl.n == 1
    f, L = np.array([1e9, 60e9]), np.linalg.norm(np.subtract(rx, tx))
    g = sbr.path_gains(pl, dev([[1.0, 0.0, 0.0]]), dev(f), None, None, sbr.POL_H).cpu().numpy()[0]
    assert np.abs(np.abs(g) - 299792458.0 / (4 * np.pi * f * L)).max() < 1e-6 * np.abs(g).max(), g


@pytest.mark.parametrize("gap", [1e-20, 1e-22])
def test_elements_that_nearly_coincide(sbr, gap):
    # a transmit element at the origin, receive elements there and a gap away: the same H
    tx, rx = (0.0, 0.0, 0.0), (2.0, 0.0, 1.0)
    bvh, pl = floor_paths(sbr, (0.0, 0.0, 0.0), rx, 0)
    assert pl.n == 1
    f = dev([60e9, 61e9])
    g = torch.full((1, 2), 1e-4 + 2e-4j, dtype=torch.complex64, device="cuda")
    te, re = dev([tx, (0.0, 0.001, 0.0)]), dev([(0.0, 0.0, 0.0), (0.0, 0.0, gap)])
    for p in (sbr.SYNTH_FP64, sbr.SYNTH_FP32, sbr.SYNTH_FP16X3, sbr.SYNTH_BF16X3):
        H = sbr.synthesize_H(pl, g, f, te, re, 0, p).cpu().numpy()
        assert np.isfinite(H).all() and np.abs(H[:, 0] - H[:, 1]).max() <= 1e-7 * np.abs(H).max(), (p, H)
