"""Capacity at the edges of the factorisation's 16-column blocks, in both
orientations, in double-float and (above about 45 dB) FP64, against the oracle.

Tolerance: an entry of W carries a relative FP32 error of at most 34 units of
2^-24 (2e-6) of the sum of its terms' magnitudes; for matrices whose extreme
eigenvalues differ by the factor 9 of an n x 4n Gaussian channel a logarithm of
an eigenvalue moves by less than 2e-5, of some 20 in a stream at 60 dB: 1e-6 of
C, bounded here by 1e-5 as for the other capacity parity tests.
"""
import numpy as np
import pytest
import torch

import oracle

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def sbr():
    import paper_2208_10006_gb300 as m
    return m


def channel(F, Nr, Nt, seed=0):
    rng = np.random.default_rng(seed)
    return ((rng.normal(size=(F, Nr, Nt)) + 1j * rng.normal(size=(F, Nr, Nt))) / 16).astype(np.complex64)


@pytest.mark.parametrize("n", [1, 2, 15, 16, 17, 31, 32, 33, 47, 48, 49, 63, 64])
@pytest.mark.parametrize("tall", [False, True])
def test_block_edges(sbr, n, tall):
    m = 4 * n + 1   # runs of 32 terms with a remainder
    H = channel(3, m, n, n) if tall else channel(3, n, m, n)
    snr = np.array([-10.0, 0.0, 30.0, 60.0])
    C = sbr.capacity(torch.as_tensor(H, device="cuda"), snr).cpu().numpy()
    Co = oracle.capacity(H.astype(np.complex128), snr)
    assert (np.abs(C - Co) < 1e-5 * np.abs(Co)).all(), (C, Co)


@pytest.mark.parametrize("F", [1, 2, 700])
def test_split_of_the_snrs_does_not_change_the_result(sbr, F):
    # few frequencies: the SNRs of one frequency run in blocks of their own;
    # a call with one SNR at a time runs each in a block that forms W again
    H = torch.as_tensor(channel(F, 5, 9), device="cuda")
    snr = [0.0, 10.0, 20.0, 50.0]
    one = [float(sbr.capacity(H, [s])[0]) for s in snr]
    assert sbr.capacity(H, snr).cpu().tolist() == one


@pytest.mark.parametrize("shift", [-45, 61])
def test_scale_of_H_cancels(sbr, shift):
    # a power of two scales every FP32 product exactly, so only the summation of
    # ||H||^2 (double-float inside, FP64 outside 2^-40 .. 2^60) can differ: 2^-44
    H = channel(4, 8, 16)
    C = sbr.capacity(torch.as_tensor(H, device="cuda"), [0.0, 20.0]).cpu().numpy()
    Hs = (H * np.float32(2.0) ** shift).astype(np.complex64)
    Cs = sbr.capacity(torch.as_tensor(Hs, device="cuda"), [0.0, 20.0]).cpu().numpy()
    assert (np.abs(C - Cs) < 1e-12 * C).all(), (C, Cs)


def test_an_infinite_or_missing_channel_is_not_a_number(sbr):
    H = torch.as_tensor(channel(3, 4, 6), device="cuda")
    assert torch.isnan(sbr.capacity(torch.zeros_like(H), [0.0, 20.0])).all()
    H[1, 2, 3] = float("inf")
    assert torch.isnan(sbr.capacity(H, [0.0, 20.0])).all()
