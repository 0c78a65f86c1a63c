"""Capacity of channels at the ends of the FP32 range. A power of two scales every
FP32 product and sum exactly while none leaves the normal range, and the
normalisation takes the scale out in FP64, so C agrees with that of the channel at
unit scale up to the wide sums (2^-44): 1e-12.
"""
import numpy as np
import pytest
import torch

from test_gpu_capacity_roundings import reference

pytestmark = pytest.mark.gpu


def signs(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    s = torch.randint(0, 2, shape + (2,), device="cuda", generator=g, dtype=torch.int8)
    return torch.view_as_complex(s.float() * 2.6 - 1.3)   # parts +-1.3


def test_many_large_entries():
    # 1024 squares of 2^118.8 in every thread's share of the power sum: 2^128.8
    import paper_2208_10006_gb300 as sbr
    H = signs((262144, 16, 16), 1)
    C = sbr.capacity(H, [0.0, 20.0]).cpu().numpy()
    Cs = sbr.capacity(H.mul_(2.0 ** 59), [0.0, 20.0]).cpu().numpy()
    assert np.isfinite(Cs).all() and (np.abs(C - Cs) < 1e-12 * C).all(), (C, Cs)


def test_gram_at_the_top_of_the_range():
    # diagonal of W 2^127.8
    import paper_2208_10006_gb300 as sbr
    H = signs((3, 8, 16), 2)
    C = sbr.capacity(H, [0.0, 20.0]).cpu().numpy()
    Cs = sbr.capacity(H * 2.0 ** 61, [0.0, 20.0]).cpu().numpy()
    assert (np.abs(C - Cs) < 1e-12 * C).all(), (C, Cs)


@pytest.mark.parametrize("n", [1, 8, 20])
def test_subnormal_gram(n):
    # entries of W of 2^-140 to 2^-127: against the same FP32 roundings on the host
    import paper_2208_10006_gb300 as sbr
    rng = np.random.default_rng(n)
    H = ((rng.normal(size=(3, n, 24)) + 1j * rng.normal(size=(3, n, 24))) * 2.0 ** -67).astype(np.complex64)
    C = sbr.capacity(torch.as_tensor(H, device="cuda"), [0.0, 20.0]).cpu().numpy()
    R = reference(H, [0.0, 20.0])
    assert (np.abs(C - R) < 1e-12 * R).all(), C / R - 1
