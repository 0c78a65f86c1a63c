"""Capacity of channels at the ends of the FP32 range. A power of two scales every
FP32 product and sum exactly while none leaves the normal range, and the
normalisation takes the scale out in FP64, so C agrees with that of the channel at
unit scale up to the wide sums (2^-44): 1e-12.
"""
import numpy as np
import pytest
import torch

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
