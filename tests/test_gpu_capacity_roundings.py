"""Capacity reproduces the FP32 roundings of its Gram product in every form of the
kernel (n = min(Nr, Nt) up to 16, 32, 48, 64; wide and tall): one fused multiply-add
a term, added to an FP32 sum over 32 terms, these sums added up beyond FP32.

The reference does the same roundings on the host and an FP64 factorisation. An
entry of W whose wide total lies within 2^-47 of a rounding boundary could be
rounded differently (once in some 2^22 entries, none for these inputs); else the
two differ by the factorisation alone, 2^-44 of a logarithm of some units: 1e-12.
"""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu
f32 = np.float32


def fma(a, b, c):
    # the product is exact in FP64
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(f32)


def reference(H, snr_db):
    F, Nr, Nt = H.shape
    tall = Nr > Nt
    n, m = min(Nr, Nt), max(Nr, Nt)
    C = np.zeros(len(snr_db))
    qbar = (np.abs(H.astype(np.complex128)) ** 2).sum() / F
    for h in H:
        h = h.T if tall else h
        xr, xi = np.ascontiguousarray(h.real), np.ascontiguousarray(h.imag)
        total = np.zeros((2, n, n))
        for p0 in range(0, m, 32):
            run = np.zeros((2, n, n), f32)
            for p in range(p0, min(m, p0 + 32)):
                ax, ay = (np.broadcast_to(v[:, p][:, None], (n, n)) for v in (xr, xi))
                bx, by = ax.T, ay.T
                run[0] += fma(ax, bx, ay * by)
                run[1] += fma(ax, by, -(ay * bx)) if tall else fma(ay, bx, -(ax * by))
            total += run
        W = total[0].astype(f32).astype(np.float64) + 1j * total[1].astype(f32).astype(np.float64)
        W = np.tril(W, -1)
        W = W + W.conj().T + np.diag(total[0].astype(f32).diagonal().astype(np.float64))
        for k, s in enumerate(snr_db):
            L = np.linalg.cholesky(np.eye(n) + 10 ** (s / 10) / Nt * (Nr * Nt / qbar) * W)
            C[k] += 2 * np.log2(L.diagonal().real).sum() / F
    return C


@pytest.mark.parametrize("n", [1, 5, 16, 17, 33, 64])
@pytest.mark.parametrize("more", [0, 35])
@pytest.mark.parametrize("tall", [False, True])
def test_gram_roundings(n, more, tall):
    import paper_2208_10006_gb300 as sbr
    rng = np.random.default_rng([n, more])
    shape = (3, n + more, n) if tall else (3, n, n + more)
    H = ((rng.normal(size=shape) + 1j * rng.normal(size=shape)) * 1e-4).astype(np.complex64)
    snr = [0.0, 20.0]
    C = sbr.capacity(torch.as_tensor(H, device="cuda"), snr).cpu().numpy()
    R = reference(H, snr)
    assert (np.abs(C - R) < 1e-12 * R).all(), C / R - 1
