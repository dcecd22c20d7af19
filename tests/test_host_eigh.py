"""The Hermitian eigensolver on the host (csrc/hostla.cpp: tridiagonalisation, implicit QR) where it can go
wrong: 1 x 1, 2 x 2, matrices that split (diagonal, blocks, zero), many equal eigenvalues, entries near the
ends of the exponent range.

Tolerance: a backward stable method is off by a small multiple of n 2^-53 |A|; 16 n of them are allowed, for
the eigenvalues, the residuals and the orthogonality (|A| the largest eigenvalue).
"""
import numpy as np
import pytest


def matrix(kind, n, rng):
    A = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    Q, _ = np.linalg.qr(A)
    if kind == "dense":
        return A + A.conj().T
    if kind == "diagonal":
        return np.diag(rng.standard_normal(n)).astype(complex)
    if kind == "zero":
        return np.zeros((n, n), complex)
    if kind == "blocks":  # splits in the middle
        A = A + A.conj().T
        A[: n // 2, n // 2 :] = 0
        A[n // 2 :, : n // 2] = 0
        return A
    if kind == "equal":  # two eigenvalues, each many times
        A = (Q * np.where(np.arange(n) % 2, 1.0, -2.0)) @ Q.conj().T
    else:  # "graded": eigenvalues over twelve orders of magnitude
        A = (Q * 10.0 ** -np.linspace(0, 12, n)) @ Q.conj().T
    return (A + A.conj().T) / 2


@pytest.mark.parametrize("scale", [1.0, 1e-290, 1e290])
@pytest.mark.parametrize("n", [1, 2, 3, 32, 63])
@pytest.mark.parametrize("kind", ["dense", "diagonal", "zero", "blocks", "equal", "graded"])
def test_host_eigh(kind, n, scale):
    import paper_1111_6288_gb300 as P

    A = matrix(kind, n, np.random.default_rng(n))
    w, Z = P.host_eigh(A * scale)
    want = np.linalg.eigvalsh(A)
    tol = 16 * n * 2.0**-53
    norm = np.abs(want).max()
    assert np.abs(w / scale - want).max() <= tol * norm
    assert np.all(np.diff(w) >= 0)
    assert np.abs(Z.conj().T @ Z - np.eye(n)).max() <= tol
    assert np.abs(A @ Z - Z * (w / scale)).max() <= tol * norm
