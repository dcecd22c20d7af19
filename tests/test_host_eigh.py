"""The Hermitian eigensolver on the host (csrc/hostla.cpp: tridiagonalisation, implicit QR) where it can go
wrong: 1 x 1, 2 x 2, matrices that split (diagonal, blocks, zero), many equal eigenvalues, entries near the
ends of the exponent range.

Couplings far below the matrix's largest entry, whose squares underflow, are one more.

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


@pytest.mark.parametrize("n", [2, 3, 5])
@pytest.mark.parametrize("tiny", [1e-155, 1e-160, 1e-165j, 1e-200j, 1e-300 + 1e-310j, 5e-324j])
@pytest.mark.parametrize("where", ["all", "first", "last"])
def test_tiny_couplings(n, tiny, where):
    """O(1) diagonals with couplings whose squares underflow: all of them, or one beside ordinary ones."""
    import paper_1111_6288_gb300 as P

    A = np.diag(1.0 + np.arange(n)).astype(complex)
    low = np.tril(np.ones((n, n)), -1) * tiny
    if where != "all" and n > 2:
        low = np.tril(0.1 * np.ones((n, n)), -1).astype(complex)
        low[(1, 0) if where == "first" else (n - 1, 0)] = tiny
        if where == "first":
            low[2:, 0] = 0
    A += low + low.conj().T
    w, Z = P.host_eigh(A)
    want = np.linalg.eigvalsh(A)
    tol = 16 * n * 2.0**-53
    norm = np.abs(want).max()
    assert np.abs(w - want).max() <= tol * norm
    assert np.abs(Z.conj().T @ Z - np.eye(n)).max() <= tol
    assert np.abs(A @ Z - Z * w).max() <= tol * norm


@pytest.mark.parametrize("bad", [np.nan, np.inf, complex(0, np.nan)])
def test_not_finite(bad):
    import paper_1111_6288_gb300 as P

    A = np.eye(3, dtype=complex)
    A[2, 1] = A[1, 2] = bad
    w, Z = P.host_eigh(A)
    assert np.isnan(w).all() and np.isnan(Z).all()
