"""The start of the SCF's diagonalisations (an FP32 eigenbasis refined in FP64, orders 4 to 240) by itself: the basis is
accepted, and the eigenpairs are those of the matrix, at the edges of its range of orders, odd
orders, and spectra whose gaps FP32 cannot resolve.

The sweeps end when off <= 1e-14 |A|_F.  On top come the products S = X^T A X and X V, n eps each, and X's own
departure from orthonormality, accepted up to 4e-16 n = 1.8 n eps off the diagonal and n eps on it: 6 n eps in all for
eigenvalues and residual; 13 n eps (the sweeps' rotations) plus these, 18 n eps, for V."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrix(n, kind):
    rng = np.random.default_rng(n)
    A = rng.normal(size=(n, n))
    Q, _ = np.linalg.qr(A)
    if kind == "random":
        A = A + A.T
    elif kind == "fock":  # deep levels and a band
        A = (A + A.T) / np.sqrt(4 * n) + np.diag(np.linspace(-1, 4, n) - 19.0 * (np.arange(n) < max(1, n // 25)))
    elif kind == "rank":
        A = (Q[:, : max(1, n // 3)] * rng.uniform(1, 2, max(1, n // 3))) @ Q[:, : max(1, n // 3)].T
    elif kind == "scaled":
        A = 1e-200 * (A + A.T)
    elif kind == "zero":
        A = np.zeros((n, n))
    elif kind == "diagonal":
        A = np.diag(rng.normal(size=n))
    else:  # groups of four, `kind` apart (0: exact multiplicities)
        w = np.repeat(rng.normal(size=(n + 3) // 4), 4)[:n] + kind * (np.arange(n) % 4)
        A = (Q * w) @ Q.T
    return 0.5 * (A + A.T)


KINDS = ["random", "fock", "rank", "scaled", "zero", "diagonal", 0.0, 1e-10, 1e-8, 1e-7, 1e-6, 1e-5, 1e-4, 1e-3]


@pytest.mark.parametrize("n", [3, 4, 5, 31, 33, 64, 101, 239, 240, 241])
@pytest.mark.parametrize("kind", KINDS, ids=str)
def test_fp32_start(n, kind):
    from paper_1708_00033_gb300 import hf
    A = _matrix(n, kind)
    w, V = np.empty(n), np.empty((n, n))
    used = ctypes.c_int32(-1)
    ctx = hf.Context(0)
    ptr = lambda a: ctypes.c_void_p(a.ctypes.data)  # noqa: E731
    rc = hf.load_library().hf_eigh_basis32(ctx._h, n, ptr(A), ptr(w), ptr(V), ctypes.byref(used), None)
    assert rc == hf.HF_OK
    assert used.value == (4 <= n <= 240)
    top = np.abs(A).max() or 1.0  # no underflow at 1e-200
    norm, resid = np.linalg.norm(A / top), np.linalg.norm((A @ V - V * w) / top)
    eps = np.finfo(float).eps
    assert np.all(np.diff(w) >= 0)
    assert np.abs(w / top - np.linalg.eigvalsh(A / top)).max() <= (2e-14 + 6 * n * eps) * norm
    assert resid <= (2e-14 + 6 * n * eps) * norm
    assert np.linalg.norm(V.T @ V - np.eye(n)) <= 18 * n * eps
