"""hf_eigh (parallel cyclic Jacobi on a matrix scaled to max |a_ij| in [1, 2)) at orders around its tile sizes, odd
ones, and on spectra with exact and near clusters, rank deficiency, zero and badly scaled matrices.

The sweeps end when off(V^T A V) <= 1e-14 |A|_F; eigenvalues and residual add the rounding of products of n terms
(n eps).  Each column of V goes through about 10 (n - 1) rotations, each changing its norm by up to 2 eps of
random sign: 2 eps sqrt(10 n) per column, 2 eps sqrt(10) n = 6.3 n eps over n columns; the bound is twice that."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _matrix(n, kind, rng):
    A = rng.normal(size=(n, n))
    Q, _ = np.linalg.qr(A)
    if kind == "random":
        return A + A.T
    if kind == "clusters":  # exact multiplicities and pairs 1e-10 apart
        w = np.repeat(rng.normal(size=(n + 3) // 4), 4)[:n]
        w[1::4] += 1e-10
        return (Q * w) @ Q.T
    if kind == "rank":
        return (Q[:, : max(1, n // 3)] * rng.uniform(1, 2, max(1, n // 3))) @ Q[:, : max(1, n // 3)].T
    if kind == "scaled":
        return 1e-200 * (A + A.T)
    if kind == "zero":
        return np.zeros((n, n))
    return np.diag(rng.normal(size=n))  # "diagonal"


@pytest.mark.parametrize("n,kind", [(1, "random"), (2, "random"), (3, "random"), (4, "random"), (5, "clusters"),
                                    (31, "random"), (33, "scaled"), (64, "clusters"), (100, "rank"), (100, "zero"),
                                    (101, "diagonal"), (239, "clusters"), (240, "random"), (241, "random"),
                                    (300, "clusters"), (512, "random"), (513, "random"), (1025, "random")])
def test_eigh_sizes_and_spectra(n, kind):
    from paper_1708_00033_gb300 import hf
    rng = np.random.default_rng(n)
    A = _matrix(n, kind, rng)
    A = 0.5 * (A + A.T)
    w, V = hf.eigh(hf.Context(0), A)
    top = np.abs(A).max() or 1.0
    norm, resid = top * np.linalg.norm(A / top), top * np.linalg.norm((A @ V - V * w) / top)  # no underflow at 1e-200
    eps = np.finfo(float).eps
    assert np.all(np.diff(w) >= 0)
    assert np.abs(w - np.linalg.eigvalsh(A)).max() <= (2e-14 + n * eps) * norm
    assert resid <= (2e-14 + n * eps) * norm
    assert np.linalg.norm(V.T @ V - np.eye(n)) <= 13 * n * eps
