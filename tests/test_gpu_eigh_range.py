"""hf_eigh at both ends of the FP64 range: the matrix is scaled by a power of two, which must itself be finite for
subnormal matrices.  Small whole numbers times 2^k are exact at these k; eigenvalues follow the sweeps' criterion
(off <= 1e-14 |A|_F) and n roundings, and are rounded to the subnormal grid 2^-1074 at the lower end."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [2, 7, 40])
@pytest.mark.parametrize("k", [-1060, -1030, -1024, -1023, -1022, 1015])
def test_eigh_extreme_scales(n, k):
    from paper_1708_00033_gb300 import hf
    B = np.random.default_rng(n).integers(-3, 4, size=(n, n)).astype(float)
    B = np.triu(B) + np.triu(B, 1).T
    w, V = hf.eigh(hf.Context(0), np.ldexp(B, k))
    eps, norm = np.finfo(float).eps, np.linalg.norm(B)
    grid = max(0.0, np.ldexp(1.0, -1074 - k))
    assert np.abs(np.ldexp(w, -k) - np.linalg.eigvalsh(B)).max() <= (2e-14 + n * eps) * norm + grid
    assert np.linalg.norm(V.T @ V - np.eye(n)) <= 13 * n * eps
    assert np.linalg.norm(B @ V - V * np.ldexp(w, -k)) <= (2e-14 + n * eps) * norm + grid * np.sqrt(n)


@pytest.mark.parametrize("n", [1, 2, 3, 8, 13, 40])
@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
@pytest.mark.parametrize("at", ["first", "last", "all"])
def test_eigh_rejects_a_matrix_that_is_not_finite(n, bad, at):
    """No eigenpairs and no answer; the context stays usable.  (The sort of NaN keys used to bring the index that pads
    it to a power of two into the permutation of the gathered columns.)"""
    from paper_1708_00033_gb300 import hf
    ctx = hf.Context(0)
    A = np.eye(n) + 0.01
    i = slice(None) if at == "all" else 0 if at == "first" else n - 1
    B = A.copy()
    B[i, i] = bad
    with pytest.raises(hf.HFError) as e:
        hf.eigh(ctx, B)
    assert e.value.code == hf.HF_E_NOCONV
    w, _ = hf.eigh(ctx, A)
    assert np.abs(w - np.linalg.eigvalsh(A)).max() <= 1e-13 * (1 + 0.01 * n)
