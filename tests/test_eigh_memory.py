"""Device memory of the eigensolver, on the recording stand-in for the CUDA runtime: the sweeps from the matrix itself
take three m x m matrices (A, its ping-pong copy, V; m = n rounded up to even) and a few vectors, at every order."""
import numpy as np
import pytest

from cuda_recorder import recorded
from paper_1708_00033_gb300 import hf


@pytest.mark.parametrize("n", [1, 2, 5, 100, 240, 241, 600, 1001])
def test_eigh_workspace(n):
    m = n + n % 2
    mp = 1 << (m - 1).bit_length()
    work = 8 * (3 * m * m + 514 + mp + 2 * m) + 4 * mp  # doubles and the permutation
    with recorded() as (lib, ctx):
        lib.rec_clear()
        idle = lib.rec_live_bytes()
        hf.eigh(ctx, np.eye(n))  # read back as converged: no sweep
        assert lib.rec_live_bytes() == idle
        assert lib.rec_peak_bytes() - idle <= work + 8 * (2 * n * n + n)  # and A, V, w of the host arrays
