"""The class launches of a build run concurrently on the context's side streams; with timing they run one
after another on the context's stream.  Both orders add the same quartets, so F, J and K agree to the
rounding of reordered FP64 additions: each element sums at most n_quartets terms of magnitude <= max|F|,
and the two sums differ by far less than 1e-12 of it for these sizes."""
import numpy as np
import pytest

from paper_1708_00033_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("waters,cutoff", [(1, 0.0), (3, 0.0), (3, 1e-4)])
def test_concurrent_class_launches_equal_serial(waters, cutoff):
    import torch

    from paper_1708_00033_gb300 import hf
    geom = inputs.water_cluster(waters, inputs.CONFIG_GUESS_EVAL, 77)
    basis = inputs.synthetic_basis(geom)
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ctx = hf.Context(0)  # the work forks from and joins a stream that is not the default one
        s = hf.System(ctx, geom, basis, schwarz_tau=1e-10, prim_tau=1e-14, fp32_cutoff=cutoff)
        A = torch.from_numpy(np.random.default_rng(waters).normal(size=(s.n_bf, s.n_bf))).cuda()
        P = (A + A.T).contiguous()
        serial = s.fock_build(P, want_J=True, want_K=True, timing=True)
        for _ in range(3):
            got = s.fock_build(P, want_J=True, want_K=True)
            for k in ("F", "J", "K"):
                scale = float(serial[k].abs().max())
                assert float((got[k] - serial[k]).abs().max()) <= 1e-12 * scale
