"""The Hermite-accumulator kernels (the FP64 default) against the Obara-Saika kernels at the places where their
code differs: one to eight primitives per shell (staircases from one row to 64 x 64, several batches of the warp
kernel), bases with more distinct exponents than the exponent table holds (direct evaluation), coincident and
distant centres, screened and unscreened, and launches of one quartet up to those that fill the GPU.

Both are FP64 evaluations of the same sums; each J or K element adds at most ~1e6 products, each within a few
hundred roundings, whose errors are independent: 1e-12 of the largest element leaves a factor of about ten."""
import numpy as np
import pytest

from paper_1708_00033_gb300 import inputs

pytestmark = pytest.mark.gpu


def _basis(n_atoms, nprim, rng, distinct):
    atom, l, npr, exps, coefs = [], [], [], [], []
    for a in range(n_atoms):
        for lq in (0, 1, 2):
            base = rng.uniform(0.2, 1.0) if distinct else 0.4
            atom.append(a)
            l.append(lq)
            npr.append(nprim)
            exps.extend(base * 2.5 ** k * (1 + (0.01 * rng.uniform() if distinct else 0.0)) for k in range(nprim))
            coefs.extend(rng.uniform(-0.3, 1.0, nprim))
    return inputs.Basis(atom=np.array(atom, np.int32), l=np.array(l, np.int32), nprim=np.array(npr, np.int32),
                        exps=np.array(exps), coefs=np.array(coefs))


@pytest.mark.parametrize("n_atoms,nprim,distinct,tau", [(1, 1, False, 0.0), (2, 3, False, 0.0), (2, 8, False, 0.0),
                                                        (3, 5, True, 0.0), (7, 8, True, 1e-10), (9, 2, False, 1e-10)])
def test_hermite_equals_obara_saika(n_atoms, nprim, distinct, tau):
    import torch

    from paper_1708_00033_gb300 import hf
    rng = np.random.default_rng(100 * n_atoms + nprim)
    xyz = rng.uniform(-4, 4, (n_atoms, 3))
    if n_atoms > 2:
        xyz[1] = xyz[0]      # coincident centres: AB = 0
        xyz[2] += 30.0       # a distant one: large Boys arguments
    geom = inputs.Geometry(Z=np.full(n_atoms, 2, np.int32), xyz=xyz)
    basis = _basis(n_atoms, nprim, rng, distinct)
    assert len(set(basis.exps)) > 53 or not distinct or n_atoms < 7
    ctx = hf.Context(0)
    s = hf.System(ctx, geom, basis, schwarz_tau=tau, prim_tau=1e-14 if tau else 0.0)
    A = torch.from_numpy(rng.normal(size=(s.n_bf, s.n_bf))).cuda()
    P = (A + A.T).contiguous()
    h = s.fock_build(P, want_J=True, want_K=True, stats=True)
    o = s.fock_build(P, want_J=True, want_K=True, rys=False, stats=True)
    assert h["stats"]["prim_quartets_fp64"] == o["stats"]["prim_quartets_fp64"] > 0
    for k in ("J", "K"):
        assert float((h[k] - o[k]).abs().max()) <= 1e-12 * float(o[k].abs().max())
    j, k = hf.fock_build_partial(s, P, 0, 3, density_screen=tau > 0)
    j2, k2 = hf.fock_build_partial(s, P, 0, 3, density_screen=tau > 0, rys=False)
    assert float((j - j2).abs().max()) <= 1e-12 * float(o["J"].abs().max())
    assert float((k - k2).abs().max()) <= 1e-12 * float(o["K"].abs().max())
