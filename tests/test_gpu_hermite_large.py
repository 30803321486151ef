"""The Hermite-accumulator kernels against the Obara-Saika kernels in launches large enough for groups of quartets per
warp (64 quartets per SM) and for sorted windows of eight rounds (1,024 per SM): whole builds, odd shards of them (a
group or window that ends short), and density-screened builds in which many quartets of a group are dead.

Both are FP64 evaluations of the same sums: each J or K element adds at most ~1e6 products, each within a few hundred
roundings, whose errors are independent: 1e-12 of the largest element leaves a factor of about ten."""
import numpy as np
import pytest

from paper_1708_00033_gb300 import inputs

pytestmark = pytest.mark.gpu


def _system(hf, n_atoms, nprim, tau):
    rng = np.random.default_rng(n_atoms)
    xyz = rng.uniform(-5, 5, (n_atoms, 3))
    xyz[1] = xyz[0]      # coincident centres
    xyz[2] += 30.0       # a distant one
    k = n_atoms * 3
    exps = (rng.uniform(0.2, 1.0, (k, 1)) * 2.5 ** np.arange(nprim)).ravel()
    basis = inputs.Basis(atom=np.repeat(np.arange(n_atoms, dtype=np.int32), 3), l=np.tile(np.arange(3, dtype=np.int32), n_atoms),
                         nprim=np.full(k, nprim, np.int32), exps=exps, coefs=rng.uniform(-0.3, 1.0, k * nprim))
    geom = inputs.Geometry(Z=np.full(n_atoms, 2, np.int32), xyz=xyz)
    return hf.System(hf.Context(0), geom, basis, schwarz_tau=tau, prim_tau=1e-14 if tau else 0.0), rng


@pytest.mark.parametrize("n_atoms,nprim,tau", [(22, 2, 0.0), (34, 3, 1e-10)])
def test_large_launches(n_atoms, nprim, tau):
    import torch

    from paper_1708_00033_gb300 import hf
    s, rng = _system(hf, n_atoms, nprim, tau)
    A = torch.from_numpy(rng.normal(size=(s.n_bf, s.n_bf))).cuda()
    P = (A + A.T).contiguous()
    h = s.fock_build(P, want_J=True, want_K=True, stats=True)
    o = s.fock_build(P, want_J=True, want_K=True, rys=False, stats=True)
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    L = [sum(map(int, k[-4:])) for k in hf.CLASS_KERNELS]
    n = h["stats"]["class_quartets_fp64"]
    assert sum(q >= 64 * sms for q, l in zip(n, L) if l >= 5) >= 3
    assert sum(q >= 1024 * sms for q, l in zip(n, L) if l <= 3) >= 1
    assert h["stats"]["prim_quartets_fp64"] == o["stats"]["prim_quartets_fp64"] > 0
    for k in ("J", "K"):
        assert float((h[k] - o[k]).abs().max()) <= 1e-12 * float(o[k].abs().max())
    # shards of odd sizes; a density over fourteen orders of magnitude, so that quartets of one group live and die
    D = torch.from_numpy(np.repeat(10.0 ** -rng.uniform(0, 7, n_atoms), 10)).cuda()
    for density, screen in ((P, False), ((D[:, None] * P * D[None, :]).contiguous(), tau > 0)):
        for shard, shards in ((1, 3), (6, 7)):
            j, k = hf.fock_build_partial(s, density, shard, shards, density_screen=screen)
            j2, k2 = hf.fock_build_partial(s, density, shard, shards, density_screen=screen, rys=False)
            assert float((j - j2).abs().max()) <= 1e-12 * float(j2.abs().max())
            assert float((k - k2).abs().max()) <= 1e-12 * float(k2.abs().max())
