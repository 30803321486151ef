"""Exponent tables on the recording stand-in for the CUDA runtime: systems and batches of one context that have the same
exponents hold one table between them, others their own, and the last owner frees it."""
import numpy as np

from cuda_recorder import recorded
from paper_1708_00033_gb300 import hf, inputs


def _molecules():
    geoms = [inputs.batch_cluster(inputs.CONFIG_BATCH, m, 1, 1) for m in range(3)]
    return geoms, [inputs.synthetic_basis(g) for g in geoms]


def test_systems_share_one_table_and_free_it():
    geoms, bases = _molecules()
    n = len(set(np.concatenate([b.exps for b in bases])))
    table = 16 * (n * (n + 1) // 2) ** 2
    assert table > 1 << 20
    with recorded() as (lib, ctx):
        idle = lib.rec_live_bytes()
        held = []

        def grown(make):
            before = lib.rec_live_bytes()
            held.append(make())
            return lib.rec_live_bytes() - before

        first = grown(lambda: hf.System(ctx, geoms[0], bases[0]))
        assert first > table
        assert [grown(lambda: hf.System(ctx, geoms[m], bases[m])) for m in (1, 2)] == 2 * [first - table - 8 * n * (n + 1) // 2]
        assert grown(lambda: hf.Batch(ctx, geoms, bases)) < table
        sp = inputs.synthetic_sp_basis(geoms[0])
        k = len(set(sp.exps))
        assert grown(lambda: hf.System(ctx, geoms[0], sp)) > 16 * (k * (k + 1) // 2) ** 2
        held.pop(0).close()  # the first owner: the others still hold the table
        assert grown(lambda: hf.System(ctx, geoms[0], bases[0])) < table
        for h in held:
            h.close()
        assert lib.rec_live_bytes() == idle
        assert grown(lambda: hf.System(ctx, geoms[0], bases[0])) == first
        held[-1].close()
