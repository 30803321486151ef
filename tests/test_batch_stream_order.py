"""A batch runs on a stream of its own; the set-up of its systems runs on the context's.  Everything the set-up
issued has to be ordered before the first batched launch, by an event or a host wait: the batched kernels index with
the pair headers that the set-up's last kernels write.  Checked on the order of the calls, without a GPU."""
import numpy as np
import pytest

from cuda_recorder import happens_before, log, recorded
from paper_1708_00033_gb300 import hf, inputs


@pytest.mark.parametrize("n_mol", [1, 3])
def test_first_batched_launch_waits_for_the_setup(n_mol):
    geoms = [inputs.batch_cluster(inputs.CONFIG_BATCH, m, 1, 2) for m in range(n_mol)]
    bases = [inputs.synthetic_basis(g) for g in geoms]
    with recorded(stream=8) as (lib, ctx):
        lib.rec_read_words(1, 1)  # every count the host reads back is one: all classes have pairs and quartets
        lib.rec_clear()
        batch = hf.Batch(ctx, geoms, bases)
        lib.rec_read_words(0, 0)
        P = np.zeros(int(batch.offsets[-1]))
        batch.fock_build(P, np.empty_like(P))
        batch.tune()
        ops = log(lib)
        batch.close()
    before = happens_before(ops)
    setup = {i for i, (op, s, what) in enumerate(ops) if op == "launch" and s == 8}
    assert sum("k_gather_headers" in ops[i][2] for i in setup) >= n_mol
    graph = next(i for i, (op, _, _) in enumerate(ops) if op == "graph")
    tuned = [i for i, (op, _, what) in enumerate(ops) if op == "launch" and "k_eri_batch" in what]
    assert tuned
    for i in [graph] + tuned:
        late = setup - before[i]
        assert not late, sorted({ops[j][2] for j in late})


class _DeviceArray:
    """A host array that the binding takes for a CUDA tensor: the stand-in's device memory is host memory."""

    is_cuda = True

    def __init__(self, a):
        self.a = a

    def data_ptr(self):
        return self.a.ctypes.data


def test_build_comes_after_the_callers_work():
    """Work is ordered on the stream given to hf_create: a density that a kernel on it still writes, or a Fock matrix
    that one still reads, when the batched build is called."""
    geom = inputs.batch_cluster(inputs.CONFIG_BATCH, 0, 1, 1)
    with recorded(stream=8) as (lib, ctx):
        lib.rec_read_words(1, 1)
        batch = hf.Batch(ctx, [geom], [inputs.synthetic_basis(geom)])
        lib.rec_read_words(0, 0)
        P = np.zeros(int(batch.offsets[-1]))
        P, F = _DeviceArray(P), _DeviceArray(np.empty_like(P))
        for build in range(2):  # a first and a repeated build
            lib.rec_clear()
            lib.rec_launch(8, b"caller")
            batch.fock_build(P, F)
            ops = log(lib)
            before = happens_before(ops)
            caller = next(i for i, op in enumerate(ops) if op == ("launch", 8, "caller"))
            issued = [i for i, (op, s, _) in enumerate(ops) if s != 8 and op in ("copy", "launch", "graph")]
            assert issued and all(caller in before[i] for i in issued), build
        batch.close()
