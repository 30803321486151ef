"""The tuning file of hf_batch_tune on the recording stand-in for the CUDA runtime (every launch takes the same time): a
file without the present header, such as one tuned for other kernels, is ignored and rewritten; one with it is taken as
it is; the candidates hold the defaults, which win a tie; kernels of one warp per block only vary their blocks per SM."""
import re
from collections import Counter

import pytest

from cuda_recorder import log, recorded
from paper_1708_00033_gb300 import hf, inputs


def _tuned(path):
    """(timed launches per kernel, info) of tuning a new batch with the file."""
    geom = inputs.batch_cluster(inputs.CONFIG_BATCH, 0, 1, 1)
    with recorded() as (lib, ctx):
        lib.rec_read_words(1, 1)
        batch = hf.Batch(ctx, [geom], [inputs.synthetic_basis(geom)])
        lib.rec_clear()
        before = batch.info()
        batch.tune(str(path))
        after = batch.info()
        counts = Counter(re.search(r"k_eri_batch_(\d{4})", w).group(1) for op, _, w in log(lib)
                         if op == "launch" and "k_eri_batch" in w)
        batch.close()
    return counts, before, after


def test_candidates_and_round_trip(tmp_path):
    path = tmp_path / "tune.txt"
    counts, before, after = _tuned(path)
    assert len(counts) == hf.NUM_CLASSES
    # warm-up and timed launch of every candidate; L = 5 and above run one warp per block
    for name, n in counts.items():
        assert n == 2 * (3 if sum(map(int, name)) > 4 else 3 * 4 * 3), name
    assert before == after
    again, _, kept = _tuned(path)
    assert not again and kept == after


@pytest.mark.parametrize("header", ["", "# hf_batch_tune format 1, recorded sm_103\n",
                                    "# hf_batch_tune format 2, another GPU\n"])
def test_other_files_are_ignored(tmp_path, header):
    path = tmp_path / "tune.txt"
    lines = "".join(f"{k[-4:]} 64 32 2\n" for k in hf.CLASS_KERNELS)
    path.write_text(header + lines)
    counts, before, after = _tuned(path)
    assert len(counts) == hf.NUM_CLASSES and after == before
    assert path.read_text().startswith("# hf_batch_tune format 2, recorded sm_103\n")


def test_chunks_below_the_sorted_window_are_for_small_batches():
    """Every class of this batch has 400,000 quartets, more than four windows per resident warp together."""
    geom = inputs.batch_cluster(inputs.CONFIG_BATCH, 0, 1, 1)
    with recorded() as (lib, ctx):
        lib.rec_read_words(1, 400_000)
        batch = hf.Batch(ctx, [geom], [inputs.synthetic_basis(geom)])
        lib.rec_clear()
        batch.tune()
        counts = Counter(re.search(r"k_eri_batch_(\d{4})", w).group(1) for op, _, w in log(lib)
                         if op == "launch" and "k_eri_batch" in w)
        batch.close()
    for name, n in counts.items():
        assert n == 2 * (3 if sum(map(int, name)) > 4 else 3 * 2 * 3), name
