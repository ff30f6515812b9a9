"""Which launches a given shape runs as, counted by kernels (the start values, the launch of the shape, and one launch
per warp per scheduler fewer that takes the last paths over), and that the autotuner times each launch once."""
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W
from tests.gpu_util import torch

pytestmark = pytest.mark.gpu
LAYER = 152 * 128       # paths that fill one warp per scheduler


def batch(**extra):
    p = cz.make_params(W.params(max_steps=300.0, **extra), cz.PREC_MIXED)
    return cz.cosmica_batch_create([p], [cz.make_species(W.PROTON)])


def alike(n):
    """All paths expected to be long."""
    return [(0, 0, 20.0, n, 0, 1)]


def spread(n):
    """One in twenty expected to be long."""
    return [(0, 0, 0.3, n // 20, 0, 1), (0, 0, 50.0, n - n // 20, n, 2)]


def kernels(b, items, tuning):
    out = cz.ExitBuffers(sum(i[3] for i in items))
    before = cz.cosmica_launch_count()
    cz.cosmica_batch_run(b, cz.make_items(items), len(items), out, tuning=tuning)
    torch().cuda.synchronize()
    return cz.cosmica_launch_count() - before


@pytest.mark.parametrize("items,n,most", [(alike, 2 * LAYER + 1, 3), (alike, 5 * LAYER, 4), (spread, 6 * LAYER + 1, 4),
                                          (spread, 9 * LAYER, 4)])
def test_shapes_that_run_as_given(items, n, most):
    """most: the launches that n paths are enough for (the hand-over's list holds at most n of them)."""
    b = batch()
    for blocks in (1, 2, 3, 4):
        assert kernels(b, items(n), cz.cosmica_tuning(128, blocks, 64, 0, 1)) == 1 + min(blocks, most), blocks
    assert kernels(b, items(n), cz.cosmica_tuning(64, 4, 64, 0, 1)) == 1 + min(2, most), "four blocks of 64"
    assert kernels(b, items(n), cz.cosmica_tuning(256, 2, 64, 0, 1)) == 1 + min(4, most), "two blocks of 256"
    cz.cosmica_batch_destroy(b)


@pytest.mark.parametrize("n", [LAYER + 1, 3 * LAYER, 6 * LAYER])
def test_shapes_that_start_at_the_last_launch(n):
    b = batch()
    for block, blocks in ((128, 1), (128, 4), (64, 8), (256, 2), (128, 0)):
        assert kernels(b, spread(n), cz.cosmica_tuning(block, blocks, 64, 0, 1)) == 2, (block, blocks)
        assert kernels(b, spread(n), cz.cosmica_tuning(block, blocks, 0, 0, 1)) == 2, (block, blocks, "as given")
    cz.cosmica_batch_destroy(b)


def test_autotuner_times_each_launch_once_and_tells_spreads_apart():
    n, b = 3 * LAYER, batch(lat_fast_deg=31.0)

    def tune(items):
        before = cz.cosmica_launch_count()
        t, rate = cz.cosmica_autotune(b, cz.make_items(items), len(items))
        return t, cz.cosmica_launch_count() - before

    t, k = tune(spread(n))
    assert t.compact_period == 0 or (t.block, t.blocks_per_sm) == (128, 1)      # a shape that runs
    # with the hand-over all of them are one launch of two kernels; without it, at most four shapes of 128 and two of 256
    assert 0 < k <= 2 * (1 + 6)
    assert tune(spread(n))[1] == 0              # cached
    assert tune(alike(n))[1] > 0                # another tail, so another class
    cz.cosmica_batch_destroy(b)
