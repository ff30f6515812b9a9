"""A launch shape given to cosmica_batch_run is the one that runs: counted by its kernels (the start values, the
launch of the shape, and one launch per warp per scheduler fewer that takes the last paths over)."""
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W
from tests.gpu_util import torch

pytestmark = pytest.mark.gpu
LAYER = 152 * 128       # paths that fill one warp per scheduler


def kernels(b, n, tuning):
    out = cz.ExitBuffers(n)
    before = cz.cosmica_launch_count()
    cz.cosmica_batch_run(b, cz.make_items([(0, 0, 20.0, n, 0, 1)]), 1, out, tuning=tuning)
    torch().cuda.synchronize()
    return cz.cosmica_launch_count() - before


@pytest.mark.parametrize("n,most", [(LAYER, 1), (LAYER + 1, 2), (2 * LAYER + 1, 3), (3 * LAYER, 4), (5 * LAYER, 4), (7 * LAYER, 4)])
def test_given_shapes_run_as_given(n, most):
    """most: the launches that n paths are enough for (the hand-over's list holds at most n of them)."""
    b = cz.cosmica_batch_create([cz.make_params(W.params(max_steps=300.0), cz.PREC_MIXED)], [cz.make_species(W.PROTON)])
    for blocks in (1, 2, 3, 4):
        assert kernels(b, n, cz.cosmica_tuning(128, blocks, 64, 0, 1)) == 1 + min(blocks, most), blocks
        assert kernels(b, n, cz.cosmica_tuning(128, blocks, 0, 0, 1)) == 2, (blocks, "no hand-over")
    assert kernels(b, n, cz.cosmica_tuning(64, 4, 64, 0, 1)) == 1 + min(2, most), "four blocks of 64"
    assert kernels(b, n, cz.cosmica_tuning(256, 2, 64, 0, 1)) == 1 + min(4, most), "two blocks of 256"
    cz.cosmica_batch_destroy(b)
