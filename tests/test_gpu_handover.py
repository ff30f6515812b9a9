"""The mixed launches that hand their last paths to fewer warps per scheduler: every model form, around the
sizes where another launch joins, equals the single launch (compact_period 0) bit for bit."""
import numpy as np
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W
from tests.gpu_util import gpu_run, torch

pytestmark = pytest.mark.gpu
LAYER = 152 * 128       # one warp per scheduler
KEYS = ("r", "th", "ph", "lnP", "s", "steps", "status", "item", "lw")

SHELLS = W.shell_params(W.solar_cycle_series(), 40, n_shells=5, R_ts=30.0, R_out=50.0)
MODELS = {
    "plain": W.params(R_out=20.0),
    "shock": W.params(R_ts=30.0, R_out=50.0, tilt_deg=60.0, polarity=-1),
    "shells": SHELLS,
    "squashed": dict(W.params(), **dict(W.SQUASHED, R_ts=30.0, R_out=50.0)),
    "any": dict(SHELLS, **{k: v for k, v in W.SQUASHED.items() if k not in ("R_ts", "R_out")}),
}


def run(b, items, tuning=None, reps=1):
    t = torch()
    for _ in range(reps):
        out = cz.ExitBuffers(sum(i[3] for i in items), with_lw=True)
        steps = t.zeros(1, dtype=t.int64, device="cuda")
        cz.cosmica_batch_run(b, cz.make_items(items), len(items), out, tuning=tuning, steps_out=steps)
        t.cuda.synchronize()
    got = out.numpy()
    assert int(steps.item()) == int(got["steps"].astype(np.int64).sum())
    return got


def same(got, ref, what):
    for k in KEYS:
        if k in ref:
            assert np.array_equal(got[k], ref[k]), (what, k)


@pytest.mark.parametrize("precision", [cz.PREC_MIXED, cz.PREC_MIXED_F64ACC])
@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("model", list(MODELS))
def test_hand_over(model, form, precision):
    """Paths of three energies, some ended by the step limit, others before the first hand-over."""
    p = dict(MODELS[model], formulation=float(form), max_steps=6000.0)
    b = cz.cosmica_batch_create([cz.make_params(p, precision)], [cz.make_species(W.HELIUM4)])
    for n in (LAYER + 1, 6 * LAYER, 6 * LAYER + 77):
        items = [(0, 0, 30.0, n - n // 3 - 5, 0, 1), (0, 0, 1.0, n // 3, 50, 2), (0, 0, 4.0, 5, 0, 3)]
        ref = run(b, items, cz.cosmica_tuning(128, 0, 0, 0, 0))
        assert len(np.unique(ref["steps"])) > 100
        same(run(b, items), ref, (n, "untuned"))
        for blocks in (2, 3, 4):
            same(run(b, items, cz.cosmica_tuning(128, blocks, 64, 0, 0)), ref, (n, blocks))
        same(run(b, items, cz.cosmica_tuning(64, 0, 16, 0, 1)), ref, (n, "blocks of 64"))
        same(run(b, items, cz.cosmica_tuning(256, 2, 1, 1, 0), reps=2), ref, (n, "blocks of 256, replayed"))
    cz.cosmica_batch_destroy(b)


@pytest.mark.parametrize("precision", [cz.PREC_MIXED, cz.PREC_MIXED_F64ACC])
def test_without_allocation(precision):
    """The fixed scratch holds shorter lists: sizes below, at and above what they hold, against the ordinary entry."""
    for n in (LAYER, LAYER + 1, 5 * LAYER, 8 * LAYER):
        job = W.Job(dict(MODELS["shock"], max_steps=3000), W.PROTON, [2.0, 20.0], [n - 999, 999], seed=5)
        ref, _, m = gpu_run(job, precision=precision)
        m.close()
        out = cz.ExitBuffers(n)
        cz.cosmica_propagate_noalloc(cz.make_params(job.params, precision), cz.make_species(W.PROTON), job.T_in,
                                     job.n_per_energy, 5, out)
        torch().cuda.synchronize()
        same(out.numpy(), ref, n)


@pytest.mark.parametrize("T", [[1.0], [0.1, 1.0, 30.0, 100.0]])
@pytest.mark.parametrize("per_lane", [1.19, 1.21, 2.5, 3.5, 6.5, 10.01])
def test_untuned_layers(T, per_lane):
    """Untuned launches on both sides of the lines between one and four warps per scheduler, all paths expected
    to be long or few of them, the last energy empty: the single launch's records."""
    n = int(per_lane * LAYER) // len(T)
    p = dict(W.params(R_out=10.0), max_steps=800.0)
    items = [(0, 0, t, n, 0, 4 + i) for i, t in enumerate(T)] + [(0, 0, 0.01, 0, 0, 9)]
    b = cz.cosmica_batch_create([cz.make_params(p, cz.PREC_MIXED)], [cz.make_species(W.PROTON)])
    ref = run(b, items, cz.cosmica_tuning(128, 0, 0, 0, 0))
    same(run(b, items), ref, "untuned")
    cz.cosmica_batch_destroy(b)
