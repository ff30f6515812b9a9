"""The FP64 path's kernels against the oracle, bit for bit: sizes on both sides of every switch between them
(four warps or four lanes a path, a lane a path with the queue, the hand-overs of the last paths), the models each form of
the step covers, starts that leave its range, and batches that mix isotropic and anisotropic sets."""
import numpy as np
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W
from tests.gpu_util import gpu_run, torch

pytestmark = pytest.mark.gpu
SM = 152        # 8 and 32 paths per SM are the switches between kernels

MODELS = {
    "isotropic": dict(W.config0().params),
    "isotropic_shock_adaptive": W.params(isotropic=1, drift_on=0, hcs_on=0, R_ts=60.0, dt_fixed=0),
    "full": W.params(),
    "shock": W.params(R_ts=30.0, R_out=50.0, tilt_deg=60.0, polarity=-1),
    "no_sheet": W.params(hcs_on=0),
    "no_drift": W.params(drift_on=0),
    "fixed_step": W.params(dt_fixed=0.02),
    "equal_winds": W.params(V_fast_kms=400.0),
    "near_pole": W.params(th0=1e-7, r0=0.5),
    "far_pole": W.params(th0=np.pi - 1e-3, r0=0.3),
    "wide_sheet": W.params(tilt_deg=70.0, dcs_min_deg=8.0),
}


def same(got, ref, with_lw=False):
    for k in ("steps", "status"):
        assert np.array_equal(got[k], ref[k]), k
    for k in ("r", "th", "ph", "lnP", "s") + (("lw",) if with_lw else ()):
        assert np.array_equal(got[k], ref[k], equal_nan=True), k


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("model", list(MODELS))
def test_models(orc, model, form):
    """A few paths to their end (four warps), and many for some steps (a lane a path, teams of four lanes)."""
    p = dict(MODELS[model], formulation=float(form))
    for n, T, steps in (([3, 2], [5.0, 60.0], 1e8), ([5000, 2001], [0.3, 20.0], 150), ([1500], [2.0], 150)):
        job = W.Job(dict(p, max_steps=steps), W.HELIUM4 if form else W.PROTON, T, n, seed=11)
        ref = orc.job_run(job)
        got, _, m = gpu_run(job, with_lw=form == 1)
        m.close()
        same(got, ref, form == 1)


@pytest.mark.parametrize("n", [1, 5, 608, 8 * SM - 1, 8 * SM, 8 * SM + 1, 32 * SM, 32 * SM + 1, 128 * SM + 17])
def test_sizes(orc, n):
    """Every path of every size, with step limits that end paths before, in and after the hand-over."""
    for steps in (1, 40, 3000):
        job = W.Job(dict(W.params(R_out=6.0, K0=60.0, max_steps=steps)), W.PROTON, [3.0, 30.0], [n - n // 3, n // 3], seed=3)
        ref = orc.job_run(job)
        got, _, m = gpu_run(job)
        m.close()
        same(got, ref)


@pytest.mark.parametrize("counts", [(40, 30, 20, 10), (900, 800, 700, 600), (3000, 2000, 1500, 1000)])
def test_mixed_models_in_a_batch(orc, counts):
    """Isotropic and anisotropic sets and both charges in one launch: each item as alone, steps summed."""
    t = torch()
    sets = [dict(MODELS[k], max_steps=400.0) for k in ("isotropic", "full", "shock", "isotropic_shock_adaptive")]
    b = cz.cosmica_batch_create([cz.make_params(p, cz.PREC_FP64) for p in sets],
                                [cz.make_species(W.PROTON), cz.make_species(W.ELECTRON)])
    items = [(i, i % 2, 4.0 + i, c, 0, 9 + i) for i, c in enumerate(counts)]
    out = cz.ExitBuffers(sum(counts))
    steps = t.zeros(1, dtype=t.int64, device="cuda")
    cz.cosmica_batch_run(b, cz.make_items(items), len(items), out, steps_out=steps)
    got = out.numpy()
    at = 0
    for i, c in enumerate(counts):
        ref = orc.job_run(W.Job(sets[i], (W.PROTON, W.ELECTRON)[i % 2], [4.0 + i], [c], seed=9 + i))
        same({k: v[at:at + c] for k, v in got.items()}, ref)
        assert np.all(got["item"][at:at + c] == i)
        at += c
    assert int(steps.item()) == int(got["steps"].astype(np.int64).sum())
    cz.cosmica_batch_destroy(b)


@pytest.mark.parametrize("n", [7, 6000])
def test_without_allocation(orc, n):
    job = W.Job(dict(W.params(R_out=8.0, max_steps=500)), W.PROTON, [2.0], [n], seed=5)
    out = cz.ExitBuffers(n)
    cz.cosmica_propagate_noalloc(cz.make_params(job.params, cz.PREC_FP64), cz.make_species(W.PROTON), [2.0], [n], 5, out)
    torch().cuda.synchronize()
    same(out.numpy(), orc.job_run(job))
