"""FP64 paths whose state or parameters leave the range of the fast step, against the oracle bit for bit, in every
kernel of the FP64 path: the four warps of a block, teams of four lanes, a lane a path."""
import numpy as np
import pytest

from paper_2502_06319_gb300 import workloads as W
from tests.gpu_util import gpu_run

pytestmark = pytest.mark.gpu
ISOTROPIC = dict(W.config0().params)
COUNTS = ([3, 2], [900, 600], [5000, 2001])


def same_as_oracle(orc, p, T, form=0, steps=60.0, counts=COUNTS):
    for n in counts:
        job = W.Job(dict(p, formulation=float(form), max_steps=steps), W.HELIUM4 if form else W.PROTON, T, n, seed=11)
        ref = orc.job_run(job)
        got, _, m = gpu_run(job, with_lw=form == 1)
        m.close()
        for k in ("steps", "status", "r", "th", "ph", "lnP", "s") + (("lw",) if form else ()):
            assert np.array_equal(got[k], ref[k], equal_nan=True), (n, k)


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("model", ["isotropic", "full", "no_sheet"])
@pytest.mark.parametrize("start", [dict(ph0=-1e9), dict(ph0=-2e6), dict(ph0=-5.0), dict(ph0=1e9), dict(th0=1e-30),
                                   dict(th0=1e-30, ph0=-1e9)], ids=str)
def test_far_angles(orc, model, start, form):
    """Longitudes far from [0, 2 pi), and a start so close to a pole that the first step throws theta away."""
    p = {"isotropic": ISOTROPIC, "full": W.params(), "no_sheet": W.params(hcs_on=0)}[model]
    same_as_oracle(orc, dict(p, **start), [5.0, 60.0], form)
