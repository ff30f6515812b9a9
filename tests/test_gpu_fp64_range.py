"""FP64 paths whose state or parameters leave the range of the fast step, against the oracle bit for bit, in every
kernel of the FP64 path: the four warps of a block, teams of four lanes, a lane a path."""
import math

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


@pytest.mark.parametrize("extra", [
    # a wind that changes over 1e-307 degrees: V is the fast one at 0.3 rad from the pole
    dict(dlat_deg=1e-307, th0=0.3, hcs_on=0, drift_on=0),
    dict(dlat_deg=1e-307, th0=0.3),
    dict(R_ts=50.0, dts_AU=1e-310),
    dict(R_ts=math.inf),
    dict(B1AU_nT=1e-300), dict(B1AU_nT=1e300), dict(K0=1e-150), dict(K0=1e150), dict(rot_period_day=1e300),
    dict(rot_period_day=1e-120), dict(V_slow_kms=1e-200), dict(kperp_r_frac=1e-250), dict(kperp_th_frac=math.inf),
    dict(eps_diff=1e-320), dict(dt_min=1e-310, dt_max=1e-309), dict(th0=1e-200), dict(lat_fast_deg=1e300)], ids=str)
def test_far_constants(orc, extra):
    """Accepted parameters whose reciprocals or products leave the FP64 range."""
    same_as_oracle(orc, W.params(**extra), [5.0, 60.0], steps=20.0)


@pytest.mark.parametrize("form", [0, 1])
@pytest.mark.parametrize("extra", [dict(R_ts=0.5, dts_AU=0.001, ts_K_factor=0.0, V_const_kms=0.0, dt_fixed=0.0),
                                   dict(R_ts=0.5, dts_AU=0.0), dict(R_ts=0.5, dts_AU=0.001, ts_K_factor=1e-300)], ids=str)
def test_far_constants_isotropic(orc, extra, form):
    """The isotropic model takes any shock, one beyond which nothing diffuses among them: its tensor has no root."""
    same_as_oracle(orc, dict(ISOTROPIC, **extra), [5.0, 60.0], form, steps=20.0)


@pytest.mark.parametrize("T", [1.32e154, 1e100, 1e20, 1e-20, 1e-100])
def test_far_energies(orc, T):
    """T (T + 2 m0) overflows while T is finite: ln P is then infinite and the path ends.  K0 keeps K0 P ordinary."""
    K0 = 11.5 / (2.0 * T if T > 1.0 else math.sqrt(2.0 * T))
    for form in (0, 1):
        for p in (ISOTROPIC, W.params()):
            same_as_oracle(orc, dict(p, K0=K0), [T, 2.0 * T], form, steps=200.0)
    same_as_oracle(orc, dict(ISOTROPIC), [T, 5.0], 1, steps=200.0)
