"""Mixed paths whose FP32 increments overflow while the rest of the state stays ordinary: the FP64-accumulated state,
which is narrowed by integer operations, ends them at the step at which the compensated state does."""
import numpy as np
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W
from tests.gpu_util import gpu_run, torch

pytestmark = pytest.mark.gpu

# Diffusion of 1e36 AU^2/day along a radial field and almost none across: A_r dt overflows, the angles hardly move.
RADIAL = dict(K0=1e36, kperp_r_frac=1.2e-38, kperp_th_frac=1.2e-38, rot_period_day=1e300, r0=100.0, R_out=122.0,
              drift_on=0, hcs_on=0, dt_fixed=2e4, max_steps=1000.0)
SQUASHED = dict(squashed=1.0, nose_th=1.5, nose_ph=3.0, hp_tail=1.5, hp_flank=1.2)
# T grows 1e21-fold in one step while r is reflected and stays inside.
HOT = dict(W.config0().params, K0=1e-20, dt_fixed=1e22, R_out=1e25, max_steps=1000.0, formulation=1.0)


def ends(job, **kw):
    out = []
    for prec in (cz.PREC_MIXED_F64ACC, cz.PREC_MIXED):
        got, _, m = gpu_run(job, precision=prec, **kw)
        m.close()
        out.append((got["steps"].tolist(), got["status"].tolist()))
    return out


@pytest.mark.parametrize("shape", [dict(), SQUASHED, dict(SQUASHED, n_shells=2.0, shell_K0=(1e36, 1e36), shell_tilt_deg=(5.0, 5.0))],
                         ids=["sphere", "squashed", "any"])
def test_infinite_radius(shape):
    a, b = ends(W.Job(W.params(**RADIAL, **shape), W.PROTON, [1.0], [64], seed=3))
    assert a == b == ([1] * 64, [cz.PATH_NONFINITE] * 64)


def test_infinite_energy():
    a, b = ends(W.Job(HOT, W.PROTON, [1e18], [64], seed=3), with_lw=True)
    assert a == b == ([2] * 64, [cz.PATH_NONFINITE] * 64)


def test_infinite_radius_at_the_server():
    p = cz.make_params(W.params(**RADIAL, **SQUASHED), cz.PREC_MIXED_F64ACC)
    s = cz.cosmica_server_create(256 << 20, cz.PREC_MIXED_F64ACC)
    bins = cz.make_bins(0.1, 1000.0, 8)
    t = cz.cosmica_server_submit(s, cz.Request(p, cz.make_species(W.PROTON), [1.0], [100], 3, bins))
    res = cz.Result(1, 8)
    cz.cosmica_server_wait(s, t, res)
    cz.cosmica_server_destroy(s)
    assert int(res.steps) == 100
    assert int(np.asarray(res.hist).reshape(-1)[8 + 2]) == 100       # none of them an exit
