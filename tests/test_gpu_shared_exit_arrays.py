"""One array given for several exit fields that the caller does not want: the other fields are as with arrays of
their own, at sizes where paths pass from kernel to kernel."""
import numpy as np
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W
from tests.gpu_util import torch

pytestmark = pytest.mark.gpu
LAYER = 152 * 128
WANTED = ("lnP", "steps", "status", "item", "lw")


def records(n, shared, lw):
    """Exit records of n particles; shared: r, theta, phi and s (and lw when it is not wanted) in one array."""
    out = cz.ExitBuffers(n, with_lw=lw)
    if shared:
        out.th = out.ph = out.s = out.r
        out.c.th = out.c.ph = out.c.s = out.c.r
    return out


def wanted(out, lw):
    got = out.numpy()
    return {k: got[k] for k in WANTED if k != "lw" or lw}


@pytest.mark.parametrize("entry", ["model", "batch", "noalloc"])
@pytest.mark.parametrize("precision,form,n", [(cz.PREC_MIXED, 0, 7 * LAYER), (cz.PREC_MIXED, 1, 2 * LAYER + 5),
                                              (cz.PREC_MIXED_F64ACC, 0, 11 * LAYER), (cz.PREC_FP64, 0, 6000),
                                              (cz.PREC_FP64, 1, 2000), (cz.PREC_FP64, 0, 500)])
def test_unwanted_fields_in_one_array(precision, form, n, entry):
    p = cz.make_params(dict(W.params(R_out=10.0, max_steps=2000.0), formulation=float(form)), precision)
    sp, T, N = cz.make_species(W.PROTON), [1.0, 30.0], [n - n // 2, n // 2]
    got = []
    for shared in (False, True):
        out = records(n, shared, form == 1)
        if entry == "model":
            m = cz.Model(p)
            cz.cosmica_propagate(m.h, sp, T, N, 5, out)
            torch().cuda.synchronize()
            m.close()
        elif entry == "batch":
            b = cz.cosmica_batch_create([p], [sp])
            items = [(0, 0, T[0], N[0], 0, 5), (0, 0, T[1], N[1], N[0], 5)]
            cz.cosmica_batch_run(b, cz.make_items(items), 2, out, tuning=cz.cosmica_tuning(128, 4, 64, 0, 1))
            torch().cuda.synchronize()
            cz.cosmica_batch_destroy(b)
        else:
            cz.cosmica_propagate_noalloc(p, sp, T, N, 5, out)
            torch().cuda.synchronize()
        got.append(wanted(out, form == 1))
    assert len(np.unique(got[0]["steps"])) > 100
    for k in got[0]:
        assert np.array_equal(got[0][k], got[1][k]), k
