"""Requests of the largest size that retire while others are suspended: their spectra are formed in the server's own
buffers, beside which the suspended particles wait."""
import numpy as np
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W
from tests.gpu_util import gpu_run, gpu_spectrum

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [cz.PREC_MIXED, cz.PREC_MIXED_F64ACC])
def test_largest_requests_beside_suspended_ones(precision):
    p = dict(W.params(R_out=20.0), max_steps=3e6)
    cases = [([0.2, 0.3], [3000, 3000], 64), (list(np.geomspace(0.5, 100.0, 256)), [40] * 256, 8192), ([5.0], [200], 8191),
             (list(np.geomspace(1.0, 50.0, 255)), [9] * 255, 4097), ([30.0] * 256, [3] * 256, 1)]
    srv = cz.cosmica_server_create(512 << 20, precision, budget_steps=128)
    reqs = [cz.Request(cz.make_params(p, precision), cz.make_species(W.PROTON), T, n, 50 + i, cz.make_bins(0.1, 1000.0, nb))
            for i, (T, n, nb) in enumerate(cases)]
    tickets = [cz.cosmica_server_submit(srv, q) for q in reqs]
    got = []
    for t, q in zip(tickets, reqs):
        r = cz.Result(q.n_energies, q.nbins)
        cz.cosmica_server_wait(srv, t, r)
        got.append(r)
    cz.cosmica_server_destroy(srv)
    assert got[0].c.t_done > got[2].c.t_done        # the first one was suspended when others retired
    for i, (T, n, nb) in enumerate(cases):
        job = W.Job(p, W.PROTON, T, n, 50 + i, bins=W.Bins(0.1, 1000.0, nb))
        ref, out, m = gpu_run(job, precision=precision)
        H, J, S = gpu_spectrum(job, out)
        m.close()
        assert np.array_equal(np.asarray(got[i].hist).reshape(len(T), nb + 3), H), i
        assert int(got[i].steps) == int(ref["steps"].astype(np.int64).sum())
        # the same sums in the same order
        assert np.allclose(got[i].J, J, rtol=1e-14, atol=0, equal_nan=True)
        assert np.allclose(got[i].sigma, S, rtol=1e-12, atol=0, equal_nan=True)
