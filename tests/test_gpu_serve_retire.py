"""Requests that retire while others are suspended: the largest ones, whose spectra are formed in the server's own
buffers beside the suspended particles, and one after which no resident set is of the kind of the freed slot's."""
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


@pytest.mark.parametrize("precision", [cz.PREC_MIXED, cz.PREC_MIXED_F64ACC])
def test_shells_after_a_plain_set_in_the_first_slot(precision):
    """A short request without shells takes the first slot and retires; the few particles of the ones with shells that
    are left share their warps with lanes that have none."""
    shells = dict(W.shell_params(W.solar_cycle_series(), 40, n_shells=5, R_ts=30.0, R_out=50.0), max_steps=3e6)
    cases = [(W.params(R_out=2.0), [50.0], [8]), (shells, [0.5], [37]), (shells, [1.0], [5])]
    srv = cz.cosmica_server_create(256 << 20, precision, budget_steps=64)
    reqs = [cz.Request(cz.make_params(p, precision), cz.make_species(W.PROTON), T, n, 9, cz.make_bins(0.1, 1000.0, 32))
            for p, T, n in cases]
    tickets = [cz.cosmica_server_submit(srv, q) for q in reqs]
    got = [cz.Result(1, 32) for _ in reqs]
    for t, r in zip(tickets, got):
        cz.cosmica_server_wait(srv, t, r)
    cz.cosmica_server_destroy(srv)
    assert got[0].c.t_done < got[1].c.t_done
    for (p, T, n), r in zip(cases, got):
        ref, _, m = gpu_run(W.Job(p, W.PROTON, T, n, 9), precision=precision)
        m.close()
        assert int(r.steps) == int(ref["steps"].astype(np.int64).sum())
