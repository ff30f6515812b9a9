"""Histogram and estimators of given exit states against plain numpy: every bin decided by the definition's
FP64 operations (values on and beside the bin edges), item orders the shared-memory rows do not cover, bin
counts on both sides of each limit, ragged sizes, and the unbinned estimator's chunks."""
import math

import numpy as np
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W

pytestmark = pytest.mark.gpu
LN10 = 2.302585092994046
M0 = W.PROTON["m0"]


def device_exits(lnP, status, item, lw=None):
    import torch
    n = len(lnP)
    out = cz.ExitBuffers(n, with_lw=lw is not None)
    for t in (out.r, out.th, out.ph, out.s):
        t.fill_(1.0)
    out.steps.fill_(1)
    out.lnP.copy_(torch.as_tensor(lnP))
    out.status.copy_(torch.as_tensor(status))
    out.item.copy_(torch.as_tensor(item.astype(np.int64)).to(torch.int32))
    if lw is not None:
        out.lw.copy_(torch.as_tensor(lw))
    return out


def table():
    T = np.logspace(-2, 4, 41)
    lnT, lnJ = np.log(T), np.log(T ** -2.7 / (1 + T ** -2.2))
    return cz.cosmica_lis(1, len(T), lnT.ctypes.data, lnJ.ctypes.data), lnT, lnJ


def lis_fn(tab):
    if tab is None:
        return lambda T: T ** -2.7 / (1 + T ** -3.7)
    return lambda T: np.exp(np.interp(np.log(T), tab[1], tab[2]))


@pytest.mark.parametrize("n,n_items,nbins,order,P_min,P_max,with_table", [
    (1, 1, 1, "sorted", 0.1, 1000.0, False),
    (257, 3, 64, "sorted", 0.1, 1000.0, True),
    (70001, 30, 512, "sorted", 0.1, 1000.0, False),
    (70001, 30, 512, "shuffled", 0.1, 1000.0, True),
    (300007, 2000, 512, "sorted", 0.1, 1000.0, False),
    (40000, 100, 333, "reversed", 0.03, 777.0, False),
    (90001, 7, 4096, "sorted", 0.1, 1000.0, False),
    (90001, 7, 4097, "sorted", 0.1, 1000.0, False),
    (20011, 4, 8189, "sorted", 0.1, 1000.0, False),
    (20011, 4, 8190, "sorted", 0.1, 1000.0, False),
    (5003, 2, 70000, "sorted", 0.1, 1000.0, False),
    (30000, 5, 512, "sorted", 2.0, 2.0001, False),
    (30000, 5, 512, "sorted", 1e-300, 1e300, False),
])
def test_binned(n, n_items, nbins, order, P_min, P_max, with_table):
    import torch
    rng = np.random.default_rng(n + nbins)
    x_lo = math.log10(P_min)
    dx = (math.log10(P_max) - x_lo) / nbins
    lnP = rng.normal(1.0, 2.0, n)
    k = n // 3           # a third on bin edges, and one unit in the last place to each side
    edge = (x_lo + rng.integers(0, nbins + 1, k) * dx) * LN10
    lnP[:k] = np.where(rng.random(k) < 0.3, edge, np.where(rng.random(k) < 0.5, np.nextafter(edge, 1e9), np.nextafter(edge, -1e9)))
    if n > 200:
        lnP[k:k + 8] = [0.0, -0.0, 15.999999, 16.0, -16.0, 700.0, -700.0, 1e-310]
    lnP = rng.permutation(lnP)
    status = np.where(rng.random(n) < 0.02, cz.PATH_STEP_LIMIT, cz.PATH_EXIT).astype(np.uint8)
    item = np.sort(rng.integers(0, n_items, n)).astype(np.uint32)
    if order == "shuffled":
        item = rng.permutation(item)
    elif order == "reversed":
        item = item[::-1].copy()
    if n > 1000:
        item[rng.integers(0, n, 5)] = n_items + 7        # out of range: not counted
    out = device_exits(lnP, status, item)
    tab = table() if with_table else None
    T = np.exp(rng.uniform(math.log(0.1), math.log(100.0), n_items))
    J, S = (torch.empty(n_items, dtype=torch.float64, device="cuda") for _ in range(2))
    H = torch.full((n_items * (nbins + 3),), -1, dtype=torch.int64, device="cuda")
    cz.cosmica_spectrum(out, cz.make_species(W.PROTON), list(T), cz.make_bins(P_min, P_max, nbins), J, S, H,
                        tab[0] if tab else None)
    with np.errstate(all="ignore"):
        b = np.floor((lnP / LN10 - x_lo) / dx)
    slot = np.where(b < 0, 0, np.where(b >= nbins, nbins + 1, b + 1)).astype(np.int64)
    slot[status != cz.PATH_EXIT] = nbins + 2
    ok = item < n_items
    want = np.bincount(item[ok].astype(np.int64) * (nbins + 3) + slot[ok], minlength=n_items * (nbins + 3))
    got = H.cpu().numpy()
    assert np.array_equal(got, want)
    if P_max > 1e10:
        return           # the bins' weights leave the double range
    with np.errstate(all="ignore"):
        Pb = 10.0 ** (x_lo + (np.arange(nbins) + 0.5) * dx)
        w = lis_fn(tab)(Pb * Pb / (np.sqrt(Pb * Pb + M0 * M0) + M0)) / Pb ** 2
        c = want.reshape(n_items, nbins + 3)[:, 1:nbins + 1].astype(np.float64)
        N = c.sum(1)
        mu = c @ w / N
        pref = T * (T + 2 * M0)
        sig = np.sqrt((c * (w - mu[:, None]) ** 2).sum(1) / (N - 1) / N)
        sig[N == 1] = 0.0
    # sums of positive terms and a few correctly rounded or 2-ulp functions: 1e-13 is far above both sides
    np.testing.assert_allclose(J.cpu().numpy(), pref * mu, rtol=1e-13, equal_nan=True)
    # sigma: the deviations w - mu lose up to mu / sigma of their digits
    np.testing.assert_allclose(S.cpu().numpy(), pref * sig, rtol=1e-13, atol=1e-13 * np.nanmax(np.append(pref * mu, 0.0)), equal_nan=True)


@pytest.mark.parametrize("form,with_table", [(0, False), (1, False), (1, True)])
@pytest.mark.parametrize("counts", [[1], [0, 2, 0, 127, 128, 129, 0], [1024, 1025, 3], [200000, 0, 1, 400001]])
def test_unbinned(counts, form, with_table):
    import torch
    rng = np.random.default_rng(sum(counts) + form)
    n, E = sum(counts), len(counts)
    lnP = rng.normal(1.0, 1.0, n)
    lw = -np.abs(rng.normal(0.5, 0.3, n))
    status = np.where(rng.random(n) < 0.01, cz.PATH_STEP_LIMIT, cz.PATH_EXIT).astype(np.uint8)
    out = device_exits(lnP, status, np.repeat(np.arange(E), counts).astype(np.uint32), lw if form else None)
    tab = table() if with_table else None
    T = np.exp(rng.uniform(math.log(0.1), math.log(100.0), E))
    J, S = (torch.empty(E, dtype=torch.float64, device="cuda") for _ in range(2))
    cz.cosmica_spectrum_unbinned(out, cz.make_species(W.PROTON), list(T), counts, form, J, S, tab[0] if tab else None)
    P = np.exp(lnP)
    En = np.sqrt(P * P + M0 * M0)
    w = lis_fn(tab)(P * P / (En + M0)) * (np.exp(lw) / (P / En) if form else 1.0 / P ** 2)
    at = np.concatenate([[0], np.cumsum(counts)])
    wJ, wS = np.full(E, np.nan), np.full(E, np.nan)
    for e in range(E):
        v = w[at[e]:at[e + 1]][status[at[e]:at[e + 1]] == cz.PATH_EXIT]
        P0 = math.sqrt(T[e] * (T[e] + 2 * M0))
        pref = P0 / math.sqrt(P0 * P0 + M0 * M0) if form else P0 * P0
        if len(v):
            wJ[e], wS[e] = pref * v.mean(), pref * v.std(ddof=1) / math.sqrt(len(v)) if len(v) > 1 else 0.0
    # a summand carries a few ulp (pow, exp, divisions), a sum of 4e5 positive terms at most 1e-13 more
    np.testing.assert_allclose(J.cpu().numpy(), wJ, rtol=1e-12, equal_nan=True)
    np.testing.assert_allclose(S.cpu().numpy(), wS, rtol=1e-12, equal_nan=True)


def test_calls_of_one_thread_on_two_streams():
    """The scratch of the handle-less calls is one per thread: calls on two streams that nothing else orders
    give what each gives alone."""
    import torch
    rng = np.random.default_rng(5)
    E, nbins, streams = 40, 2048, [torch.cuda.Stream() for _ in range(2)]
    T = list(np.exp(rng.uniform(-2.0, 4.0, E)))
    jobs = []
    for n in (4000000, 40000):
        item = np.sort(rng.integers(0, E, n)).astype(np.uint32)
        out = device_exits(rng.normal(1.0, 1.0, n), np.ones(n, np.uint8), item, -np.abs(rng.normal(0.5, 0.3, n)))
        jobs.append((out, [int(c) for c in np.bincount(item, minlength=E)]))
    sp, bins = cz.make_species(W.PROTON), cz.make_bins(0.1, 1000.0, nbins)

    def call(job, stream):
        out, counts = job
        r = [torch.empty(E, dtype=torch.float64, device="cuda") for _ in range(4)]
        H = torch.empty(E * (nbins + 3), dtype=torch.int64, device="cuda")
        stream.wait_stream(torch.cuda.current_stream())
        cz.cosmica_spectrum(out, sp, T, bins, r[0], r[1], H, stream=stream)
        cz.cosmica_spectrum_unbinned(out, sp, T, counts, 1, r[2], r[3], stream=stream)
        return r + [H]

    alone = []
    for j in jobs:
        alone.append(call(j, streams[0]))
        torch.cuda.synchronize()
    together = [[call(j, s) for j, s in zip(jobs, streams)] for _ in range(10)]
    torch.cuda.synchronize()
    for pair in together:
        for got, ref in zip(pair, alone):
            assert all(torch.equal(a, b) for a, b in zip(got, ref))
