"""The work a user has this framework do, one case per way of using it.

A case is one pass through the public entry points (`paper_2502_06319_gb300.cosmica`): exit states and
spectra of a set of quasi-particles, a batch of heliospheres, a set of served requests, or the spectra
of exit states that are already there.  The kinds:

  propagate   one heliosphere and species: cosmica_propagate (or its orbit or allocation-free entry) and
              the binned spectrum, or the unbinned one in the energy form
  batch       many heliospheres x species x energies: cosmica_batch_run and cosmica_batch_spectrum
  serve       spectrum requests handed to the continuous-batching server together
  binned      cosmica_batch_spectrum of given exit states
  unbinned    cosmica_spectrum_unbinned of given exit states
"""
import math

import numpy as np
import torch

from paper_2502_06319_gb300 import cosmica as cz
from paper_2502_06319_gb300 import workloads as W

PREC = {"fp64": cz.PREC_FP64, "mixed": cz.PREC_MIXED, "f64acc": cz.PREC_MIXED_F64ACC}


def listed():
    return [
        # the plain method on the spherically symmetric model: 1e4 protons of 1 GeV, fixed step (workloads.config0)
        dict(name="fp64_isotropic", kind="propagate", entry="model", model="isotropic", prec="fp64", form=0,
             species="proton", n_e=1, T_lo=1.0, T_hi=1.0, n=10000, uneven=False, nbins=64),
        # a handful of FP64 paths of the full model, as one checks a heliosphere or another precision with
        dict(name="fp64_few", kind="propagate", entry="model", model="full", prec="fp64", form=0,
             species="proton", n_e=4, T_lo=5.0, T_hi=100.0, n=24, uneven=False, nbins=512),
        # an FP64 spectrum of the full model: workloads.config1 at its higher energies and half its counts
        dict(name="fp64_spectrum", kind="propagate", entry="model", model="full", prec="fp64", form=0,
             species="proton", n_e=10, T_lo=5.0, T_hi=100.0, n=2500, uneven=False, nbins=512),
        # the smallest mixed call: three energies with a few quasi-particles each, one heliosphere
        dict(name="mixed_few", kind="propagate", entry="model", model="full", prec="mixed", form=0,
             species="proton", n_e=3, T_lo=0.3, T_hi=10.0, n=200, uneven=False, nbins=512),
        # one spectrum at its usual size (workloads.config2: 30 energies x 20 000)
        dict(name="mixed_spectrum", kind="propagate", entry="model", model="full", prec="mixed", form=0,
             species="proton", n_e=30, T_lo=0.1, T_hi=100.0, n=20000, uneven=False, nbins=512),
        # heliospheres with a shock, FP32 coefficients and FP64 accumulation (workloads.config3 as it names it)
        dict(name="batch_f64acc", kind="batch", model="shock", prec="f64acc", form=0, n_sets=4, n_e=30,
             scale=0.025, graph=False),
        # a batch of heliospheres at its usual precision: a quarter of workloads.config3's sets, uneven counts
        dict(name="batch_mixed", kind="batch", model="shock", prec="mixed", form=0, n_sets=16, n_e=30,
             scale=0.1, graph=False),
        # a year of observations through 15 radial shells, replayed as a graph (workloads.config_shells)
        dict(name="batch_shells", kind="batch", model="shells", prec="mixed", form=0, n_sets=13, n_e=30,
             scale=0.02, graph=True),
        # the energy form in a nose-squashed heliosphere seen along an orbit, odd and uneven counts, unbinned
        dict(name="orbit_energy_squashed", kind="propagate", entry="orbit", model="squashed", prec="mixed", form=1,
             species="he4", n_e=13, T_lo=0.2, T_hi=50.0, n=1501, uneven=True, nbins=512),
        # requests that arrive together at the server (workloads.config4 at a tenth of its counts)
        dict(name="serve", kind="serve", prec="mixed", n_req=4, scale=0.1),
        # spectra of a whole batch from its exit states: 64 heliospheres x 3 species x 30 energies
        dict(name="spectra_binned", kind="binned", n_items=5760, n=16000001, nbins=512, table=False),
        # the unbinned, loss-weighted estimator on one spectrum's exit states (30 energies x 20 000)
        dict(name="spectra_unbinned", kind="unbinned", n_items=30, n=600000, form=1, table=False),
    ]


def _log(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def _log_int(rng, lo, hi):
    return int(round(_log(rng, lo, hi)))


def draw(rng):
    kind = rng.choice(("propagate", "propagate", "propagate", "batch", "batch", "serve", "binned", "unbinned"))
    if kind == "propagate":
        prec = rng.choice(("fp64", "mixed", "mixed", "f64acc"))
        model = rng.choice(("isotropic", "full", "full", "shock", "shells", "squashed"))
        n_e = rng.randint(1, 30)
        c = dict(kind=kind, entry=rng.choice(("model", "model", "orbit", "noalloc")), model=model, prec=prec,
                 form=rng.choice((0, 0, 1)), species=rng.choice(("proton", "he4", "electron")), n_e=n_e,
                 T_lo=_log(rng, 0.1, 1.0), T_hi=_log(rng, 10.0, 100.0), uneven=rng.random() < 0.5,
                 nbins=_log_int(rng, 32, 1024))
        if prec == "fp64":
            # plain FP64 paths are run at the energies whose paths are short
            c.update(T_lo=_log(rng, 3.0, 10.0), T_hi=_log(rng, 20.0, 100.0), n=max(1, _log_int(rng, 24, 10000) // n_e))
            if model != "isotropic":
                c.update(model="full", species="proton")
        elif prec == "f64acc":
            c.update(n=max(1, _log_int(rng, 100, 60000) // n_e))
        else:
            c.update(n=max(1, _log_int(rng, 100, 400000) // n_e))
        return c
    if kind == "batch":
        prec = rng.choice(("mixed", "mixed", "f64acc"))
        model = rng.choice(("shock", "shock", "shells", "squashed"))
        n_sets = _log_int(rng, 2, 40) if model != "shells" else rng.randint(2, 13)
        n_e = rng.randint(5, 30)
        most = 700000 if prec == "mixed" else 100000          # particles
        per = n_sets * (2 if model == "shells" else 3) * n_e * 12500.0   # of scale 1
        return dict(kind=kind, model=model, prec=prec, form=rng.choice((0, 0, 0, 1)), n_sets=n_sets, n_e=n_e,
                    scale=_log(rng, 2000, most) / per, graph=rng.random() < 0.5)
    if kind == "serve":
        return dict(kind=kind, prec=rng.choice(("mixed", "mixed", "f64acc")), n_req=rng.randint(1, 6),
                    scale=_log(rng, 0.002, 0.03))
    if kind == "binned":
        return dict(kind=kind, n_items=_log_int(rng, 1, 5760), n=_log_int(rng, 1000, 16000000),
                    nbins=_log_int(rng, 32, 1024), table=rng.random() < 0.5)
    return dict(kind=kind, n_items=_log_int(rng, 1, 200), n=_log_int(rng, 1000, 2000000), form=rng.choice((0, 1)),
                table=rng.random() < 0.5)


# ------------------------------------------------------------------ inputs --
def _model(case):
    """Parameter record of the case's heliosphere."""
    m = case["model"]
    shock = dict(R_ts=85.0, ts_K_factor=0.5, R_out=122.0)
    if m == "isotropic":
        p = dict(W.config0().params)
    elif m == "full":
        p = W.params()
    elif m == "shock":
        p = W.params(tilt_deg=35.0, polarity=-1.0, **shock)
    elif m == "shells":
        p = W.shell_params(W.solar_cycle_series(), 40)
    else:
        p = W.params(tilt_deg=35.0, **shock, **W.SQUASHED)
    return dict(p, formulation=float(case["form"]))


def _energies(case):
    n = case["n_e"]
    return [case["T_lo"]] if n == 1 else W.logspace(case["T_lo"], case["T_hi"], n)


def _counts(case):
    if not case["uneven"]:
        return [case["n"]] * case["n_e"]
    f = np.exp(np.random.default_rng(case["n_e"]).uniform(math.log(0.25), math.log(2.0), case["n_e"]))
    return [max(1, int(round(case["n"] * x))) for x in f]


def _spectra(n, nbins):
    J = torch.empty(n, dtype=torch.float64, device="cuda")
    return J, torch.empty_like(J), torch.empty(n * (nbins + 3), dtype=torch.int64, device="cuda")


def _exit_dict(out):
    d = {k: getattr(out, k) for k in ("r", "th", "ph", "lnP", "s", "steps", "status", "item")}
    if out.lw is not None:
        d["lw"] = out.lw
    return d


class _Handle:
    """A batch or server handle that is given back with its owner."""

    def __init__(self, h, destroy):
        self.h, self._destroy = h, destroy

    def __del__(self):
        try:
            self._destroy(self.h)
        except Exception:
            pass


def _jobs(case, seed):
    """A batch's jobs: energies and counts of the workload, heliospheres and particle identities of the seed."""
    n = case["n_sets"]
    if case["model"] == "shells":
        jobs = W.config_shells(n_obs=n, n_e=case["n_e"], scale=case["scale"])
        sets = [W.shell_params(W.solar_cycle_series(seed), 40 + i) for i in range(n)]
    else:
        jobs = W.config3(n_sets=n, n_e=case["n_e"], scale=case["scale"])
        shape = W.SQUASHED if case["model"] == "squashed" else {}
        sets = [dict(p, **{k: float(v) for k, v in shape.items()}) for p in W.config3_param_sets(seed, n)]
    for i, j in enumerate(jobs):
        j.params = dict(sets[i * n // len(jobs)], formulation=float(case["form"]))
        j.seed += 1000 * seed
    return jobs


def _requests(case, seed):
    """Requests of the serving stream: its species, energies and counts, heliospheres and identities of the seed."""
    jobs = [q.job for q in W.config4(n_requests=case["n_req"], scale=case["scale"])]
    for p, j in zip(W.config3_param_sets(seed, len(jobs)), jobs):
        j.params, j.seed = p, j.seed + 1000 * seed
    return jobs


_TABLE_T = np.logspace(-2.0, 4.0, 61)     # a tabulated local interstellar spectrum [GeV/n]


def _lis():
    """A log-log table of a local interstellar spectrum; the arrays stay with the record."""
    lnT = np.ascontiguousarray(np.log(_TABLE_T))
    lnJ = np.ascontiguousarray(np.log(_TABLE_T ** -2.7 / (1.0 + 0.8 * _TABLE_T ** -2.5)))
    rec = cz.cosmica_lis(1, len(lnT), lnT.ctypes.data, lnJ.ctypes.data)
    return rec, lnT, lnJ


def _exit_items(case, seed):
    """(T, n) per item of given exit states: uneven counts that add up to the case's n."""
    n_items, n = case["n_items"], case["n"]
    rng = np.random.default_rng(seed)
    w = np.exp(rng.uniform(0.0, math.log(50.0), n_items))
    cut = np.floor(np.cumsum(w) / w.sum() * n).astype(np.int64)
    cut[-1] = n
    return np.exp(rng.uniform(math.log(0.1), math.log(100.0), n_items)), np.diff(np.concatenate([[0], cut]))


def _given_exits(case, seed):
    """Exit states as a propagation leaves them: ln P above the start's by an energy-dependent spread."""
    T, counts = _exit_items(case, seed)
    n = case["n"]
    g = torch.Generator(device="cuda").manual_seed(seed)
    out = cz.ExitBuffers(n, with_lw=case["kind"] == "unbinned" and case["form"] == 1)
    item = torch.repeat_interleave(torch.arange(len(T), device="cuda"), torch.as_tensor(counts, device="cuda"))
    P0 = torch.as_tensor(0.5 * np.log(T * (T + 2 * W.PROTON["m0"])), device="cuda")
    rise = torch.as_tensor(0.9 / (1.0 + T), device="cuda")
    z = torch.randn(n, dtype=torch.float64, device="cuda", generator=g)
    out.lnP.copy_(P0[item] + (0.05 + rise[item]) * torch.exp(0.35 * z))
    u = torch.rand(n, dtype=torch.float64, device="cuda", generator=g)
    out.status.copy_(torch.where(u < 1e-3, cz.PATH_STEP_LIMIT, cz.PATH_EXIT))
    out.item.copy_(item)
    for t, v in ((out.r, 122.0), (out.th, 1.5), (out.ph, 3.0), (out.s, 100.0)):
        t.fill_(v)
    out.steps.fill_(1000)
    if out.lw is not None:
        out.lw.copy_(-2.0 * (out.lnP - P0[item]))
    return T, counts, out


def prepare(case, seed):
    kind = case["kind"]
    s = {"kind": kind}
    if kind == "propagate":
        s["params"] = cz.make_params(_model(case), PREC[case["prec"]])
        s["entry"], s["form"], s["seed"] = case["entry"], case["form"], 1 + seed
        s["species"] = cz.make_species(W.SPECIES[case["species"]])
        s["T"] = _energies(case)
        s["N"] = _counts(case)
        if s["entry"] != "noalloc":
            s["model"] = cz.Model(s["params"])
        s["orbit"] = W.polar_orbit()
        s["bins"] = cz.make_bins(0.1, 1000.0, case["nbins"])
        s["out"] = cz.ExitBuffers(sum(s["N"]), with_lw=case["form"] == 1)
        s["J"], s["S"], s["H"] = _spectra(len(s["T"]), case["nbins"])
    elif kind == "batch":
        params, species, items = W.items_of(_jobs(case, seed))
        pc = [cz.make_params(p, PREC[case["prec"]]) for p in params]
        s["batch"] = _Handle(cz.cosmica_batch_create(pc, [cz.make_species(x) for x in species]), cz.cosmica_batch_destroy)
        s["items"], s["n_items"] = cz.make_items(items), len(items)
        s["out"] = cz.ExitBuffers(sum(it[3] for it in items), with_lw=case["form"] == 1)
        s["bins"] = cz.make_bins(0.1, 1000.0, 512)
        s["J"], s["S"], s["H"] = _spectra(len(items), 512)
        # a program that replays its launch as a graph runs on a stream of its own
        s["tuning"] = cz.cosmica_tuning(128, 4, 64, 1, 1) if case["graph"] else None
        s["stream"] = torch.cuda.Stream() if case["graph"] else None
    elif kind == "serve":
        s["server"] = _Handle(cz.cosmica_server_create(1 << 30, PREC[case["prec"]]), cz.cosmica_server_destroy)
        bins = cz.make_bins(0.1, 1000.0, 512)
        s["requests"] = [cz.Request(cz.make_params(j.params, PREC[case["prec"]]), cz.make_species(j.species),
                                    j.T_in, j.n_per_energy, j.seed, bins) for j in _requests(case, seed)]
    else:
        T, counts, s["out"] = _given_exits(case, seed)
        s["T"], s["N"] = [float(t) for t in T], [int(n) for n in counts]
        s["lis"] = _lis() if case["table"] else None
        s["species"] = cz.make_species(W.PROTON)
        if kind == "binned":
            s["batch"] = _Handle(cz.cosmica_batch_create([cz.make_params(W.params(), cz.PREC_MIXED)], [s["species"]]),
                                 cz.cosmica_batch_destroy)
            s["items"] = cz.make_items([(0, 0, t, n, 0, 1) for t, n in zip(s["T"], s["N"])])
            s["bins"] = cz.make_bins(0.1, 1000.0, case["nbins"])
            s["J"], s["S"], s["H"] = _spectra(len(T), case["nbins"])
        else:
            s["form"] = case["form"]
            s["J"], s["S"], _ = _spectra(len(T), 1)
    return s


# --------------------------------------------------------------- one pass --
def run(s):
    kind = s["kind"]
    if kind == "propagate":
        out = s["out"]
        if s["entry"] == "model":
            cz.cosmica_propagate(s["model"].h, s["species"], s["T"], s["N"], s["seed"], out)
        elif s["entry"] == "orbit":
            cz.cosmica_propagate_orbit(s["model"].h, s["species"], s["T"], s["N"], s["orbit"], s["seed"], out)
        else:
            cz.cosmica_propagate_noalloc(s["params"], s["species"], s["T"], s["N"], s["seed"], out)
        r = _exit_dict(out)
        if s["form"] == 1:
            cz.cosmica_spectrum_unbinned(out, s["species"], s["T"], s["N"], 1, s["J"], s["S"])
        else:
            cz.cosmica_spectrum(out, s["species"], s["T"], s["bins"], s["J"], s["S"], s["H"])
            r["hist"] = s["H"]
        return dict(r, J=s["J"], sigma=s["S"])
    if kind == "batch":
        if s["stream"] is not None:
            s["stream"].wait_stream(torch.cuda.current_stream())
        cz.cosmica_batch_run(s["batch"].h, s["items"], s["n_items"], s["out"], s["tuning"], stream=s["stream"])
        cz.cosmica_batch_spectrum(s["batch"].h, s["items"], s["n_items"], s["out"], s["bins"], s["J"], s["S"], s["H"],
                                  stream=s["stream"])
        if s["stream"] is not None:
            torch.cuda.current_stream().wait_stream(s["stream"])
        return dict(_exit_dict(s["out"]), J=s["J"], sigma=s["S"], hist=s["H"])
    if kind == "serve":
        tickets = [cz.cosmica_server_submit(s["server"].h, q) for q in s["requests"]]
        got = []
        for t, q in zip(tickets, s["requests"]):
            res = cz.Result(q.n_energies, q.nbins)
            cz.cosmica_server_wait(s["server"].h, t, res)
            got.append({"J": res.J, "sigma": res.sigma, "hist": res.hist.view(np.int64), "steps": int(res.steps)})
        return got
    lis = s["lis"][0] if s["lis"] else None
    if kind == "binned":
        cz.cosmica_batch_spectrum(s["batch"].h, s["items"], len(s["T"]), s["out"], s["bins"], s["J"], s["S"], s["H"], lis)
        return {"J": s["J"], "sigma": s["S"], "hist": s["H"]}
    cz.cosmica_spectrum_unbinned(s["out"], s["species"], s["T"], s["N"], s["form"], s["J"], s["S"], lis)
    return {"J": s["J"], "sigma": s["S"]}


# ------------------------------------------------------ what a pass needs --
_STEP_FLOPS = 382      # operations of one step of the full model with a shock, each function call as one


def _mean_steps(model, T, charge_polarity=1.0):
    """Mean steps of a path (a fit to measured means of the workloads' models, within a factor of two)."""
    if model == "isotropic":
        return 812.0
    x = math.log(T)
    far = 0.0 if model == "full" else 0.5
    return max(1400.0, math.exp(9.5 + far - 0.55 * x - 0.04 * x * x + 0.01 * x ** 3 + (1.0 if charge_polarity < 0 else 0.0)))


def work(case):
    kind = case["kind"]
    if kind == "propagate":
        N = _counts(case)
        sign = -1.0 if case["model"] == "shock" else 1.0
        if case["species"] == "electron":
            sign = -sign
        steps = sum(n * _mean_steps(case["model"], T, sign) for n, T in zip(N, _energies(case)))
        return {"bytes": 49.0 * sum(N) + 8.0 * case["n_e"] * (case["nbins"] + 5), "flops": steps * _STEP_FLOPS}
    if kind == "batch":
        steps = n = items = 0
        for j in _jobs(case, 1):
            q = j.params["polarity"] * (1.0 if j.species["Z"] > 0 else -1.0)
            steps += sum(c * _mean_steps(case["model"], T, q) for T, c in zip(j.T_in, j.n_per_energy))
            n += j.n_particles
            items += len(j.T_in)
        return {"bytes": 49.0 * n + items * (64.0 + 8.0 * 517), "flops": steps * _STEP_FLOPS}
    if kind == "serve":
        steps = items = 0
        for j in _requests(case, 1):
            s = j.params["polarity"] * (1.0 if j.species["Z"] > 0 else -1.0)
            steps += sum(c * _mean_steps("shock", T, s) for T, c in zip(j.T_in, j.n_per_energy))
            items += len(j.T_in)
        return {"bytes": items * 8.0 * 517, "flops": steps * _STEP_FLOPS}
    if kind == "binned":      # status, ln P and item of every exit state; histogram, J and sigma
        return {"bytes": 13.0 * case["n"] + 8.0 * case["n_items"] * (case["nbins"] + 5), "flops": 10.0 * case["n"]}
    # status, ln P and, in the energy form, the loss weight of every exit state; J and sigma
    return {"bytes": (17.0 if case["form"] else 9.0) * case["n"] + 16.0 * case["n_items"], "flops": 30.0 * case["n"]}


# ------------------------------------------------ the same in 64 bits -----
def _slots(lnP, nbins):
    """Histogram slot of each exit rigidity on [0.1, 1000) GV."""
    return np.clip(np.floor((lnP / math.log(10.0) + 1.0) / (4.0 / nbins)), -1, nbins).astype(np.int64) + 1


def _spectrum_of_bins(hist, nbins, T0, A, Z, m0, lis):
    """J and sigma of one item's histogram row, by the estimator's definition."""
    c = hist[1:nbins + 1].astype(np.float64)
    N = c.sum()
    if N == 0:
        return math.nan, math.nan
    dx = 4.0 / nbins
    Pb = 10.0 ** (-1.0 + (np.arange(nbins) + 0.5) * dx)
    pn = Pb * abs(Z) / A
    w = lis(pn * pn / (np.sqrt(pn * pn + m0 * m0) + m0)) / Pb ** 2
    pref = (A / abs(Z)) ** 2 * T0 * (T0 + 2 * m0)
    mu = (c * w).sum() / N
    return pref * mu, pref * math.sqrt((c * (w - mu) ** 2).sum() / (N - 1.0) / N) if N > 1 else 0.0


def _lis_value(table):
    if not table:
        return lambda T: T ** -2.7 / (1.0 + T ** -3.7)
    _, lnT, lnJ = _lis()
    return lambda T: np.exp(np.interp(np.log(T), lnT, lnJ))


def _philox(c0, pid, seed):
    """Philox4x32-10 of the counters (c0, pid, 0, 0) with a 32-bit key, as float64 uniforms on (0, 1)."""
    lo = np.uint64(0xFFFFFFFF)
    x = [c0.astype(np.uint64), pid.astype(np.uint64), np.zeros_like(pid, dtype=np.uint64), np.zeros_like(pid, dtype=np.uint64)]
    k0, k1 = seed & 0xFFFFFFFF, seed >> 32
    for _ in range(10):
        a, b = np.uint64(0xD2511F53) * x[0], np.uint64(0xCD9E8D57) * x[2]
        x = [(b >> np.uint64(32)) ^ x[1] ^ np.uint64(k0), b & lo, (a >> np.uint64(32)) ^ x[3] ^ np.uint64(k1), a & lo]
        k0, k1 = (k0 + 0x9E3779B9) & 0xFFFFFFFF, (k1 + 0xBB67AE85) & 0xFFFFFFFF
    return [(w.astype(np.float64) + 0.5) * 2.0 ** -32 for w in x]


def _isotropic_paths(p, m0, T, n, seed):
    """Exit radius, ln P and time of the isotropic model with a fixed step: Euler-Maruyama in float64 (the angles
    of a path that comes close to a pole separate like those of a path through the current sheet)."""
    dt, R, r_in = p["dt_fixed"], p["R_out"], p["r_in"]
    V = p["V_const_kms"] * 86400.0 / 1.495978707e8
    pid = np.concatenate([np.arange(sum(n[:e]), sum(n[:e + 1])) for e in range(len(n))])
    lnP = np.concatenate([np.full(c, 0.5 * math.log(t * (t + 2 * m0))) for t, c in zip(T, n)])
    r, th, ph = np.full(len(pid), p["r0"]), np.full(len(pid), p["th0"]), np.full(len(pid), p["ph0"])
    out = {k: np.empty(len(pid)) for k in ("r", "lnP", "s")}
    live, k, s, sdt = np.arange(len(pid)), 0, 0.0, math.sqrt(dt)
    while len(live):
        u = _philox(np.full(len(live), k), pid[live], seed)
        rho0, rho2 = np.sqrt(-2.0 * np.log(u[0])), np.sqrt(-2.0 * np.log(u[2]))
        z = rho0 * np.cos(2 * math.pi * u[1]), rho0 * np.sin(2 * math.pi * u[1]), rho2 * np.cos(2 * math.pi * u[3])
        P = np.exp(lnP)
        K = p["K0"] * P / np.sqrt(P * P + m0 * m0) * P
        L, sn = np.sqrt(2.0 * K) * sdt, np.sin(th)
        dr = (2.0 * K / r - V) * dt + L * z[0]
        dth = K * np.cos(th) / sn / r ** 2 * dt + L * z[1] / r
        dph = L * z[2] / (r * sn)
        lnP = lnP + 2.0 * V / (3.0 * r) * dt
        r, th, ph = r + dr, th + dth, ph + dph
        r = np.where(r < r_in, 2 * r_in - r, r)
        th = th - 2 * math.pi * np.floor(th / (2 * math.pi))
        ph = np.where(th > math.pi, ph + math.pi, ph)
        th = np.where(th > math.pi, 2 * math.pi - th, th)
        ph = ph - 2 * math.pi * np.floor(ph / (2 * math.pi))
        k, s = k + 1, s + dt
        end = r >= R
        for a, v in zip(("r", "lnP"), (r, lnP)):
            out[a][live[end]] = v[end]
        out["s"][live[end]] = s
        r, th, ph, lnP, live = r[~end], th[~end], ph[~end], lnP[~end], live[~end]
    return out


def exact(case, seed):
    """Outputs that plain numpy can give: spectra of given exit states, and the isotropic model's paths in
    FP64.  Paths through the wavy current sheet separate on the first differing rounding, and mixed paths
    are FP32 steps, so the other cases have no such value."""
    kind = case["kind"]
    m0 = W.PROTON["m0"]
    if kind in ("binned", "unbinned"):
        T, counts, out = _given_exits(case, seed)
        lnP, ok = out.lnP.cpu().numpy(), out.status.cpu().numpy() == cz.PATH_EXIT
        lis = _lis_value(case["table"])
        J, S = np.empty(len(T)), np.empty(len(T))
        at = np.concatenate([[0], np.cumsum(counts)])
        if kind == "binned":
            nb = case["nbins"]
            b = np.where(ok, _slots(lnP, nb), nb + 2)
            for e in range(len(T)):
                J[e], S[e] = _spectrum_of_bins(np.bincount(b[at[e]:at[e + 1]], minlength=nb + 3), nb, T[e], 1, 1, m0, lis)
            return {"J": J, "sigma": S, "hist": None}
        P = np.exp(lnP)
        En = np.sqrt(P * P + m0 * m0)
        w = lis(P * P / (En + m0))
        if case["form"]:
            w = w * np.exp(out.lw.cpu().numpy()) / (P / En)
        else:
            w = w / P ** 2
        for e in range(len(T)):
            v = w[at[e]:at[e + 1]][ok[at[e]:at[e + 1]]]
            P0 = math.sqrt(T[e] * (T[e] + 2 * m0))
            pref = P0 / math.sqrt(P0 * P0 + m0 * m0) if case["form"] else P0 * P0
            J[e] = pref * v.mean() if len(v) else math.nan
            S[e] = (pref * v.std(ddof=1) / math.sqrt(len(v)) if len(v) > 1 else 0.0) if len(v) else math.nan
        return {"J": J, "sigma": S}
    if kind != "propagate" or case["model"] != "isotropic" or case["prec"] != "fp64" or case["entry"] == "orbit" \
            or case["form"] != 0 or case["species"] != "proton":
        return None
    T, N = _energies(case), _counts(case)
    if sum(n * t for n, t in zip(N, T)) > 2e5:     # a path's steps fall with T, the noise's cost does not
        return None
    nb = case["nbins"]
    paths = _isotropic_paths(_model(case), m0, T, N, 1 + seed)
    slots = np.split(_slots(paths["lnP"], nb), np.cumsum(N)[:-1])
    J, S = np.array([_spectrum_of_bins(np.bincount(b, minlength=nb + 3), nb, t, 1, 1, m0, _lis_value(False))
                     for b, t in zip(slots, T)]).T
    return dict(dict.fromkeys(("th", "ph", "steps", "status", "item", "hist")), J=J, sigma=S, **paths)
