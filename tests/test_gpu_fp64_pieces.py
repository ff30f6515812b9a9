"""The pieces of the fast FP64 step against what they replace, bit for bit: the quotient against IEEE division
(quotients nearest a rounding boundary among them), floor, the uniforms and the elementary functions against
those of the definition, over the ranges that the step uses and at their ends."""
import numpy as np
import pytest

from paper_2502_06319_gb300 import cosmica as cz
from tests.gpu_util import torch

pytestmark = pytest.mark.gpu


def piece(name, x, b=None):
    t = torch()
    dx, db = t.as_tensor(x, device="cuda"), None if b is None else t.as_tensor(b, device="cuda")
    y = t.empty_like(dx)
    cz.cosmica_debug_step64(name, dx, y, db)
    return y.cpu().numpy()


def definition(name, x):
    t = torch()
    dx = t.as_tensor(x, device="cuda")
    y = t.empty_like(dx)
    cz.cosmica_debug_fn64(name, dx, y)
    return y.cpu().numpy()


def same(got, want):
    bad = np.flatnonzero(got.view(np.uint64) != want.view(np.uint64))
    assert len(bad) == 0, (len(bad), bad[:3], got[bad[:3]], want[bad[:3]])


def nearest_midpoints(rng, B):
    """(a, b) with integer b and a / b as near as it gets to the middle of two neighbouring doubles: a 2^k = Q b +- 1
    with an odd Q of 54 bits."""
    a, b = [], []
    for v in B:
        v = int(v)
        for k in range(53, 57):
            inv = pow(2, -k, v)
            a += [inv, v - inv]
            b += [v, v]
    return np.array(a, float), np.array(b, float)


def test_quotients():
    rng = np.random.default_rng(1)
    n = 1 << 21
    m = lambda: rng.integers(2 ** 52, 2 ** 53, n).astype(float)
    sign = np.where(rng.random(n) < 0.5, -1.0, 1.0)
    # all mantissas, exponents over the whole range with a normal quotient
    eb = rng.integers(-999, 999, n)
    ea = np.clip(eb + rng.integers(-900, 900, n), -950, 999)
    a, b = np.ldexp(m(), ea - 53) * sign, np.ldexp(m(), eb - 53)
    with np.errstate(all="ignore"):
        ok = (np.abs(a / b) > 1e-300) & (np.abs(a / b) < 1e300)
    assert ok.mean() > 0.5
    same(piece("quotient", a[ok], b[ok]), a[ok] / b[ok])
    # exact quotients and their neighbours
    q, b = m(), rng.integers(1, 2 ** 20, n) * 2.0 + 1.0
    a = q * b
    for x in (a, np.nextafter(a, 0.0), np.nextafter(a, np.inf)):
        same(piece("quotient", x, b), x / b)
    ends = np.array([0.0, -0.0, 1.0, 3.0]), np.array([3.0, 3.0, 2.0 ** -999, 2.0 ** 999])
    same(piece("quotient", *ends), ends[0] / ends[1])


def test_quotients_next_to_midpoints():
    rng = np.random.default_rng(2)
    B = rng.integers(2 ** 51, 2 ** 52, 20000) * 2 + 1
    a, b = nearest_midpoints(rng, B)
    e = rng.integers(-300, 300, len(a))
    same(piece("quotient", np.ldexp(a, e), b), np.ldexp(a, e) / b)


def test_integers_and_scaling():
    rng = np.random.default_rng(3)
    k = rng.integers(-2 ** 20 + 1, 2 ** 20, 200000).astype(float)
    x = np.concatenate([k, np.nextafter(k, np.inf), np.nextafter(k, -np.inf), rng.uniform(-1.0, 1.0, 200000) * 2.0 ** 20,
                        rng.uniform(-2.0, 2.0, 100000), [0.0, -0.0, 1e-300, -1e-300, 5e-324, -5e-324, 0.5, -0.5, 1.0, -1.0,
                                                         2.0 ** 20 - 2.0 ** -33, -2.0 ** 20 + 2.0 ** -33]])
    x = x[np.abs(x) < 2.0 ** 20]
    same(piece("floor", x), np.floor(x) + 0.0)          # an integer has no negative zero
    w = np.concatenate([rng.integers(0, 2 ** 32, 500000), [0, 1, 2, 3, 2 ** 31 - 1, 2 ** 31, 2 ** 32 - 2, 2 ** 32 - 1],
                        2 ** np.arange(32), 2 ** np.arange(1, 33) - 1]).astype(float)
    same(piece("uniform", w), (w + 0.5) * 2.3283064365386963e-10)
    x = np.concatenate([np.exp(rng.uniform(-700, 700, 100000)), [0.0, -0.0, 2.3e-308]])
    same(piece("twice", np.concatenate([x, -x])), 2.0 * np.concatenate([x, -x]))


@pytest.mark.parametrize("name,fn,x", [
    ("exp", "exp", lambda r: np.concatenate([r.uniform(-40, 40, 500000), r.uniform(-699, 699, 500000), [0.0, -0.0, 40.0, 1e-300]])),
    ("log", "log", lambda r: np.concatenate([np.exp(r.uniform(-700, 700, 500000)), 1.0 - r.random(200000), 1.0 + r.random(200000),
                                             [1.0, np.sqrt(2.0), np.nextafter(np.sqrt(2.0), 2.0), np.nextafter(np.sqrt(2.0), 1.0),
                                              2.0 ** -33, 1.0 - 2.0 ** -33, 2.3e-308, 1.7e308]])),
    ("sin", "sin", lambda r: np.concatenate([r.uniform(0, 7, 500000), r.uniform(-1e6, 1e6, 500000), [0.0, np.pi, np.pi / 2]])),
    ("cos", "cos", lambda r: np.concatenate([r.uniform(0, 7, 500000), r.uniform(-1e6, 1e6, 500000), [0.0, np.pi, np.pi / 2]])),
    ("cos alone", "cos", lambda r: np.concatenate([r.uniform(0, 7, 500000), r.uniform(-1e6, 1e6, 500000), [0.0, np.pi, np.pi / 2]])),
    ("atan", "atan", lambda r: np.concatenate([r.uniform(-2, 2, 500000), np.exp(r.uniform(-600, 600, 300000)),
                                               -np.exp(r.uniform(-600, 600, 300000)),
                                               [0.0, 1.0, -1.0, 0.66817863791929891, 0.19891236737965800, 60.0, -60.0]])),
])
def test_functions(name, fn, x):
    x = x(np.random.default_rng(4))
    same(piece(name, x), definition(fn, x))
