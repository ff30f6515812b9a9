"""The vote of the FP64-accumulated step on the new radius (csrc/f64bits.h): when it passes, the FP64 radius lies
between the boundaries, also after a step from far out that ends beside the inner one."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "f64bits.h"
using namespace cosmica::f64bits;
extern "C" void vote(const float *fr, const float *dr, float r_in, float R, int sphere, uint8_t *o, int n)
{
    const float lo = vote_floor(r_in, R), hi = vote_ceiling(R);
    for (int i = 0; i < n; ++i) {
        const float nr = fr[i] + dr[i];
        o[i] = (nr > lo) & (sphere ? nr < hi : dr[i] < kMostRise);
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("vote")
    (d / "t.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2502_06319_gb300", "csrc"), str(d / "t.cpp"), "-o", str(d / "t.so")], check=True)
    return C.CDLL(str(d / "t.so"))


@pytest.mark.parametrize("r_in,R", [(0.1, 100.0), (0.05, 122.0), (0.3, 20.0), (1e-3, 1e5)])
def test_passed_radii_are_inside(lib, r_in, R):
    f = np.float32
    rng = np.random.default_rng(7)
    n = 1 << 21
    inner = np.float64(f(r_in))
    r = np.exp(rng.uniform(np.log(inner), np.log(R), n))
    fr = r.astype(f)
    o = np.empty(n, np.uint8)
    p = lambda a: a.ctypes.data_as(C.c_void_p)
    passed = 0
    # steps that end within a few roundings of a boundary, by the old radius, by the boundary, or anywhere
    for target in (inner + rng.uniform(-3e-7, 3e-7, n) * r, inner * (1.0 + rng.uniform(-3e-6, 3e-6, n)),
                   R * (1.0 + rng.uniform(-3e-6, 3e-6, n)), np.exp(rng.uniform(np.log(inner), np.log(R), n)),
                   r * (1.0 + rng.uniform(-0.1, 0.1, n))):
        dr = (target - r).astype(f)
        lib.vote(p(fr), p(dr), C.c_float(r_in), C.c_float(R), 1, p(o), n)
        new = r + dr.astype(np.float64)
        assert np.all((new[o == 1] >= inner) & (new[o == 1] < R))
        passed += int(o.sum())
    if R < 1e4 * r_in:
        assert o.mean() > 0.9 and passed > 1.5 * n      # and it passes what is well inside
    for bad in (np.inf, -np.inf, np.nan):
        dr = np.full(n, bad, f)
        lib.vote(p(fr), p(dr), C.c_float(r_in), C.c_float(R), 0, p(o), n)
        assert not o.any()
