"""The quotient of the CP-ALS solves (csrc/fcs_div.cuh), compiled for the host,
against float32 division: within one unit in the last place, and the same
infinities, zeros and NaN."""
from __future__ import annotations

import ctypes as C
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))),
                    "paper_2106_13062_gb300", "csrc")

SOURCE = """
#include "fcs_div.cuh"
extern "C" void quotients(long n, const float *x, const float *g, int inf, float *out) {
  for (long i = 0; i < n; ++i)
    out[i] = inf ? fcs::quotient<true>(x[i], g[i], 1.f / g[i])
                 : fcs::quotient<false>(x[i], g[i], 1.f / g[i]);
}
"""


@pytest.fixture(scope="module")
def quotients(tmp_path_factory):
    d = tmp_path_factory.mktemp("quotient")
    (d / "q.cpp").write_text(SOURCE)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC",
                    f"-I{CSRC}", "-o", str(d / "q.so"), str(d / "q.cpp")], check=True)
    lib = C.CDLL(str(d / "q.so"))

    def run(x, g, inf):
        x, g = (np.ascontiguousarray(a, dtype=np.float32) for a in (x, g))
        out = np.empty_like(x)
        x_, g_, out_ = (C.c_void_p(a.ctypes.data) for a in (x, g, out))
        lib.quotients(C.c_long(x.size), x_, g_, C.c_int(inf), out_)
        return out

    return run


@pytest.mark.parametrize("inf", [False, True])
def test_within_one_ulp_of_division(quotients, inf):
    """Divisors over the range of the solves' pivots (square roots of a Gram
    entry or of its floor 1e-30), right-hand sides of any size for which the
    quotient and the residual stay normal."""
    r = np.random.default_rng(3)
    n = 1_000_000
    x = (r.uniform(1, 2, n) * r.choice([-1, 1], n) * 2.0 ** r.integers(-60, 60, n)).astype(np.float32)
    g = (r.uniform(1, 2, n) * 2.0 ** r.integers(-50, 64, n)).astype(np.float32)
    q, d = quotients(x, g, inf), x / g
    assert np.all(np.abs(q.view(np.int32) - d.view(np.int32)) <= 1)


def test_infinities_zeros_nan(quotients):
    inf, nan = np.inf, np.nan
    with np.errstate(all="ignore"):
        x = np.float32([inf, -inf, inf, 1, -3, 0, 0, nan, 1, inf, 3e38, -3e38])
        g = np.float32([2, 1e-15, 1e18, inf, inf, inf, 5, 2, nan, inf, 1e-15, 0.5])
        np.testing.assert_array_equal(quotients(x, g, True), x / g)
