"""The limit at which a trial's objective may end early, against the test (2.3) that
the trial has to fail: compiled from the header that the kernels and the host loop
share, and held against exact rationals.  The right-hand side is a difference of
larger terms, so the cases cancel down to 1e-13 of them."""
import ctypes
import os
import subprocess
from fractions import Fraction as Fr

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SHIM = """
#include "fbl_linesearch.h"
extern "C" double rhs(double s, double r, double g, double d, double a) { return fbl::ls_rhs(s, r, g, d, a); }
extern "C" double limit(double s, double r) { return fbl::ls_limit(s, r); }
extern "C" double objective(double s, double r) { return fbl::ls_objective(s, r); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("ls")
    (d / "s.cpp").write_text(SHIM)
    so = str(d / "s.so")
    subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-shared", "-fPIC", "-I",
                    os.path.join(ROOT, "paper_2605_12085_gb300", "csrc"), str(d / "s.cpp"), "-o", so], check=True)
    out = ctypes.CDLL(so)
    for f, n in ((out.rhs, 5), (out.limit, 2), (out.objective, 2)):
        f.restype, f.argtypes = ctypes.c_double, [ctypes.c_double] * n
    return out


def cases(n=4000):
    """(scale, rho0, gTd, dd, alpha) whose right-hand side cancels to 10^-e of its terms."""
    rng = np.random.default_rng(8)
    for _ in range(n):
        scale, rho0 = float(rng.integers(1, 721)) / float(rng.integers(1, 41)), 10.0 ** rng.uniform(-6, 20)
        alpha, f = 0.5 ** int(rng.integers(0, 30)), 0.5 * scale * rho0
        quad = f * rng.uniform(0.2, 5)
        left = f * 10.0 ** -rng.uniform(0, 13) * rng.choice([1, 1, -1])
        yield scale, rho0, left - f - quad, 2.0 * alpha * quad, alpha


def test_a_partial_sum_above_the_limit_fails_the_test(lib):
    for scale, rho0, gTd, dd, alpha in cases():
        rhs = lib.rhs(scale, rho0, gTd, dd, alpha)
        lim = lib.limit(scale, rhs)
        # the sum that is compared with the limit and the one the decision takes may each be
        # off by n 2^-53 (n = 2^31 blocks)
        least = Fr(np.nextafter(lim, np.inf)) * (1 - Fr(2 ** 32, 2 ** 53))
        assert lib.objective(scale, float(least)) > rhs
        # and the limit costs no early end worth having
        assert lim <= max(rhs, 0.0) / (0.5 * scale) * (1 + 2e-6)


def test_a_contracted_right_hand_side_would_not_do(lib):
    """The reason for one shared form: with f_N(x) and g^T d in one FMA, as a compiler
    contracts them, the two right-hand sides differ by more than a relative margin of 1e-9."""
    worst = 0.0
    for scale, rho0, gTd, dd, alpha in cases():
        rhs = lib.rhs(scale, rho0, gTd, dd, alpha)
        fma = float(Fr(0.5 * scale) * Fr(rho0) + Fr(gTd))
        worst = max(worst, abs(fma + dd / (2.0 * alpha) - rhs) / max(abs(rhs), 1e-300))
    assert worst > 1e-9
