"""psi and its derivative's exponential as the FP64 adjoint takes them (lbm_fixed.cuh), compiled for the
host, against long double and the formulas -expm1(-rho / rho0), exp(-rho / rho0): as good at small and
large densities as there.  No GPU needed."""
import ctypes
import math
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def numbers(tmp_path_factory):
    out = tmp_path_factory.mktemp("numbers") / "libnumbershost.so"
    src = os.path.join(ROOT, "tests", "native", "numbers_host.cpp")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "paper_1402_6019_gb300", "csrc"), src, "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    dp = ctypes.POINTER(ctypes.c_double)
    for f in (lib.number_psi, lib.number_exp):
        f.argtypes, f.restype = [ctypes.c_double, ctypes.c_double, dp], None
    lib.coef_taken.argtypes, lib.coef_taken.restype = [dp], ctypes.c_int
    lib.number_bits57.argtypes, lib.number_bits57.restype = [ctypes.c_double], ctypes.c_longlong
    return lib


def measure(f, rho, rho0):
    out = np.zeros(4)
    f(rho, rho0, out.ctypes.data_as(ctypes.POINTER(ctypes.c_double)))
    return out


@pytest.mark.parametrize("rho0", [1.0, 0.83, 1e6, 1e-3])
@pytest.mark.parametrize("low,high", [(-12, -5), (-5, -2), (-2, -1), (-1, 0), (0, 1.6)])
def test_no_further_off_than_the_formulas(numbers, rho0, low, high):
    """Over decades of rho / rho0: the largest and the root-mean-square error no larger than the
    formula's, but for the 2^-60 of the fixed-point exponential (2^-7 of the unit here; 2^-5 at the
    smallest psi formed with it)."""
    rng = np.random.default_rng(7)
    rho = rho0 * 10.0 ** rng.uniform(low, high, 4000)
    for f, own in ((numbers.number_psi, 2.0 ** -2), (numbers.number_exp, 2.0 ** -6)):
        e = np.array([measure(f, r, rho0)[2:] for r in rho])
        assert e[:, 0].max() <= max(e[:, 1].max(), 1.0 + own)
        assert np.sqrt((e[:, 0] ** 2).mean()) <= np.sqrt((e[:, 1] ** 2).mean()) * (1 + own)


def test_the_ends_of_the_range(numbers):
    """Densities that are zero, negative, tiny, huge or not finite give what the formulas give."""
    for r in (0.0, -0.0, -0.7, -3.0, 5e-324, 1e-300, 1e-290, 1e290, 1e300, math.inf, -math.inf, math.nan, 45.0, 700.0, 745.0):
        for f in (numbers.number_psi, numbers.number_exp):
            with np.errstate(over="ignore"):
                out = measure(f, r, 1.0)
            assert out[0] == out[1] or (math.isnan(out[0]) and math.isnan(out[1])) or abs(out[0] / out[1] - 1) < 1e-15, r


def test_a_psi_on_the_57_bit_scale_is_exact(numbers):
    rng = np.random.default_rng(3)
    for p in [2.0 ** -5, 1.0, math.nextafter(1.0, 0), math.nextafter(2.0 ** -5, 1), 0.5, math.nextafter(0.5, 0)] + \
            list(rng.uniform(2.0 ** -5, 1.0, 2000)) + list(2.0 ** rng.uniform(-5, 0, 2000)):
        assert numbers.number_bits57(p) * 2.0 ** -57 == p and math.ldexp(p, 57) == int(math.ldexp(p, 57))


def test_couplings_beyond_the_fixed_point_range_are_refused(numbers):
    for top, want in ((0.0, 1), (1.0, 1), (2.0 ** -900, 1), (2.0 ** -901, 0), (2.0 ** 900, 1), (2.0 ** 901, 0),
                      (5e-324, 0), (1.7e308, 0), (math.inf, 0), (math.nan, 0)):
        for c in ([top, 0, 0, 0, 0], [0.0, -top, 0, 0, 0], [0, 0, 0, 0, top]):
            a = np.array(c, dtype=np.float64)
            assert numbers.coef_taken(a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))) == want, c
