"""The FP64 step's fixed-point pseudopotential, force and stresses (lbm_fixed.cuh), compiled for the
host, against long double and against the FP64 forms.  No GPU needed."""
import ctypes
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

from paper_1402_6019_gb300 import lbm as L
from paper_1402_6019_gb300 import workloads as W

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def fixed(tmp_path_factory):
    out = tmp_path_factory.mktemp("fixed") / "libfixedhost.so"
    src = os.path.join(ROOT, "tests", "native", "fixed_host.cpp")
    subprocess.run(["g++", "-std=c++17", "-O1", "-fPIC", "-shared", "-ffp-contract=off",
                    "-I", os.path.join(ROOT, "include"),
                    "-I", os.path.join(ROOT, "paper_1402_6019_gb300", "csrc"), src, "-o", str(out)], check=True)
    lib = ctypes.CDLL(str(out))
    dp = ctypes.POINTER(ctypes.c_double)
    lib.fixed_psi.argtypes = [ctypes.c_double, ctypes.c_double, dp]
    lib.fixed_psi.restype = ctypes.c_double
    lib.fixed_rcp.argtypes = [ctypes.c_double]
    lib.fixed_rcp.restype = ctypes.c_double
    lib.fixed_scaled.argtypes = [ctypes.c_longlong, ctypes.c_int]
    lib.fixed_scaled.restype = ctypes.c_double
    lib.fixed_site.argtypes = [ctypes.POINTER(L.lbm_params), ctypes.c_int] + [dp] * 7
    return lib


def _p(a):
    return a.ctypes.data_as(ctypes.POINTER(ctypes.c_double))


@pytest.mark.parametrize("rho0", [1.0, 0.83, 3.7, 1e-3])
def test_psi_is_within_its_resolution(fixed, rho0):
    """Within 2^-56 (the argument's 57 fraction bits, the polynomial's remainder and the roundings of
    lbm_fixed.cuh add up to less than 2^-57 + 2^-59), from tiny densities to ones whose exponential
    underflows, at the exact powers of two and their neighbours."""
    out = np.zeros(2)
    rng = np.random.default_rng(3)
    rho = list(10.0 ** rng.uniform(-12, 3, 20000)) + list(rng.uniform(0.01, 3.0, 20000))
    for e in range(-60, 12):
        rho += [math.ldexp(1.0, e), math.nextafter(math.ldexp(1.0, e), 0), math.nextafter(math.ldexp(1.0, e), 9e9)]
    rho += [1e-290, 1e-250, 1e250, 1e290, 5e-324, 1.7e308]
    for r in rho:
        assert fixed.fixed_psi(r, rho0, _p(out)) <= 1.0, r
        assert 0.0 <= out[0] <= 1.0 and abs(out[0] - out[1]) <= 4e-16, r


def test_psi_of_an_invalid_density_is_zero(fixed):
    out = np.zeros(2)
    for r in (0.0, -1.0, -1e300, math.nan, -math.inf):
        fixed.fixed_psi(r, 1.0, _p(out))
        assert out[0] == 0.0, r
    fixed.fixed_psi(math.inf, 1.0, _p(out))
    assert out[0] == 1.0


def test_reciprocal_is_within_an_ulp(fixed):
    """Against exact rationals: error below 2^-53 of the value (the last rounding) plus 2^-62 (the
    iteration's remainder and its own roundings), over mantissas and exponents, at powers of two
    and their neighbours."""
    rng = np.random.default_rng(5)
    xs = list(rng.uniform(1e-3, 8.0, 5000)) + list(2.0 ** rng.uniform(-900, 900, 2000))
    for e in range(-40, 41):
        xs += [2.0 ** e, math.nextafter(2.0 ** e, 0.0), math.nextafter(2.0 ** e, 9e99), -(2.0 ** e) * 1.7]
    for x in xs:
        want = 1 / Fraction(x)
        assert abs(Fraction(fixed.fixed_rcp(x)) - want) <= abs(want) * (Fraction(1, 2 ** 53) + Fraction(1, 2 ** 62)), x


def test_scaled_double_rounds_to_nearest(fixed):
    rng = np.random.default_rng(4)
    for v in [0, 1, -1, 2 ** 62, -2 ** 62, 2 ** 53 + 1, 2 ** 62 - 1, -(2 ** 63 - 1)] + \
            [int(x) >> int(k) for x, k in zip(rng.integers(-2 ** 62, 2 ** 62, 5000), rng.integers(0, 62, 5000))]:
        got = Fraction(fixed.fixed_scaled(v, -60))  # exact: v itself may have more digits than a double
        assert abs(got - Fraction(v, 2 ** 60)) <= abs(Fraction(v, 2 ** 60)) / 2 ** 53, v


@pytest.mark.parametrize("preset", [0, 1])
@pytest.mark.parametrize("params", [W.EMULSION_PARAMS, W.FILM_PARAMS, dict(W.EMULSION_PARAMS, G1=(-60.0, 0.0), G2=(0.0, 0.0))])
def test_force_and_stress_are_no_further_off_than_fp64(fixed, preset, params):
    """Against long double over random windows (smooth, noisy, droplet edges, uniform): the
    fixed-point sums' root-mean-square error is no larger than that of the FP64 forms."""
    p = L.lbm_params()
    p.weight_norm, p.weight_preset = params["weight_norm"], preset
    for k in range(2):
        p.tau[k], p.G1[k], p.G2[k], p.rho0[k] = 1.0, params["G1"][k], params["G2"][k], params["rho0"][k]
    rng = np.random.default_rng(11)
    err = np.zeros((2, 5))
    for i in range(3000):
        kind = i % 4
        rho = {0: 0.05 + 1.2 * rng.random(25), 1: 1.0 + 0.01 * rng.uniform(-1, 1, 25),
               2: np.where(rng.random(25) < 0.5, 1.2, 0.05), 3: np.full(25, 0.05 + rng.random())}[kind]
        F, S, F64, S64, FL, SL = np.zeros(2), np.zeros(3), np.zeros(2), np.zeros(3), np.zeros(2), np.zeros(3)
        fixed.fixed_site(ctypes.byref(p), i % 2, _p(np.ascontiguousarray(rho)), _p(F), _p(S), _p(F64), _p(S64), _p(FL), _p(SL))
        want = np.concatenate([FL, SL])
        err[0] += (np.concatenate([F, S]) - want) ** 2
        err[1] += (np.concatenate([F64, S64]) - want) ** 2
    assert np.all(err[0] <= err[1]), np.sqrt(err / 3000)


def test_force_is_exactly_odd(fixed):
    """A window turned by 180 degrees gives exactly the reversed force, a uniform one exactly none:
    the rounding of the fixed-point products has no preferred direction."""
    p = L.lbm_params()
    p.weight_norm = W.FILM_PARAMS["weight_norm"]
    for k in range(2):
        p.tau[k], p.G1[k], p.G2[k], p.rho0[k] = 1.0, -20.4, 16.0, 1.0
    rng = np.random.default_rng(13)
    scratch = [np.zeros(3) for _ in range(5)]

    def force(rho):
        F = np.zeros(2)
        fixed.fixed_site(ctypes.byref(p), 0, _p(np.ascontiguousarray(rho)), _p(F), *[_p(a) for a in scratch])
        return F

    for _ in range(500):
        rho = 0.05 + 1.4 * rng.random(25)
        assert np.array_equal(force(rho), -force(rho[::-1]))
        assert np.array_equal(force(np.full(25, rho[0])), np.zeros(2))
