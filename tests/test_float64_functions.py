"""The float64 functions of the kernels' law header, compiled for the host with models of the fast float32 functions
that they start from (tests/host/float64_functions.cpp), against 80-bit arithmetic: every result has to hold for every
error that CUDA documents for those starts."""
import ctypes
import os
import shutil
import subprocess

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
ROOT = os.path.dirname(HERE)
TILTS = [(a, b) for a in (-1.0, 0.0, 1.0) for b in (-1.0, 0.0, 1.0)]
LD = np.longdouble


def _cuda_include():
    nvcc = shutil.which(os.environ.get("NVCC", "nvcc")) or "/usr/local/cuda/bin/nvcc"
    return os.path.join(os.path.dirname(os.path.dirname(os.path.realpath(nvcc))), "include")


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    so = str(tmp_path_factory.mktemp("host") / "float64_functions.so")
    subprocess.run(["g++", "-std=c++17", "-O2", "-ffp-contract=off", "-w", "-shared", "-fPIC", "-I" + _cuda_include(),
                    "-I" + os.path.join(ROOT, "include"), "-I" + os.path.join(ROOT, "paper_2004_08503_gb300", "csrc"),
                    os.path.join(HERE, "host", "float64_functions.cpp"), "-o", so], check=True)
    return ctypes.CDLL(so)


def _p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def _tilt(lib, t):
    lib.set_tilt(ctypes.c_double(t[0]), ctypes.c_double(t[1]))


def _psi(u, K, gamma):
    u = u.astype(LD)
    return u[:, 3] - (u[:, 1] ** 2 + u[:, 2] ** 2) / (2 * u[:, 0]) - K.astype(LD) * u[:, 0] ** LD(gamma)


def _psi_at(u, w, s, K, gamma):
    return _psi(u.astype(LD) + s * w.astype(LD), K, gamma)


def _states(rng, n, gamma, decades):
    """States of all densities, Mach numbers up to 3, K just below the state's own sigma."""
    rho = 10.0 ** rng.uniform(-decades, decades, n)
    rhoe = rho * 10.0 ** rng.uniform(-1, 1, n)
    c = np.sqrt(gamma * (gamma - 1.0) * rhoe / rho)
    v = c[:, None] * rng.uniform(-2, 2, (n, 2))
    u = np.column_stack([rho, rho[:, None] * v, rhoe + 0.5 * rho * np.sum(v * v, axis=1)])
    K = (_psi(u, np.zeros(n), gamma) * (1 - 10.0 ** rng.uniform(-8, -2, n)) / rho.astype(LD) ** LD(gamma)).astype(float)
    w = u * 10.0 ** rng.uniform(-7, -1, (n, 1)) * rng.uniform(-1, 1, (n, 4))
    return u, K, w


def _screen(lib, gamma, u, K, w, sc, tcap):
    out = np.empty(len(u), np.int32)
    lib.screen(len(u), ctypes.c_double(gamma), _p(u), _p(K), _p(w), ctypes.c_double(sc), ctypes.c_double(tcap), _p(out))
    return out.astype(bool)


@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0, 1.1])
@pytest.mark.parametrize("decades", [1, 4, 12, 17.5])
def test_screen_passes_no_inadmissible_candidate(lib, gamma, decades):
    """Candidates with psi_K below zero by 1e-9 to 1e-4 of rho e: none of them may be called certain."""
    rng = np.random.default_rng(int(10 * decades))
    u, K, w = _states(rng, 40000, gamma, decades)
    sc, tcap = 0.37, 0.9
    target = -(10.0 ** rng.uniform(-9, -4, len(u))) * _psi(u, np.zeros(len(u)), gamma)
    s = LD(sc) * LD(tcap)
    for _ in range(2):  # psi is affine in the energy: move the candidate onto its target
        w[:, 3] += ((target - _psi_at(u, w, s, K, gamma)) / s).astype(float)
    bad = _psi_at(u, w, s, K, gamma) < 0
    assert bad.mean() > 0.99
    for t in TILTS:
        _tilt(lib, t)
        undecided = _screen(lib, gamma, u, K, w, sc, tcap)
        wrong = bad & ~undecided
        assert not wrong.any(), (t, int(wrong.sum()), float((target[wrong] / _psi(u, np.zeros(len(u)), gamma)[wrong]).min()))


def test_screen_decides_clear_candidates(lib):
    """The screen is worth its cost: candidates with psi_K above zero by 1e-4 of rho E are certain."""
    rng = np.random.default_rng(3)
    u, K, w = _states(rng, 20000, 1.4, 12)
    K, w = 0.9 * K, 1e-3 * w
    ok = _psi_at(u, w, LD(0.5), K, 1.4) > 1e-4 * u[:, 3]
    assert ok.mean() > 0.9
    for t in TILTS:
        _tilt(lib, t)
        assert not _screen(lib, 1.4, u, K, w, 1.0, 0.5)[ok].any(), t


@pytest.mark.parametrize("gamma", [1.4, 5.0 / 3.0, 1.1])
def test_sigma_certainly_above_is_certain(lib, gamma):
    """States with sigma below K by 1e-9 to 1e-3: none may be called certainly above."""
    rng = np.random.default_rng(4)
    u, K, _ = _states(rng, 40000, gamma, 17.5)
    sig = _psi(u, np.zeros(len(u)), gamma) / u[:, 0].astype(LD) ** LD(gamma)
    K = (sig * (1 + 10.0 ** rng.uniform(-9, -3, len(u)))).astype(float)
    out = np.empty(len(u), np.int32)
    for t in TILTS:
        _tilt(lib, t)
        lib.certainly_above(len(u), ctypes.c_double(gamma), _p(u), _p(K), _p(out))
        assert not out.any(), (t, int(out.sum()))


def test_minima_and_sign_tests(lib):
    """The integer forms against fmax, fmin and the comparisons, NaN of both signs, infinities, zeros and denormals among
    the operands; every result bit for bit but for the sign of a zero and which NaN comes out of two."""
    rng = np.random.default_rng(5)
    v = np.concatenate([[0.0, -0.0, 5e-324, -5e-324, 2.2e-308, 1.0, -1.0, 1.0 + 2e-16, 1e308, -1e308, np.inf, -np.inf, np.nan,
                         -np.nan, np.copysign(np.nan, -1.0)], rng.normal(size=20) * 10.0 ** rng.uniform(-300, 300, 20)])
    a, b = (np.ascontiguousarray(m.ravel()) for m in np.meshgrid(v, v))
    out = np.empty((5, a.size))
    lib.compare_ops(a.size, _p(a), _p(b), _p(out))
    for got, exp in zip(out, (np.fmax(a, b), np.fmin(a, b), np.fmax(a, 0.0), np.fmin(a, 0.0), (a > 0).astype(float))):
        np.testing.assert_array_equal(got, exp)
    a, b = np.where(np.isnan(a), a, np.abs(a)), np.where(np.isnan(b), b, np.abs(b))  # >= +0, or a NaN of either sign
    out = np.empty((2, a.size))
    lib.compare_ops_nonneg(a.size, _p(a), _p(b), _p(out))
    for got, exp in zip(out, (np.fmax(a, b), np.fmin(a, b))):
        np.testing.assert_array_equal(got, exp)


def test_quotients_and_roots_round_like_ieee(lib):
    """a / b, 1 / b and the root over all exponents: within half an ulp and 1e-5 of the 80-bit value (whose own
    resolution is 2^-11 ulp) where the result is normal, and the IEEE results for zeros, infinities, NaN, overflow and denormals."""
    rng = np.random.default_rng(6)
    n = 100000
    for decades in (1, 28, 307):
        a, b = (rng.choice([-1.0, 1.0], n) * rng.uniform(1, 2, n) * 10.0 ** rng.uniform(-decades, decades, n) for _ in range(2))
        b[: n // 2] = np.abs(b[: n // 2])
        out = np.empty((3, n))
        with np.errstate(all="ignore"):
            exact = [a.astype(LD) / b, 1 / b.astype(LD), np.sqrt(b.astype(LD))]
            ieee = [a / b, 1 / b, np.sqrt(b)]
        for t in TILTS[::3]:
            _tilt(lib, t)
            lib.quotients(n, _p(a), _p(b), _p(out))
            for got, x, i in zip(out, exact, ieee):
                normal = np.isfinite(i) & (np.abs(i) > 1e-290)
                ulps = np.abs(got[normal] - x[normal]) / np.spacing(np.abs(i[normal]))
                assert ulps.max() <= 0.5 + 2.0 ** -11 + 1e-5, (decades, t, float(ulps.max()))
                np.testing.assert_allclose(got[~normal], i[~normal], rtol=0, atol=5e-324)
    v = np.array([0.0, -0.0, 5e-324, 1e-310, 1e-300, 1e-40, 1.0, -3.0, 1e40, 1e300, np.inf, -np.inf, np.nan])
    a, b = (np.ascontiguousarray(m.ravel()) for m in np.meshgrid(v, v))
    out = np.empty((3, a.size))
    _tilt(lib, (0.0, 0.0))
    lib.quotients(a.size, _p(a), _p(b), _p(out))
    with np.errstate(all="ignore"):
        for got, exp in zip(out, (a / b, 1 / b, np.sqrt(b))):
            np.testing.assert_array_equal(got, exp)


@pytest.mark.parametrize("gamma", [1.4, np.nextafter(1.4, 2), 1.4 + 2e-14, 1.4 - 2e-14])
@pytest.mark.parametrize("decades", [0.5, 3, 24.9])
def test_powers_round_no_worse_than_pow(lib, decades, gamma):
    """x^-e, x^-gamma, x^gamma and x^(1/e) against the 80-bit power of the float64 exponent.  CUDA's pow is 0.25 to 0.34 ulp
    off in the mean and 1.05 to 1.25 at most over these arguments (measured)."""
    rng = np.random.default_rng(7)
    x = rng.uniform(0.9, 1, 50000) * 10.0 ** rng.uniform(-decades, decades, 50000)
    exact = [x.astype(LD) ** LD(e) for e in (-(gamma - 1) / (2 * gamma), -gamma, gamma, 2 * gamma / (gamma - 1))]
    out = np.empty((4, x.size))
    for t in TILTS:
        _tilt(lib, t)
        lib.powers(x.size, ctypes.c_double(gamma), _p(x), _p(out))
        for got, e in zip(out, exact):
            ulps = np.abs(got - e) / np.spacing(e.astype(float))
            assert ulps.mean() <= 0.29 and ulps.max() <= 1.25, (t, float(ulps.mean()), float(ulps.max()))


@pytest.mark.parametrize("gamma", [1.4, 1.2, 5.0 / 3.0])
def test_powers_of_extreme_arguments(lib, gamma):
    """Arguments outside the range of the closed forms, and exponents without one, take pow itself."""
    x = np.array([1e-300, 1e-28, 1e28, 1e40, np.inf, 0.0, np.nan, -1.0])
    out = np.empty((4, x.size))
    _tilt(lib, (0.0, 0.0))
    lib.powers(x.size, ctypes.c_double(gamma), _p(x), _p(out))
    with np.errstate(all="ignore"):
        for got, e in zip(out, (-(gamma - 1) / (2 * gamma), -gamma, gamma, 2 * gamma / (gamma - 1))):
            np.testing.assert_allclose(got, x ** e, rtol=4e-16)
