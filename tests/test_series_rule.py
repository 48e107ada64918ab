"""Stopping rule of the FP32 inner series (csrc/series.cuh) on recorded shapes of its update."""
import ctypes
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
RUNNING, STOPPED, PLATEAU, EXHAUSTED, ABORTED, NOT_FINITE = range(6)

SOURCE = """
#include "series.cuh"
using namespace dyson_detail;
extern "C" int run(const double* upd, int n, int max_sweeps, double target, double abort_peak, int plateau, int* sweeps) {
  SeriesState S = series_start(plateau != 0);
  for (int k = 0; k < n && S.run; ++k) series_step(S, upd[k], max_sweeps, target, abort_peak);
  *sweeps = S.sweeps;
  return S.outcome;
}
extern "C" int served(double res, double prev) { return plateau_served(res, prev); }
extern "C" double share(double dt, double u, double eps, double j) { return accept_share(dt, u, eps, j); }
extern "C" int more(double res, double tol, double prev, double share, int last) { return refine_once_more(res, tol, prev, share, last); }
"""


@pytest.fixture(scope="module")
def rule(tmp_path_factory):
    d = tmp_path_factory.mktemp("rule")
    (d / "rule.cpp").write_text(SOURCE)
    so = str(d / "rule.so")
    subprocess.run(["g++", "-std=c++17", "-O1", "-shared", "-fPIC", "-I" + os.path.join(ROOT, "paper_1309_5994_gb300", "csrc"),
                    str(d / "rule.cpp"), "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.run.argtypes = [ctypes.POINTER(ctypes.c_double), ctypes.c_int, ctypes.c_int, ctypes.c_double, ctypes.c_double,
                        ctypes.c_int, ctypes.POINTER(ctypes.c_int)]
    lib.served.argtypes = [ctypes.c_double, ctypes.c_double]

    lib.share.argtypes = [ctypes.c_double] * 4
    lib.share.restype = ctypes.c_double
    lib.more.argtypes = [ctypes.c_double] * 4 + [ctypes.c_int]

    def go(upd, max_sweeps=400, target=4e-7, abort_peak=1e5, plateau=1):
        s = ctypes.c_int()
        out = lib.run((ctypes.c_double * len(upd))(*upd), len(upd), max_sweeps, target, abort_peak, plateau, ctypes.byref(s))
        return out, s.value

    go.served = lambda res, prev: bool(lib.served(res, prev))
    go.share = lib.share
    go.more = lambda *a: bool(lib.more(*a))
    return go


def _transient(peak, sweeps):
    """growth to the peak and the start of the decay, as the real-time series has them"""
    up = [peak ** (k / 19.0) for k in range(20)]
    return up + [peak * 0.85 ** k for k in range(1, sweeps - 19)]


def test_an_oscillating_update_that_rests_above_the_floor_goes_on(rule):
    """Twelve sweeps above a minimum at 9.2e-3 of the peak, then the decay goes on to the target (a lattice with
    disorder, 10x10 sites, 256 contour points)."""
    head = [u for u in _transient(3.7e4, 60) if u > 350.0][:-1] + [340.0]
    rest = [430.0 + 20.0 * (k % 3) for k in range(12)]
    tail = [310.0 * 0.8 ** k for k in range(100)]
    out, sweeps = rule(head + rest + tail)
    assert out == STOPPED and sweeps > len(head) + len(rest) + 20


def test_a_floor_above_the_stall_line_ends_the_series(rule):
    """A rounding floor at 1e-3 of the peak: the series ends long before its budget."""
    head = [u for u in _transient(1e4, 60) if u > 12.0]
    floor = [10.0 * (1.0 + 0.05 * (k * 7 % 5)) for k in range(400)]
    out, sweeps = rule(head + floor, target=1e-6)
    assert out == PLATEAU and sweeps <= len(head) + 25
    assert rule(head + floor, target=1e-6, plateau=0) == (EXHAUSTED, 400)


def test_a_plateau_has_to_gain_a_digit(rule):
    """With less, the solve goes to GMRES or to the whole budget, as it did before the rule."""
    inf = float("inf")
    assert rule.served(0.09, inf) and not rule.served(0.3, inf)
    assert rule.served(1e-5, 1e-3) and not rule.served(4e-4, 1e-3)


def test_other_ends_of_a_series(rule):
    assert rule([1.0, 0.5, 1e-8])[0] == STOPPED
    assert rule([10.0 ** k for k in range(9)])[0] == ABORTED
    assert rule([1.0, float("inf")]) == (NOT_FINITE, 2)
    assert rule([1.0, float("nan")]) == (NOT_FINITE, 2)
    assert rule([1.0, 0.9, 0.8], max_sweeps=3) == (EXHAUSTED, 3)
    assert rule([1.0, 1e-3, 1e-5, 1.1e-5, 1.2e-5, 1.1e-5, 1.2e-5])[0] == STOPPED


def test_a_loose_tolerance_is_met_by_the_observables_too(rule):
    """The share of the tolerance follows from how much the double occupancy amplifies a residual."""
    assert rule.share(0.05, 20.0, 10.0, 1.0) == pytest.approx(20.0 / (2 / 0.05 + 10.0 + 4.0))
    assert rule.share(0.005, 4.0, 2.0, 1.0) == pytest.approx(4.0 / (2 / 0.005 + 2.0 + 4.0))
    assert rule.share(0.05, 0.0, 1.0, 1.0) < 1e-200 and rule.share(10.0, 50.0, 1.0, 1.0) == 1.0
    inf = float("inf")
    assert rule.more(0.5e-6, 1e-6, inf, 0.37, 0) and not rule.more(0.3e-6, 1e-6, inf, 0.37, 0)
    assert rule.more(0.3e-6, 1e-6, inf, 0.01, 0)
    assert not rule.more(0.5e-6, 1e-6, 0.9e-6, 0.37, 0)                # only one more
    assert not rule.more(0.5e-6, 1e-6, inf, 0.37, 1) and not rule.more(0.5e-10, 1e-10, 1e-6, 0.37, 0)
