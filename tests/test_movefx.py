"""The integer form of the folded z move (csrc/rlt2_movefx.cuh), compiled for the
host, against the exact move in rational arithmetic; and on the GPU the ascent
that uses it (dual_mode 1) against the FP64 form (dual_mode 2) at the sizes
where its (p, q, r) groups have remainders.

Error bound of one entry: w_b is rounded once (2^-53 |w_b|), which enters D'_b
directly and, times phi, through the other five; the grid step is at most 2^-58
of the largest input, and cutting and scaling lose less than 8 steps; D'_b is
rounded once."""
import ctypes
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HDR = os.path.join(ROOT, "paper_1710_03732_gb300", "csrc")
SHIM = r"""
#include "rlt2_movefx.cuh"
extern "C" int move_one(double* D, const double* w, double phi) {
  return rlt2::move_class_fx(D, w, rlt2::fx_factor(phi)) ? 1 : 0;
}
"""
U = Fraction(1, 2**53)


@pytest.fixture(scope="module")
def move(tmp_path_factory):
    d = tmp_path_factory.mktemp("movefx")
    src, lib = d / "shim.cpp", d / "libmovefx.so"
    src.write_text(SHIM)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-fPIC", "-shared", "-I" + HDR, str(src), "-o", str(lib)],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(str(lib))
    dp = ctypes.POINTER(ctypes.c_double)
    L.move_one.argtypes = [dp, dp, ctypes.c_double]

    def run(D, w, phi=0.2):
        D = np.array(D, dtype=np.float64)
        w = np.ascontiguousarray(w, dtype=np.float64)
        return L.move_one(D.ctypes.data_as(dp), w.ctypes.data_as(dp), phi), D
    return run


def _exact(D, w, phi):
    s = [Fraction(d) - x for d, x in zip(D, w)]
    S = sum(s)
    return [x + Fraction(phi) * (S - y) for x, y in zip(w, s)]


def _classes(kind, rng, count):
    for _ in range(count):
        xi, psi, slack = rng.normal(0, 300, 6), rng.normal(0, 300, 6), rng.exponential(50, 6)
        if kind == "integers":
            xi, psi, slack = np.rint(xi), np.rint(psi), np.rint(slack)
        elif kind == "ranges":
            scale = 2.0 ** rng.integers(-60, 61, 6)
            xi, psi, slack = xi * scale, psi * scale, slack * scale
        elif kind == "sparse":
            keep = rng.random((3, 6)) < 0.4
            xi, psi, slack = xi * keep[0], psi * keep[1], slack * keep[2]
        elif kind == "large":
            xi, psi, slack = xi * 2.0**1005, psi * 2.0**1005, slack * 2.0**1005
        elif kind == "small":
            xi, psi, slack = xi * 2.0**-950, psi * 2.0**-950, slack * 2.0**-950
        yield xi + psi + slack, xi, psi


@pytest.mark.parametrize("kind", ["plain", "integers", "ranges", "sparse", "large", "small"])
def test_class_move_within_its_bound(move, kind):
    rng = np.random.default_rng(7)
    taken = 0
    for D, xi, psi in _classes(kind, rng, 400):
        w = xi + psi
        ok, got = move(D, w)
        if not ok:
            continue
        taken += 1
        we = [Fraction(a) + Fraction(b) for a, b in zip(xi, psi)]
        ref = _exact(D, we, 0.2)
        step = Fraction(max(np.abs(D).max(), np.abs(w).max())) / 2**58
        for b in range(6):
            others = sum(abs(we[c]) for c in range(6) if c != b)
            bound = U * (abs(we[b]) + Fraction(0.2) * others + abs(ref[b])) + 8 * step
            assert abs(Fraction(got[b]) - ref[b]) <= bound
    assert taken >= 300


def test_class_move_keeps_exact_cases(move):
    # D = w: no slack, nothing moves; equal slacks: phi (S - s) = s up to phi's own rounding
    ok, got = move(np.arange(6.0), np.arange(6.0))
    assert ok and np.array_equal(got, np.arange(6.0))
    ok, got = move([-0.0, 3.0, 0.0, 0.0, 0.0, -7.0], [0.0, 3.0, -0.0, 0.0, 0.0, -7.0])
    assert ok and np.array_equal(got, [0.0, 3.0, 0.0, 0.0, 0.0, -7.0])


@pytest.mark.parametrize("x", [0.0, 5e-324, 1e-300, 2.0**1023, np.inf, -np.inf, np.nan])
def test_exponent_ends_are_left_to_fp64(move, x):
    ok, got = move([x] + [0.0] * 5, [0.0] * 6)
    assert not ok and np.array_equal(got, [x] + [0.0] * 5, equal_nan=True)


@pytest.mark.gpu
@pytest.mark.parametrize("n", [3, 4, 5, 7, 8, 9, 11, 13, 18, 21])
def test_ascent_integer_move_against_fp64_form(n):
    from paper_1710_03732_gb300 import instances as I
    from paper_1710_03732_gb300 import rlt2
    inst = I.random_instance(n, 40 + n, with_b=True, asymmetric=True)
    iters, out = 4, {}
    for mode in (1, 2):
        with rlt2.Context(inst.F, inst.D, inst.B, prm=rlt2.params(dual_mode=mode, feas_tol=0.0)) as ctx:
            bounds, done = ctx.iterate(iters)
            assert done == iters
            out[mode] = (bounds, *ctx.export_state())
    # LAP grid 2^-47 of a tile's magnitude, at most 2 m entries on a dual's path,
    # at most fourfold growth of a difference per iteration (D' = w + phi (S - s))
    for a, b in zip(out[1], out[2]):
        scale = max(1.0, np.abs(out[2][1]).max(), np.abs(out[2][2]).max(), np.abs(b).max())
        assert np.abs(a - b).max() <= 2 * max(n - 2, 1) * 2.0**-47 * 4**iters * scale
