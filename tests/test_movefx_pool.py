"""The z move's pool in integers (csrc/rlt2_movefx.cuh): compiled for the host,
against the exact move in rational arithmetic and beside the FP64 form, on classes
whose members are alike and on classes whose members are far apart; and the
device's move of a whole D^ against the host's, bit for bit.

Error of one entry: s_c = (D_c - xi_c) - psi_c is rounded twice, which enters D'_b
with weight 1 for c = b and phi for the others; the cuts onto the class's grid lose
less than one step for s_b, one for the phi share of the other five and three in
the product, a step being at most 2^-58 of the largest |s|; the change of D_b and
D'_b are rounded once each."""
import ctypes
import itertools
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

import oracle as O

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
HDR = os.path.join(ROOT, "paper_1710_03732_gb300", "csrc")
SHIM = r"""
#include <cmath>
#include "rlt2_movefx.cuh"
// classes of six entries each: the integer form (FP64 where it declines), and the FP64 form alone
static void fp64(double* D, const double* s, double phi) {
  double S = s[0];
  for (int b = 1; b < 6; ++b) S += s[b];
  for (int b = 0; b < 6; ++b) D[b] = std::fma(-(1.0 + phi), s[b], std::fma(phi, S, D[b]));
}
extern "C" long long move_all(long long n, double* D, const double* xi, const double* psi, double phi, int form) {
  long long taken = 0;
  for (long long c = 0; c < n; ++c, D += 6, xi += 6, psi += 6) {
    double s[6];
    for (int b = 0; b < 6; ++b) {
      const double t = D[b] - xi[b];
      s[b] = t - psi[b];
    }
    if (form && rlt2::pool_class_fx(D, s, rlt2::fx_factor(phi))) ++taken;
    else fp64(D, s, phi);
  }
  return taken;
}
"""
PHI = Fraction(0.2)
U = Fraction(1, 2**53)


@pytest.fixture(scope="module")
def move(tmp_path_factory):
    d = tmp_path_factory.mktemp("movefxpool")
    src, so = d / "shim.cpp", d / "libpool.so"
    src.write_text(SHIM)
    r = subprocess.run(["g++", "-O2", "-std=c++17", "-ffp-contract=off", "-fPIC", "-shared", "-I" + HDR, str(src), "-o",
                        str(so)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    L = ctypes.CDLL(str(so))
    dp = ctypes.POINTER(ctypes.c_double)
    L.move_all.argtypes = [ctypes.c_longlong, dp, dp, dp, ctypes.c_double, ctypes.c_int]
    L.move_all.restype = ctypes.c_longlong

    def run(D, xi, psi, form=1):
        D, xi, psi = (np.array(x, dtype=np.float64).reshape(-1, 6) for x in (D, xi, psi))
        taken = L.move_all(len(D), *(x.ctypes.data_as(dp) for x in (D, xi, psi)), 0.2, form)
        return D, taken
    return run


KINDS = ["plain", "tight", "integers", "first", "spread3", "spread9", "far3", "far6", "far9", "bound2", "large", "small"]


def _classes(kind, count):
    """(D, xi, psi) of `count` classes as ascents meet them, and members far apart."""
    rng = np.random.default_rng([11, KINDS.index(kind)])
    shape = (count, 6)
    xi, psi, slack = rng.normal(0, 300, shape), rng.normal(0, 300, shape), rng.exponential(50, shape)
    if kind == "tight":  # most members at their duals
        slack *= rng.random(shape) < 0.4
    elif kind == "integers":
        xi, psi, slack = np.rint(xi), np.rint(psi), np.rint(slack)
    elif kind.startswith("spread"):  # each member on its own scale
        f = 10.0 ** (int(kind[-1]) * rng.random(shape))
        xi, psi, slack = xi * f, psi * f, slack * f
    elif kind.startswith("far"):  # one member far above the others and without slack, exactly
        f = 10.0 ** int(kind[-1])
        xi[:, 0], psi[:, 0], slack[:, 0] = np.rint(xi[:, 0] * f), np.rint(psi[:, 0] * f), 0.0
    elif kind == "bound2":  # one slack far above the others
        slack[:, 3] = 1e7
    elif kind in ("large", "small"):
        f = 2.0**1005 if kind == "large" else 2.0**-940
        xi, psi, slack = xi * f, psi * f, slack * f
    D = np.zeros(shape) if kind == "first" else xi + psi + slack
    return D, xi, psi


def _exact(D, xi, psi):
    s = [Fraction(d) - Fraction(a) - Fraction(b) for d, a, b in zip(D, xi, psi)]
    S = sum(s)
    return [Fraction(d) - x + PHI * (S - x) for d, x in zip(D, s)], s


@pytest.mark.parametrize("kind", KINDS)
def test_error_within_its_bound_and_the_fp64_forms(move, kind):
    D, xi, psi = _classes(kind, 1500)
    got, taken = move(D, xi, psi)
    assert taken >= 1450
    plain, _ = move(D, xi, psi, form=0)
    sums = np.zeros((2, 2))  # squares, (class scale, member scale) x (integer form, FP64 form)
    for c in range(len(D)):
        ref, s = _exact(D[c], xi[c], psi[c])
        ds = [U * (abs(Fraction(D[c, b]) - Fraction(xi[c, b])) + abs(s[b])) for b in range(6)]
        step = max(abs(x) for x in s) / 2**58
        top = max(abs(x) for x in ref) or 1
        for b in range(6):
            bound = (ds[b] + PHI * (sum(ds) - ds[b]) + 5 * step + U * (abs(ref[b] - Fraction(D[c, b])) + abs(ref[b])))
            err = [abs(Fraction(x[c, b]) - ref[b]) for x in (got, plain)]
            assert err[0] <= bound * (1 + Fraction(1, 2**40)), (c, b)
            own = abs(Fraction(D[c, b])) + abs(Fraction(xi[c, b])) + abs(Fraction(psi[c, b])) + abs(ref[b]) or 1
            for k in range(2):
                sums[0, k] += float(err[k] / top) ** 2
                sums[1, k] += float(err[k] / own) ** 2
    # 9,000 entries: 5 % is more than their sampling error
    assert (np.sqrt(sums[:, 0]) <= 1.05 * np.sqrt(sums[:, 1])).all(), np.sqrt(sums / D.size)


def _members(n):
    fac = np.array(list(itertools.combinations(range(n), 3)))
    loc = np.array(list(itertools.permutations(range(n), 3)))
    out = []
    for o in [(0, 1, 2), (0, 2, 1), (1, 0, 2), (1, 2, 0), (2, 0, 1), (2, 1, 0)]:
        f = fac[:, o][:, None, :] + np.zeros((1, len(loc), 1), dtype=int)
        x = loc[:, o][None, :, :] + np.zeros((len(fac), 1, 1), dtype=int)
        i, j, k, p, q, r = (a.reshape(-1) for a in (f[..., 0], f[..., 1], f[..., 2], x[..., 0], x[..., 1], x[..., 2]))
        t = ((i * n + p) * (n - 1) + j - (j > i)) * (n - 1) + q - (q > p)
        out.append((t, k - (k > i) - (k > j), r - (r > p) - (r > q), i * n + p))
    return [np.stack(a, axis=1) for a in zip(*out)]  # each [classes, 6]


@pytest.mark.gpu
@pytest.mark.parametrize("spread", [0, 3, 60])
@pytest.mark.parametrize("n", [3, 4, 5, 6, 8, 9, 11, 13, 15])
def test_device_move_equals_host_move(move, n, spread):
    from paper_1710_03732_gb300 import instances as I
    from paper_1710_03732_gb300 import rlt2 as R
    inst = I.random_instance(n, 30 + n, with_b=True, asymmetric=True)
    m = n - 2
    rng = np.random.default_rng([n, spread])
    # whole tiles on their own binary scales: the members of a class lie in six tiles
    D0 = rng.normal(0, 100, (O.num_tiles(n), m, m)) * 2.0 ** rng.integers(-spread, spread + 1, (O.num_tiles(n), 1, 1))
    D0[::5, 0] = 0.0
    D0 = D0.reshape(-1)
    with R.Context(inst.F, inst.D, inst.B, prm=R.params(dual_mode=1, feas_tol=0.0)) as ctx:
        ctx.import_state(D0, ctx.export_state()[1])
        ctx.iterate(1)
        du, red = ctx.duals(), ctx.reduced_costs()
        assert np.array_equal(ctx.export_state()[0], D0)  # its move is pending
        ctx.iterate(1)
        D1 = ctx.export_state()[0]
    t, row, col, ip = _members(n)
    term = (0.5 / m) * red["pi_y"] + (1.0 / ((n - 1) * m)) * np.repeat(red["pi_x"].reshape(-1), (n - 1) ** 2)
    psi = (du["psi"].reshape(-1, m) - term[:, None]).reshape(-1)
    at = (t * m + row) * m + col
    got, taken = move(D0[at], du["xi"].reshape(-1)[t * m + row], psi[t * m + col])
    assert taken > 0.9 * len(t)
    ref = np.empty_like(D0)
    ref[at.reshape(-1)] = got.reshape(-1)
    assert np.array_equal(D1, ref)
