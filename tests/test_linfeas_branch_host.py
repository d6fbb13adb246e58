"""CPU tests of the branch subproblem of the linear projection (eq. linfeas),
from a host build of the device header (tests/host/linfeas_helpers.cpp),
against exact rational arithmetic: minimisers inside the box, on its edges, and
within 1e-1 to 1e-14 of an edge or a corner, for short and long lines."""
import ctypes as C
import os
import shutil
import subprocess
from fractions import Fraction as Q

import numpy as np
import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
DP = C.POINTER(C.c_double)


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if shutil.which("g++") is None:
        pytest.skip("g++ not available")
    out = str(tmp_path_factory.mktemp("host") / "linfeas_helpers.so")
    subprocess.check_call(["g++", "-O2", "-shared", "-fPIC", "-o", out, os.path.join(HERE, "host", "linfeas_helpers.cpp")])
    return C.CDLL(out)


@pytest.fixture(scope="module")
def solve(lib):
    def run(P):
        P = np.ascontiguousarray(P)
        v = np.zeros((len(P), 4))
        lib.host_lf_branch(len(P), P.ctypes.data_as(DP), v.ctypes.data_as(DP))
        return v

    return run


def _rows(Y):
    """The four flow rows over (w_i, w_j, wR, wI)."""
    gii, bii, gij, bij, gji, bji, gjj, bjj = Y
    return [[gii, 0, gij, bij], [-bii, 0, -bij, gij], [0, gjj, gji, -bji], [0, -bjj, -bji, -gji]]


def _exact(p):
    p = [Q(float(v)) for v in p]
    F, rho = _rows(p[:8]), p[8]
    yf = [p[15], p[16], p[18], p[19]]
    H = [[rho * sum(F[r][a] * F[r][b] for r in range(4)) for b in range(4)] for a in range(4)]
    c = [sum(F[r][a] * yf[r] for r in range(4)) for a in range(4)]
    for a, (h, g) in enumerate(((rho, p[17]), (rho, p[20]), (2, -p[9]), (2, -p[10]))):
        H[a][a] += h
        c[a] += g
    d = H[2][2]
    assert H[2][3] == 0 and H[3][3] == d
    T = [[H[a][2] / d, H[a][3] / d] for a in (0, 1)]
    S = [[H[a][b] - d * (T[a][0] * T[b][0] + T[a][1] * T[b][1]) for b in (0, 1)] for a in (0, 1)]
    s = [c[a] - T[a][0] * c[2] - T[a][1] * c[3] for a in (0, 1)]
    lo, hi = (p[11], p[13]), (p[12], p[14])
    det = S[0][0] * S[1][1] - S[0][1] ** 2
    w = [-(S[1][1] * s[0] - S[0][1] * s[1]) / det, -(S[0][0] * s[1] - S[0][1] * s[0]) / det]
    if not all(lo[a] <= w[a] <= hi[a] for a in (0, 1)):
        best = None
        for a in (0, 1):
            for v in (lo[a], hi[a]):
                o = 1 - a
                t = [None, None]
                t[a], t[o] = v, min(max(-(s[o] + S[0][1] * v) / S[o][o], lo[o]), hi[o])
                f = sum(t[i] * (s[i] + (S[i][0] * t[0] + S[i][1] * t[1]) / 2) for i in (0, 1))
                if best is None or f < best[0]:
                    best = (f, t)
        w = best[1]
    v = w + [-(c[2 + k] / d + T[0][k] * w[0] + T[1][k] * w[1]) for k in (0, 1)]
    return [float(x) for x in v], [float(sum(F[r][a] * v[a] for a in range(4))) for r in range(4)]


def _problems(rng, n, size, where):
    """Lines of admittance `size` and y such that the unconstrained minimiser is
    about a chosen w."""
    P = np.zeros((n, 21))
    for p in P:
        ph, tap, sh = rng.uniform(0.05, 1.5), rng.uniform(0.95, 1.05), rng.uniform(-0.05, 0.05)
        y, bc = size * np.exp(-1j * ph), 1j * rng.uniform(0, 0.3)
        yii, yjj = (y + bc) / tap ** 2, y + bc
        yij, yji = -y / tap * np.exp(1j * sh), -y / tap * np.exp(-1j * sh)
        p[:8] = [f(v) for v in (yii, yij, yji, yjj) for f in (np.real, np.imag)]
        p[8] = rho = np.exp(rng.uniform(np.log(0.05), np.log(50)))
        p[11], p[12], p[13], p[14] = 0.9, 1.1, 0.9, 1.1
        if rng.random() < 0.1:
            p[13] = p[14] = 1.0  # a fixed voltage
        w = np.array([rng.uniform(0.85, 1.15), rng.uniform(0.85, 1.15), rng.uniform(0.9, 1.1), rng.uniform(-0.1, 0.1)])
        if where == "near":
            for k in range(2):
                if k == 0 or rng.random() < 0.7:
                    w[k] = p[11 + 2 * k + rng.integers(2)] + rng.choice((-1, 1)) * 10 ** -rng.uniform(1, 14)
        F = np.array(_rows(p[:8]))
        yf = -rho * F @ (w + rng.uniform(-0.01, 0.01, 4)) + rng.uniform(-5, 5, 4)
        g = F.T @ (rho * F @ w + yf)
        p[9:11] = g[2:] + 2 * w[2:]
        p[15:17], p[18:20] = yf[:2], yf[2:]
        p[17], p[20] = -(g[0] + rho * w[0]), -(g[1] + rho * w[1])
    return P


@pytest.mark.parametrize("size", [3, 30, 300, 3000])
@pytest.mark.parametrize("where", ["anywhere", "near"])
def test_branch_subproblem_against_exact_arithmetic(solve, size, where):
    P = _problems(np.random.default_rng(size), 1500, float(size), where)
    V = solve(P)
    # the linear term carries about ten roundings and the eigenvalues of S are
    # rho and rho |Y|^2 apart: 10 |Y|^2 2^-53, which is 1e-12 at |Y| = 30
    tol = 10 * max(size, 10) ** 2 * 2.0 ** -53
    at = 0
    for p, v in zip(P, V):
        want, flows = _exact(p)
        at += any(want[a] in (p[11 + 2 * a], p[12 + 2 * a]) for a in (0, 1))
        for a in (0, 1):
            assert p[11 + 2 * a] <= v[a] <= p[12 + 2 * a]
        assert np.max(np.abs(v - want)) <= tol, (p, v, want)
        assert np.max(np.abs(np.array(_rows(p[:8])) @ v - flows)) <= tol
    assert at > 500


def test_branch_subproblem_keeps_nan(solve):
    P = _problems(np.random.default_rng(1), 12, 30.0, "near")
    for k, j in enumerate((15, 16, 18, 19)):
        P[3 * k:3 * k + 3, j] = np.nan
    assert np.isnan(solve(P)).any(axis=1).all()


def test_quotient_from_a_kept_reciprocal(lib):
    rng = np.random.default_rng(9)
    n = 200000
    a = rng.standard_normal(n) * 10.0 ** rng.uniform(-12, 12, n)
    b = 10.0 ** rng.uniform(-6, 8, n)
    a[:6] = np.inf, -np.inf, np.nan, 0.0, 1e300, -1e300
    out = np.zeros(n)
    lib.host_quot_kept(n, a.ctypes.data_as(DP), b.ctypes.data_as(DP), out.ctypes.data_as(DP))
    np.testing.assert_array_equal(out, a / b)
