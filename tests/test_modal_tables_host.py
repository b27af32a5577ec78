"""The sensor's modal tables (host build of modal_tables.h; no GPU needed)
against their definitions in exact rational arithmetic: the Legendre
coefficients of the basis functions by integration of monomials, the
continuation m_j(x + 1) and the semi-norm matrix.  Every entry is off by at
most a few roundings (8 of 2^-53); at the LGL points, whose float64 values are
themselves rounded, by 2^-48."""
import os
import shutil
import subprocess
from decimal import Decimal, getcontext
from fractions import Fraction as Q
from math import comb

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
getcontext().prec = 60


def _mul(a, b):
    r = [Q(0)] * (len(a) + len(b) - 1)
    for i, x in enumerate(a):
        for j, y in enumerate(b):
            r[i + j] += x * y
    return r


def _int(a):
    return sum(c / (i + 1) for i, c in enumerate(a))


def _diff(a, k):
    for _ in range(k):
        a = [i * c for i, c in enumerate(a)][1:] or [Q(0)]
    return a


def _at_next(a):
    return [sum(c * comb(i, m) for i, c in enumerate(a)) for m in range(len(a))]


LEG = [[Q((-1) ** (k + i) * comb(k, i) * comb(k + i, i)) for i in range(k + 1)] for k in range(5)]


def _basis(p, lgl):
    if not lgl:
        out = []
        for a in range(p + 1):
            q = [Q(comb(p, a))]
            for f in [[Q(0), Q(1)]] * a + [[Q(1), Q(-1)]] * (p - a):
                q = _mul(q, f)
            out.append(q)
        return out
    z = Q((Decimal(1) / 5 if p == 3 else Decimal(3) / 7).sqrt()) / 2
    x = {1: [Q(0), Q(1)], 2: [Q(0), Q(1, 2), Q(1)], 3: [Q(0), Q(1, 2) - z, Q(1, 2) + z, Q(1)],
         4: [Q(0), Q(1, 2) - z, Q(1, 2), Q(1, 2) + z, Q(1)]}[p]
    out = []
    for a in range(p + 1):
        q = [Q(1)]
        for b in range(p + 1):
            if b != a:
                q = _mul(q, [-x[b] / (x[a] - x[b]), 1 / (x[a] - x[b])])
        out.append(q)
    return out


@pytest.fixture(scope="module")
def tables(tmp_path_factory):
    nvcc = shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"
    if not os.path.exists(nvcc):
        pytest.skip("nvcc not available")
    exe = str(tmp_path_factory.mktemp("modal") / "modal_tables_check")
    subprocess.run([nvcc, "-std=c++17", "-O2", "-o", exe, os.path.join(HERE, "native", "modal_tables_check.cu")],
                   check=True, capture_output=True)
    out = {}
    for line in subprocess.run([exe], capture_output=True, text=True, check=True).stdout.split("\n"):
        if line:
            name, *at, v = line.split()
            out[(name, *map(int, at))] = float.fromhex(v)
    return out


@pytest.mark.parametrize("basis", [0, 1])
@pytest.mark.parametrize("p", [1, 2, 3, 4])
def test_modal_tables(tables, p, basis):
    n = p + 1
    tol = Q(8, 2 ** 53) if not basis else Q(1, 2 ** 48)
    B = _basis(p, basis)
    L = [[(2 * k + 1) * _int(_mul(LEG[k], B[a])) for a in range(n)] for k in range(n)]

    def near(key, exact):
        got = Q(tables[key])
        assert abs(got - exact) <= tol * max(abs(exact), Q(1, 2 ** 20)), (key, float(got), float(exact))

    pairs = (p + 1) // 2
    for k in range(n):
        for j in (1, 2):
            if j < pairs + (1 if k % 2 == 0 and p % 2 == 0 else 0):
                near(("mf", basis, p, k, j - 1), L[k][p - j] / L[k][p])
        for j in range(n):
            c = (2 * k + 1) * _int(_mul(_at_next(LEG[j]), LEG[k])) * L[j][p] / L[k][p]
            near(("mc", basis, p, k, j), c if j > k else Q(int(j == k)))
    S = [[[_int(_mul(_diff(LEG[k], d), _diff(LEG[m], d))) for m in range(n)] for k in range(n)] for d in range(n)]
    for i in range(n * n):
        for j in range(n * n):
            k, kk, m, mm = i % n, i // n, j % n, j // n
            s = sum(S[a][k][m] * S[b][kk][mm] for a in range(n) for b in range(n - a) if a + b >= 1)
            near(("m2", basis, p, i, j), s * L[k][p] * L[m][p] * L[kk][p] * L[mm][p] * (1 if i == j else 2))
