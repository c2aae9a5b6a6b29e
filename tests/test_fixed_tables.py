"""The integer tables compiled into the fixed-point kernels, against the float64 tables."""
import numpy as np
import pytest


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
def test_fixed_point_tables(native, n):
    """The integer tables of the fixed-point operators against the float64 tables of
    dg_ref_tables, within the float64 rounding of the latter (1e-13 of the largest entry)."""
    import os
    import re
    path = os.path.join(os.path.dirname(native.__file__), "csrc", "dg_fixed_tables.cuh")
    src = open(path).read()
    t = native.ref_tables(n)
    w = t["w"] / 2
    rw = 1 / np.sqrt(w)
    want = {"deriv": (t["C0"], t["muR"], t["lL"], -t["muL"], t["lR"]),
            "stiff": (rw[:, None] * t["A1cc"] * rw, rw * t["betaA"], rw * t["lL"], rw * t["lL"], rw * t["betaA"]),
            "lap": (t["A1cc"] / w[:, None], t["betaA"] / w, t["lL"], t["lL"] / w, t["betaA"])}
    for name, (M, a, r, d, s) in want.items():
        body = re.search(r"fx_%s<%d>\(\) \{\s*return \{(.*?)\};\s*\}" % (name, n), src, re.S).group(1)
        e, er, es = (int(v) for v in body.split(",")[:3])
        v = np.array([int(h) * 2 ** 30 + int(lo) for h, lo in re.findall(r"\{(-?\d+),(-?\d+)\}", body)], dtype=object)
        v = (v.astype(object) / 2 ** 60).astype(float)
        m = n * n
        got = (v[:m].reshape(n, n) * 2.0 ** e, v[m:m + n] * 2.0 ** (e - er), v[m + n:m + 2 * n] * 2.0 ** er,
               v[m + 2 * n:m + 3 * n] * 2.0 ** (e - es), v[m + 3 * n:m + 4 * n] * 2.0 ** es)
        for g, x in zip(got, (M, a, r, d, s)):
            assert np.abs(g - x).max() <= 1e-13 * max(1.0, np.abs(M).max()), (name, n)
        # the bound the accumulators rely on: rows, the traces' sums included, below 1
        row = np.abs(got[0]).sum(1) + np.abs(got[1]) * np.abs(got[2]).sum() + np.abs(got[3]) * np.abs(got[4]).sum()
        assert row.max() < 2.0 ** e and np.abs(got[2]).sum() <= 2.0 ** er and np.abs(got[4]).sum() <= 2.0 ** es


def _exact_tables(n):
    """The same operators with 60 decimal digits, from Lagrange bases on the Gauss nodes: for each its
    row sums' parts M, a, r, d, s and, of the first cell at a Dirichlet boundary, Mf, af, sf."""
    from decimal import Decimal as D, getcontext
    getcontext().prec = 60
    R = range(n)
    x = []
    for x0 in np.polynomial.legendre.leggauss(n)[0]:  # Newton's method on the Legendre polynomial
        t = D(float(x0))
        for _ in range(7):
            p, q = D(1), t
            for k in range(2, n + 1):
                p, q = q, ((2 * k - 1) * t * q - (k - 1) * p) / k
            dq = n * (t * q - p) / (t * t - 1)
            t -= q / dq
        x.append((t, 2 / ((1 - t * t) * dq * dq)))
    x, w = [v[0] for v in x], [v[1] / 2 for v in x]  # weights of a cell of size 1

    def prod(v):
        out = D(1)
        for u in v:
            out *= u
        return out
    den = [prod(x[j] - x[m] for m in R if m != j) for j in R]
    lL = [prod(-1 - x[m] for m in R if m != j) / den[j] for j in R]
    lR = [prod(1 - x[m] for m in R if m != j) / den[j] for j in R]
    d = [[sum((prod(x[i] - x[m] for m in R if m not in (j, k)) for k in R if k != j), D(0)) / den[j] for j in R]
         for i in R]
    half = D(1) / 2
    C = [[2 * d[i][j] - half * (lR[i] * lR[j] - lL[i] * lL[j]) / w[i] for j in R] for i in R]
    F = [[2 * d[i][j] - lR[i] * lR[j] / w[i] for j in R] for i in R]            # flux from the right cell
    Ff = [[F[i][j] + lL[i] * lL[j] / w[i] for j in R] for i in R]               # first cell at a boundary
    up = [lR[i] / w[i] for i in R]

    def gram(A, last):
        return [[sum((w[k] * A[k][i] * A[k][j] for k in R), D(0)) + last * lL[i] * lL[j] *
                 sum((w[k] * up[k] * up[k] for k in R), D(0)) for j in R] for i in R]
    K, Kf = gram(F, 1), gram(Ff, 0)
    Kf = [[Kf[i][j] + lL[i] * lL[j] for j in R] for i in R]                     # boundary penalty 1 / h
    be, bf = ([sum((A[k][i] * lR[k] for k in R), D(0)) for i in R] for A in (F, Ff))
    rw = [1 / v.sqrt() for v in w]
    zero = [D(0)] * n
    scale = lambda v, c: [v[i] * c[i] for i in R]
    iw = [1 / v for v in w]
    return {"deriv": (C, [half * v for v in up], lL, [-half * lL[i] / w[i] for i in R], lR, [zero] * n, zero, zero),
            "stiff": ([[rw[i] * K[i][j] * rw[j] for j in R] for i in R], scale(be, rw), scale(lL, rw), scale(lL, rw),
                      scale(be, rw), [[rw[i] * Kf[i][j] * rw[j] for j in R] for i in R], scale(bf, rw), scale(bf, rw)),
            "lap": ([[iw[i] * K[i][j] for j in R] for i in R], scale(be, iw), lL, scale(lL, iw), be,
                    [[iw[i] * Kf[i][j] for j in R] for i in R], scale(bf, iw), bf)}


@pytest.mark.parametrize("n", [1, 2, 3, 4, 5])
def test_fixed_point_tables_are_rounded_to_one_unit(native, n):
    """Every entry, the first Dirichlet cell's included, is the coefficient rounded to an integer (half a
    unit), and the rows of the inner, the first and the second cell keep the accumulators' bounds."""
    import os
    import re
    from decimal import Decimal as D
    src = open(os.path.join(os.path.dirname(native.__file__), "csrc", "dg_fixed_tables.cuh")).read()
    for name, (M, a, r, d, s, Mf, af, sf) in _exact_tables(n).items():
        body = re.search(r"fx_%s<%d>\(\) \{\s*return \{(.*?)\};\s*\}" % (name, n), src, re.S).group(1)
        e, er, es = (int(v) for v in body.split(",")[:3])
        v = [int(h) * 2 ** 30 + int(lo) for h, lo in re.findall(r"\{(-?\d+),(-?\d+)\}", body)]
        want = [(x, e) for row in M for x in row]
        for part, k in ((a, e - er), (r, er), (d, e - es), (s, es)):
            want += [(x, k) for x in part]
        if name != "deriv":  # the derivative takes ghost traces at a boundary
            want += [(x, e) for row in Mf for x in row] + [(x, e - er) for x in af] + [(x, es) for x in sf]
        assert len(v) == len(want)
        off = [abs(D(i) - x * D(2) ** (60 - k)) for i, (x, k) in zip(v, want)]
        assert max(off) <= D("0.5001"), (name, max(off))
        # |row| <= 2^e with the traces' own sums, |r| and |s| (sf) below 2^er and 2^es
        S = lambda u: sum(map(abs, u))
        assert S(r) <= 2 ** er and max(S(s), S(sf)) <= 2 ** es
        for m, lift, trace in ((M, a, s), (Mf, af, s), (M, a, sf)):
            assert max(S(m[i]) + abs(lift[i]) * S(r) + abs(d[i]) * S(trace) for i in range(n)) < 2 ** e, name
