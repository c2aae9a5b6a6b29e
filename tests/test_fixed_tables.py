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
