"""The sweep's fixed-point reconstructions (csrc/ase_df_fixed.cuh), compiled for the host: constants to the
bit, mirrored, negated and scaled data alike, what does not fit refused, and an rms error against
exact sums that is no larger than the FP64 chain's for every kind of stencil that is let in."""
import os
import shutil
import subprocess
from fractions import Fraction

import pytest

from test_fixed_weights import nodes, polynomial

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_2410_05489_gb300", "csrc")


def exact_weights():
    """Per order: f (normal, W_-k .. W_k), e and o (even and odd Gauss-point weights) as doubles, then as long
    doubles (a double and its remainder)."""
    rows = []
    for order in (3, 5, 7, 9):
        k = (order - 1) // 2
        P = polynomial(k)
        at = lambda xi: [sum(xi ** q * P[q][i] for q in range(order)) for i in range(order)]  # noqa: B023, E731
        f = at(Fraction(0)) + [Fraction(0)] * (9 - order)
        e = [[Fraction(0)] * 5 for _ in range(2)]
        o = [[Fraction(0)] * 5 for _ in range(2)]
        G = 1 if order == 3 else k
        for g, x in enumerate(nodes(G)):
            w = at(x - 1)
            for t in range(k + 1):
                e[g][t] = (w[k + t] + w[k - t]) / 2 if t else w[k]
                o[g][t] = (w[k + t] - w[k - t]) / 2 if 2 * g + 1 != G else Fraction(0)
        dbl = lambda v: float(v).hex()  # noqa: E731
        ldbl = lambda v: "%sL + %sL" % (float(v).hex(), float(v - Fraction(float(v))).hex())  # noqa: E731
        vec = lambda v, s: "{" + ", ".join(s(x) for x in v) + "}"  # noqa: E731
        mat = lambda m, s: "{" + ", ".join(vec(r, s) for r in m) + "}"  # noqa: E731
        rows.append("{" + ", ".join(h(x, s) for s in (dbl, ldbl) for h, x in ((vec, f), (mat, e), (mat, o))) + "}")
    return ("struct Exact { double f[9], e[2][5], o[2][5]; long double F[9], E[2][5], O[2][5]; };\n"
            "static const Exact kExact[4] = {\n" + ",\n".join(rows) + "};\n")


def test_reconstructions_on_the_host(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("g++ not found")
    (tmp_path / "cuda_runtime.h").write_text("")  # the check defines the few intrinsics itself
    (tmp_path / "exact_weights.h").write_text(exact_weights())
    exe = str(tmp_path / "fixed_check")
    subprocess.run([cxx, "-std=c++17", "-O2", "-ffp-contract=off", "-fwrapv", "-I", str(tmp_path), "-I", CSRC,
                    os.path.join(HERE, "fixed_check.cpp"), "-o", exe], check=True, capture_output=True, text=True)
    res = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert res.returncode == 0, res.stdout + res.stderr
    assert res.stdout.endswith("ok\n"), res.stdout
