"""sqrt(T) e1 by quadrature (csrc/tridiag_quad.h), compiled here for the host,
against numpy's eigendecomposition: sizes from 1, spectra over nine decades,
and the cases it must leave to QR."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2510_02135_gb300", "csrc")
MAIN = r"""
#include <cstdio>
#include "tridiag_quad.h"
int main() {
    lmk::SqrtQuadrature q;
    int m;
    while (std::scanf("%d", &m) == 1) {
        std::vector<double> a(m), b(m), z(m, 0.0);
        for (double& v : a) if (std::scanf("%lf", &v) != 1) return 1;
        for (int i = 0; i + 1 < m; ++i) if (std::scanf("%lf", &b[i]) != 1) return 1;
        const bool ok = q.solve(m, a.data(), b.data(), z.data());
        std::printf("%d", ok ? 1 : 0);
        for (double v : z) std::printf(" %.17g", v);
        std::printf("\n");
    }
}
"""


@pytest.fixture(scope="module")
def solve(tmp_path_factory):
    d = tmp_path_factory.mktemp("quad")
    src, exe = str(d / "q.cpp"), str(d / "q")
    with open(src, "w") as f:
        f.write(MAIN)
    subprocess.run(["g++", "-O2", "-std=c++17", "-I", CSRC, src, "-o", exe], check=True)

    def run(systems):
        text = "\n".join(" ".join(["%d" % len(a)] + ["%.17g" % v for v in [*a, *b]]) for a, b in systems)
        out = subprocess.run([exe], input=text, capture_output=True, text=True, check=True).stdout.splitlines()
        return [(int(ln.split()[0]), np.array(ln.split()[1:], float)) for ln in out]

    return run


def lanczos_t(rng, m, kappa):
    """alpha, beta of m Lanczos steps on a diagonal with condition number kappa."""
    n = max(4 * m, 40)
    ev = 3.0 * kappa ** (-np.arange(n) / (n - 1.0))
    v = rng.standard_normal(n)
    V, al, be = [v / np.linalg.norm(v)], [], []
    for _ in range(m):
        w = ev * V[-1]
        al.append(w @ V[-1])
        for _ in range(2):
            w -= np.array(V).T @ (np.array(V) @ w)
        be.append(np.linalg.norm(w))
        V.append(w / be[-1])
    return np.array(al), np.array(be[:m - 1])


def test_matches_eigendecomposition(solve):
    rng = np.random.default_rng(4)
    systems = [lanczos_t(rng, m, kappa) for kappa in (1.5, 1e2, 1e4, 1e6, 1e9) for m in (1, 2, 3, 17, 64, 130)]
    # one sequence as the caller makes it: m = 1, 2, 3, ... of one matrix (the bound carries over)
    al, be = lanczos_t(rng, 40, 1e5)
    systems += [(al[:m], be[:m - 1]) for m in range(1, 41)]
    for (a, b), (ok, z) in zip(systems, solve(systems)):
        ev, ec = np.linalg.eigh(np.diag(a) + np.diag(b, 1) + np.diag(b, -1))
        ref = ec @ (np.sqrt(np.maximum(ev, 0.0)) * ec[0])
        assert ok == 1
        # eigh's own root: an eigenvalue error of m eps |T| enters as its square root only below sqrt(eps) |T|
        assert np.linalg.norm(z - ref) <= 1e-12 * np.sqrt(a[0]) * max(1.0, len(a) / 10.0), len(a)


def test_leaves_indefinite_and_extreme_to_qr(solve):
    systems = [([1.0, -1e-3], [0.1]), ([1.0, 1.0], [1.0]), ([0.0], []), ([1e-200], []), ([1e150, 1e150], [1.0]),
               ([1.0, 1e-13], [0.0])]
    for ok, z in solve(systems):
        assert ok == 0 and not z.any()
