"""The rational approximation of the square root (csrc/sqrt_nodes.h), compiled with g++ on the CPU."""
import math
import os
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1612_00474_gb300", "csrc")
SRC = """#include <cstdio>
#include "sqrt_nodes.h"
int main() { const rpb::SqrtNodes r = rpb::sqrt_nodes();
for (int j = 0; j < rpb::kSqrtNodes; ++j) printf("%.17g %.17g\\n", r.s[j], r.w[j]); }
"""


@pytest.fixture(scope="module")
def nodes(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("nodes")
    (d / "n.cpp").write_text(SRC)
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", CSRC, str(d / "n.cpp"), "-o", str(d / "n")], check=True)
    out = subprocess.run([str(d / "n")], check=True, capture_output=True, text=True).stdout
    return np.array([[float(x) for x in line.split()] for line in out.splitlines()]).T


def test_square_roots(nodes):
    s, w = nodes
    assert np.all(s > 0) and np.all(w > 0) and np.all(np.diff(s) > 0)
    for lam in np.geomspace(1e-19, 1.0, 400):
        # 128 positive terms: their rounding, a few units in the last place of the sum
        assert abs(math.fsum(w * lam / (lam + s)) / math.sqrt(lam) - 1.0) < 4e-15
    # below the interval: at most the root of its end
    assert math.fsum(w * 1e-26 / (1e-26 + s)) < 1e-10


@pytest.mark.parametrize("kappa,k", [(10.0, 1), (10.0, 2), (1e3, 8), (1e4, 20), (1e6, 40)])
def test_tridiagonal(nodes, kappa, k):
    """The shifted eliminations of the kernel in numpy against the eigen-decomposition."""
    s, w = nodes
    rng = np.random.default_rng(k)
    lam = np.geomspace(1.0, 1.0 / kappa, k + 10)
    v = rng.standard_normal(k + 10)
    V, al, be = [v / np.linalg.norm(v)], [], []
    for _ in range(k):
        x = lam * V[-1]
        for _ in range(2):
            c = np.array(V) @ x
            x = x - c @ np.array(V)
            al.append(c[-1])
        al[-2:] = [al[-2] + al[-1]]
        be.append(np.linalg.norm(x))
        V.append(x / be[-1])
    T = np.diag(al) + np.diag(be[:-1], 1) + np.diag(be[:-1], -1)
    e, Q = np.linalg.eigh(T)
    ref = Q @ (np.sqrt(e) * Q[0])
    M = np.abs(T).sum(1).max()
    c = np.full(s.size, al[-1])
    r = [1.0 / (c + M * s)]
    for i in range(k - 2, -1, -1):
        c = al[i] - be[i] ** 2 * r[0]
        r.insert(0, 1.0 / (c + M * s))
    x0 = w * r[0]
    z, y = -M * s * x0, [np.sum(c * x0)]
    for i in range(1, k):
        z = -be[i - 1] * r[i] * z
        y.append(np.sum(z))
    # the reference's own error: rounding over the smallest eigenvalue's square root
    assert np.linalg.norm(math.sqrt(M) * np.array(y) - ref) <= 1e-15 * math.sqrt(kappa) * 20 * np.linalg.norm(ref)
