"""The end of the float32 column sums (csrc/float_sums.h), compiled with g++ on the CPU, against exact rationals: float64's
rounding of the total, whatever cancels."""
import os
import shutil
import subprocess
from fractions import Fraction

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1612_00474_gb300", "csrc")
SRC = r"""#include <cstdio>
#include "float_sums.h"
int main() {  // two sums of four chains each and their corrections, joined
    float s[4], c[4];
    rpb::FloatSum f[2];
    for (int k = 0; scanf("%a %a %a %a %a %a %a %a", s, s + 1, s + 2, s + 3, c, c + 1, c + 2, c + 3) == 8; k ^= 1) {
        f[k] = rpb::join_sums(s, c);
        printf("%a\n", f[k].value());
        if (k) {
            f[0].add(f[1]);
            printf("%a\n", f[0].value());
        }
    }
}
"""

WIDEN = r"""#include <initializer_list>
#include "float_sums.h"
int main() {  // every exponent and sign with some mantissas, against the conversion, bit for bit
    for (uint64_t k = 0; k < ((uint64_t)1 << 32); k += 509) {
        for (uint32_t b : {(uint32_t)k, (uint32_t)k & 0xff800000u, (uint32_t)k | 0x007fffffu, (uint32_t)k & 0x807fffffu}) {
            float x;
            std::memcpy(&x, &b, 4);
            const double y = rpb::widen(x), z = x;
            if (x == x ? std::memcmp(&y, &z, 8) != 0 : y == y) return 1;
        }
    }
}
"""


def _compiled(tmp_path, src):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    (tmp_path / "t.cpp").write_text(src)
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")], check=True)
    return str(tmp_path / "t")


def test_widen(tmp_path):
    assert subprocess.run([_compiled(tmp_path, WIDEN)]).returncode == 0


def test_join(tmp_path):
    exe = _compiled(tmp_path, SRC)
    rng = np.random.default_rng(1)
    rows = []
    for k in range(4000):
        s = rng.normal(size=4) * 2.0 ** rng.integers(-12, 13, 4)
        if k % 4 == 1:  # the sums cancel, the corrections are what is left
            s[1], s[3] = -s[0], -s[2]
        if k % 4 == 2:
            s[1] = -s[0] * (1 + 2.0 ** -20)
        c = rng.normal(size=4) * 2.0 ** -24 * np.abs(s)
        rows.append(np.concatenate([s, c]).astype(np.float32))
    rows += [np.zeros(8, np.float32)] * 2
    text = "\n".join(" ".join(float(x).hex() for x in r) for r in rows)
    out = subprocess.run([exe], input=text, check=True, capture_output=True, text=True).stdout.split()
    f = [[Fraction(float(x)) for x in r] for r in rows]
    groups = []
    for k in range(0, len(rows), 2):
        groups += [[f[k]], [f[k + 1]], [f[k], f[k + 1]]]
    assert len(out) == len(groups)
    for g, y in zip(groups, out):
        exact = sum(sum(r[:4]) - sum(r[4:]) for r in g)
        # one rounding of the total; the remainder, 2^-46 of the largest, has been added up in float32
        bound = abs(exact) * Fraction(1, 2 ** 53) + max(abs(x) for r in g for x in r) * Fraction(1, 2 ** 67)
        assert abs(Fraction(float.fromhex(y)) - exact) <= bound
