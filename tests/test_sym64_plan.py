"""Work split of the float64 symmetric pass (csrc/sym64_plan.h), compiled with g++ on the CPU: the runs cover the
triangle of tiles once, in row order, and every plan stays inside the scratch of a larger context."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1612_00474_gb300", "csrc")
SRC = r"""#include <cstdio>
#include <cstdlib>
#include <set>
#include <utility>
#include "sym64_plan.h"
using namespace rpb;
int main(int argc, char **argv) {
    const int sms = atoi(argv[1]);
    for (int k = 2; k < argc; ++k) {
        const int64_t N = atoll(argv[k]);
        const Sym64Plan p = sym64_plan(N, sms);
        std::set<std::pair<int, int>> seen;
        std::set<int64_t> slots;
        int64_t top = -1;
        for (int64_t r = 0; r < p.runs; ++r) {
            const int b = sym64_row_of(p, r), t0 = b + (int)(r - sym64_row_run(p, b)) * p.L;
            const int t1 = t0 + p.L < p.nb ? t0 + p.L : p.nb;
            if (b < 0 || b >= p.nb || t0 < b || t0 >= t1) return 1;
            for (int t = t0; t < t1; ++t) {
                if (!seen.insert({b, t}).second) return 2;
                for (int s = 0; t > b && s < p.qs; ++s) {
                    const int64_t q = sym64_col_slot(p, b, t, s);
                    if (q < 0 || !slots.insert(q).second) return 3;
                    if (q > top) top = q;
                }
            }
        }
        if ((int64_t)seen.size() != (int64_t)p.nb * (p.nb + 1) / 2) return 4;
        if (sym64_row_run(p, 0) != 0 || sym64_row_run(p, p.nb) != p.runs) return 5;
        for (int64_t M : {N, N + 1, 2 * N, N + 1000})
            if (p.runs * p.qs * 96 > sym64_tgt_elems(M, sms) || (top + 1) * 96 > sym64_src_elems(M, sms)) return 6;
        for (int part = 0; part < 4 * p.qs; ++part)  // every part of a unit has a whole number of rotations, all 32 in all
            if (32 * (part + 1) / (4 * p.qs) < 32 * part / (4 * p.qs)) return 7;
    }
    return 0;
}
"""


@pytest.mark.parametrize("sms", [1, 4, 152])
def test_plan(tmp_path, sms):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    (tmp_path / "p.cpp").write_text(SRC)
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", CSRC, str(tmp_path / "p.cpp"), "-o", str(tmp_path / "p")], check=True)
    sizes = list(range(1, 140)) + [256, 511, 512, 513, 700, 1000, 1024, 2047, 3001, 4096, 4097, 10007]
    assert subprocess.run([str(tmp_path / "p"), str(sms), *map(str, sizes)]).returncode == 0
