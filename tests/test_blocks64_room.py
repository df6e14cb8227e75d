"""Room for the pair blocks of a float64 Lanczos solve (csrc/sym64_plan.h), compiled with g++ on the CPU: enough for the
solve or none, at most 8 GB, and an eighth of the device left free."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.abspath(__file__)), "..", "paper_1612_00474_gb300", "csrc")
SRC = r"""#include <initializer_list>
#include "sym64_plan.h"
using namespace rpb;
int main() {
    const int64_t GB = (int64_t)1 << 30;
    for (int64_t total : {2 * GB, 80 * GB, 280 * GB})
        for (int64_t max_N : {1, 32, 33, 1000, 4096, 16500, 200000})
            for (int64_t N : {1, 33, 1000, 1200, 4096, 16000, 16500, 150000})
                for (int64_t held : {0, 31, 990, 1000, 4000, 16000})
                    for (int64_t used : {(int64_t)0, total / 2, total * 7 / 8 - 1000, total}) {
                        if (N > max_N || held >= N || blocks64_bytes(held) > used) continue;
                        const int64_t room = blocks64_room(N, held, max_N, total - used, total);
                        const int64_t left = total - used + (held ? blocks64_bytes(held) : 0);
                        const bool fits = blocks64_bytes(N) <= 8 * GB && left - blocks64_bytes(N) >= total / 8;
                        if ((room > 0) != fits) return 1;
                        if (!room) continue;
                        if (room < N || room > max_N) return 2;
                        if (held == 0 && room != N) return 3;
                        if (room > N && room > held + held / 4) return 4;
                        if (blocks64_bytes(room) > 8 * GB || left - blocks64_bytes(room) < total / 8) return 5;
                    }
    // 64 bytes for both spheres of each ordered pair of the triangle's units
    return blocks64_bytes(4096) == (int64_t)128 * 129 / 2 * 1024 * 64 && blocks64_bytes(1) == 65536 ? 0 : 6;
}
"""


def test_room(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    (tmp_path / "r.cpp").write_text(SRC)
    subprocess.run([gxx, "-O1", "-std=c++17", "-I", CSRC, str(tmp_path / "r.cpp"), "-o", str(tmp_path / "r")], check=True)
    assert subprocess.run([str(tmp_path / "r")]).returncode == 0
