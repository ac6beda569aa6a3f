"""The multiplication and shift that stand for the division of an element's index by the
row length (laps_rows.cuh), against the division: every row length a target or a batch
problem can have, indices at both ends of rows over the whole 31 bits.  Host code, no GPU."""
import os
import subprocess

from conftest import ROOT

MAIN = r"""
#include <cstdio>
#include "laps_rows.cuh"
int main() {
    unsigned long long bad = 0, seen = 0;
    unsigned rnd = 1;
    for (int w = 1; w <= 10304; ++w) {
        const laps::RowIndex r = laps::row_index(0x7fffffff / w, w);
        const uint32_t rows = 0x7fffffffu / w;
        for (int t = 0; t < 400; ++t) {
            rnd = rnd * 1664525u + 1013904223u;
            const uint32_t q = t < 20 ? t : t < 40 ? rows - (t - 20) : rnd % rows;
            for (int e = -1; e <= 1; ++e) {
                const int64_t k = (int64_t)q * w + e;
                if (k < 0 || k > 0x7ffffffe) continue;
                uint32_t row;
                int col;
                laps::row_of(r, (uint32_t)k, row, col);
                ++seen;
                if (row != (uint32_t)k / w || col != (int)((uint32_t)k % w)) ++bad;
            }
        }
    }
    printf("%llu %llu\n", seen, bad);
    return 0;
}
"""


def test_row_and_column_of_an_index(tmp_path):
    from paper_2601_16696_gb300 import build
    src, exe = tmp_path / "rows.cu", tmp_path / "rows"
    src.write_text(MAIN)
    cmd = [build._nvcc(), *build.FLAGS, "-I", os.path.join(ROOT, "paper_2601_16696_gb300", "csrc"), str(src), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    assert r.returncode == 0, r.stdout + r.stderr
    seen, bad = map(int, subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.split())
    assert seen > 10 ** 7 and bad == 0
