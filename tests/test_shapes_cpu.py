"""The launchers' shape rules, on the CPU."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2506_18408_gb300", "csrc")

PROGRAM = r"""
#include "shapes.h"
#include <cstdio>
using namespace sfg;
// limit: CTAs of the largest cluster the device holds, unstaged; staged: the same for a staged slice
static void line(int P, int s, int m, size_t left, int staged, int plain) {
    int asked = 0;
    const QrShape q = qr_shape(P, s, m, left, false, [&](const QrShape& c) {
        ++asked;
        return c.cluster <= (c.staged ? staged : plain);
    });
    std::printf("%d %d %d %d %d %zu\n", q.cluster, q.staged ? 1 : 0, q.nrp, q.slice, asked, qr_smem(q, m, m - 1));
}
int main() {
    const size_t big = 226 * 1024;
    line(1, 1000, 200, big, 16, 16);
    line(1, 1000, 200, big, 8, 16);
    line(1, 1000, 200, big, 8, 8);
    line(1, 1000, 200, 20000, 16, 16);
    line(1, 1000, 200, 20000, 16, 8);
    line(1, 120, 30, big, 0, 0);
    line(16, 1000, 200, big, 0, 0);
    line(4, 400, 100, big, 8, 8);
    for (int i : {0, 8, 16, 30}) std::printf("%d ", qr_long(120, 4, i));
    for (int i : {1, 16, 32, 33, 59}) std::printf("%d ", qr_long(240, 4, i));
    for (int i : {1, 16, 17, 99}) std::printf("%d ", qr_long(1000, 16, i));
    std::printf("\n");
}
"""


def test_clusters_fall_back_to_what_the_device_places(tmp_path):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("no g++")
    src, exe = tmp_path / "shapes.cpp", tmp_path / "shapes"
    src.write_text(PROGRAM)
    r = subprocess.run([gxx, "-std=c++17", "-I", CSRC, "-o", str(exe), str(src)], capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    *got, parts = [tuple(map(int, ln.split())) for ln in
                   subprocess.run([str(exe)], capture_output=True, text=True, check=True).stdout.splitlines()]
    # 64^2 (30 rows: at most 8 a group, 30 columns in four groups); 60 rows in 8, 4 or 2 groups, 59 columns in two; 63 rows in
    # 8 groups up to 8 columns' worth of threads, then 4 (16 rows) and 2 (32 rows)
    assert parts == (0, 0, 0, 0) + (0, 0, 0, 1, 1) + (0, 0, 0, 1)
    kind = [(c, st, asked) for c, st, _, _, asked, _ in got]
    assert kind == [(16, 1, 1),   # held as wanted
                    (16, 0, 2),   # not with its slice in shared memory: the same cluster, so the same sums, from L2
                    (8, 1, 2),    # not at all: the portable size, whose slices of 125 rows fit
                    (16, 0, 1),   # no room for the slice beside the step
                    (8, 0, 1),
                    (4, 1, 0),    # portable sizes are not asked about
                    (8, 1, 0),
                    (8, 1, 2)]
    for (P, s, m), (c, st, nrp, slice_, _, smem) in zip([(1, 1000, 200)] * 5 + [(1, 120, 30), (16, 1000, 200), (4, 400, 100)], got):
        assert nrp % 2 == 1 and c * nrp >= s and slice_ >= nrp * m and slice_ % 2 == 0
        assert smem == 8 * ((((m - 1) * nrp + 1) // 2 * 2 if st else 0) + 2 * nrp + 3 * m)
