"""How a batch is split into runs, against batches that were timed either way on a GB300: whether libraries of several k
share runs (mixed_runs_pay) and whether a large one runs alone (runs_alone). CPU: C++ programs ask the built library."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

K2, K3, K4 = (21, 31), (21, 25, 31), (25, 29, 31, 55)
K12 = (17, 19, 21, 23, 25, 27, 29, 31, 33, 41, 51, 55)
# (libraries, bases of each, k in turn, ms in mixed runs, ms grouped by k), those that differ by 6 % or more
TIMED = [
    (6, 20_000, K2, 0.709, 0.772), (6, 20_000, K12, 0.660, 1.354), (6, 1_000_000, K3, 0.995, 1.175),
    (6, 4_000_000, K2, 1.701, 1.596), (6, 4_000_000, K12, 1.746, 1.964), (6, 10_000_000, K4, 3.361, 2.902),
    (12, 200_000, K2, 1.142, 1.351), (12, 1_000_000, K12, 1.622, 3.026), (12, 4_000_000, K3, 3.231, 2.884),
    (12, 4_000_000, K12, 3.277, 3.830), (12, 10_000_000, K12, 7.106, 6.184), (24, 200_000, K3, 1.993, 2.214),
    (24, 1_000_000, K3, 2.949, 2.779), (24, 1_000_000, K4, 2.830, 3.035), (24, 1_000_000, K12, 2.911, 4.260),
    (24, 4_000_000, K4, 6.324, 5.473), (48, 200_000, K2, 3.740, 4.054), (48, 1_000_000, K2, 5.880, 5.426),
    (48, 1_000_000, K3, 5.906, 5.541), (48, 1_000_000, K12, 5.833, 6.483), (48, 4_000_000, K2, 14.971, 10.176),
]

BODY = """
#include <cstdio>
#include <vector>
#include "host.h"
int main() {
    int libraries, n_k;
    unsigned long long bases;
    while (scanf("%d %llu %d", &libraries, &bases, &n_k) == 3) {
        std::vector<int> k(n_k);
        for (int &x : k)
            if (scanf("%d", &x) != 1) return 1;
        const uint64_t offsets[2] = {0, bases};
        std::vector<turtle_job> jobs(libraries);
        std::vector<size_t> idx;
        for (int i = 0; i < libraries; i++) {
            jobs[i] = turtle_job{nullptr, offsets, 1, k[i % n_k], 2};
            idx.push_back(i);
        }
        printf("%d\\n", (int)mixed_runs_pay(jobs.data(), idx));
    }
}
"""


def _ask(tmp_path, body, asked):
    if not shutil.which("g++"):
        pytest.skip("no C++ compiler")
    import paper_1305_1861_gb300 as pkg
    from paper_1305_1861_gb300 import _nvcc

    pkg.build()
    cuda = os.path.dirname(os.path.dirname(shutil.which("nvcc") or "/usr/local/cuda/bin/nvcc"))
    src, exe = tmp_path / "choice.cpp", tmp_path / "choice"
    src.write_text(body)
    subprocess.run(["g++", "-std=c++17", str(src), "-I", os.path.join(ROOT, "paper_1305_1861_gb300", "csrc"), "-I",
                    os.path.join(ROOT, "include"), "-I", os.path.join(cuda, "include"), _nvcc.LIB,
                    "-Wl,-rpath," + os.path.dirname(_nvcc.LIB), "-o", str(exe)], check=True)
    return subprocess.run([str(exe)], input=asked, check=True, capture_output=True, text=True).stdout.split()


def test_the_faster_way_is_chosen(tmp_path):
    asked = "".join("%d %d %d %s\n" % (n, b, len(ks), " ".join(map(str, ks))) for n, b, ks, _, _ in TIMED)
    assert _ask(tmp_path, BODY, asked) == [str(int(mixed < grouped)) for _, _, _, mixed, grouped in TIMED]


ALONE = """
#include <cstdio>
#include "host.h"
int main() {
    unsigned form;
    unsigned long long bases;
    while (scanf("%u %llu", &form, &bases) == 2) {
        const uint64_t offsets[2] = {7, bases + 7};
        turtle_params p;
        turtle_params_default(&p);
        p.compact = form;
        printf("%d\\n", (int)runs_alone(turtle_job{nullptr, offsets, 1, 31, 2}, p));
    }
}
"""


def test_large_libraries_run_alone_where_that_is_faster(tmp_path):
    """From 64 MiB by tiles and in the hash-table form; shared in the global one (and in what a batch runs as it)."""
    at = [(form, bases) for form in range(4) for bases in (1, (64 << 20) - 1, 64 << 20, 200_000_000)]
    got = _ask(tmp_path, ALONE, "".join("%d %d\n" % x for x in at))
    assert got == [str(int(form in (0, 2) and bases >= 64 << 20)) for form, bases in at]
