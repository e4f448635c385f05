"""The rule that chooses between the two tensor-core kNN kernels, at sizes where both were timed (us: CTAs
per 128 rows, units of 256): it must take the faster one wherever they differ by a tenth, with the list
length that the rows' kind gives (integers k, others a margin more)."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1707_00143_gb300", "csrc")

# n, queries, k, integer rows, self join, us by CTAs, us by units
TIMED = [
    (6000, 8000, 1, 0, 0, 1239, 1981), (8000, 8000, 64, 1, 1, 1357, 2292), (12000, 300, 10, 0, 0, 1403, 1544),
    (12000, 1500, 10, 0, 0, 1442, 1722), (12000, 1500, 10, 1, 0, 902, 659), (18000, 1500, 10, 0, 0, 1700, 1300),
    (26000, 300, 100, 0, 0, 3861, 2788), (26000, 26000, 100, 1, 1, 5340, 4319), (26000, 24000, 200, 1, 0, 9742, 15484),
    (40000, 40000, 100, 0, 1, 12861, 20223), (40000, 10000, 100, 0, 0, 4845, 6763), (40000, 1500, 100, 1, 0, 3321, 1064),
    (40000, 4000, 100, 1, 0, 3360, 1598), (40000, 40000, 100, 1, 1, 9160, 7000), (20000, 20000, 10, 0, 1, 2604, 4156),  # the last: rows in tight clusters
    (1000000, 1000, 100, 0, 0, 47300, 6500), (10000, 100, 10, 1, 0, 760, 490),
]


@pytest.mark.skipif(shutil.which("g++") is None, reason="needs g++")
def test_rule_takes_the_faster_kernel(tmp_path):
    src = tmp_path / "rule.cpp"
    src.write_text("""#include <cstdio>
#include <initializer_list>
#include "knn_rule.h"
struct T { long n, nq; int k, integers, self; };
int main() {
    for (T t : {%s}) {
        const int margin = t.k / 2 > 32 ? t.k / 2 : 32, KL = t.integers ? t.k : t.k + margin < 256 ? t.k + margin : 256;
        const bool bounded = nsg::knn_sample_tiles((t.n + 127) / 128, KL + t.self) > 0;
        std::printf("%%d\\n", nsg::knn_small(t.n, t.nq, KL, bounded, 152));
    }
}
""" % ", ".join("T{%d, %d, %d, %d, %d}" % t[:5] for t in TIMED))
    exe = tmp_path / "rule"
    subprocess.run(["g++", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    got = [int(x) for x in subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout.split()]
    for t, small in zip(TIMED, got):
        assert small == (t[5] < t[6]), t
