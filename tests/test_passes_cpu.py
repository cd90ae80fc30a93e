"""How a call's steps are cut into passes of several steps: every step is
taken, for the largest step count that a call accepts too."""
import subprocess

from paper_1806_10241_gb300 import build

PROGRAM = """
#include "lb_internal.h"
#include <cstdio>
#include <climits>
int main() {
    for (int T = 1; T <= 4; ++T)
        for (long long n : {1LL, 2LL, 3LL, 4LL, 5LL, 7LL, 12LL, 500LL, (long long)INT_MAX - 2, (long long)INT_MAX - 1, (long long)INT_MAX})
            std::printf("%d %lld %lld\\n", T, n, (long long)lbk::pass_count(n, T));
}
"""


def test_passes_take_every_step(tmp_path):
    src = tmp_path / "passes.cu"
    src.write_text(PROGRAM)
    subprocess.run([build.NVCC, "-std=c++17", "-I", build.CSRC, "-o", str(tmp_path / "passes"), str(src)], check=True)
    out = subprocess.run([str(tmp_path / "passes")], check=True, capture_output=True, text=True).stdout
    rows = [tuple(map(int, line.split())) for line in out.splitlines()]
    assert len(rows) == 44
    for T, n, m in rows:
        assert 1 <= m <= n and (n - m) % 2 == 0
        # passes of n // m and n // m + 1 steps
        assert n // m + (1 if n % m else 0) <= T and m * (n // m) + n % m == n
        assert m <= -(-n // T) + 1
