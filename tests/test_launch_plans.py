"""Launch rules that are plain host arithmetic, compiled from the headers that hold them (no GPU needed)."""
import os
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2603_09215_b200", "csrc")

MAIN = """
#include <cstdio>
#include "sparsk_gemm.cuh"
int main()
{
    const int sms[] = {1, 2, 74, 132, 148};
    for (int n : sms)
        for (int F = 8; F <= 65536; F += 8) printf("%d %d %d\\n", n, F, sparsk::gateup_unit_rows(F, n));
}
"""


def _up(a, b):
    return -(-a // b)


@pytest.mark.skipif(shutil.which("nvcc") is None, reason="needs nvcc")
def test_gateup_units_are_dealt_evenly_without_more_rounds(tmp_path):
    """The height of a gate/up unit is a multiple of 8 rows in 32..128, no SM takes more units one after
    another than with 128 rows, and 8 rows less would make one do so (lower units cost as many MMAs as
    high ones)."""
    src, exe = tmp_path / "plan.cu", str(tmp_path / "plan")
    src.write_text(MAIN)
    subprocess.run(["nvcc", "-std=c++17", "-gencode", "arch=compute_100a,code=sm_100a", "-I", CSRC, "-o", exe, str(src)], check=True)
    rows = [tuple(map(int, l.split())) for l in subprocess.run([exe], check=True, capture_output=True, text=True).stdout.splitlines()]
    assert len(rows) == 5 * 8192
    for n, F, r in rows:
        rounds = _up(_up(F, 128), n)
        assert r % 8 == 0 and 32 <= r <= 128
        assert _up(_up(F, r), n) == rounds, (n, F, r)
        assert r == 32 or _up(_up(F, r - 8), n) > rounds, (n, F, r)
