"""Counts of tiles at the last positions a state can have (2^31 - 2): the helper of
kmc_internal.h that the filtered search runs on, on the CPU."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SRC = r"""
#include "kmc_internal.h"
#include <stdio.h>
int main() {
    const int32_t last = 2147483646;
    const int32_t ends[] = {1, 7, 8, 9, 63, 64, 65, 1000, 1 << 30, last - 65, last - 64, last - 63, last - 8, last - 7, last - 1, last};
    for (int32_t size : {8, 64})
        for (int32_t q1 : ends)
            for (int32_t q0 : ends)
                printf("%d %d %d %d\n", size, q0, q1, kmc::pieces_touched(q0, q1, size));
}
"""


def test_pieces_up_to_the_last_position(tmp_path):
    src, exe = tmp_path / "t.cpp", str(tmp_path / "t")
    src.write_text(SRC)
    cuda = os.path.join(os.environ.get("CUDA_HOME", "/usr/local/cuda"), "include")
    subprocess.run(["g++", "-std=c++17", "-fsanitize=undefined", "-fno-sanitize-recover=all", "-I", cuda, "-I",
                    os.path.join(ROOT, "paper_1210_8084_gb300", "csrc"), str(src), "-o", exe], check=True)
    lines = subprocess.run([exe], check=True, capture_output=True, text=True).stdout.split("\n")[:-1]
    assert len(lines) == 2 * 16 * 16
    for line in lines:
        size, q0, q1, touched = map(int, line.split())
        assert touched == (-(-q1 // size) - q0 // size if q1 > q0 else 0)
