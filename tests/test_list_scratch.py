"""Scratch of the list builder (csrc/list_scratch.cuh): what is sized for some
capacities holds every chunk built with these or smaller ones.  Compiled for
the host."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(__file__), "..", "paper_1807_10459_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "list_scratch.cuh"
using namespace idtx;
int main()
{
    const int64_t ns[] = {9, 200, 1000, 2049, 4097, 9995, 18501, 65537, 99850, 2000000};
    const int caps[] = {32, 64, 1024, 1504, 1536, 1568, 2016, 2048, 2080, 3072, 4064, 4096};
    int bad = 0;
    for (int64_t n : ns)
        for (int a : caps)
            for (int b : caps)
                for (int a2 : caps)
                    for (int b2 : caps)
                        if (a <= 2048 && a2 <= a && (b2 <= b) &&
                            (chunk_bytes(n, a2, b2) > list_scratch_bytes(n, a, b) ||
                             chunk_bytes(n, a2, 0) > list_scratch_bytes(n, a, b)))
                            if (bad++ < 5)
                                std::printf("n %lld: %d, %d in scratch for %d, %d\n", (long long)n, a2, b2, a, b);
    for (int cap = 32; cap < 4096; cap += 32)
        if (buf_of(cap, 1 << 20) > buf_of(cap + 32, 1 << 20) || buf_of(cap, 1 << 20) < cap + 32) ++bad;
    return bad != 0;
}
"""


def test_scratch_holds_smaller_capacities(tmp_path):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    src = tmp_path / "t.cpp"
    src.write_text(PROGRAM)
    exe = str(tmp_path / "t")
    subprocess.run(["g++", "-std=c++17", "-O1", "-I", CSRC, str(src), "-o", exe], check=True)
    r = subprocess.run([exe], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
