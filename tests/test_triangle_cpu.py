"""Packed-triangle indices of the B_opt solver on the host: every entry's row and column, up to columns of
more members than 32-bit products hold."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2302_00414_gb300", "csrc")

PROGRAM = r"""
#define __host__
#define __device__
#define __forceinline__ inline
#include "triangle.cuh"
#include <cstdio>
using namespace infft;
static int check(long long e) {
    long long r = -1, c = -1;
    tri_rc(e, &r, &c);
    if (r >= 0 && c >= 0 && c <= r && r < (1LL << 31) && tri(r, c) == e) return 0;
    printf("entry %lld: row %lld, column %lld\n", e, r, c);
    return 1;
}
int main() {
    int bad = 0;
    for (long long e = 0; e < 100000; ++e) bad += check(e);
    // the first and last entries of rows around every power of two, and around the limit of 32-bit products
    for (long long r = 64; r < 200000 && bad < 10; r = r * 9 / 8 + 1)
        for (long long q = r - 1; q <= r + 1; ++q) bad += check(tri(q, 0)) + check(tri(q, q)) + check(tri(q, q / 2));
    for (long long r = 46330; r < 46350 && bad < 10; ++r) bad += check(tri(r, 0)) + check(tri(r, 1)) + check(tri(r, r));
    for (long long e = (1LL << 30) - 3; e < (1LL << 30) + 3 && bad < 10; ++e) bad += check(e);
    return bad != 0;
}
"""


def test_rows_and_columns(tmp_path):
    cc = shutil.which("g++")
    if cc is None:
        pytest.skip("no host compiler")
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(PROGRAM)
    subprocess.run([cc, "-O1", "-fwrapv", "-std=c++17", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    r = subprocess.run([str(exe)], capture_output=True, text=True, timeout=60)
    assert r.returncode == 0, r.stdout
