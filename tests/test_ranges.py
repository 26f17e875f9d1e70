"""The kernels' index arithmetic at the largest row count of a context
(2^31 - 1), on the CPU: the header that the kernels use, compiled for the host."""
import ctypes
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2608_20532_gb300", "csrc")
MAX = 2 ** 31 - 1

SRC = """
#include "ranges.cuh"
extern "C" {
int chunk_exists(int f, int k, int c, int n) { return f2::chunk_exists(f, k, c, n); }
int step_to(int a, int s, int n) { return f2::step_to(a, s, n); }
int chunk_count(int f, int c, int n) { return f2::chunk_count(f, c, n); }
int item_in(int a, int j, int n) { return f2::item_in(a, j, n); }
int all_rows(long long r) { return f2::all_rows(r); }
int rows_of(int c) { return f2::rows_of(c); }
int table_entries(int n, int m) { return f2::table_entries(n, m); }
}
"""


@pytest.fixture(scope="module")
def ranges(tmp_path_factory):
    d = tmp_path_factory.mktemp("ranges")
    (d / "r.cpp").write_text(SRC)
    # signed overflow traps, so that a sum that leaves 32 bits does not pass by luck
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-ftrapv", "-shared", "-fPIC", "-I", CSRC, str(d / "r.cpp"),
                           "-o", str(d / "r.so")])
    lib = ctypes.CDLL(str(d / "r.so"))
    lib.all_rows.argtypes = [ctypes.c_longlong]
    return lib


COUNTS = (1, 2, 63, 64, 1023, 1024, 1025, 2 ** 30, MAX - 1024, MAX - 1, MAX)


@pytest.mark.parametrize("n", COUNTS)
def test_chunks(ranges, n):
    for chunk in (1024, 2048):
        for start in {0, 1, n // 2, max(0, n - chunk), n - 1, n}:
            want = -(-(n - start) // chunk)
            assert ranges.chunk_count(start, chunk, n) == want
            # CTAs claim chunks past the last: at least one each
            for k in {0, 1, want - 1, want, want + 1, want + 456, want + 5000}:
                if k >= 0:
                    assert ranges.chunk_exists(start, k, chunk, n) == (start + k * chunk < n)


@pytest.mark.parametrize("n", COUNTS)
def test_steps(ranges, n):
    for step in (32, 128, 256, 512, 1024, 4096, 16384):
        for at in {0, 1, n // 2, max(0, n - step), max(0, n - step - 1), n - 1, n}:
            assert ranges.step_to(at, step, n) == min(at + step, n)
            for j in (0, 1, step - 1, step, 2 * step - 1):
                assert ranges.item_in(at, j, n) == (at + j < n)


@pytest.mark.parametrize("n", COUNTS)
def test_row_counts_and_tables(ranges, n):
    code = ranges.all_rows(n)
    assert code <= -2 and ranges.rows_of(code) == n
    for most in (512, 2048, 8192):
        want = 64
        while want < 2 * n and want < most:
            want *= 2
        assert ranges.table_entries(n, most) == want


def test_kernels_use_it():
    """The claims, chunk ends and row steps of the kernels go through the header."""
    with open(os.path.join(CSRC, "learn.cu")) as f:
        learn = f.read()
    with open(os.path.join(CSRC, "elim.cuh")) as f:
        elim = f.read()
    assert "* CHECK_CHUNK <" not in learn and "+ CHECK_CHUNK <" not in learn and "CHECK_CHUNK - 1) / CHECK" not in learn
    assert learn.count("chunk_exists(") == 3 and "chunk_count(" in learn
    assert "st.base +=" not in elim and "item_in(" in elim
