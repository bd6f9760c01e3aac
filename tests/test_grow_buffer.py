"""Growth of a scratch buffer (csrc/grow.h) with a fake allocator, compiled for
the host: the old buffer is released only once the new one is there, and a
failed allocation leaves buffer and capacity as they were."""
import os
import subprocess

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

SOURCE = r"""
#include "grow.h"
#include <cstdio>
int main() {
    static int store[8];
    int next = 0, fail = 0, released = 0, allocated = 0;
    int *last = nullptr;
    auto alloc = [&](int **q, size_t) { if (fail) return 2; ++allocated; *q = store + next++; return 0; };
    auto release = [&](int *old) { ++released; last = old; return 0; };
    int *p = nullptr;
    size_t cap = 0;
    fail = 1;
    if (oct::grow_buffer(&p, &cap, 4, alloc, release) != 2 || p || cap || released) return 1;  // nothing yet
    fail = 0;
    if (oct::grow_buffer(&p, &cap, 4, alloc, release) || p != store || cap != 4 || released) return 2;
    if (oct::grow_buffer(&p, &cap, 9, alloc, release) || p != store + 1 || cap != 9 || last != store) return 3;
    fail = 1;
    if (oct::grow_buffer(&p, &cap, 20, alloc, release) != 2) return 4;
    if (p != store + 1 || cap != 9 || released != 1 || allocated != 2) return 5;  // the old one still serves
    return 0;
}
"""


def test_failed_growth_keeps_the_buffer(tmp_path):
    src, exe = tmp_path / "grow.cpp", tmp_path / "grow"
    src.write_text(SOURCE)
    csrc = os.path.join(ROOT, "paper_1705_01022_gb300", "csrc")
    subprocess.run(["g++", "-std=c++17", "-Wall", "-Werror", f"-I{csrc}", str(src), "-o", str(exe)], check=True)
    assert subprocess.run([str(exe)]).returncode == 0


def test_row_records_grow_through_it():
    """Every growth of the batch's stream-ordered scratch takes that form: no
    free stands before its allocation."""
    src = open(os.path.join(ROOT, "paper_1705_01022_gb300", "csrc", "batch.cu")).read()
    assert "cudaFreeAsync(b->d_rows" not in src and "cudaFreeAsync(*p" not in src
    assert "grow_async(&b->d_rows, &b->rows_cap" in src
