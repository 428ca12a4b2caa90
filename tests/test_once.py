"""Constants that a handle makes once (csrc/xc_once.h), compiled for the host with a buffer and a launch that
can fail: after an error the next call starts again instead of taking an unfilled buffer for made."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1801_09803_gb300", "csrc")
PROGRAM = r"""
#include <assert.h>
#include <stdlib.h>
#include "xc_once.h"
enum Err { OK = 0, NOMEM = 2, LAUNCH = 9 };
struct Buf {
    void *p = nullptr;
    bool full = false;
    Err ensure(size_t n) { if (full) return NOMEM; p = malloc(n); return OK; }
    void release() { free(p); p = nullptr; }
};
int main() {
    Buf b;
    int made = 0;
    auto ok = [&] { ++made; return OK; };
    auto bad = [&] { ++made; return LAUNCH; };
    b.full = true;
    assert(xc::make_once(b, 64, ok) == NOMEM && !b.p && made == 0);
    b.full = false;
    assert(xc::make_once(b, 64, bad) == LAUNCH && !b.p && made == 1);
    assert(xc::make_once(b, 64, ok) == OK && b.p && made == 2);
    assert(xc::make_once(b, 64, bad) == OK && b.p && made == 2);   // made: not made again
    b.release();
}
"""


def test_nothing_half_made_is_kept(tmp_path):
    cxx = shutil.which("g++")
    if not cxx:
        pytest.skip("no host compiler")
    (tmp_path / "t.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(tmp_path / "t.cpp"), "-o", str(tmp_path / "t")], check=True)
    subprocess.run([str(tmp_path / "t")], check=True)


def test_every_matrix_of_a_handle_goes_through_it():
    for f in ("xc_tree.cu", "xc_tree64.cu"):
        assert "make_once(" in open(os.path.join(CSRC, f)).read(), f
