"""Working memory made by its first user (csrc/ready.h), on the CPU with calls
that fail: what was allocated but not filled is filled before it is used."""
import os
import subprocess

from tests.conftest import ROOT

MAIN = r"""
#include "ready.h"
#include <cassert>
int main()
{
    msd::WorkArea w;
    unsigned char mem[1] = {0};
    int allocs = 0, fills = 0, alloc_error = 2, fill_error = 0;
    auto call = [&] {
        return msd::make_ready(
            w, [&](unsigned char *&p) { allocs++; if (!alloc_error) p = mem; return alloc_error; },
            [&](unsigned char *p) { assert(p == mem); fills++; if (!fill_error) *p = 7; return fill_error; });
    };
    assert(call() == 2 && allocs == 1 && fills == 0 && !w.ready);
    alloc_error = 0;
    fill_error = 5;
    assert(call() == 5 && allocs == 2 && fills == 1 && !w.ready);
    fill_error = 0;
    assert(call() == 0 && allocs == 2 && fills == 2 && w.ready && mem[0] == 7);
    assert(call() == 0 && allocs == 2 && fills == 2);
    return 0;
}
"""


def test_filled_before_use(tmp_path):
    src, exe = tmp_path / "t.cpp", tmp_path / "t"
    src.write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-I", os.path.join(ROOT, "paper_2303_07819_gb300", "csrc"), str(src), "-o", str(exe)],
                   check=True)
    subprocess.run([str(exe)], check=True)
