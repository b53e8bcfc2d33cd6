"""The choice of the memory pool for a call's scratch, on the CPU (csrc/thin_pool.h is host logic).

A program that goes back and forth between the device's primary context and another one makes one pool
in all; the primary context created anew makes another; a failed creation is tried again by the next call."""
import os
import shutil
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1603_09180_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "thin_pool.h"
int main()
{
    thin::PoolSlot<int> slot;
    int made = 0;
    bool fail = false;
    unsigned long long primary = 7;
    auto ask = [&](unsigned long long ctx) {
        return thin::pool_for(slot, ctx, [&] { return ctx == primary; }, [&](int *p) { if (fail) return false; *p = ++made; return true; });
    };
    if (ask(0) != 0 || made != 0) return 1;                        // no context: no pool
    fail = true;
    if (ask(7) != 0 || slot.pool != 0) return 2;
    fail = false;
    if (ask(7) != 1 || ask(7) != 1) return 3;                      // made once, kept
    for (int k = 0; k < 100; ++k)
        if (ask(9 + k % 2) != 0 || ask(7) != 1) return 4;          // other contexts in between: the default pool
    if (made != 1) return 5;
    primary = 12;                                                  // the primary context has been created anew
    if (ask(12) != 2 || ask(12) != 2 || ask(7) != 0 || made != 2) return 6;
    return 0;
}
"""


def test_pool_for(tmp_path):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "p.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-I", CSRC, str(tmp_path / "p.cpp"), "-o", str(tmp_path / "p")], check=True)
    assert subprocess.run([str(tmp_path / "p")]).returncode == 0
