"""The kernels' decision table against the oracle's point test, on the CPU.

The table is generated at compile time (csrc/thin_common.cuh), so a host
compiler can print it.  Entry sum t_d 3^d holds, one bit per mode, whether a
point whose neighbour d is not lower (t = 0), lower by at most lambda (1) or
lower by more (2) may be lowered.  Every entry is compared in every mode with
the oracle on values of those states; with lambda = 0 no neighbour is in state 1."""
import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1603_09180_gb300", "csrc")


@pytest.fixture(scope="module")
def table(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("table")
    src = d / "t.cpp"
    src.write_text('#include <cstdio>\n#include "thin_common.cuh"\n'
                   "int main() { fwrite(thin::kDecisionTable.v, 1, thin::kDecisions, stdout); }\n")
    subprocess.run([cxx, "-std=c++17", "-fconstexpr-ops-limit=200000000", "-I", CSRC, str(src), "-o", str(d / "t")], check=True)
    return np.frombuffer(subprocess.run([str(d / "t")], check=True, capture_output=True).stdout, np.uint8)


@pytest.mark.parametrize("mode", range(8))
def test_every_state(table, mode):
    rule, op, adj = mode & 1, (mode >> 1) & 1, mode >> 2
    assert table.size == 3 ** 8
    for i in range(3 ** 8):
        t = [(i // 3 ** d) % 3 for d in range(8)]
        got = (int(table[i]) >> mode) & 1
        nb = [(100, 90, 89)[s] for s in t]  # lambda = 10: equal, lower by 10, lower by 11
        assert got == int(bool(oracle.lowerable(nb, 100, 10, rule, op, adj)[0])), (t, mode)
        if 1 not in t:
            nb = [(101, 0, 99)[s] for s in t]
            assert got == int(bool(oracle.lowerable(nb, 100, 0, rule, op, adj)[0])), (t, mode)
