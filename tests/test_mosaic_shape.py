"""The mosaic engine's choice of a tile shape against what its kernel can exchange, on the CPU.

The choice is host arithmetic (csrc/thin_layout.h), so a host compiler can run it: every shape it
returns, for one to 16 images of either type on GPUs of 152 and of 148 SMs, lies within the turns in
which a block moves its rims' side columns (2 es 16-byte vectors a row, a thread to a vector) and within
the other bounds of the kernel, which a launch checks; shapes just past a bound are refused."""
import math
import os
import random
import shutil
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1603_09180_gb300", "csrc")
LIMIT = 115456  # shared memory of a block, two to an SM of 228 KiB

MAIN = r"""
#include <cstdio>
#include <vector>
#include "thin_layout.h"
struct Job { int w, h; };
int main()
{
    int n, es, sms, limit;
    while (scanf("%d %d %d %d", &n, &es, &sms, &limit) == 4) {
        std::vector<Job> jobs(n);
        for (Job &j : jobs)
            if (scanf("%d %d", &j.w, &j.h) != 2) return 1;
        thin::MosaicShape s = {0, 0, 0};
        const bool ok = thin::mosaic_search(jobs.data(), n, es == 2, sms, limit, &s);
        printf("%d %d %d %d %d %d\n", int(ok), s.tw, s.th, s.halo, thin::mosaic_side_turns(es) * thin::kThreads,
               int(thin::mosaic_shape_fits(es, s)));
    }
}
"""


@pytest.fixture(scope="module")
def search(tmp_path_factory):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    d = tmp_path_factory.mktemp("shape")
    (d / "s.cpp").write_text(MAIN)
    subprocess.run([cxx, "-std=c++17", "-O1", "-fconstexpr-ops-limit=200000000", "-I", CSRC, str(d / "s.cpp"), "-o", str(d / "s")],
                   check=True)

    def run(calls):
        text = "\n".join("%d %d %d %d %s" % (len(sizes), es, sms, LIMIT, " ".join("%d %d" % s for s in sizes))
                         for sizes, es, sms in calls)
        out = subprocess.run([str(d / "s")], input=text, check=True, capture_output=True, text=True).stdout
        return np.array([[int(v) for v in line.split()] for line in out.splitlines()])

    return run


def calls(es, sms):
    rng = random.Random(10 * sms + es)
    side = lambda hi: int(round(math.exp(rng.uniform(math.log(3), math.log(hi)))))  # noqa: E731
    out = [([(s, s)], es, sms) for s in range(3, 4200, 7)]
    out += [([(side(20000), side(20000))], es, sms) for _ in range(4000)]
    out += [([(s, s)] * n, es, sms) for n in (2, 4, 16) for s in range(16, 2200, 16)]
    return out + [([(side(2000), side(2000)) for _ in range(rng.randint(2, 16))], es, sms) for _ in range(1000)]


@pytest.mark.parametrize("es", [1, 2])
@pytest.mark.parametrize("sms", [148, 152])
def test_side_columns_of_every_shape_are_exchanged(search, es, sms):
    got = search(calls(es, sms))
    tw, th, halo, vectors, fits = got[got[:, 0] == 1][:, 1:].T
    assert len(tw) > 3000 and th.max() > 192
    assert (2 * es * th <= vectors).all()
    assert fits.all()


@pytest.mark.parametrize("es,tw,th,halo,ok", [
    (1, 32, 16, 15, 1), (2, 32, 16, 15, 1), (1, 224, 304, 15, 1), (2, 224, 304, 15, 1), (1, 16, 16, 1, 1),
    (1, 224, 306, 15, 0), (2, 32, 312, 15, 0), (1, 240, 64, 15, 0), (2, 240, 64, 15, 0), (1, 40, 64, 15, 0),
    (1, 32, 15, 3, 0), (1, 32, 14, 15, 0), (1, 0, 64, 15, 0), (1, 32, 64, 16, 0), (1, 32, 64, 0, 0)])
def test_bounds(tmp_path, es, tw, th, halo, ok):
    cxx = shutil.which("g++")
    if cxx is None:
        pytest.skip("no host compiler")
    (tmp_path / "b.cpp").write_text('#include "thin_layout.h"\n'
                                    "static_assert(thin::mosaic_shape_fits(%d, thin::MosaicShape{%d, %d, %d}) == %s, \"\");\n"
                                    % (es, tw, th, halo, "true" if ok else "false"))
    subprocess.run([cxx, "-std=c++17", "-fsyntax-only", "-fconstexpr-ops-limit=200000000", "-I", CSRC, str(tmp_path / "b.cpp")],
                   check=True)
