"""Host side of the fixed-point factors: e^{i ph} in units of 2^-62 against the
C library, over all phases a potential table can hold."""
import math
import os
import random
import shutil
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include <cinttypes>
#include <cstdio>
#include "fix64_host.h"
int main() {
    double ph;
    while (std::scanf("%la", &ph) == 1) {
        int64_t c, s;
        soft::fx_cis_host(soft::fx_turns_host(ph), &c, &s);
        std::printf("%" PRId64 " %" PRId64 "\n", c, s);
    }
}
"""


@pytest.fixture(scope="module")
def exe(tmp_path_factory):
    if not shutil.which("g++"):
        pytest.skip("no g++")
    d = tmp_path_factory.mktemp("fix64")
    (d / "cis.cpp").write_text(SRC)
    subprocess.run(["g++", "-O1", "-std=c++17", "-I", os.path.join(ROOT, "paper_1505_06707_gb300", "csrc"),
                    "-o", str(d / "cis"), str(d / "cis.cpp")], check=True)
    return str(d / "cis")


@pytest.mark.parametrize("lo,hi", [(-60, 0), (0, 30), (30, 50), (50, 64), (64, 1000)])
def test_phases(exe, lo, hi):
    """To half a unit of a double's cosine and the same again for the reduction."""
    rng = random.Random(lo)
    ph = [math.ldexp(rng.uniform(-1, 1), rng.randint(lo, hi)) for _ in range(2000)]
    ph += [s * math.ldexp(1.0, k) for k in (lo, hi) for s in (1, -1)]
    out = subprocess.run([exe], input="\n".join(v.hex() for v in ph), capture_output=True, text=True, check=True)
    for v, line in zip(ph, out.stdout.splitlines(), strict=True):
        c, s = (int(w) * 2.0 ** -62 for w in line.split())
        assert abs(c - math.cos(v)) < 4.5e-16 and abs(s - math.sin(v)) < 4.5e-16, v
        assert abs(c * c + s * s - 1) < 1e-15
