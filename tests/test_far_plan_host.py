"""The passes of the far-field sum over its directions (csrc/far_plan.h), compiled on the host: the
scratch of a pass, tables included, stays within 256 MB above the waves' own tables and partial
sums of 64 directions, whatever the number of directions."""

import itertools
import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(HERE, "..", "paper_1408_4495_gb300", "csrc")

PROG = r"""
#include <cstdio>
#include "far_plan.h"
int main() {
  int d, n, r, k;
  while (std::scanf("%d %d %d %d", &d, &n, &r, &k) == 4)
    std::printf("%d %zu\n", ls::far_chunk(d, n, r, k), ls::far_scratch_elems(d, n, r, k));
}
"""


@pytest.fixture(scope="module")
def plans(tmp_path_factory):
    cxx = shutil.which(os.environ.get("CXX", "g++"))
    if cxx is None:
        pytest.skip("no C++ compiler")
    tmp = tmp_path_factory.mktemp("far")
    src, exe = tmp / "p.cpp", tmp / "p"
    src.write_text(PROG)
    subprocess.run([cxx, "-std=c++17", "-O2", "-I", CSRC, str(src), "-o", str(exe)], check=True)
    cases = [(d, n, r, k) for d, ns in ((2, (16, 32, 48, 128, 512, 2048)), (3, (8, 24, 64, 128)))
             for n, r, k in itertools.product(ns, (1, 3, 32, 512), (1, 64, 9000, 100000, 1048577, 2147483647))]
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True,
                         input="\n".join(" ".join(map(str, c)) for c in cases)).stdout
    return [c + tuple(int(v) for v in line.split()) for c, line in zip(cases, out.splitlines(), strict=True)]


def test_scratch_is_bounded(plans):
    for d, n, r, k, chunk, elems in plans:
        lines = n ** (d - 1)
        tiles = -(-lines // 16)
        assert 1 <= chunk <= k
        # inc, outer, cs and the partial sums of a full pass, 16 bytes each
        need = r * d * n + chunk * ((d - 1) * n + n // 2 + r * tiles)
        assert elems >= need
        floor = r * d * n + 64 * ((d - 1) * n + n // 2 + r * tiles)
        assert elems * 16 <= max(floor * 16, (256 << 20) + r * d * n * 16)


def test_tiles_fit_the_grid(plans):
    assert max(-(-chunk // 16) for *_, chunk, _ in plans) <= 65535  # k_far_sum's gridDim.z at 16 directions a CTA
