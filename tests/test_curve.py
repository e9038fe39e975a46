"""The sort keys' Hilbert curve (csrc/sk_curve.h), compiled with the host compiler:
every cell of the 8 x 8 x 8 corner grid at each scale gets its own key, keys that
follow one another belong to cells that share a face, and the lowest and highest
cells stay below 2^30 (the key of a source without weight is the largest)."""

import os
import shutil
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_2310_13908_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include "sk_curve.h"
int main() {
  unsigned x, y, z;
  while (std::scanf("%u %u %u", &x, &y, &z) == 3) std::printf("%u\n", sk::hilbert_key(x, y, z));
}
"""


@pytest.fixture(scope="module")
def keys(tmp_path_factory):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("needs a host C++ compiler")
    d = tmp_path_factory.mktemp("curve")
    (d / "program.cpp").write_text(PROGRAM)
    subprocess.run([cxx, "-std=c++17", "-O1", "-I", CSRC, str(d / "program.cpp"), "-o",
                    str(d / "program")], check=True)

    def run(q):
        text = "".join(f"{a} {b} {c}\n" for a, b, c in q)
        out = subprocess.run([str(d / "program")], input=text, capture_output=True, text=True,
                             check=True).stdout.split()
        return np.array([int(v) for v in out], dtype=np.int64)

    return run


@pytest.mark.parametrize("shift", [0, 3, 7])
@pytest.mark.parametrize("corner", [(0, 0, 0), (1016, 1016, 1016), (512, 0, 504), (8, 1000, 128)])
def test_curve_visits_neighbouring_cells(keys, shift, corner):
    size = 8 << shift
    if any(c % size for c in corner):
        corner = (0, 0, 0)
    cells = np.stack(np.meshgrid(*[np.arange(8)] * 3, indexing="ij"), -1).reshape(-1, 3)
    q = cells * (1 << shift) + np.array(corner)
    k = keys(q)
    assert k.min() >= 0 and k.max() < 1 << 30
    place = k >> (3 * shift)               # the cell's place at this scale
    order = np.argsort(place)
    assert np.array_equal(place[order], place.min() + np.arange(512))
    assert np.all(np.abs(np.diff(cells[order], axis=0)).sum(1) == 1)
