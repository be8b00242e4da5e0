"""The geometry of the search grid (csrc/grid_spec.cuh), compiled for the host:
for boxes from a point to the largest accepted coordinates, flat and thin ones
and ones of subnormal extent, and from 1 to 2^30 points, the cells fit the
arrays that hold their counts, the counts index within 32 bits, and the cell
edge and its reciprocal are finite."""
import os
import subprocess

import numpy as np
import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_1902_01061_gb300", "csrc")

MAIN = r"""
#include <cstdio>
#include "grid_spec.cuh"
int main() {
  float e[3];
  int n;
  while (std::scanf("%a %a %a %d", &e[0], &e[1], &e[2], &n) == 4) {
    const float lo[3] = {0.f, 0.f, 0.f};
    scgr::GridSpec g;
    scgr::make_grid_spec(lo, e, n, &g);
    std::printf("%d %d %d %d %a %a %zu\n", g.g[0], g.g[1], g.g[2], g.ncell, g.h, g.inv_h, scgr::grid_start_entries(n));
  }
}
"""


@pytest.fixture(scope="module")
def spec(tmp_path_factory):
    d = tmp_path_factory.mktemp("grid_spec")
    (d / "main.cpp").write_text(MAIN)
    subprocess.run(["g++", "-std=c++17", "-O1", "-ffp-contract=off", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")], check=True)

    def run(boxes):
        text = "\n".join(" ".join([*(float(v).hex() for v in b[:3]), str(b[3])]) for b in boxes)
        out = subprocess.run([str(d / "main")], input=text, capture_output=True, text=True, check=True).stdout
        rows = [r.split() for r in out.splitlines()]
        assert len(rows) == len(boxes)
        return [([int(v) for v in r[:4]], float.fromhex(r[4]), float.fromhex(r[5]), int(r[6])) for r in rows]

    return run


def boxes():
    rng = np.random.default_rng(5)
    out = []
    for e in (0.0, 1e-45, 1e-39, 2.9e-39, 3e-39, 1e-38, 1e-31, 1e-30, 1e-12, 1.0, 2e18):
        for f in ((1, 0, 0), (1, 1e-3, 1e-3), (1, 1, 0), (1, 1, 1)):
            for n in (1, 3, 500, 20000, 10**6, 10**8, 2**29, 2**29 + 1, 2**30):
                out.append((*(np.float32(e * v) for v in f), n))
    for _ in range(4000):
        e = 10.0 ** rng.uniform(-44, 18) * 10.0 ** rng.uniform(-6, 0, 3)
        out.append((*np.float32(e), int(round(2.0 ** rng.uniform(0, 30)))))
    return out


def test_cells_fit_their_arrays(spec):
    for box, (g, h, inv_h, entries) in zip(bs := boxes(), spec(bs)):
        cells = g[0] * g[1] * g[2]
        assert min(g[:3]) >= 1 and max(g[:3]) <= 2**16 + 1, (box, g)
        assert cells == g[3], (box, g)
        assert cells + 1 <= entries, (box, g, entries)
        # the count scan walks blocks of 4,096 entries with 32-bit positions
        assert entries + 4096 < 2**31, (box, entries)
        assert 0.0 < h < np.inf and 0.0 < inv_h < np.inf, (box, h, inv_h)


def test_every_point_of_the_box_has_a_cell(spec):
    """The far corner's unclamped cell is the last one at most (the kernels
    clamp; a box that its cells did not cover would be searched wrongly)."""
    for box, (g, h, inv_h, _) in zip(bs := boxes(), spec(bs)):
        for a in range(3):
            assert np.floor(np.float32(box[a]) * np.float32(inv_h)) <= g[a], (box, g)
