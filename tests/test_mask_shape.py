"""csrc/ns_mask.h (face codes, solid cells, solid surface and separate fluid
regions of a mask) against plain numpy: random masks of every density, sealed rooms, rooms
joined only through a periodic axis, walls and wraps, extents down to 2.  No GPU
needed."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

from test_masked_mg_emulation import FC_FLUID, _codes

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
CSRC = os.path.join(ROOT, "paper_1705_06149_gb300", "csrc")

MAIN = """#include <cstdio>
#include <cstdlib>
#include "ns_mask.h"
int main(int, char** argv) {
    int n[3];
    bool per[3];
    for (int a = 0; a < 3; ++a) n[a] = atoi(argv[1 + a]), per[a] = atoi(argv[4 + a]) != 0;
    std::vector<uint8_t> s((size_t)n[0] * n[1] * n[2]);
    FILE* f = fopen(argv[7], "rb");
    if (!f || fread(s.data(), 1, s.size(), f) != s.size()) return 2;
    const MaskShape m = mask_shape(n, per, s.data());
    printf("%lld %lld %lld\\n", m.solid, m.faces, m.rooms);
    const std::vector<uint8_t> c = mask_face_codes(n, per, s.data(), 64);
    f = fopen(argv[8], "wb");
    fwrite(c.data(), 1, c.size(), f);
    fclose(f);
    return 0;
}
"""


@pytest.fixture(scope="module")
def driver(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("mask")
    (d / "main.cpp").write_text(MAIN)
    r = subprocess.run([gxx, "-std=c++17", "-O1", "-Wall", "-Werror", "-fsanitize=address,undefined",
                        "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr[-2000:]
    return str(d / "main"), d


def _shape(solid, periodic):
    """The same by label propagation: every fluid cell takes the smallest label
    around it until none changes."""
    fluid = solid == 0
    label = np.where(fluid, np.arange(1, solid.size + 1).reshape(solid.shape), 0)
    pairs = []
    for a in range(3):
        ax, n = 2 - a, solid.shape[2 - a]
        lo, hi = list(range(n - 1)), list(range(1, n))
        if periodic[a]:
            lo.append(n - 1)
            hi.append(0)
        pairs.append((ax, lo, hi))
    faces = sum(int((np.take(fluid, lo, ax) != np.take(fluid, hi, ax)).sum()) for ax, lo, hi in pairs)
    while True:
        old = label.copy()
        for ax, lo, hi in pairs:
            v = np.moveaxis(label, ax, 0)
            for i, j in list(zip(lo, hi)) + list(zip(lo, hi))[::-1]:
                both = (v[i] > 0) & (v[j] > 0)
                m = np.minimum(v[i], v[j])
                v[i] = np.where(both, m, v[i])
                v[j] = np.where(both, m, v[j])
        if (label == old).all():
            break
    _, count = np.unique(label[label > 0], return_counts=True)
    return int((~fluid).sum()), faces, int((count > 1).sum())


def _masks():
    rng = np.random.default_rng(0)
    for dims in ((9, 7, 8), (2, 5, 3), (13, 2, 2)):
        for share in (0.0, 0.1, 0.3, 0.5, 0.7, 1.0):
            yield (rng.random(dims[::-1]) < share).astype(np.uint8)
    room = np.zeros((9, 9, 12), np.uint8)
    room[2:7, 2:7, 2:7] = 1
    room[3:6, 3:6, 3:6] = 0
    yield room
    room[4, 4, 6] = 0  # a door
    yield room
    cell = np.zeros((6, 6, 6), np.uint8)
    cell[2:5, 2:5, 2:5] = 1
    cell[3, 3, 3] = 0
    yield cell
    for ax in range(3):  # two halves, one with a periodic axis across them
        half = np.zeros((6, 8, 10), np.uint8)
        np.moveaxis(half, ax, 0)[3] = 1
        yield half


@pytest.mark.parametrize("periodic", [(0, 0, 0), (1, 0, 0), (0, 1, 0), (0, 0, 1), (1, 1, 1)])
def test_mask_shape_matches_numpy(driver, periodic):
    exe, d = driver
    for solid in _masks():
        solid.tofile(d / "s.bin")
        r = subprocess.run([exe, *map(str, solid.shape[::-1]), *map(str, periodic),
                            str(d / "s.bin"), str(d / "c.bin")], capture_output=True, text=True)
        assert r.returncode == 0, r.stderr[-2000:]
        assert tuple(map(int, r.stdout.split())) == _shape(solid, periodic), (solid.shape, periodic)
        code = np.fromfile(d / "c.bin", dtype=np.uint8).reshape(solid.shape)
        assert FC_FLUID == 64
        assert (code == _codes(solid, ["periodic" if p else "wall" for p in periodic])).all()
