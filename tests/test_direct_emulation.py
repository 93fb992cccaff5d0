"""The direct solve of the pressure correction (k_dir_xy forward, k_dir_z,
k_dir_xy inverse) run on the host: the kernels' source and that of the plan,
compiled as C++ with every CTA as host threads (tests/emu/) under
AddressSanitizer and UBSan, against the 7-point Neumann / periodic Laplacian:
the residual r - L e of one application is the rounding of e times the
conditioning of L.  Odd and even extents, extents below one tile, columns of
one and several chunks (the last one short), several column blocks per plane,
walls, slip and periodic axes.  An inactive state stays untouched.  No GPU
needed."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

from test_mg_block_emulation import CSRC, EMU, _extract
from test_refine_emulation import _source

BC = {"wall": 0, "periodic": 1, "slip": 2}


def _direct_source() -> str:
    cl = open(os.path.join(CSRC, "ns_mg_cluster.cuh")).read()
    a = cl.index("// Four consecutive x cells")
    b = cl.index("template <typename T> __device__ __forceinline__ void q2_ld")
    src = open(os.path.join(CSRC, "ns_direct.cuh")).read()
    body = src[src.index("constexpr int DIR_MAX_THREADS"):src.rindex("}  // namespace nsk")]
    shared = "extern __shared__ __align__(16) unsigned char smem_raw[];"
    assert shared in body
    return ("struct float4 {\n    float x, y, z, w;\n};\n" + cl[a:b] + "\n\n" +
            body.replace(shared, "unsigned char* smem_raw = emu_smem;"))


@pytest.fixture(scope="module")
def emulator(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("direct_emu")
    cpp = d / "direct_emu.cpp"
    cpp.write_text('#include "block_emu.h"\n\n' + _source() + "\n\n" + _direct_source() + "\n\n" +
                   open(os.path.join(EMU, "direct_emu_main.cpp")).read())
    exe = d / "direct_emu"
    cmd = [gxx, "-std=c++20", "-O1", "-g", "-fsanitize=address,undefined",
           "-fno-sanitize-recover=undefined", "-fno-omit-frame-pointer", "-pthread",
           "-I", EMU, str(cpp), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0 and "barrier" in r.stderr and "No such file" in r.stderr:
        pytest.skip("the host compiler has no <barrier>")
    assert r.returncode == 0, r.stderr[-3000:]
    return str(exe), d


def _lap(p, h, bc):
    out = np.zeros_like(p)
    for d in range(3):
        ax = 2 - d
        if bc[d] == "periodic":
            out += (np.roll(p, 1, ax) + np.roll(p, -1, ax) - 2 * p) / h[d] ** 2
        else:
            df = np.diff(p, axis=ax) / h[d] ** 2
            z = np.zeros_like(np.take(p, [0], ax))
            out += np.diff(np.concatenate([z, df, z], ax), axis=ax)
    return out


# (cells, boundaries, box, planes of a call: below 152 two column blocks)
CASES = [
    ((16, 16, 16), ("wall",) * 3, (1.0, 1.0, 1.0), 16),
    ((2, 2, 2), ("wall",) * 3, (1.0, 1.0, 1.0), 2),
    ((2, 2, 2), ("periodic",) * 3, (1.0, 1.0, 1.0), 500),
    ((19, 13, 11), ("wall",) * 3, (1.0, 1.3, 0.8), 500),
    ((45, 7, 9), ("wall", "slip", "wall"), (2.0, 1.0, 1.0), 9),
    ((12, 37, 17), ("periodic", "wall", "periodic"), (1.0, 3.0, 1.0), 500),
    ((9, 10, 3), ("periodic", "periodic", "wall"), (1.0, 1.0, 0.1), 500),
    ((64, 34, 8), ("wall",) * 3, (1.0, 1.0, 1.0), 500),
    ((6, 5, 130), ("wall", "periodic", "wall"), (1.0, 1.0, 20.0), 500),   # long chunks
    ((5, 6, 133), ("wall", "wall", "periodic"), (1.0, 1.0, 20.0), 500),
    ((72, 128, 2), ("slip", "wall", "wall"), (1.0, 2.0, 0.1), 500),       # FP64: column blocks
]


@pytest.mark.parametrize("prec", ["f", "d"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_direct_solve_inverts_the_laplacian(emulator, case, prec):
    exe, d = emulator
    n, bc, box, planes = CASES[case]
    t = np.float32 if prec == "f" else np.float64
    h = [box[a] / n[a] for a in range(3)]
    rng = np.random.default_rng(case)
    r = rng.normal(size=(2,) + n[::-1])
    r -= r.mean(axis=(1, 2, 3), keepdims=True)
    r = r.astype(t)
    fin, fout = d / "r.bin", d / "e.bin"
    r.tofile(fin)
    args = [exe, prec, *map(str, n), *(str(BC[x]) for x in bc), *map(repr, box), str(planes),
            str(fin), str(fout)]
    out = subprocess.run(args, capture_output=True, text=True, timeout=600)
    assert out.returncode == 0, (out.returncode, out.stderr[-3000:])
    e = np.fromfile(fout, dtype=t).reshape(r.shape).astype(np.float64)
    assert not e[1].any()
    res = r[0].astype(np.float64) - _lap(e[0], h, bc)
    res -= res.mean()
    # rounding of e, at most a few units in the last place of its largest mode,
    # seen through L: eps times the condition number of L (about 0.1 of that
    # is measured)
    low = min(4 * np.sin((np.pi if bc[a] == "periodic" else np.pi / 2) / n[a]) ** 2 / h[a] ** 2
              for a in range(3))
    cond = sum(4 / x ** 2 for x in h) / low
    bound = max(np.finfo(t).eps * cond, 8 * np.finfo(t).eps)
    assert np.linalg.norm(res) <= bound * np.linalg.norm(r[0]), (np.linalg.norm(res) /
                                                                 np.linalg.norm(r[0]), bound)
