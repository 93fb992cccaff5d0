"""The direct solve of the pressure correction (k_dir_xy forward, k_dir_z,
k_dir_xy inverse) run on the host: the kernels' source and that of the plan,
compiled as C++ with every CTA as host threads (tests/emu/) under
AddressSanitizer and UBSan, against the 7-point Neumann / periodic Laplacian:
the residual r - L e of one application is the rounding of e times the
conditioning of L; and the FP32 step kernels around it (k_dir_start,
k_dir_refine, k_dir_correct) against FP64.  Odd and even extents, extents below one tile, columns of
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


def _build(tmp_path_factory, name):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp(name)
    cpp = d / f"{name}.cpp"
    cpp.write_text('#include "block_emu.h"\n\n' + _source() + "\n\n" + _direct_source() + "\n\n" +
                   open(os.path.join(EMU, f"{name}_main.cpp")).read())
    exe = d / name
    cmd = [gxx, "-std=c++20", "-O1", "-g", "-fsanitize=address,undefined",
           "-fno-sanitize-recover=undefined", "-fno-omit-frame-pointer", "-pthread",
           "-I", EMU, str(cpp), "-o", str(exe)]
    r = subprocess.run(cmd, capture_output=True, text=True)
    if r.returncode != 0 and "barrier" in r.stderr and "No such file" in r.stderr:
        pytest.skip("the host compiler has no <barrier>")
    assert r.returncode == 0, r.stderr[-3000:]
    return str(exe), d


@pytest.fixture(scope="module")
def emulator(tmp_path_factory):
    return _build(tmp_path_factory, "direct_emu")


@pytest.fixture(scope="module")
def step_emulator(tmp_path_factory):
    return _build(tmp_path_factory, "direct_step_emu")


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


# (cells, boundaries, box, planes of a call: below 152 two column blocks, 0: the
# transforms one axis at a time)
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
    ((19, 33, 9), ("wall", "slip", "wall"), (1.0, 1.5, 0.5), 0),
    ((70, 10, 5), ("periodic", "wall", "wall"), (3.0, 0.5, 0.3), 0),      # ragged line blocks
    ((4, 2, 6), ("wall", "periodic", "periodic"), (1.0, 1.0, 1.0), 0),
]


@pytest.mark.parametrize("prec", ["f", "d", "m"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_direct_solve_inverts_the_laplacian(emulator, case, prec):
    exe, d = emulator
    n, bc, box, planes = CASES[case]
    t = np.float64 if prec == "d" else np.float32
    h = [box[a] / n[a] for a in range(3)]
    rng = np.random.default_rng(case)
    r = rng.normal(size=(2,) + n[::-1])
    r -= r.mean(axis=(1, 2, 3), keepdims=True)
    r = r.astype(np.float32 if prec == "f" else np.float64)
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


# (cells, boundaries, applications before the correction, tile_z)
STEP_CASES = [
    ((12, 12, 12), ("wall",) * 3, 0, 0),
    ((40, 10, 9), ("wall",) * 3, 1, 8),          # two x tiles, a short last batch
    ((13, 9, 5), ("periodic", "wall", "slip"), 2, 3),
    ((8, 16, 10), ("wall", "periodic", "periodic"), 3, 0),   # the oldest is folded
    ((2, 2, 2), ("wall",) * 3, 5, 0),
    ((70, 3, 4), ("slip", "periodic", "wall"), 4, 2),
]


@pytest.mark.parametrize("case", range(len(STEP_CASES)))
def test_step_kernels_match_fp64(step_emulator, case):
    exe, d = step_emulator
    n, bc, steps, tile_z = STEP_CASES[case]
    lbox, dt = 1.3, 2e-3
    h = [lbox / m for m in n]
    rng = np.random.default_rng(40 + case)
    shp = [tuple(n[a] + (1 if a == c and bc[a] != "periodic" else 0) for a in (2, 1, 0))
           for c in range(3)]
    cshape = n[::-1]

    def faces(scale):
        out = []
        for c in range(3):
            v = rng.normal(size=shp[c]) * scale
            if bc[c] != "periodic":
                np.moveaxis(v, 2 - c, 0)[[0, -1]] = 0.0
            out.append(v.astype(np.float32))
        return out

    inc, vel = faces(1e-2), faces(1.0)
    p = 100.0 + rng.normal(size=cshape)
    ring = (1e-2 * rng.normal(size=(4,) + cshape)).astype(np.float32)
    fin, fout = d / "in.bin", d / "out.bin"
    with open(fin, "wb") as f:
        p.tofile(f)
        for a in inc + vel + [ring]:
            a.tofile(f)
    args = [exe, *map(str, n), *(str(BC[x]) for x in bc), repr(lbox), repr(dt), str(steps),
            str(tile_z), str(fin), str(fout)]
    out = subprocess.run(args, capture_output=True, text=True, timeout=300)
    assert out.returncode == 0, (out.returncode, out.stderr[-3000:])
    raw = open(fout, "rb").read()
    off = 0

    def take(shape, dtype=np.float32):
        nonlocal off
        a = np.frombuffer(raw, dtype=dtype, count=int(np.prod(shape)), offset=off).reshape(shape)
        off += a.nbytes
        return a.astype(np.float64)

    def pair():
        return take(cshape) + take(cshape)

    def div(f):
        o = 0.0
        for a in range(3):
            x = f[a].astype(np.float64)
            hi = np.roll(x, -1, 2 - a) if bc[a] == "periodic" else np.take(
                x, range(1, n[a] + 1), 2 - a)
            o = o + (hi - np.take(x, range(n[a]), 2 - a)) / h[a]
        return o

    norm = np.linalg.norm
    # the increment's divergence is taken in FP32 (unit roundoff 6e-8 of its
    # terms); everything after it in float-float (2^-45 of the magnitudes)
    b0, b1 = div(inc) / dt, div([a.astype(np.float64) + v for a, v in zip(inc, vel)]) / dt
    lp = _lap(p, h, bc)
    fp32 = 2e-7 * sum(norm(a) / x for a, x in zip(inc, h)) * 2 / dt
    top = 4 * sum(1 / x ** 2 for x in h)
    ff = 2.0 ** -45 * (top * norm(p) + norm(b1))
    r0, r1 = pair(), pair()
    assert norm(r0 - (b0 - lp)) <= fp32 + ff
    assert norm(r1 - (b1 - lp)) <= fp32 + ff
    r2, base = pair(), pair()
    e = ring[steps % 4].astype(np.float64)
    assert norm(r2 - (r1 - r1.mean() - _lap(e, h, bc))) <= 2.0 ** -40 * (norm(r1) + top * norm(e))
    want = p + (ring[(steps + 1) % 4] if steps >= 3 else 0.0)
    assert norm(base - want) <= 2.0 ** -45 * norm(p)
    u = [take(s) for s in shp]
    w, q = pair(), pair()
    pout = take(cshape, np.float64)
    num = take((6,), np.float64)
    made = steps + 1
    full = base + sum(ring[(made - m) % 4].astype(np.float64) for m in range(1, min(made, 3) + 1))
    # the mean the library keeps: of the warm start plus that of every
    # application seen by k_dir_refine (here one)
    mean = p.mean() + e.mean()
    assert norm(q - (full - mean)) <= 1e-6 * norm(full - mean) and norm(pout - q) <= 1e-12 * norm(p)
    assert norm(w - (2 * q - p)) <= 2.0 ** -40 * norm(p)
    for c in range(3):
        ax = 2 - c
        if bc[c] == "periodic":
            g = (full - np.roll(full, 1, ax)) / h[c]
        else:
            g = np.zeros(shp[c])
            np.moveaxis(g, ax, 0)[1:-1] = np.moveaxis(np.diff(full, axis=ax) / h[c], ax, 0)
        want = vel[c].astype(np.float64) + (inc[c] - dt * g)
        assert norm(u[c] - want) <= 4e-7 * (norm(want) + norm(dt * g))
    bb = norm(b1 - b1.mean()) ** 2
    assert abs(num[0] - bb) <= 1e-5 * bb + 1e-5 * fp32 ** 2
    rr = norm(r1 - r1.mean()) ** 2
    assert abs(num[1] - rr) <= 1e-5 * rr
    assert abs(num[2] - norm(r2 - r2.mean()) ** 2) <= 1e-5 * num[2]
    assert abs(num[3] - (p.sum() + e.sum())) <= 1e-9 * abs(p).sum()
    assert num[4] == made
