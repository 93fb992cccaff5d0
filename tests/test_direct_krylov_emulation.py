"""The kernels that apply a direct solve's result, run on the host like
test_direct_emulation.py runs the transforms: k_dir_update (x += e, r -= L e +
mean(r) of an FP64 grid; FP32 corrections come in the power-of-two scale of the
residual, whatever its size) against FP64, and the conjugate gradients around
the solid cells (k_cg_dot, k_cg_lap, k_cg_update, the direction kept across an
outer correction) against the same recurrences in numpy, on ragged tiles,
periodic and slip axes, two x tiles.  No GPU needed."""
from __future__ import annotations

import subprocess

import numpy as np
import pytest

from test_direct_emulation import BC, _build, _lap
from test_masked_mg_emulation import _codes, _lap_masked

DIMS = [((20, 9, 11), ("wall",) * 3), ((36, 5, 8), ("periodic", "wall", "slip")),
        ((6, 12, 17), ("wall", "periodic", "periodic"))]


@pytest.fixture(scope="module")
def emulator(tmp_path_factory):
    return _build(tmp_path_factory, "direct_krylov_emu")


def _run(exe, *args):
    r = subprocess.run([exe, *map(str, args)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-3000:])


@pytest.mark.parametrize("power", [0, -20, -30, -400, 300])
@pytest.mark.parametrize("prec", ["f", "d"])
@pytest.mark.parametrize("case", range(len(DIMS)))
def test_update_applies_a_correction_of_any_size(emulator, case, prec, power):
    exe, d = emulator
    n, bc = DIMS[case]
    h = [1.0 / m for m in n]
    rng = np.random.default_rng(case)
    size = 2.0 ** power
    r = rng.normal(size=n[::-1])
    r -= r.mean()
    r *= size
    x = 1e-2 * size * rng.normal(size=r.shape)
    e = (1e-2 * rng.normal(size=r.shape)).astype(np.float32)
    # the scale: half the distance of the exponents of (r, r) and of the cells, none
    # below 24
    rr, rmean = float((r * r).sum()), 1e-3 * size
    half = int((np.frexp(rr)[1] - 1 - int(np.log2(r.size))) / 2)
    up = np.ldexp(1.0, half if abs(half) > 24 else 0)
    with open(d / "in.bin", "wb") as f:
        x.tofile(f)
        r.tofile(f)
        (e if prec == "f" else e.astype(np.float64) * up).tofile(f)
    _run(exe, "update", prec, *n, *(BC[b] for b in bc), repr(rr), repr(rmean), d / "in.bin",
         d / "out.bin")
    out = np.fromfile(d / "out.bin")
    C = r.size
    e64 = e.astype(np.float64) * up
    want_x, want_r = x + e64, r - _lap(e64, h, bc) - rmean
    # FP64 rounding of sums of a few terms; L of FP32 corrections in float-float
    top = 4 * sum(1 / a ** 2 for a in h) * np.abs(e64).max()
    assert np.abs(out[:C] - want_x.ravel()).max() <= 4e-16 * np.abs(want_x).max()
    assert np.abs(out[C:2 * C] - want_r.ravel()).max() <= (2.0 ** -44 if prec == "f" else 2.0 ** -50) * top
    assert abs(out[2 * C] / (want_r ** 2).sum() - 1) <= 1e-10
    assert abs(out[2 * C + 1] - want_x.sum()) <= 1e-12 * np.abs(want_x).sum()
    assert abs(out[2 * C + 2] - want_r.mean()) <= 1e-12 * top
    assert list(out[2 * C + 3:]) == [0.0, 1.0]  # still iterating, one application


@pytest.mark.parametrize("case", range(len(DIMS)))
def test_conjugate_gradients_match_numpy(emulator, case):
    exe, d = emulator
    n, bc = DIMS[case]
    shape = n[::-1]
    solid = np.zeros(shape, dtype=np.uint8)
    solid[2:4, 1:4, 2:5] = 1      # a box, and one that touches two walls (or a seam)
    solid[-2:, -2:, -1:] = 1
    code = _codes(solid, bc)
    fluid = solid == 0
    w = [float(m) * m for m in n]
    rng = np.random.default_rng(50 + case)

    def field():
        a = np.where(fluid, rng.normal(size=shape), 0.0)
        return np.where(fluid, a - a.sum() / fluid.sum(), 0.0).astype(np.float32)

    r0, r1 = field(), field()
    diag = (0.5 + rng.random(shape)).astype(np.float32) / np.float32(4 * sum(w))
    junk = rng.normal(size=shape).astype(np.float32)  # z in solid cells takes no part
    with open(d / "in.bin", "wb") as f:
        code.tofile(f)
        for a in (r0, diag, r1, junk):
            a.tofile(f)
    its, more = 5, 3
    _run(exe, "cg", *n, *(BC[b] for b in bc), its, more, d / "in.bin", d / "out.bin")
    raw = open(d / "out.bin", "rb").read()
    C = r0.size
    got = np.frombuffer(raw, np.float32, 4 * C).astype(np.float64).reshape((4,) + shape)
    num = np.frombuffer(raw, np.float64, offset=16 * C)

    p = q = None
    for solve, (r, k) in enumerate(((r0, its), (r1, more))):
        r, x = r.astype(np.float64), np.zeros(shape)
        for _ in range(k):
            z = np.where(fluid, diag * r, 0.0)
            p = z if p is None else z - (z * q).sum() / (p * q).sum() * p
            q = _lap_masked(p, code, w)
            a = (r * p).sum() / (p * q).sum()
            x, r = x + a * p, r - a * q
        # FP32 sums and products over a handful of iterations
        assert np.linalg.norm(got[2 * solve] - x) <= 2e-5 * np.linalg.norm(x)
        assert np.linalg.norm(got[2 * solve + 1] - r) <= 2e-5 * np.linalg.norm((r0, r1)[solve])
        assert not got[2 * solve][~fluid].any()
        assert abs(num[2 * solve] / (r * r).sum() - 1) <= 1e-3
        assert abs(num[2 * solve + 1] - x.sum()) <= 2e-5 * np.abs(x).sum()
