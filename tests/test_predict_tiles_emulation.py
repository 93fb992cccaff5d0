"""The default predictor tiles that the tile option does not offer (16 columns,
one plane, a march longer than the grid), run on the host like
test_predict_emulation.py runs the others: FP64 to 1e-13 of the oracle, on grids
that leave a remainder along every axis, walls with the lid, periodic and slip
axes.  No GPU needed."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

from paper_1705_06149_gb300 import inputs

from test_mg_block_emulation import EMU
from test_predict_emulation import BC, _run_predictor, _source


@pytest.fixture(scope="module", params=[16, 32])
def emulator(request, tmp_path_factory):
    return _build(tmp_path_factory, request.param, lambda s: s)


def _build(tmp_path_factory, width, edit):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    main = open(os.path.join(EMU, "predict_emu_main.cpp")).read()
    for a, b in (("PT_X", str(width)), ("ptile_elems<PY, PZ>", f"ptile_elems<PY, PZ, {width}>"),
                 ("PY, PZ>(G", f"PY, PZ, {width}>(G"),
                 ("case 408: run(I4{}, I8{})", "case 401: run(I4{}, std::integral_constant<int, 1>{})"),
                 ("case 808: run(I8{}, I8{})", "case 832: run(I8{}, std::integral_constant<int, 32>{})")):
        assert a in main
        main = main.replace(a, b)
    main = edit(main)
    d = tmp_path_factory.mktemp("predict_tiles")
    cpp, exe = d / "emu.cpp", d / "emu"
    cpp.write_text('#include "block_emu.h"\n\n' + _source() + "\n\n" + main)
    r = subprocess.run([gxx, "-std=c++20", "-O1", "-g", "-fsanitize=address,undefined",
                        "-fno-sanitize-recover=undefined", "-fno-omit-frame-pointer", "-pthread",
                        "-I", EMU, str(cpp), "-o", str(exe)], capture_output=True, text=True)
    if r.returncode != 0 and "barrier" in r.stderr and "No such file" in r.stderr:
        pytest.skip("the host compiler has no <barrier>")
    assert r.returncode == 0, r.stderr[-3000:]
    return str(exe), d


@pytest.mark.parametrize("tile", [(4, 1), (8, 32)])
@pytest.mark.parametrize("dims,bc", [((17, 9, 5), ("wall",) * 3),
                                     ((33, 5, 35), ("periodic", "slip", "wall")),
                                     ((2, 3, 2), ("wall", "wall", "periodic"))])
@pytest.mark.parametrize("incr", [False, True])
def test_default_tiles_match_oracle(emulator, dims, bc, tile, incr):
    _run_predictor(emulator, dims, bc, False, incr, tile)


def test_fp32_increment_carries_no_coefficient_rounding(tmp_path_factory):
    """FP32 increment of a velocity u(y, z) so small that only diffusion counts:
    its projection on the exact one is 1 up to the random rounding of each
    value (about 1e-7 over the root of 2304 columns, 2e-9); the rounding of
    dt / (Re h^2) to FP32 (here -5.5e-8) would be in every value alike."""

    def as_float(s):
        for a, b in (("const double* u = in.data();",
                      "std::vector<float> in32(in.begin(), in.end());\n    const float* u = in32.data();"),
                     ("const double* v =", "const float* v ="), ("const double* w =", "const float* w ="),
                     ("std::vector<double> out(", "std::vector<float> out("),
                     ("double* fu", "float* fu"), ("double* fv", "float* fv"),
                     ("double* fw", "float* fw"), ("k_predict_tile<double", "k_predict_tile<float"),
                     ("k_predict_masked<double", "k_predict_masked<float"),
                     ("fwrite(out.data(), sizeof(double)", "fwrite(out.data(), sizeof(float)")):
            assert a in s, a
            s = s.replace(a, b)
        return s

    exe, d = _build(tmp_path_factory, 32, as_float)
    dims, bc, re, dt = (2, 48, 48), ("periodic",) * 3, 194.0, 7e-4
    line = np.random.default_rng(2).standard_normal((48, 48, 1)) * 1e-6
    u = (line + np.zeros((48, 48, 2))).astype(np.float32).astype(np.float64)
    zero = [np.zeros(a.shape) for a in inputs.random_state(*dims, seed=1, sigma=1.0, bc=bc)[1:3]]
    fin, fout = d / "in.bin", d / "out.bin"
    np.concatenate([np.ravel(a) for a in [u] + zero]).tofile(fin)
    r = subprocess.run([exe, *map(str, dims), *(str(BC[b]) for b in bc), repr(re), "0.0", repr(dt),
                        "1", str(fin), "-", str(fout), "8", "32"], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-3000:])
    got = np.fromfile(fout, dtype=np.float32)[:u.size].astype(np.float64).reshape(u.shape)
    want = sum(np.roll(u, s, a) - u for s in (1, -1) for a in (0, 1)) * (dt / re * 48.0 ** 2)
    assert abs((got * want).sum() / (want * want).sum() - 1.0) <= 1e-8
