"""The default predictor tiles that the tile option does not offer (16 columns,
one plane, a march longer than the grid), run on the host like
test_predict_emulation.py runs the others: FP64 to 1e-13 of the oracle, on grids
that leave a remainder along every axis, walls with the lid, periodic and slip
axes.  No GPU needed."""
from __future__ import annotations

import os
import shutil
import subprocess

import pytest

from test_mg_block_emulation import EMU
from test_predict_emulation import _run_predictor, _source


@pytest.fixture(scope="module", params=[16, 32])
def emulator(request, tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    main = open(os.path.join(EMU, "predict_emu_main.cpp")).read()
    for a, b in (("PT_X", str(request.param)), ("ptile_elems<PY, PZ>", f"ptile_elems<PY, PZ, {request.param}>"),
                 ("PY, PZ>(G", f"PY, PZ, {request.param}>(G"),
                 ("case 408: run(I4{}, I8{})", "case 401: run(I4{}, std::integral_constant<int, 1>{})"),
                 ("case 808: run(I8{}, I8{})", "case 832: run(I8{}, std::integral_constant<int, 32>{})")):
        assert a in main
        main = main.replace(a, b)
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
