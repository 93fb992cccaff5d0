"""The predictor of a grid with solid cells as the tiles of k_predict_tile and the
faces that k_list_faces lists (k_predict_faces), run on the host in FP64 against
the oracle to 1e-13: boxes that touch walls, wrap a periodic axis, leave channels
one or two cells wide; every face that is not listed is then one whose stencil
no solid cell changes.  No GPU needed."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_1705_06149_gb300 import inputs
from test_mg_block_emulation import EMU
from test_predict_emulation import BC, CSRC, _source


def _full_source() -> str:
    ker = open(os.path.join(CSRC, "ns_kernels.cuh")).read()
    a = ker.index("// Does a solid cell take part in face f")
    b = ker.index("// ---------------------------------------------------------------------------\n// b = D F*")
    return _source() + "\n\n" + ker[a:b]


@pytest.fixture(scope="module")
def emulator(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    main = open(os.path.join(EMU, "predict_emu_main.cpp")).read()
    # the tiles always, then the listed faces
    main = main.replace("if (G.solid == nullptr) {", "{")
    a = main.index("    } else {\n        if (incr)")
    b = main.index("    f = fopen(argv[13]")
    main = main[:a] + """    }
    const long long total = G.cnt[0] + G.cnt[1] + G.cnt[2];
    std::vector<long long> list(total, -1);
    unsigned long long count = 0;
    launch((int)((total + 255) / 256), 256, [&] { k_list_faces(G, list.data(), &count); }, true);
    launch((int)((count + NTHREADS - 1) / NTHREADS), NTHREADS, [&] {
        if (incr) k_predict_faces<double, true>(G, u, v, w, fu, fv, fw, dt, list.data(), (long long)count);
        else k_predict_faces<double, false>(G, u, v, w, fu, fv, fw, dt, list.data(), (long long)count);
    });
    printf("%llu\\n", count);
""" + main[b:]
    add = """inline unsigned long long atomicAdd(unsigned long long* p, unsigned long long v) {
    return __atomic_fetch_add(p, v, __ATOMIC_SEQ_CST);
}
"""
    d = tmp_path_factory.mktemp("predict_faces")
    cpp, exe = d / "emu.cpp", d / "emu"
    cpp.write_text('#include "block_emu.h"\n' + add + _full_source() + "\n\n" + main)
    r = subprocess.run([gxx, "-std=c++20", "-O1", "-g", "-fsanitize=address,undefined",
                        "-fno-sanitize-recover=undefined", "-fno-omit-frame-pointer", "-pthread",
                        "-I", EMU, str(cpp), "-o", str(exe)], capture_output=True, text=True)
    if r.returncode != 0 and "barrier" in r.stderr and "No such file" in r.stderr:
        pytest.skip("the host compiler has no <barrier>")
    assert r.returncode == 0, r.stderr[-3000:]
    return str(exe), d


BOXES = [((3, 6), (2, 5), (4, 6)), ((7, 9), (2, 5), (4, 6)), ((0, 2), (7, 9), (0, 3)),
         ((10, 12), (0, 10), (3, 4))]


@pytest.mark.parametrize("incr", [False, True])
@pytest.mark.parametrize("bc", [("wall",) * 3, ("periodic", "wall", "slip"),
                                ("wall", "periodic", "periodic")])
def test_tiles_and_listed_faces_match_the_oracle(emulator, bc, incr):
    exe, d = emulator
    dims, re, u_lid, dt = (12, 10, 8), 50.0, 1.0, 2e-3
    solid = np.zeros(dims[::-1], dtype=np.uint8)
    for x, y, z in BOXES:
        solid[z[0]:z[1], y[0]:y[1], x[0]:x[1]] = 1
    rs = inputs.random_state(*dims, seed=9, sigma=1.0, bc=bc, solid=solid)
    want = oracle.Grid(*dims, re=re, u_lid=u_lid, bc=bc, solid=solid).predict(*rs[:3], dt)
    fin, fsol, fout = d / "in.bin", d / "solid.bin", d / "out.bin"
    np.concatenate([np.ravel(a) for a in rs[:3]]).astype(np.float64).tofile(fin)
    solid.tofile(fsol)
    r = subprocess.run([exe, *map(str, dims), *(str(BC[b]) for b in bc), repr(re), repr(u_lid),
                        repr(dt), "1" if incr else "0", str(fin), str(fsol), str(fout)],
                       capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-3000:])
    assert 0 < int(r.stdout) < sum(a.size for a in want)
    out, o = np.fromfile(fout, dtype=np.float64), 0
    for c in range(3):
        got = out[o:o + want[c].size].reshape(want[c].shape)
        o += want[c].size
        err = np.max(np.abs(got + (rs[c] if incr else 0.0) - want[c])) / np.max(np.abs(want[c]))
        assert err <= 1e-13, (c, err)
