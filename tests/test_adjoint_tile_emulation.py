"""k_adj_tile (the reverse step lambda = mu + dt (dR/du)^T mu from a staged tile,
with the per-CTA partials of (dR/du_lid)^T mu summed by k_adj_sum_block) run on
the host like test_adjoint_emulation.py runs the gather, against the oracle's
scatter: grids of one to three tiles per axis with remainders, the smallest
sizes, every boundary type; FP64 to 1e-12 and FP32 to 2e-5 of the largest
entry (the bounds derived there).  No GPU needed."""
from __future__ import annotations

import os
import shutil
import subprocess

import numpy as np
import pytest

import oracle
from paper_1705_06149_gb300 import inputs
from test_mg_block_emulation import CSRC, EMU

BC = {"wall": 0, "periodic": 1, "slip": 2}
DT = 1.0


def _source() -> str:
    dev = open(os.path.join(CSRC, "ns_device.cuh")).read()
    adj = open(os.path.join(CSRC, "ns_adjoint.cuh")).read()
    body = (dev[dev.index("enum { BC_WALL"):dev.index("}  // namespace nsk")] + "\n\n" +
            adj[adj.index("// Tile of k_adj_tile"):adj.rindex("}  // namespace nsk")])
    shared = "extern __shared__ __align__(16) unsigned char asm_raw[];"
    assert shared in body
    return body.replace(shared, "unsigned char* asm_raw = emu_smem;")


def _main() -> str:
    main = open(os.path.join(EMU, "adj_emu_main.cpp")).read()
    a = main.index("    const int ctas = G.fbx")
    b = main.index("    out.assign(")
    return main[:a] + """
    const int tbx = (G.n[0] + TX - 1) / TX, tby = (G.n[1] + TY - 1) / TY;
    const int ctas = tbx * tby * ((G.n[2] + AT_Z - 1) / AT_Z);
    std::vector<double> part(ctas, -7.0);
    std::vector<unsigned char> smem(6 * AT_N * sizeof(T));
    emu_smem = smem.data();
    gridDim.x = (unsigned)ctas;
    launch(ctas, [&] {
        k_adj_tile<T>(G, u.data(), u.data() + G.cnt[0], u.data() + G.cnt[0] + G.cnt[1],
                      mu.data(), mu.data() + G.cnt[0], mu.data() + G.cnt[0] + G.cnt[1],
                      o.data(), o.data() + G.cnt[0], o.data() + G.cnt[0] + G.cnt[1], 1.0, tbx,
                      tby, part.data());
    });
    launch(1, [&] { k_adj_sum_block(part.data(), ctas, &dlid, 0); });
""" + main[b:]


@pytest.fixture(scope="module")
def emulator(tmp_path_factory):
    gxx = shutil.which("g++")
    if gxx is None:
        pytest.skip("g++ not available")
    d = tmp_path_factory.mktemp("adj_tile")
    cpp, exe = d / "emu.cpp", d / "emu"
    cpp.write_text('#include "block_emu.h"\n\n' + _source() + "\n\n" + _main())
    r = subprocess.run([gxx, "-std=c++20", "-O1", "-g", "-fsanitize=address,undefined",
                        "-fno-sanitize-recover=undefined", "-fno-omit-frame-pointer", "-pthread",
                        "-I", EMU, str(cpp), "-o", str(exe)], capture_output=True, text=True)
    if r.returncode != 0 and "barrier" in r.stderr and "No such file" in r.stderr:
        pytest.skip("the host compiler has no <barrier>")
    assert r.returncode == 0, r.stderr[-3000:]
    return str(exe), d


@pytest.mark.parametrize("prec", ["d", "f"])
@pytest.mark.parametrize("dims,bc", [((12, 12, 12), ("wall",) * 3),
                                     ((33, 5, 9), ("wall",) * 3),
                                     ((35, 6, 5), ("periodic", "wall", "slip")),
                                     ((8, 16, 6), ("wall", "periodic", "periodic")),
                                     ((3, 2, 4), ("wall", "slip", "periodic")),
                                     ((2, 3, 2), ("periodic", "wall", "wall")),
                                     ((2, 2, 2), ("wall", "wall", "periodic"))])
def test_adjoint_tile_matches_oracle(emulator, dims, bc, prec):
    exe, d = emulator
    re, u_lid = 40.0, 1.0
    rnd = (lambda a: np.asarray(a, np.float32).astype(np.float64)) if prec == "f" else np.asarray
    st = [rnd(a) for a in inputs.random_state(*dims, seed=17, sigma=0.5, bc=bc)]
    mu = [rnd(a) for a in inputs.random_state(*dims, seed=18, sigma=1.0, bc=bc)[:3]]
    og = oracle.Grid(*dims, re=re, u_lid=u_lid, bc=bc)
    want, want_dl = og.rhs_adjoint(*st[:3], mu)
    tol = 1e-12 if prec == "d" else 2e-5
    tag = "_".join(map(str, dims)) + prec
    fin, fout = d / f"in_{tag}.bin", d / f"out_{tag}.bin"
    np.concatenate([np.ravel(a) for a in list(st[:3]) + list(mu)]).tofile(fin)
    r = subprocess.run([exe, prec, *map(str, dims), *(str(BC[x]) for x in bc), repr(re),
                        repr(u_lid), str(fin), str(fout)], capture_output=True, text=True,
                       timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-3000:])
    out = np.fromfile(fout, dtype=np.float64)
    o = 0
    for c in range(3):
        got = out[o:o + want[c].size].reshape(want[c].shape)
        o += want[c].size
        lam = mu[c] + DT * want[c]
        if bc[c] != "periodic":  # wall faces
            lam = lam.copy()
            idx = [slice(None)] * 3
            for end in (0, -1):
                idx[2 - c] = end
                lam[tuple(idx)] = 0.0
        err = np.max(np.abs(got - lam)) / np.max(np.abs(want[c]))
        assert err <= tol, (c, err)
    assert abs(out[-1] - want_dl) <= tol * max(abs(want_dl), np.max(np.abs(want[0])))


def test_lid_derivative_carries_no_coefficient_rounding(emulator):
    """FP32, u = 0, mu near one: the lid's part is 2 / (Re h^2) sum mu over the
    faces under it.  A face's sum rounds at random (2^-24 of it at most, 2e-9 of
    the total of 600 faces at one standard deviation); the coefficient's own
    rounding would be in every face alike (6.6e-8 here as FP32 factors)."""
    exe, d = emulator
    dims, bc, re = (40, 6, 15), ("periodic", "wall", "periodic"), 44.0
    shapes = [a.shape for a in inputs.random_state(*dims, seed=1, sigma=1.0, bc=bc)]
    rng = np.random.default_rng(3)
    mu = [np.zeros(s) for s in shapes[:3]]
    mu[0] = (1.0 + 0.1 * rng.random(shapes[0])).astype(np.float32).astype(np.float64)
    zero = [np.zeros(s) for s in shapes[:3]]
    fin, fout = d / "in_lid.bin", d / "out_lid.bin"
    np.concatenate([np.ravel(a) for a in zero + mu]).tofile(fin)
    r = subprocess.run([exe, "f", *map(str, dims), *(str(BC[x]) for x in bc), repr(re), "1.0",
                        str(fin), str(fout)], capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, (r.returncode, r.stderr[-3000:])
    want = oracle.Grid(*dims, re=re, u_lid=1.0, bc=bc).rhs_adjoint(*zero, mu)[1]
    assert abs(np.fromfile(fout, dtype=np.float64)[-1] / want - 1.0) <= 1e-8
