"""bench.py's byte model names and counts the kernels that a profile saw run: the
direct solve's where they ran (FP32 corrections of FP64 residuals on large FP64
grids), the preconditioned BiCGStab's elsewhere.  No GPU needed."""
import os
import sys

import pytest

sys.path.insert(0, os.path.dirname(os.path.dirname(os.path.abspath(__file__))))
import bench  # noqa: E402
from paper_1705_06149_gb300._native import KERNEL_KINDS  # noqa: E402

CELLS = 32 * 64 ** 3


def _prof(**launches):
    assert set(launches) <= set(KERNEL_KINDS)
    return {k: {"launches": launches.get(k, 0)} for k in KERNEL_KINDS}


# two calls of 50 steps, two applications a step
DIRECT = _prof(predict=100, inner_init=2, solve_init=100, direct_xy=400, direct_z=200, refine=200,
               correct=100)
MG = _prof(predict=100, divergence=100, solve_init=100, krylov_A=500, krylov_B=500, krylov_C=500,
           refine=300, correct=100)


def test_direct_solve_is_counted_as_it_runs():
    b, names, solver = bench.traffic_model("fp32_refine", "multigrid", DIRECT, CELLS)
    # k_dir_refine reads r (8) and e (4), writes r (8); k_dir_start reads the
    # increments (12) and w (8), writes r (8)
    assert (b["refine"], b["solve_init"], b["direct_xy"], b["direct_z"]) == (20, 28, 8, 8)
    # 49 of 50 corrections read u, increments, base, two applications, q, write
    # u, w, q; the last writes p in the place of w and q and reads no q
    assert b["correct"] == pytest.approx(0.98 * 76 + 0.02 * 60)
    half = bench.traffic_model("fp32_refine", "multigrid", DIRECT, CELLS, 0.5)[0]["correct"]
    assert half == pytest.approx(b["correct"] - 4)  # one application less apart
    assert names["refine"] == "k_dir_refine" and names["solve_init"] == "k_dir_start"
    assert names["correct"] == "k_dir_correct"
    assert "direct" in solver and "BiCGStab" not in solver
    # no kernel of the launch list (64^3 x 32 states, us) above the HBM peak
    for kind, us in (("predict", 159), ("solve_init", 109), ("direct_xy", 46), ("direct_z", 23),
                     ("refine", 60), ("correct", 120)):
        assert b[kind] * CELLS / (us * 1e-6) / 1e9 <= 6785, kind


def test_fp64_direct_solve_counts_fp32_corrections():
    big = bench.traffic_model("fp64", "multigrid", DIRECT, CELLS)
    small = bench.traffic_model("fp64", "multigrid", DIRECT, 16 ** 3)
    assert (big[0]["direct_xy"], big[0]["direct_z"], big[0]["refine"]) == (10, 8, 36)
    assert (small[0]["direct_xy"], small[0]["direct_z"], small[0]["refine"]) == (16, 16, 40)
    assert big[1]["refine"] == "k_dir_update" and "FP32 corrections" in big[2]
    assert "FP32" not in small[2]


def test_multigrid_and_plain_paths_keep_their_model():
    b, names, solver = bench.traffic_model("fp32_refine", "multigrid", MG, CELLS)
    assert (b["refine"], b["correct"], b["krylov_C"], b["mg_block"]) == (44, 76, 32, 4)
    assert names["refine"] == "k_mg_refine_update_ff" and "BiCGStab + multigrid" in solver
    b, _, solver = bench.traffic_model("fp64", "none", MG, CELLS)
    assert b == {"krylov_A": 48, "krylov_B": 24, "krylov_C": 64} and solver == "BiCGStab"


def test_every_counted_kind_has_a_name():
    for prec, pc, prof in (("fp32_refine", "multigrid", DIRECT), ("fp64", "multigrid", DIRECT),
                           ("fp32_refine", "multigrid", MG), ("fp64", "none", MG)):
        b, names, _ = bench.traffic_model(prec, pc, prof, CELLS)
        assert set(b) - set(names) <= {"mg_coarse", "mg_block", "mg_cluster"}


def test_launches_that_states_leave_at_once_are_not_counted():
    assert bench.share_of(200 * 32, DIRECT, 32) == 1.0
    assert bench.share_of(150 * 32, DIRECT, 32) == 0.75
    assert bench.share_of(400 * 32, MG, 32) == 0.8
    assert bench.share_of(0, _prof(), 32) == 1.0
