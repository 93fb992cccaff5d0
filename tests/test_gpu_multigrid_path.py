"""The multigrid-preconditioned BiCGStab on boxes without solid cells: the solver
of grids that the direct solve does not take (NS_DIRECT=0 in the environment, a
tolerance below 1e-14, planes and matrices beyond shared memory).  The tests of
the default path run again with the direct solve turned off: solves and steps
against the oracle, the captured conditional loops, the pipelined schedule, the
gradient.
"""
import pytest

import test_gpu_adjoint as A
import test_gpu_graph as G
import test_gpu_parity as P
from paper_1705_06149_gb300 import Grid, inputs

pytestmark = pytest.mark.gpu

PRECS = ["fp64", "fp32_refine"]


@pytest.fixture(autouse=True)
def multigrid(monkeypatch):
    monkeypatch.setenv("NS_DIRECT", "0")
    g = Grid(16, 16, 16)
    st = g.state_from(inputs.random_state(16, 16, 16, seed=1, sigma=0.2))
    g.profile(True)
    g.step_fine(st, 1e-3, 1)
    prof = g.profile_read()
    g.close()
    assert prof["krylov_A"]["launches"] > 0 and prof["direct_xy"]["launches"] == 0


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("dims", [(24, 20, 18), (32, 16, 8), (64, 64, 64)])
def test_poisson_solve(prec, dims):
    P.test_poisson_solve_matches_oracle(prec, dims, "multigrid")


@pytest.mark.parametrize("prec", PRECS)
@pytest.mark.parametrize("dims,bc", [((12, 12, 12), ("wall",) * 3),
                                     ((16, 12, 8), ("periodic", "wall", "slip"))])
def test_fine_steps(dims, bc, prec):
    P.test_fine_steps_match_oracle(dims, bc, prec, "multigrid")


@pytest.mark.parametrize("prec", PRECS)
def test_chunked_parareal(prec):
    P.test_chunked_parareal_is_bit_identical(prec, "multigrid")


@pytest.mark.parametrize("prec", PRECS)
def test_pipelined_parareal_stops(prec):
    P.test_pipelined_parareal_stops_at_the_tolerance(prec)


@pytest.mark.parametrize("prec", PRECS)
def test_nonfinite_slice(prec):
    P.test_nonfinite_slice_in_pipelined_parareal_is_reported(prec)


@pytest.mark.parametrize("prec", PRECS)
def test_iteration_limit(prec):
    P.test_iteration_limit_is_reported(prec, "multigrid")


def test_resume():
    P.test_parareal_resume_and_tolerance()


@pytest.mark.parametrize("prec", PRECS)
def test_graph_reproduces_the_stream_path(prec):
    G.test_graph_reproduces_the_stream_path_bit_for_bit(prec)


@pytest.mark.parametrize("prec", PRECS)
def test_graph_counts(prec):
    G.test_graph_counts_steps_solves_and_iterations(prec)


@pytest.mark.parametrize("prec", PRECS)
def test_graph_above_the_one_cta_levels(prec):
    G.test_graph_matches_the_oracle_above_the_one_cta_levels(prec)


@pytest.mark.parametrize("prec", PRECS)
def test_step_fine_many(prec):
    G.test_step_fine_many_reproduces_the_stream_path(prec)


@pytest.mark.parametrize("moving", [False, True])
def test_adjoint(moving):
    A.test_adjoint_matches_oracle(moving)


def test_fp32_adjoint():
    A.test_fp32_refine_adjoint_matches_oracle()
