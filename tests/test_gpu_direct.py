"""Pressure corrections by the direct solve (boxes without solid cells)
against the FP64 oracle, at the sizes where its kernels change: odd extents,
extents below a tile, several column blocks and column chunks, every boundary
type, grids the multigrid hierarchy cannot halve, and the graph path."""
import numpy as np
import pytest

import oracle
from paper_1705_06149_gb300 import Grid, NSError, StepGraph, inputs
from paper_1705_06149_gb300 import _native as N

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

TOL = {"fp64": 1e-10, "fp32_refine": 1e-5}

CASES = [((6, 3, 5), ("wall", "periodic", "wall")),
         ((19, 13, 11), ("wall",) * 3),
         ((45, 37, 21), ("wall", "slip", "wall")),
         ((33, 10, 9), ("periodic", "periodic", "wall")),
         ((12, 20, 40), ("wall", "wall", "periodic")),
         ((10, 6, 150), ("wall",) * 3),
         ((72, 100, 6), ("slip", "wall", "periodic"))]


def rel(a, b):
    n = np.linalg.norm(np.ravel(b))
    return np.linalg.norm(np.ravel(a) - np.ravel(b)) / (n if n > 0 else 1.0)


@pytest.mark.parametrize("prec", ["fp64", "fp32_refine"])
@pytest.mark.parametrize("case", range(len(CASES)))
def test_direct_steps_and_solves_match_the_oracle(case, prec):
    dims, bc = CASES[case]
    B = 2
    box = [d / max(dims) for d in dims]  # cubic cells: cond(L) stays that of the extents
    og = oracle.Grid(*dims, *box, re=100.0, bc=bc, rtol=1e-13)
    g = Grid(*dims, *box, re=100.0, bc=bc, precision=prec, batch=B, poisson_rtol=1e-13)
    inits = [inputs.random_state(*dims, seed=30 + s, sigma=0.2, bc=bc) for s in range(B)]
    st = g.state_from([np.stack([i[c] for i in inits]) for c in range(4)])
    g.profile(True)
    g.step_fine(st, 2e-4, 3)
    prof = g.profile_read()
    g.profile(False)
    assert prof["direct_xy"]["launches"] > 0 and prof["krylov_A"]["launches"] == 0
    got = st.numpy()
    for s in range(B):
        want = oracle.copy_state(inits[s])
        og.step(want, 2e-4, 3)
        vg = np.concatenate([np.ravel(got[c][s]) for c in range(3)])
        vw = np.concatenate([np.ravel(want[c]) for c in range(3)])
        assert rel(vg, vw) <= TOL[prec], (s, rel(vg, vw))
        assert rel(got[3][s], want[3]) <= TOL[prec], (s, rel(got[3][s], want[3]))
    b = np.random.default_rng(case).normal(size=(B,) + og.shape(3))
    bt = torch.tensor(b, device="cuda")
    pt = torch.zeros_like(bt)
    assert g.poisson_solve(bt, pt) >= 1
    for s in range(B):
        want, _ = og.poisson(b[s], rtol=1e-13)
        # both sides stop at a relative residual (FP32+refine 1e-10), which the
        # condition number of L (at most a few 1e4 here) turns into p's error
        assert rel(pt[s].cpu().numpy(), want) <= (1e-9 if prec == "fp64" else 1e-6)
    g.close()


def test_a_grid_the_hierarchy_cannot_halve_still_refuses_graphs():
    g = Grid(45, 37, 21, precision="fp32_refine")
    with pytest.raises(NSError) as e:
        StepGraph([(g, g.zeros(1), 1e-3, 1)])
    assert e.value.status == N.NS_ERR_ARG
    g.close()


@pytest.mark.parametrize("prec", ["fp64", "fp32_refine"])
def test_direct_solve_off_gives_the_multigrid_result(prec, monkeypatch):
    dims = (32, 24, 16)
    init = inputs.random_state(*dims, seed=4, sigma=0.2)
    out = []
    for env in ("1", "0"):
        monkeypatch.setenv("NS_DIRECT", env)
        g = Grid(*dims, re=200.0, precision=prec, poisson_rtol=1e-13)
        st = g.state_from(init)
        g.profile(True)
        g.step_fine(st, 1e-3, 3)
        assert (g.profile_read()["direct_xy"]["launches"] > 0) == (env == "1")
        out.append(st.numpy())
        g.close()
    for c in range(4):
        assert rel(out[0][c], out[1][c]) <= TOL[prec]


# conjugate gradients around the direct solve: remainders of its tiles, one and
# several chunks of a column, every boundary type, a dense mask (whose predictor
# takes every face by the solid cells' rules)
@pytest.mark.parametrize("dims,bc,count,edge",
                         [((16, 12, 8), ("wall",) * 3, 3, (0.15, 0.3)),
                          ((36, 20, 24), ("periodic", "wall", "slip"), 3, (0.1, 0.2)),
                          ((8, 12, 144), ("wall", "slip", "periodic"), 3, (0.1, 0.3)),
                          ((20, 16, 12), ("wall",) * 3, 1, (0.6, 0.6))])
def test_obstacle_steps_match_the_oracle(dims, bc, count, edge, monkeypatch):
    box = [d / max(dims) for d in dims]
    _, solid = inputs.obstacle_boxes(dims, seed=5, count=count, edge=edge)
    og = oracle.Grid(*dims, *box, re=100.0, bc=bc, solid=solid, rtol=1e-13)
    init = inputs.random_state(*dims, seed=3, sigma=0.2, bc=bc, solid=solid)
    want = oracle.copy_state(init)
    og.step(want, 2e-4, 3)
    for env in ("1", "0"):
        monkeypatch.setenv("NS_DIRECT", env)
        g = Grid(*dims, *box, re=100.0, bc=bc, solid=solid, precision="fp32_refine")
        st = g.state_from(init)
        g.profile(True)
        g.step_fine(st, 2e-4, 3)
        assert (g.profile_read()["direct_xy"]["launches"] > 0) == (env == "1")
        got = st.numpy()
        vg = np.concatenate([np.ravel(got[c][0]) for c in range(3)])
        vw = np.concatenate([np.ravel(want[c]) for c in range(3)])
        assert rel(vg, vw) <= TOL["fp32_refine"]
        assert rel(got[3][0], want[3]) <= TOL["fp32_refine"]
        g.close()


# FP64 solves whose corrections are FP32 (393216 cells and more per grid): right
# sides and boxes far outside FP32's range solve as their scaled copies do
MIXED = (64, 64, 48)


def _solve(b, box=(1.0, 1.0, 1.0), batch=2):
    g = Grid(*MIXED, *box, batch=batch, poisson_rtol=1e-12)
    p = torch.zeros_like(b)
    its = g.poisson_solve(b, p)
    g.close()
    return p, its


@pytest.mark.parametrize("power", [-400, 300])
def test_fp64_solves_do_not_depend_on_the_size_of_the_right_side(power):
    b = torch.tensor(np.random.default_rng(1).normal(size=(2,) + MIXED[::-1]), device="cuda")
    p, its = _solve(b)
    q, its_q = _solve(b * 2.0 ** power)
    # powers of two: every operation rounds alike
    assert its_q == its and torch.equal(q * 2.0 ** -power, p)


def test_fp64_solves_of_a_box_beyond_fp32():
    b = torch.tensor(np.random.default_rng(2).normal(size=(2,) + MIXED[::-1]), device="cuda")
    p, _ = _solve(b)
    q, _ = _solve(b, box=(2.0 ** -70,) * 3)  # h^-2 about 2^152
    # both stop at a relative residual of 1e-12, seen through L (a few 1e3)
    assert rel((q * 2.0 ** 140).cpu().numpy(), p.cpu().numpy()) <= 1e-8


def _room(dims, door):
    solid = np.zeros(dims[::-1], np.uint8)
    solid[2:14, 2:14, 2:14] = 1
    solid[3:13, 3:13, 3:13] = 0
    if door:
        solid[7:9, 7:9, 13] = 0
    return solid


def _specks(dims):
    return (np.random.default_rng(1).random(dims[::-1]) < 0.05).astype(np.uint8)


# which solid cells keep the V-cycle: a sealed room (a second region of fluid,
# which conjugate gradients around the box solve do not converge on) and, on large
# planes, scattered single cells
@pytest.mark.parametrize("dims,mask,direct",
                         [((32, 24, 16), lambda d: _room(d, False), False),
                          ((32, 24, 16), lambda d: _room(d, True), True),
                          ((32, 32, 16), _specks, True),
                          ((128, 72, 8), _specks, False)])
def test_masks_that_keep_the_multigrid_solve(dims, mask, direct):
    solid = mask(dims)
    init = inputs.random_state(*dims, seed=3, sigma=0.2, solid=solid)
    box = [d / max(dims) for d in dims] if dims[0] > 32 else (1.0, 1.0, 1.0)
    g = Grid(*dims, *box, precision="fp32_refine", solid=solid)
    st = g.state_from(init)
    g.profile(True)
    g.project(st)
    prof = g.profile_read()
    assert (prof["direct_xy"]["launches"] > 0) == direct
    assert (prof["krylov_A"]["launches"] > 0) != direct
    want = oracle.Grid(*dims, *box, solid=solid, rtol=1e-13).project(*init[:3])
    got = st.numpy()
    vg = np.concatenate([np.ravel(got[c][0]) for c in range(3)])
    vw = np.concatenate([np.ravel(want[c]) for c in range(3)])
    assert rel(vg, vw) <= 1e-6
    # tens of iterations, where a solve that stalls takes its corrections' limit
    # of 40 solves times 20 max(n) iterations
    assert g.stats()["krylov_iters"] <= 100
    g.close()


# what include/ns.h says of the bits: one grid gives a state the same ones whatever
# the batch of a call and its place in it; grids of another capacity agree at
# rounding level (FP64 from 393216 cells on: FP32 corrections, so within the
# solves' tolerance)
@pytest.mark.parametrize("prec,dims,caps", [("fp32_refine", (64, 64, 32), (1, 5, 24)),
                                            ("fp64", (64, 64, 48), (1, 3)),
                                            ("fp64", (20, 12, 16), (1, 5))])
def test_bits_of_a_state_belong_to_its_grid(prec, dims, caps):
    inits = [inputs.random_state(*dims, seed=60 + s, sigma=0.2) for s in range(3)]
    out = {}
    for cap in caps:
        g = Grid(*dims, re=500.0, precision=prec, batch=cap)
        alone = [g.state_from(i) for i in inits]
        for st in alone:
            g.step_fine(st, 5e-4, 3)
        if cap >= 3:
            both = g.state_from([np.stack([i[c] for i in inits]) for c in range(4)])
            g.step_fine(both, 5e-4, 3)
            for c in range(4):
                for s in range(3):
                    assert torch.equal(both.fields()[c][s], alone[s].fields()[c][0]), (cap, c, s)
        out[cap] = [torch.cat([st.fields()[c] for st in alone]).double() for c in range(4)]
        g.close()
    for cap in caps[1:]:
        # FP32: a rounding of the stored velocity; its divergence over dt in p.
        # FP64: residuals of 1e-12 through L's condition number (a few 1e3)
        for c in range(4):
            a, b = out[cap][c], out[caps[0]][c]
            tol = 1e-8 if prec == "fp64" else (1e-6 if c < 3 else 1e-5)
            assert float((a - b).norm()) <= tol * float(b.norm()), (cap, c)
