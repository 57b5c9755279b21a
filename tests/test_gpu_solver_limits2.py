"""Further limits of the step kernel's solvers against the oracle: FP64 row blocks on both sides of 19,456 vertices (128 and
256 rows) and past 38,912 (more blocks than SMs, the last one short), the dense inverse and the direct Newton solve with
per-component constraints, and all of them in one-cluster teams.

Tolerances are those of the parity tests: 1e-10 of the displacement in FP64, 1e-6 with FP32 and refinement, 1e-9 for
Newton's iterations.
"""
import dataclasses

import numpy as np
import pytest

import shellgen as sg
from oracle import newton as nw
from oracle import system as osys

gb = pytest.importorskip("paper_2502_10872_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gb.load_library()


def rel(a, b, ref):
    return np.linalg.norm(a - b) / max(np.linalg.norm(ref), 1e-300)


def plate(nx, ny, model, E=1e6, fixed=None):
    """Plate held by the vertices of one side, moving; fixed: (side, component bits) of further vertices."""
    xy, tris = sg.grid(nx, ny)
    rest = sg.flat3(xy)
    pinned = np.zeros(len(rest), np.uint8)
    pinned[sg.grid_side_vertices(nx, ny, "x0")] = 1
    v0 = 0.1 * np.sin(3.0 * rest[:, [0, 1, 0]] + rest[:, [1, 0, 1]])
    bits = np.where(pinned, 7, 0).astype(np.uint8)
    for side, b in fixed or ():
        bits[sg.grid_side_vertices(nx, ny, side)] |= b
    v0[((bits[:, None] >> np.arange(3)) & 1).astype(bool)] = 0.0
    sc = sg.plate_clamped_x0(8, model=model, E=E, dt=1e-2)
    return dataclasses.replace(sc, tris=tris, rest=rest, x0=rest.copy(), v0=v0, pinned=pinned,
                               clamped_edges=np.zeros((0, 2), np.int32), fixed_dofs=bits if fixed else None)


@pytest.mark.parametrize("nx,ny", [(127, 151), (128, 151), (199, 200)])   # 19,456, 19,608 and 40,200 vertices
def test_fp64_row_blocks_of_large_meshes(nx, ny):
    sc = plate(nx, ny, "EP")
    xo, _ = osys.step(osys.from_scenario(sc), sc.x0, sc.v0, 1)
    h = gb.create_from_scenario(sc, precision="fp64")
    gb.shell_step(h, 1)
    x, _ = gb.shell_get_state(h)
    assert rel(x, xo, xo - sc.rest) <= 1e-10


FIXED = [("x1", 1), ("y0", 2)]   # x held on the far side, y along one edge


@pytest.mark.parametrize("nx,ny,model", [(16, 16, "EP"), (31, 15, "SP")])
def test_dense_inverse_with_fixed_components(nx, ny, model):
    """The inverse is that of the matrix with the constrained vertices' diagonals doubled, and the solves are projected."""
    sc = plate(nx, ny, model, fixed=FIXED)
    xo, _ = osys.step(osys.from_scenario(sc), sc.x0, sc.v0, 3)
    bits = ((sc.fixed_dofs[:, None] >> np.arange(3)) & 1).astype(bool)
    for precision, tol in (("fp64", 1e-10), ("fp32_refine", 1e-6)):
        h = gb.create_from_scenario(sc, precision=precision)
        assert gb.shell_info(h)["amg_levels"] == 1
        gb.shell_step(h, 3)
        x, _ = gb.shell_get_state(h)
        assert np.array_equal(x[bits], sc.x0[bits])
        assert rel(x, xo, xo - sc.x0) <= tol


def newton(sc):
    h = gb.create_from_scenario(sc, precision="fp64")
    gb.shell_set_nonlinear(h, 40, 1e-11)
    gb.shell_set_newton(h, True)
    return h


@pytest.mark.parametrize("nx,ny,model", [(12, 2, "FP"), (30, 1, "EP")])
def test_direct_newton_with_fixed_components(nx, ny, model):
    sc = plate(nx, ny, model, E=1e5, fixed=FIXED)
    xo, vo, its = nw.step_newton(osys.from_scenario(sc, factor=False), sc.x0, sc.v0, 1, max_iters=40, rtol=1e-11)
    h = newton(sc)
    st = gb.shell_step(h, 1)
    x, v = gb.shell_get_state(h)
    bits = ((sc.fixed_dofs[:, None] >> np.arange(3)) & 1).astype(bool)
    assert np.array_equal(x[bits], sc.x0[bits])
    assert rel(x, xo, xo - sc.x0) <= 1e-9 and rel(v, vo, vo) <= 1e-9
    assert abs(st["nl_iterations"] - its[0]) <= 1 and st["pcg_iterations"] <= 2 * st["nl_iterations"]


@pytest.mark.parametrize("kind", ["fp64", "fp32_refine", "newton"])
def test_one_cluster_teams_do_not_change_results(kind):
    scs = {"newton": [plate(12, 2, "FP", E=1e5), plate(30, 1, "EP", E=1e5, fixed=FIXED)]}.get(
        kind, [plate(16, 16, "EP"), plate(31, 15, "SP"), plate(9, 4, "FP"), plate(76, 63, "SP")])
    make = newton if kind == "newton" else lambda sc: gb.create_from_scenario(sc, precision=kind)
    alone = []
    for sc in scs:
        h = make(sc)
        gb.shell_step(h, 2)
        alone.append(gb.shell_get_state(h))
    for group in [list(range(len(scs)))] + [[k] for k in range(len(scs))]:   # a batch of all, then each in a cluster
        b = gb.shell_batch_create(1 << 40)
        gb.shell_batch_set_launch(b, 2, 1.0, True)
        hs = [make(scs[k]) for k in group]
        slots = [gb.shell_batch_admit(b, h) for h in hs]
        rc, stats = gb.shell_batch_step(b, 2)
        assert rc == 0
        assert len(group) > 1 or stats[slots[0]]["team_ctas"] == 8
        x, v = gb.shell_batch_get_states(b)
        _, offs = gb.shell_batch_state_layout(b)
        for q, k in enumerate(group):
            xs, vs = x[offs[q]:offs[q + 1]], v[offs[q]:offs[q + 1]]
            assert np.array_equal(xs, alone[k][0]) and np.array_equal(vs, alone[k][1]), (group, k)
        gb.shell_batch_destroy(b)
