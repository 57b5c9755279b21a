"""Direct solve of small Newton systems (FP64 instances of one row block whose band fits shared memory) against the
oracle's Newton steps, and its limits: meshes whose band does not fit iterate as before. The Newton matrix itself
is tested by the iteration counts: with its factor as the preconditioner a linear solve takes one or two iterations,
with any other matrix many.
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


def strip(nx, ny, model, seed=4):
    """Strip of nx x ny cells held by the vertices of one end, falling with a random initial velocity."""
    xy, tris = sg.grid(nx, ny)
    rest = sg.flat3(xy)
    pinned = np.zeros(len(rest), np.uint8)
    pinned[sg.grid_side_vertices(nx, ny, "x0")] = 1
    v0 = 0.1 * np.random.default_rng(seed).standard_normal(rest.shape)
    v0[pinned.astype(bool)] = 0.0
    sc = sg.plate_clamped_x0(8, model=model, E=1e5, dt=1e-2)
    return dataclasses.replace(sc, tris=tris, rest=rest, x0=rest.copy(), v0=v0, pinned=pinned,
                               clamped_edges=np.zeros((0, 2), np.int32))


# the smallest mesh, a ragged one, one close below the limit of the band (85 vertices of an edge-hinge strip), and one
# past it
@pytest.mark.parametrize("nx,ny,model,direct", [(1, 1, "EP", True), (2, 1, "FP", True), (13, 2, "SS", True),
                                                (42, 1, "EP", True), (15, 14, "SP", False)])
def test_small_newton_steps_match_oracle(nx, ny, model, direct):
    sc = strip(nx, ny, model)
    m = osys.from_scenario(sc, factor=False)
    xo, vo, its = nw.step_newton(m, sc.x0, sc.v0, 2, max_iters=60, rtol=1e-11)
    h = gb.create_from_scenario(sc, precision="fp64")
    gb.shell_set_nonlinear(h, 60, 1e-11)
    gb.shell_set_newton(h, True)
    per_solve = []
    for k in range(2):
        st = gb.shell_step(h, 1)
        per_solve.append(st["pcg_iterations"] / st["nl_iterations"])
        assert abs(st["nl_iterations"] - its[k]) <= 1
    x, v = gb.shell_get_state(h)
    assert rel(x, xo, xo - sc.x0) <= 1e-9
    assert rel(v, vo, vo) <= 1e-9
    assert (max(per_solve) <= 2.0) == direct


def test_direct_newton_alone_and_in_a_batch_is_the_same():
    scs = [strip(12, 2, "FP"), strip(9, 1, "EP", seed=5)]

    def make(sc):
        h = gb.create_from_scenario(sc, precision="fp64")
        gb.shell_set_nonlinear(h, 8, 1e-9)
        gb.shell_set_newton(h, True)
        return h

    alone = []
    for sc in scs:
        h = make(sc)
        gb.shell_step(h, 2)
        alone.append(gb.shell_get_state(h))
    b = gb.shell_batch_create(1 << 40)
    hs = [make(sc) for sc in scs]
    for h in hs:
        gb.shell_batch_admit(b, h)
    rc, _ = gb.shell_batch_step(b, 2)
    assert rc == 0
    x, v = gb.shell_batch_get_states(b)
    _, offs = gb.shell_batch_state_layout(b)
    for k in range(2):
        xs, vs = x[offs[k]:offs[k + 1]], v[offs[k]:offs[k + 1]]
        assert np.array_equal(xs, alone[k][0]) and np.array_equal(vs, alone[k][1]), k
    gb.shell_batch_destroy(b)
