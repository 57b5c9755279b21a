"""Small Newton systems whose band factorisation is rejected: the solve falls back to the iteration.

An unloaded membrane of vanishing thickness, held at one end and compressed in its plane, has no stiffness across the
sheet: its bending (t / h)^2 and its inertia M / (dt^2 K) lie below 1e-17 of the membrane's entries, and the tangent's
rotation terms are clamped at zero, so that the pivots of the transverse components are the rounding left by the
cancellation of equal entries. They have either sign, and one that is not positive rejects the factor. In the plane
the problem is well posed and its solution known: the sheet goes back to rest (inertia cannot hold it), and since
nothing acts across the sheet it stays plane exactly. The iteration counts tell that the solve did iterate: with the
factor a solve takes one or two.

Tolerance: a Newton residual of 1e-9 of the first, times the condition of the strip's in-plane stiffness (below 1e3).
"""
import dataclasses

import numpy as np
import pytest

import shellgen as sg

gb = pytest.importorskip("paper_2502_10872_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gb.load_library()


def membrane(nx, ny, model):
    xy, tris = sg.grid(nx, ny)
    rest = sg.flat3(xy)
    pinned = np.zeros(len(rest), np.uint8)
    pinned[sg.grid_side_vertices(nx, ny, "x0")] = 1
    x0 = rest.copy()
    x0[:, 0] *= 0.98
    sc = sg.plate_clamped_x0(8, model=model, E=1e5, dt=1e8, thickness=1e-11)
    return dataclasses.replace(sc, tris=tris, rest=rest, x0=x0, v0=np.zeros_like(rest), pinned=pinned,
                               clamped_edges=np.zeros((0, 2), np.int32), gravity=(0.0, 0.0, 0.0))


def handle(sc):
    h = gb.create_from_scenario(sc, precision="fp64")
    gb.shell_set_nonlinear(h, 40, 1e-9)
    gb.shell_set_newton(h, True)
    return h


SIZES = [(6, 2, "EP"), (12, 2, "FP"), (9, 3, "SP")]


@pytest.mark.parametrize("nx,ny,model", SIZES)
def test_rejected_factor_iterates(nx, ny, model):
    sc = membrane(nx, ny, model)
    h = handle(sc)
    st = gb.shell_step(h, 1)
    x, _ = gb.shell_get_state(h)
    assert st["pcg_iterations"] > 4 * st["nl_iterations"]   # at least one solve iterated
    assert np.all(x[:, 2] == 0.0)
    assert np.linalg.norm(x - sc.rest) <= 1e-6 * np.linalg.norm(sc.x0 - sc.rest)


def test_rejected_factor_in_teams_of_one_and_of_a_cluster():
    scs = [membrane(*s) for s in SIZES]
    alone = []
    for sc in scs:
        h = handle(sc)
        gb.shell_step(h, 1)
        alone.append(gb.shell_get_state(h))
    for clusters in (False, True):   # a queue of one-CTA instances; one-cluster teams for one instance at a time
        for group in ([0, 1, 2],) if not clusters else ([0], [1], [2]):
            b = gb.shell_batch_create(1 << 40)
            gb.shell_batch_set_launch(b, 2, 1.0, clusters)
            hs = [handle(scs[k]) for k in group]
            for h in hs:
                gb.shell_batch_admit(b, h)
            rc, _ = gb.shell_batch_step(b, 1)
            assert rc == 0
            x, v = gb.shell_batch_get_states(b)
            _, offs = gb.shell_batch_state_layout(b)
            for q, k in enumerate(group):
                xs, vs = x[offs[q]:offs[q + 1]], v[offs[q]:offs[q + 1]]
                assert np.array_equal(xs, alone[k][0]) and np.array_equal(vs, alone[k][1]), (clusters, k)
            gb.shell_batch_destroy(b)
