"""Sizes at which the step kernel changes its solver or its split of the work, against the oracle: the dense inverse of
small meshes (256 to 512 vertices), the FP64 row blocks of 32 to 256 rows (a chunk per SM up to 4,864, 9,728 and 19,456
rows), and both in batches, where the teams differ and the results may not.

Tolerances are those of the parity tests: 1e-10 of the displacement in FP64, 1e-6 with FP32 and refinement.
"""
import dataclasses

import numpy as np
import pytest

import shellgen as sg
from oracle import system as osys

gb = pytest.importorskip("paper_2502_10872_gb300")
pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _cuda():
    import torch
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    gb.load_library()


def plate(nx, ny, model):
    xy, tris = sg.grid(nx, ny)
    rest = sg.flat3(xy)
    pinned = np.zeros(len(rest), np.uint8)
    pinned[sg.grid_side_vertices(nx, ny, "x0")] = 1
    v0 = 0.1 * np.sin(3.0 * rest[:, [0, 1, 0]] + rest[:, [1, 0, 1]])
    v0[pinned.astype(bool)] = 0.0
    sc = sg.plate_clamped_x0(8, model=model, E=1e6, dt=1e-2)
    return dataclasses.replace(sc, tris=tris, rest=rest, x0=rest.copy(), v0=v0, pinned=pinned,
                               clamped_edges=np.zeros((0, 2), np.int32))


@pytest.mark.parametrize("nx,ny,model,dense", [(16, 14, "EP", False), (15, 15, "EP", True), (31, 15, "SP", True),
                                               (26, 18, "FP", False)])
def test_dense_inverse_of_small_meshes(nx, ny, model, dense):
    sc = plate(nx, ny, model)
    m = osys.from_scenario(sc)
    xo, vo = osys.step(m, sc.x0, sc.v0, 3)
    for precision, tol in (("fp64", 1e-10), ("fp32_refine", 1e-6)):
        h = gb.create_from_scenario(sc, precision=precision)
        st = gb.shell_step(h, 3)
        x, _ = gb.shell_get_state(h)
        assert np.linalg.norm(x - xo) <= tol * np.linalg.norm(xo - sc.rest)
        assert (gb.shell_info(h)["amg_levels"] == 1) == dense
        if dense:
            assert st["pcg_iterations"] <= 2 * max(1, st["refine_rounds"])


@pytest.mark.parametrize("nx,ny", [(30, 8), (75, 63), (76, 63), (138, 69)])   # 279, 4,864, 4,928 and 9,730 vertices
def test_fp64_row_blocks(nx, ny):
    sc = plate(nx, ny, "EP")
    m = osys.from_scenario(sc)
    xo, _ = osys.step(m, sc.x0, sc.v0, 2)
    h = gb.create_from_scenario(sc, precision="fp64")
    gb.shell_step(h, 2)
    x, _ = gb.shell_get_state(h)
    assert np.linalg.norm(x - xo) <= 1e-10 * np.linalg.norm(xo - sc.rest)


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
def test_teams_do_not_change_results(precision):
    scs = [plate(15, 15, "EP"), plate(31, 15, "SP"), plate(9, 4, "FP"), plate(76, 63, "SP"), plate(40, 33, "EP")]
    alone = []
    for sc in scs:
        h = gb.create_from_scenario(sc, precision=precision)
        gb.shell_step(h, 3)
        alone.append(gb.shell_get_state(h))
    for ctas, share in ((1, 8.0), (2, 1.0)):   # few CTAs for the large instances, then many
        b = gb.shell_batch_create(1 << 40)
        gb.shell_batch_set_launch(b, ctas, share)
        hs = [gb.create_from_scenario(sc, precision=precision) for sc in scs]
        for h in hs:
            gb.shell_batch_admit(b, h)
        gb.shell_batch_step(b, 3)
        x, v = gb.shell_batch_get_states(b)
        _, offs = gb.shell_batch_state_layout(b)
        for k in range(len(scs)):
            xs, vs = x[offs[k]:offs[k + 1]], v[offs[k]:offs[k + 1]]
            assert np.array_equal(xs, alone[k][0]) and np.array_equal(vs, alone[k][1]), (ctas, k)
        gb.shell_batch_destroy(b)
