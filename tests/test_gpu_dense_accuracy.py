"""Where an FP32 solve with a dense inverse (small stiff meshes) ends: at 0.07 of the refinement target, as far as one
further round gets it, and not just under the target, where its error lies in the smooth modes."""
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


def moving(sc, seed):
    v0 = np.random.default_rng(seed).standard_normal((3, 3)) @ np.sin(3.0 * sc.rest.T + seed)
    v0 = 0.2 * v0.T * sc.rest[:, :1]
    v0[sc.pinned.astype(bool)] = 0.0
    return dataclasses.replace(sc, v0=np.ascontiguousarray(v0))


@pytest.mark.parametrize("sc", [sg.plate_clamped_x0(16, model="EP"), sg.plate_clamped_x0(21, model="SP"),
                                sg.plate_clamped_x0(15, model="FP")], ids=lambda sc: sc.name)
def test_rounds_end_below_the_target(sc):
    for seed in range(4):
        s = moving(sc, seed)
        xo, _ = osys.step(osys.from_scenario(s), s.x0, s.v0, 1)
        h = gb.create_from_scenario(s, precision="fp32_refine")
        assert gb.shell_info(h)["amg_levels"] == 1
        st = gb.shell_step(h, 1)
        x, _ = gb.shell_get_state(h)
        assert st["refine_rounds"] >= 1 and st["rel_residual"] <= 0.0708 * 3e-7
        # FP32 forces of a sheet moving through rest: below 1e-7 of the displacement
        assert np.linalg.norm(x - xo) <= 1e-7 * np.linalg.norm(xo - s.x0)
        # one round allowed: its result counts as before; a target near FP64's own rounding is reached as before
        for kw in ({"refine_max": 1, "refine_rtol": 1e-5}, {"refine_rtol": 1e-12}):
            h = gb.create_from_scenario(s, precision="fp32_refine", **kw)
            st = gb.shell_step(h, 1)
            assert st["status"] == 0 and st["rel_residual"] <= kw["refine_rtol"]


def test_chord_iterations_end_below_the_target():
    """Without a nonlinear tolerance each solve refers to its own residual; an error of one of them stays in the modes that
    the constant matrix overestimates."""
    for seed in range(4):
        s = moving(sg.plate_clamped_x0(16, model="EP"), seed)
        h = gb.create_from_scenario(s, precision="fp32_refine")
        gb.shell_set_nonlinear(h, 3, 0.0)
        st = gb.shell_step(h, 1)
        assert st["nl_iterations"] == 3 and st["rel_residual"] <= 0.0708 * 3e-7
