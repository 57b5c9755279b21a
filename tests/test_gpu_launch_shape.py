"""Launch shapes set by the caller or tried by the autotuner."""
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


@pytest.mark.parametrize("precision", ["fp64", "fp32_refine"])
def test_the_share_sets_the_team_of_an_instance_alone(precision):
    """Shares at which a second CTA costs more than it saves in the planner's model (25 and more) give one CTA."""
    for share, one in ((1.0, False), (20.0, False), (30.0, True)):
        h = gb.create_from_scenario(sg.cylinder_panel(48, "FS", ny=40), precision=precision)
        b = gb.shell_batch_create(1 << 40)
        slot = gb.shell_batch_admit(b, h)
        gb.shell_batch_set_launch(b, 2, share)
        for _ in range(2):
            rc, stats = gb.shell_batch_step(b, 1)
            assert rc == 0 and (stats[slot]["team_ctas"] == 1) == one, share
        gb.shell_batch_destroy(b)


def test_the_autotuner_tries_three_occupancies_in_fp32():
    b = gb.shell_batch_create(1 << 40)
    hs = [gb.create_from_scenario(sc, precision="fp32_refine") for sc in sg.mixed_batch(6, seed=3, side_lo=6, side_hi=40)]
    for h in hs:
        gb.shell_batch_admit(b, h)
    info = gb.shell_batch_autotune(b, 1)
    assert all(ms > 0.0 for ms in info["trial_ms"][:9])
    assert info["ctas_per_sm"] in (2, 3, 4)
    gb.shell_batch_destroy(b)


# 64, 72, 128 and 132 vertices; a narrow band (129 vertices) is one row block for the direct Newton solve in any case
@pytest.mark.parametrize("nx,ny,newton,one", [(7, 7, True, True), (7, 8, True, False), (15, 7, False, True),
                                              (11, 10, False, False), (42, 2, False, True)])
def test_small_fp64_instances_take_one_cta(nx, ny, newton, one):
    sc = sg.cylinder_panel(nx, "FS", ny=ny)

    def make():
        h = gb.create_from_scenario(sc, precision="fp64", pcg_rtol=1e-8)
        if newton:
            gb.shell_set_nonlinear(h, 3, 0.0)
            gb.shell_set_newton(h, True)
        return h

    states = []
    for batch in (1, 3):
        hs = [make() for _ in range(batch)]
        b = gb.shell_batch_create(1 << 40)
        slots = [gb.shell_batch_admit(b, h) for h in hs]
        for _ in range(2):
            rc, stats = gb.shell_batch_step(b, 1)
            assert rc == 0 and all((stats[k]["team_ctas"] == 1) == one for k in slots)
        states.append(gb.shell_batch_get_states(b)[0][:sc.n_verts])
        gb.shell_batch_destroy(b)
    h = make()
    st = gb.shell_step_noalloc(h, 2)
    assert (st["team_ctas"] == 1) == one
    states.append(gb.shell_get_state(h)[0])
    assert (states[0] == states[1]).all() and (states[0] == states[2]).all()
