"""What a call enqueues besides its steps, counted from the CUDA activity of repeated calls."""
import collections

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


def activity(fn):
    """Number of CUDA operations by kind: "Memcpy HtoD", "Memcpy DtoH", kernels by the start of their name."""
    import torch
    from torch.profiler import ProfilerActivity, profile
    counts = collections.Counter()
    for warm in (True, False):   # a process's first session may start too late to record anything
        with profile(activities=[ProfilerActivity.CUDA]) as p:
            if warm:
                torch.ones(8, device="cuda").sum().item()
            else:
                fn()
            torch.cuda.synchronize()
    for e in p.events():
        counts[e.name.split(" (")[0].strip()] += 1
    if counts["Memcpy DtoH"] == 0:   # every step call reads its statuses back
        pytest.skip("no CUDA activity recorded")
    return counts


def test_a_large_instance_alone_is_planned_once():
    """352 row blocks, more than the CTAs of one launch: the team is set by the machine, so that after the first
    measured call repeated calls upload no tables."""
    h = gb.create_from_scenario(sg.jittered_plate(300, steps=1), precision="fp32_refine")
    for _ in range(3):
        gb.shell_step(h, 1)
    assert activity(lambda: [gb.shell_step(h, 1) for _ in range(3)])["Memcpy HtoD"] == 0


def chord(sc, iters):
    h = gb.create_from_scenario(sc, precision="fp32_refine")
    gb.shell_set_nonlinear(h, iters, 0.0)   # no tolerance: every iteration runs
    return h


def test_a_group_of_chord_iterations_reads_the_statuses_at_once():
    """60 iterations are five groups: four reads between them and the call's own, two copies each, however many
    instances the batch holds."""
    b = gb.shell_batch_create(1 << 40)
    hs = [chord(sg.plate_clamped_x0(9 + k, model="EP"), 60) for k in range(8)]
    for h in hs:
        gb.shell_batch_admit(b, h)
    gb.shell_batch_step(b, 1)
    counts = activity(lambda: gb.shell_batch_step(b, 1))
    assert sum(n for k, n in counts.items() if "k_solve" in k) == 60
    assert counts["Memcpy DtoH"] <= 10
    gb.shell_batch_destroy(b)


def test_a_wait_that_gave_up_ends_the_chord_iterations():
    """A team whose barrier wait runs out (1 ns) launches no further group, commits nothing, and steps on after."""
    sc = sg.cylinder_panel(48, "FS", ny=40)
    ref, h = chord(sc, 60), chord(sc, 60)
    b = gb.shell_batch_create(1 << 40)
    slot = gb.shell_batch_admit(b, h)
    gb.shell_batch_step(b, 1)
    gb.shell_batch_set_wait_limit(b, 1)
    out = []
    counts = activity(lambda: out.append(gb.shell_batch_step(b, 1, check=False)))
    rc, stats = out[0]
    assert rc == gb.SHELL_ERR_TIMEOUT and stats[slot]["steps_done"] == 0
    assert sum(n for k, n in counts.items() if "k_solve" in k) == 12
    gb.shell_batch_set_wait_limit(b, 0)
    rc, stats = gb.shell_batch_step(b, 1)
    assert rc == 0 and stats[slot]["steps_done"] == 1
    gb.shell_step(ref, 2)
    for a, c in zip(gb.shell_get_state(ref), gb.shell_batch_get_states(b)):
        assert (a == c).all()
    gb.shell_batch_destroy(b)
