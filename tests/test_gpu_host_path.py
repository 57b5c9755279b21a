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
