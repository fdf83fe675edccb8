"""Captures of steps that fail (the test hook: on the host, after the first step of
the capture): one capture of several steps is given up for good and single steps
are replayed, no capture at all means direct launches; results and launch counts
are those of an undisturbed run."""

import numpy as np
import pytest

from paper_1408_4675_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kw():
    from paper_1408_4675_gb300 import build, kwgb
    build.build()
    kwgb.load()
    return kwgb


# steps before the hook, failures asked for, of which are left after 45 steps more
@pytest.mark.parametrize("before,faults,left", [(2, 5, 4), (1, 1, 0), (1, 5, 4), (0, 5, 4), (40, 5, 5)])
def test_failed_capture_is_not_tried_again(kw, before, faults, left):
    cfg = inputs.make_config(2, n=32, n_steps=90)
    plain, ids = kw.from_config(cfg)
    plain.step(before + 45)
    sim, _ = kw.from_config(cfg)
    if before:
        sim.step(before)
    assert sim.L.kwgb_debug_capture_fault(sim.h, faults) == 0
    sim.step(45)
    assert sim.L.kwgb_debug_capture_fault(sim.h, 0) == left
    assert sim.steps_done == plain.steps_done and sim.launch_count == plain.launch_count and sim.status() == 0
    sim.step(1)
    plain.step(1)
    assert sim.launch_count == plain.launch_count
    assert np.array_equal(sim.read_field("p"), plain.read_field("p"))
    assert np.array_equal(sim.read(ids[0], kw.P_RMS), plain.read(ids[0], kw.P_RMS))
    sim.close()
    plain.close()
