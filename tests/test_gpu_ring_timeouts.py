"""Bounded waits of the passes of 64-point lines and longer, whose tiles go through
a ring of buffers shared by several groups of threads: with every load expecting
more bytes than arrive (the test hook, no fault), each group gives up, the loads
that are under way are waited for, tensor memory is given back, the status is
KWGB_ERR_TIMEOUT, and the same results as before come from the same context
afterwards.  Sizes: more tiles per CTA than the ring holds."""

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

TIMEOUT = -5


@pytest.fixture(scope="module")
def kw():
    from paper_1408_4675_gb300 import build, kwgb
    build.build()
    kwgb.load()
    return kwgb


def _sim(kw, shape):
    sim = kw.Simulation(shape, (1e-4,) * 3, 2e-8, 1500.0, flags=kw.NONLINEAR)
    sim.set_medium(1500.0, 1000.0, 5.0)
    return sim


def _gradient(kw, sim, f):
    import torch
    outs = [torch.empty_like(f) for _ in range(3)]
    sim.apply_operator(kw.OP_GRAD_FWD, f, outs)
    torch.cuda.synchronize()
    return outs


@pytest.mark.parametrize("shape", [(64, 64, 1024), (256, 256, 256)])
def test_operator_gives_up_and_context_survives(kw, shape):
    import torch
    f = torch.from_numpy(np.random.default_rng(3).standard_normal(shape).astype(np.float32)).cuda()
    sim = _sim(kw, shape)
    before = _gradient(kw, sim, f)
    assert sim.status() == 0
    assert sim.L.kwgb_debug_wait_fault(sim.h, 1) == 0
    _gradient(kw, sim, f)
    assert sim.status() == TIMEOUT
    sim.close()
    sim = _sim(kw, shape)
    after = _gradient(kw, sim, f)
    assert sim.status() == 0
    assert all(torch.equal(a, b) for a, b in zip(before, after))
    sim.close()


def test_summing_pass_gives_up_and_context_survives(kw):
    shape = (64, 64, 512)
    src, obj = np.array([20 * 64 * 512 + 32 * 512 + 200]), np.array([22 * 64 * 512 + 32 * 512 + 203])

    def forward():
        sim = _sim(kw, shape)
        sim.add_source(src, np.full(4, 1e5, np.float32))
        sim.adjoint_forward(obj, 1, checkpoint_every=1)
        return sim

    sim = forward()
    before = sim.adjoint_backward()
    sim.close()
    sim = forward()
    assert sim.L.kwgb_debug_wait_fault(sim.h, 1) == 0
    with pytest.raises(kw.KwgbError) as e:
        sim.adjoint_backward()
    assert e.value.code == TIMEOUT
    sim.close()
    sim = forward()
    after = sim.adjoint_backward()
    assert all(np.array_equal(a, b) for a, b in zip(before, after))
    sim.close()
