"""Device memory as an allocator leaves it: every allocation comes filled with NaN.
What a simulation computes is bitwise what it computes in cleared memory, so
nothing is read before it is written and no padding column reaches a valid one
(operators, lossless and absorbing steps, an adjoint, every precision form)."""

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


def _sim(kw, shape, flags, fill):
    import torch
    sim = kw.Simulation(shape, (1e-4,) * 3, 2e-8, 1550.0, (2, 2, 2), (2.0,) * 3, flags=flags, alpha_power=1.3,
                        use_torch_allocator=False)
    held = {}

    def alloc(nbytes, ctx):
        t = torch.full(((nbytes + 255) // 4,), fill, dtype=torch.float32, device="cuda")
        torch.cuda.synchronize()
        held[t.data_ptr()] = t
        return t.data_ptr()

    def free(p, ctx):
        held.pop(p, None)

    sim._test_refs = (kw.ALLOC_FN(alloc), kw.FREE_FN(free))
    assert sim.L.kwgb_set_allocator(sim.h, *sim._test_refs, None) == 0
    c0 = inputs.smooth_random_field(shape, 1450.0, 1550.0, 7, 1.0).astype(np.float32)
    sim.set_medium(c0, 1000.0, 5.0, 1e-9 if flags & 2 else None)
    return sim


def _run(kw, shape, flags, fill):
    import torch
    sim, out = _sim(kw, shape, flags, fill), []
    f = torch.from_numpy(np.random.default_rng(1).standard_normal(shape).astype(np.float32)).cuda()
    for op in (kw.OP_GRAD_FWD, kw.OP_ABS_ETA) if flags & 2 else (kw.OP_GRAD_BWD,):
        o = [torch.empty_like(f) for _ in range(3 if op < 2 else 1)]
        sim.apply_operator(op, f, o)
        torch.cuda.synchronize()
        out += [x.cpu().numpy() for x in o]
    nz, ny, nx = shape
    sim.add_source(np.array([nx * (ny * (nz // 2) + ny // 2) + nx // 2]), np.full(8, 1e5, np.float32))
    s = sim.add_sensor(None, kw.P_MAX | kw.P_RMS)
    if flags & (4 | 8):
        sim.step(3)
    else:
        out.append(np.array([sim.adjoint_forward(np.array([nx * ny * (nz // 2) + 5]), 3, checkpoint_every=2)]))
        out += [np.asarray(g) for g in sim.adjoint_backward()]
    out += [sim.read(s, kw.P_MAX), sim.read(s, kw.P_RMS), sim.read_field("p"), sim.read_field("ux")]
    assert sim.status() == 0
    sim.close()
    return out


@pytest.mark.parametrize("shape", [(16, 32, 8), (64, 64, 64), (32, 128, 128), (256, 64, 512), (16, 64, 1024)])
@pytest.mark.parametrize("flags", [1, 3, 3 | 4, 3 | 8])
def test_results_do_not_depend_on_what_memory_held(kw, shape, flags):
    for a, b in zip(_run(kw, shape, flags, float("nan")), _run(kw, shape, flags, 0.0)):
        assert np.isfinite(a).all() and np.array_equal(a, b)
