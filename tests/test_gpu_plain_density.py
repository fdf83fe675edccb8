"""The density pass of lossless media on short rows, on either side of the rule that
takes small grids to its side-by-side form (16 plain CTAs per SM), and runs of just
enough steps to replay several of them per graph (the first step is launched
directly).  Against the float64 oracle, tolerance of the short heterogeneous runs
(1e-4 / 5e-4, test_gpu_parity.py); replayed steps bitwise against single ones."""

import numpy as np
import pytest

from helpers import linf, oracle_from_config, rel_l2
from paper_1408_4675_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kw():
    from paper_1408_4675_gb300 import build, kwgb
    build.build()
    kwgb.load()
    return kwgb


def _config(kw, shape, flags, steps):
    nz, ny, nx = shape
    c0 = inputs.smooth_random_field(shape, 1450.0, 1550.0, 61, 1.0)
    dx, c_ref = 1e-4, float(c0.max())
    dt = 0.3 * dx / c_ref
    plane = inputs.linear_index(shape, np.full((ny, nx), 2), np.arange(ny)[:, None], np.arange(nx)[None, :]).ravel()
    sig = 1e5 * np.sin(2 * np.pi * 2e6 * (np.arange(steps) + 0.5) * dt)
    return dict(shape=shape, d=(dx,) * 3, dt=dt, c_ref=c_ref, flags=flags, alpha_power=1.3, c0=c0, rho0=1000.0, bona=6.0,
                alpha0=1e-9 if flags & 2 else 0.0, p0=None, pml_size=(0, 0, 2), pml_alpha=(2.0,) * 3,
                sources=[(plane, sig)], sensors=[(None, kw.P_MAX | kw.P_RMS | kw.P_MIN)])


# plain CTAs per SM (152): 27, 13.5, 27, 13.5, 54
@pytest.mark.parametrize("shape", [(256, 128, 128), (128, 128, 128), (512, 256, 32), (256, 256, 32), (1024, 1024, 8)])
@pytest.mark.parametrize("flags", [0, 1])
def test_lossless_density_pass_on_both_sides_of_the_rule(kw, shape, flags):
    steps = 3
    cfg = _config(kw, shape, flags, steps)
    sim, (sid,) = kw.from_config(cfg)
    sim.step(steps)
    ref, (rid,) = oracle_from_config(cfg)
    ref.step(steps)
    for which in (kw.P_MAX, kw.P_RMS, kw.P_MIN):
        got, exp = sim.read(sid, which), ref.read(rid, which)
        assert rel_l2(got, exp) <= 1e-4 and linf(got, exp) <= 5e-4, (which, rel_l2(got, exp), linf(got, exp))
    sim.close()


@pytest.mark.parametrize("steps", [33, 34, 36, 37])
def test_first_replay_of_several_steps(kw, steps):
    cfg = _config(kw, (16, 16, 32), 3, steps)
    many, (sid,) = kw.from_config(cfg)
    many.step(steps)
    one, _ = kw.from_config(cfg)
    for _ in range(steps):
        one.step(1)
    assert many.steps_done == one.steps_done == steps and many.launch_count == one.launch_count
    for f in ("p", "uy", "rhox"):
        assert np.array_equal(many.read_field(f), one.read_field(f))
    assert np.array_equal(many.read(sid, kw.P_RMS), one.read(sid, kw.P_RMS))
    many.close()
    one.close()
