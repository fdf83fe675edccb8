"""The paths that small grids take, at the edges of their rules: x_dens with its
three row transforms side by side (rows of 8 to 128 reals, row counts that do not
fill a CTA, beside the plain form of grids just beyond the rule), runs long
enough to replay several steps per graph, and sensors whose rows are full of
entries.  Against the float64 oracle, tolerance of the short heterogeneous runs
(1e-4 / 5e-4, test_gpu_parity.py)."""

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


def _config(kw, shape, flags, steps, mass=True):
    nz, ny, nx = shape
    c0 = inputs.smooth_random_field(shape, 1450.0, 1550.0, 61, 1.0)
    rho0 = inputs.smooth_random_field(shape, 950.0, 1050.0, 62, 1.0)
    dx, c_ref = 1e-4, float(c0.max())
    dt = 0.3 * dx / c_ref
    plane = inputs.linear_index(shape, np.full((ny, nx), 2), np.arange(ny)[:, None], np.arange(nx)[None, :]).ravel()
    sig = 1e5 * np.sin(2 * np.pi * 2e6 * (np.arange(steps) + 0.5) * dt)
    xz = inputs.linear_index(shape, np.arange(nz)[:, None], np.full((nz, nx), ny // 2), np.arange(nx)[None, :]).ravel()
    rec = kw.P_MAX | kw.P_RMS | kw.P_MIN
    return dict(shape=shape, d=(dx,) * 3, dt=dt, c_ref=c_ref, flags=flags, alpha_power=1.3, c0=c0, rho0=rho0, bona=6.0,
                alpha0=1e-9 if flags & 2 else 0.0, p0=None if mass else 1e4 * (c0 - 1500.0), pml_size=(0, 0, 2), pml_alpha=(2.0,) * 3,
                sources=[(plane, sig)] if mass else [], sensors=[(None, rec), (xz, rec), (xz[::-1].copy(), rec)])


@pytest.mark.parametrize("shape", [(8, 8, 8), (16, 8, 16), (32, 16, 32), (64, 128, 8), (32, 64, 64), (64, 32, 128), (16, 64, 128),
                                   (64, 256, 32)])
@pytest.mark.parametrize("flags", [0, 1, 3])
def test_rows_side_by_side_and_full_sensors_match_oracle(kw, shape, flags):
    steps = 8
    cfg = _config(kw, shape, flags, steps)
    sim, ids = kw.from_config(cfg)
    sim.step(steps)
    ref, rids = oracle_from_config(cfg)
    ref.step(steps)
    for i, r in zip(ids, rids):
        for which in (kw.P_MAX, kw.P_RMS, kw.P_MIN):
            got, exp = sim.read(i, which), ref.read(r, which)
            assert rel_l2(got, exp) <= 1e-4 and linf(got, exp) <= 5e-4, (which, rel_l2(got, exp), linf(got, exp))
    sim.close()


@pytest.mark.parametrize("steps", [32, 35, 70])
def test_steps_replayed_together_equal_single_steps(kw, steps):
    cfg = _config(kw, (16, 16, 32), 3, steps)
    many, ids = kw.from_config(cfg)
    many.step(steps)
    one, _ = kw.from_config(cfg)
    for _ in range(steps):
        one.step(1)
    assert many.steps_done == one.steps_done == steps and many.launch_count == one.launch_count
    for f in ("p", "ux", "rhoz"):
        assert np.array_equal(many.read_field(f), one.read_field(f))
    for i in ids:
        assert np.array_equal(many.read(i, kw.P_RMS), one.read(i, kw.P_RMS))
    many.close()
    one.close()
