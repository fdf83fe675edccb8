"""Accuracy of the Eq. 8 operator k^{y-2} in float32, where its power is steepest.

Tolerance: six transforms of at most 1024 points, 1.1e-7 relative L2 each at
random rounding (2.7e-7 together), and the power: the rounding of a base-2 logarithm
near 16 (5e-7 rms of it half a unit in the last place) times (2 - y) / 2 ln 2 = 0.31,
1.6e-7, in white noise weighted by k^{y-2}: sqrt(2.7^2 + 1.6^2) = 3.1e-7, taken as 3.3e-7.  A
logarithm a unit in the last place worse alone doubles the second term (4.2e-7)."""

import numpy as np
import pytest

import oracle
from helpers import rel_l2

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shape", [(64, 1024, 64), (1024, 64, 64), (64, 64, 64), (256, 256, 256)])
def test_power_of_k_is_as_accurate_as_float32_allows(shape):
    import torch
    from paper_1408_4675_gb300 import build, kwgb
    build.build()
    kwgb.load()
    nz, ny, nx = shape
    d, dt, y = (2e-4,) * 3, 3.6e-8, 1.1
    sim = kwgb.Simulation(shape, d, dt, 1650.0, flags=kwgb.ABSORBING, alpha_power=y)
    sim.set_medium(1500.0, 1000.0, 5.0, 1e-9)
    f = np.random.default_rng(17).standard_normal(shape).astype(np.float32)
    dev = torch.from_numpy(f).cuda()
    out = torch.empty_like(dev)
    sim.apply_operator(kwgb.OP_ABS_TAU, dev, [out])
    torch.cuda.synchronize()
    ref, = oracle.apply_operator(oracle.Grid(nx, ny, nz, *d, dt, 1650.0, flags=kwgb.ABSORBING, alpha_power=y),
                                 kwgb.OP_ABS_TAU, f.astype(np.float64))
    err = rel_l2(out.cpu().numpy(), ref)
    assert err <= 3.3e-7, err
    sim.close()
