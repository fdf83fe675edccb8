"""Source lists of every kind at the sizes where the row loop can go wrong: rows
that are full of points (several batches per thread), points with several
contributions of different lengths, rows with one point, short and long rows
(one and two warps per row).  Against the float64 oracle, tolerance of the
short heterogeneous runs (1e-4 / 5e-4, test_gpu_parity.py)."""

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


@pytest.mark.parametrize("shape", [(16, 8, 8), (8, 16, 64), (8, 8, 256), (8, 8, 1024)])
@pytest.mark.parametrize("mode,amp", [(0, 1e5), (2, 1e9), (4, 2e4)])
def test_full_rows_and_repeated_points_match_oracle(kw, shape, mode, amp):
    nz, ny, nx = shape
    rng = np.random.default_rng(nx + mode)
    c0 = inputs.smooth_random_field(shape, 1450.0, 1550.0, 91, 1.0)
    rho0 = inputs.smooth_random_field(shape, 950.0, 1050.0, 92, 1.0)
    dx, c_ref = 1e-4, float(c0.max())
    dt, steps = 0.3 * dx / c_ref, 6
    sig = lambda rows, nt: amp * rng.uniform(-1.0, 1.0, (rows, nt))
    x = np.arange(nx)
    full = inputs.linear_index(shape, np.full(nx, 3), np.full(nx, 2), x)           # a whole row, its own signals
    pairs = inputs.linear_index(shape, np.full(nx, 3), np.full(nx, 2), x // 2)      # points twice in one source
    single = inputs.linear_index(shape, [5], [4], [nx - 1])
    sources = [(full, sig(nx, 6), mode), (pairs, sig(1, 3), mode), (single, sig(1, 6), mode), (full[::3], sig(1, 5), mode)]
    cfg = dict(shape=shape, d=(dx,) * 3, dt=dt, c_ref=c_ref, flags=3, alpha_power=1.3, c0=c0, rho0=rho0, bona=6.0,
               alpha0=1e-9, p0=None, pml_size=(0, 0, 0), pml_alpha=(0.0,) * 3, sources=sources, sensors=[(None, 1)])
    sim, ids = kw.from_config(cfg)
    sim.step(steps)
    ref, rids = oracle_from_config(cfg)
    ref.step(steps)
    got, exp = sim.read(ids[0], kw.P_MAX), ref.read(rids[0], 1)
    assert rel_l2(got, exp) <= 1e-4 and linf(got, exp) <= 5e-4, (rel_l2(got, exp), linf(got, exp))
    p = sim.read_field("p")
    assert rel_l2(p, ref.p) <= 1e-4, rel_l2(p, ref.p)
    sim.close()
