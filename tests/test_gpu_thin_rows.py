"""Rows of 8 and 16 reals: one tile to a line, dealt out to the CTAs one by one
(fewer tiles than CTAs, as many, a remainder), and on large grids the 1024-point
y lines of 8-real rows on the one-column kernel.  Tolerances as for every
operator (test_gpu_parity.py): 1e-5 relative L2, 5e-5 relative L-inf."""

import numpy as np
import pytest

import oracle
from helpers import linf, rel_l2

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kw():
    from paper_1408_4675_gb300 import build, kwgb
    build.build()
    kwgb.load()
    return kwgb


@pytest.mark.parametrize("shape", [(64, 64, 8), (8, 128, 16), (128, 256, 16), (256, 512, 8), (64, 1024, 8), (512, 1024, 8)])
@pytest.mark.parametrize("op", [0, 1, 3])
def test_one_tile_to_a_line(kw, shape, op):
    import torch
    nz, ny, nx = shape
    d, dt, y = (1e-4, 1.25e-4, 0.8e-4), 2e-8, 1.3
    sim = kw.Simulation(shape, d, dt, 1500.0, flags=kw.ABSORBING, alpha_power=y)
    sim.set_medium(1500.0, 1000.0)
    f = np.random.default_rng(sum(shape) + op).standard_normal(shape).astype(np.float32)
    dev = torch.from_numpy(f).cuda()
    outs = [torch.empty_like(dev) for _ in range(3 if op < 2 else 1)]
    sim.apply_operator(op, dev, outs)
    torch.cuda.synchronize()
    ref = oracle.apply_operator(oracle.Grid(nx, ny, nz, *d, dt, 1500.0, flags=kw.ABSORBING, alpha_power=y), op,
                                f.astype(np.float64))
    for got, r in zip(outs, ref):
        got = got.cpu().numpy()
        assert rel_l2(got, r) <= 1e-5 and linf(got, r) <= 5e-5, (shape, op, rel_l2(got, r), linf(got, r))
    sim.close()
