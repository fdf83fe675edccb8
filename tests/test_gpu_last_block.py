"""The last block of a spectrum's columns (which is never full): from 64 MB on its
tiles come through a tensor map that ends with the last column, below that with
the padding beside it, which holds anything.  Operators on either side of that
line, for a Nyquist column alone, for a whole spectrum in one block, and for
lines of the short and of the tensor-core passes, with the scratch spectra's
padding written over by an initial pressure first.

Tolerances as for every operator (test_gpu_parity.py): 1e-5 relative L2 and 5e-5
relative L-inf against float64, the bfloat16 form 1e-4 / 1e-3."""

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


# (nz, ny, nx): 67, 67, 71, 75 and 84 MB spectra, then 34, 34 and 50 MB
@pytest.mark.parametrize("shape", [(256, 1024, 32), (1024, 512, 8), (64, 256, 1024), (16, 1024, 512), (256, 256, 256),
                                   (1024, 256, 8), (256, 1024, 16), (1024, 128, 64)])
@pytest.mark.parametrize("form,op", [(0, 0), (0, 1), (0, 2), (8, 0), (4, 3)])
def test_last_block_clipped_or_padded(kw, shape, form, op):
    import torch
    if form and min(shape[:2]) < 16:
        pytest.skip("the tensor-core forms take lines of 16 points and more")
    nz, ny, nx = shape
    d, dt, y = (1e-4, 1.25e-4, 0.8e-4), 2e-8, 1.3
    sim = kw.Simulation(shape, d, dt, 1500.0, flags=kw.ABSORBING | form, alpha_power=y)
    sim.set_medium(1500.0, 1000.0)
    f = np.random.default_rng(sum(shape) + op).standard_normal(shape).astype(np.float32)
    sim.set_initial_pressure(1e30 * f)
    dev = torch.from_numpy(f).cuda()
    outs = [torch.empty_like(dev) for _ in range(3 if op < 2 else 1)]
    sim.apply_operator(op, dev, outs)
    torch.cuda.synchronize()
    ref = oracle.apply_operator(oracle.Grid(nx, ny, nz, *d, dt, 1500.0, flags=kw.ABSORBING, alpha_power=y), op,
                                f.astype(np.float64))
    l2, li = (1e-4, 1e-3) if form == 4 else (1e-5, 5e-5)
    for got, r in zip(outs, ref):
        got = got.cpu().numpy()
        assert rel_l2(got, r) <= l2 and linf(got, r) <= li, (shape, op, rel_l2(got, r), linf(got, r))
    sim.close()
