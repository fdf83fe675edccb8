"""The reverse step's density pass on rows of every length class (components side
by side up to 512 reals, one after another beyond; row counts that fill a CTA and
that do not), lossless and absorbing, against the oracle adjoint: dJ/ds 2e-3
relative L2 (test_gpu_adjoint.py)."""

import numpy as np
import pytest

from helpers import oracle_from_config, rel_l2
from oracle import adjoint as oadj
from paper_1408_4675_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kw():
    from paper_1408_4675_gb300 import build, kwgb
    build.build()
    kwgb.load()
    return kwgb


@pytest.mark.parametrize("shape", [(16, 8, 8), (16, 16, 32), (16, 8, 128), (16, 8, 512), (16, 8, 1024)])
@pytest.mark.parametrize("absorbing", [False, True])
@pytest.mark.parametrize("k", [6, 20])
def test_density_pass_of_every_row_length_matches_oracle(kw, shape, absorbing, k):
    nz, ny, nx = shape
    steps, dx = 20, 1e-4
    c0 = inputs.smooth_random_field(shape, 1450.0, 1550.0, 51, 1.0)
    rho0 = inputs.smooth_random_field(shape, 950.0, 1050.0, 52, 1.0)
    c_ref = float(c0.max())
    dt = 0.3 * dx / c_ref
    idx = [np.sort(inputs.linear_index(shape, [5] * 2, [2 + e] * 2, [nx // 2 - 1, nx // 2])) for e in range(3)]
    sig = [1e5 * np.sin(2 * np.pi * 2e6 * (np.arange(steps) + 0.5) * dt + e) for e in range(3)]
    cfg = dict(shape=shape, d=(dx,) * 3, dt=dt, c_ref=c_ref, flags=1 | (2 if absorbing else 0), alpha_power=1.5, c0=c0,
               rho0=rho0, bona=5.0, alpha0=inputs.db_to_neper(0.8, 1.5) if absorbing else 0.0, p0=None, pml_size=(0, 0, 2),
               pml_alpha=(2.0,) * 3, sources=list(zip(idx, sig)), sensors=[])
    focal = inputs.linear_index(shape, [8, 8, 9], [3, 4, 3], [nx // 2] * 3)
    sim, _ = kw.from_config(cfg)
    J, g = sim.adjoint(focal, steps, checkpoint_every=k)
    sim.close()
    ref, _ = oracle_from_config(cfg)
    value, dJdp = oadj.mean_abs_pressure(focal, steps)
    rec = oadj.forward_record(ref, steps)
    Jo = value(rec)
    go = np.stack([v.sum(axis=0) for v in oadj.backward(ref, rec, dJdp)])
    assert abs(J - Jo) <= 1e-3 * abs(Jo)
    assert rel_l2(np.stack([v[0] for v in g]), go) <= 2e-3
