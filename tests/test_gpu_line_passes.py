"""The strided passes of 64- to 1024-point lines (tiles handled in turn by the
thread groups of one CTA out of a ring of buffers) and the blocked spectra, at
the sizes where they can go wrong: rings that wrap, ragged last tiles, one
tile per CTA, kappa arguments beyond its short series.

Tolerances: one float32 FFT round trip against float64, 1e-5 relative L2 and
5e-5 relative L-inf, as for every operator (test_gpu_parity.py); dJ/ds 2e-3
relative L2 against the oracle adjoint (test_gpu_adjoint.py)."""

import numpy as np
import pytest

import oracle
from helpers import linf, rel_l2
from paper_1408_4675_gb300 import inputs

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def kw():
    from paper_1408_4675_gb300 import build, kwgb
    build.build()
    kwgb.load()
    return kwgb


def _check(kw, shape, op, dt=2e-8, seed=0):
    import torch
    nz, ny, nx = shape
    d, y = (1e-4, 1.25e-4, 0.8e-4), 1.3
    sim = kw.Simulation(shape, d, dt, 1500.0, flags=kw.ABSORBING, alpha_power=y)
    sim.set_medium(1500.0, 1000.0)
    f = np.random.default_rng(seed + sum(shape) + op).standard_normal(shape).astype(np.float32)
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


# (nz, ny, nx): tiles per CTA from below one to beyond twice the ring of every line length on either axis
@pytest.mark.parametrize("shape", [(64, 64, 1024), (128, 32, 1024), (16, 128, 512), (256, 64, 512), (64, 256, 256),
                                   (512, 64, 256), (128, 512, 128), (1024, 32, 128), (64, 1024, 64), (64, 128, 8),
                                   (512, 8, 8), (1024, 1024, 8)])
@pytest.mark.parametrize("op", [0, 1, 2, 3])
def test_operator_on_rings_of_every_length(kw, shape, op):
    _check(kw, shape, op)


@pytest.mark.parametrize("shape", [(64, 16, 16), (16, 256, 32), (512, 8, 16), (1024, 8, 64)])
@pytest.mark.parametrize("dt", [4e-8, 1.2e-7])              # largest (c_ref k dt / 2)^2: about 4.5 and 40
@pytest.mark.parametrize("op", [0, 1])
def test_operator_beyond_the_short_kappa_series(kw, shape, dt, op):
    _check(kw, shape, op, dt=dt)


def test_summing_pass_over_a_wrapping_ring_matches_oracle(kw):
    """The adjoint's z passes on 256-point lines with seven tiles per CTA."""
    from oracle import adjoint as oadj
    from helpers import oracle_from_config
    shape, steps, zs = (256, 64, 256), 20, 12
    c0 = inputs.smooth_random_field(shape, 1450.0, 1550.0, 81, 1.5)
    dx, c_ref = 1e-4, float(c0.max())
    dt = 0.3 * dx / c_ref
    idx = [np.sort(inputs.linear_index(shape, [zs] * 2, [30 + e, 31 + e], [126 + e, 127 + e])) for e in range(3)]
    sig = [1e5 * np.sin(2 * np.pi * 2e6 * (np.arange(steps) + 0.5) * dt + e) for e in range(3)]
    cfg = dict(shape=shape, d=(dx,) * 3, dt=dt, c_ref=c_ref, flags=1, alpha_power=1.5, c0=c0, rho0=1000.0, bona=5.0,
               alpha0=0.0, p0=None, pml_size=(4, 4, 10), pml_alpha=(2.0,) * 3, sources=list(zip(idx, sig)), sensors=[])
    focal = inputs.box_mask(shape, (zs + 3, 32, 128), 1)
    sim, _ = kw.from_config(cfg)
    J, g = sim.adjoint(focal, steps, checkpoint_every=steps)
    sim.close()
    ref, _ = oracle_from_config(cfg)
    value, dJdp = oadj.mean_abs_pressure(focal, steps)
    rec = oadj.forward_record(ref, steps)
    Jo = value(rec)
    go = np.stack([v.sum(axis=0) for v in oadj.backward(ref, rec, dJdp)])
    assert abs(J - Jo) <= 1e-3 * abs(Jo)
    assert rel_l2(np.stack([v[0] for v in g]), go) <= 2e-3


@pytest.mark.parametrize("shape", [(8, 16, 64), (16, 8, 128), (8, 8, 1024)])
def test_snapshot_holds_the_spectrum_as_whole_rows(kw, shape):
    """A snapshot's pressure spectrum is [nz][ny][nx/2 + 1 rounded up to 16] complex,
    whatever the layout on the device."""
    nz, ny, nx = shape
    sim = kw.Simulation(shape, (1e-4,) * 3, 2e-8, 1500.0)
    sim.set_medium(1500.0, 1000.0)
    p0 = np.random.default_rng(5).standard_normal(shape).astype(np.float32)
    sim.set_initial_pressure(p0)
    buf = sim.save_state()
    n, nhp = nz * ny * nx, (nx // 2 + 1 + 15) // 16 * 16
    assert buf.size == 80 + 6 * 4 * n + 8 * nz * ny * nhp
    P = buf[80 + 24 * n:].view(np.complex64).reshape(nz, ny, nhp)[:, :, :nx // 2 + 1]
    assert np.linalg.norm(P - np.fft.rfft(p0.astype(np.float64), axis=2)) <= 1e-6 * np.linalg.norm(P)
    sim.load_state(buf)
    assert np.array_equal(sim.save_state()[80:80 + 24 * n], buf[80:80 + 24 * n])
    again = sim.save_state()[80 + 24 * n:].view(np.complex64).reshape(nz, ny, nhp)[:, :, :nx // 2 + 1]
    assert np.array_equal(again, P)
    sim.close()
