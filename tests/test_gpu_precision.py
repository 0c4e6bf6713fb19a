"""Rounding that a step repeats in every node and every step, which no tolerance of a few
steps sees.

* Velocity: the collision hands on the momentum rho u times 12 (w/12).  A binary32 w/12 is
  off by up to 2^-25 (3.0e-8 at tau = 1), which grows the velocity by that much a step.
  Without it a decaying shear wave keeps its amplitude to the biases of the stencil weights
  (1/9 and 1/36 in binary32: 7.5e-9 each, in the viscous and pressure terms that change a
  wave of this length by far less than itself) and to random roundings: bound 1e-8 a step.
* Batched jobs start at rest: a standing density wave, half of whose energy is motion, so
  half of the bound.
* Density of a binary64 state: the moving populations are added first, so the sum is off by
  half an ulp of the density and the roundings of sums of the moving populations.
* LBM_FP32: the resident schedule is as accurate as the fused one.
"""
from __future__ import annotations

import numpy as np
import pytest

from helpers import gpu_problem, oracle_problem, seeded_mixture, smooth_rho

pytestmark = pytest.mark.gpu

FP64, FP32DEV, FP32 = 0, 1, 2
AUTO, THREEPASS, FUSED, MULTIPASS = 0, 1, 2, 3


@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("nc", [1, 4])
@pytest.mark.parametrize("precision,schedule,lattice,shape", [
    (FP32DEV, AUTO, 0, (1, 32, 32)), (FP32DEV, FUSED, 0, (1, 32, 32)), (FP32DEV, MULTIPASS, 0, (1, 32, 32)),
    (FP32DEV, MULTIPASS, 1, (4, 32, 8)), (FP32, AUTO, 0, (1, 32, 32)), (FP32, FUSED, 0, (1, 32, 32)),
    (FP64, THREEPASS, 0, (1, 32, 32))],
    ids=["dev-resident", "dev-fused", "dev-multipass", "dev-d3q19", "fp32-resident", "fp32-fused", "fp64"])
def test_amplitude_of_a_shear_wave(precision, schedule, lattice, shape, nc, tau):
    steps = 100
    c = seeded_mixture(540 + nc, nc, lattice, shape, Tfac=1.5)
    rng = np.random.default_rng(540)
    rho = (0.15 / nc) / np.asarray(c["b"])[:, None, None, None] * np.ones((nc,) + shape)
    rho *= 1 + 1e-3 * rng.uniform(-1, 1, rho.shape)  # rounds differently in every node
    D = 2 + lattice
    y = 2 * np.pi * (np.arange(shape[1]) + 0.3) / shape[1]
    u = np.zeros((D,) + shape)
    u[0] = 0.02 * np.cos(y)[None, :, None]

    def velocity(**kw):
        with gpu_problem(c, lattice, shape, tau=tau, tune=0, **kw) as gp:
            gp.init_fields(rho, u)
            gp.step(steps)
            return gp.moments(want=("u",))["u"][0]

    ref = velocity(precision=FP64, schedule=THREEPASS)
    got = velocity(precision=precision, schedule=schedule)
    wave = np.cos(y)[None, :, None]
    amp = [(v * wave).sum() for v in (ref, got)]
    assert abs(amp[1] / amp[0] - 1) < 1e-8 * steps, amp[1] / amp[0] - 1


@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_amplitude_of_a_batched_density_wave(tau):
    from paper_2306_10652_gb300 import lbmfug
    nc, shape, parts = 3, (1, 4, 64), (100, 50, 50, 50, 50)
    c = seeded_mixture(550, nc, 0, shape, Tfac=1.5)
    rng = np.random.default_rng(550)
    wave = np.cos(2 * np.pi * (np.arange(shape[2]) + 0.3) / shape[2])[None, None, :]
    rho = (0.15 / nc) / np.asarray(c["b"])[:, None, None, None] * (1 + 0.02 * wave[None])
    rho = rho * (1 + 1e-3 * rng.uniform(-1, 1, (nc,) + shape))
    with gpu_problem(c, 0, shape, tau=tau, precision=FP64) as gp, \
            lbmfug.Batch(c["a"], c["b"], c["omega"], c["kij"], tau, [(c["T"], rho[:, 0])], precision=FP32DEV) as bt:
        gp.init_fields(rho)
        start, done = (rho * wave).sum(axis=(1, 2, 3)), 0
        for n in parts:
            gp.step(n)
            bt.run(max_steps=n, check_every=n, tol=0.0)
            done += n
            ref = (gp.moments(want=("rho",))["rho"] * wave).sum(axis=(1, 2, 3))
            got = (bt.state(0)["rho"][:, None] * wave).sum(axis=(1, 2, 3))
            assert (np.abs(got - ref) <= 0.5e-8 * done * start).all(), (done, (got - ref) / start)


@pytest.mark.parametrize("schedule,lattice,shape", [(AUTO, 0, (1, 8, 21)), (THREEPASS, 0, (1, 20, 33)),
                                                    (THREEPASS, 1, (5, 6, 7))], ids=["resident", "d2q9", "d3q19"])
def test_binary64_density_rounds_once(schedule, lattice, shape):
    nc = 3
    c = seeded_mixture(560, nc, lattice, shape, Tfac=1.2)
    rho = smooth_rho(560, c, shape)
    with gpu_problem(c, lattice, shape, schedule=schedule) as gp:
        gp.init_fields(rho)
        gp.step(5)
        g = gp.get_state()
        got = gp.moments(want=("rho",))["rho"]
    ref = g.astype(np.longdouble).sum(axis=1)
    moving = np.abs(g[:, 1:]).sum(axis=1)
    bound = 0.5 * np.spacing(np.abs(got)) + (g.shape[1] - 2) * 0.5 * np.spacing(moving)
    assert (np.abs(got - ref) <= bound).all()
    assert (bound < np.spacing(np.abs(got))).mean() > 0.5  # the case is met: small moving populations


@pytest.mark.parametrize("nc,seed", [(2, 571), (4, 572), (8, 573)])
def test_resident_binary32_is_as_accurate_as_fused(nc, seed):
    shape, steps = (1, 4, 128), 200
    c = seeded_mixture(seed, nc, 0, shape, Tfac=1.2)
    rho = smooth_rho(seed, c, shape)
    orc = oracle_problem(c, 0, shape)
    ref = orc.step(orc.init_equilibrium(rho), steps).sum(axis=1)
    err = {}
    for schedule in (AUTO, FUSED):
        with gpu_problem(c, 0, shape, precision=FP32, schedule=schedule, tune=0) as gp:
            gp.init_fields(rho)
            gp.step(steps)
            err[schedule] = np.sqrt(((gp.moments(want=("rho",))["rho"] - ref) ** 2).mean())
    assert err[AUTO] <= 1.25 * err[FUSED], err
