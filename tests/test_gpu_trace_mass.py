"""Component mass over a step in which single populations exceed the density of the node
that they leave or enter: a trace component in every other column, or pair of columns,
whose terms in grad rho_i come from the columns between.  In pairs of columns, beside a
moving fluid, they are 2^24 times the density and more, which a sum that is exact only
for smaller terms loses.

The density moves by what left and arrived, every population with its rounding error:
what is lost is the rounding of the sum of these errors, at most Q times 2^-25 of Q
errors of 2^-25 of the largest partial sum for what left and for what arrived (Q = 18),
and a few roundings of the pair's low word: below 256 x 2^-48 of the largest value that a
node's sums meet.  A density that is itself lost to a population beside it is 2^-34 of the
largest here.
"""
from __future__ import annotations

import numpy as np
import pytest

from helpers import gpu_problem, seeded_mixture, smooth_rho

pytestmark = pytest.mark.gpu

FP32DEV, FP32 = 1, 2


@pytest.mark.parametrize("width,trace,speed", [(1, 1e-10, 0.0), (2, 2e-11, 0.1)], ids=["columns", "pairs"])
@pytest.mark.parametrize("tau", [1.0, 0.8])
@pytest.mark.parametrize("nc", [2, 3])
@pytest.mark.parametrize("precision,schedule,lattice,shape", [
    (FP32DEV, 3, 1, (6, 5, 24)), (FP32DEV, 3, 0, (1, 11, 40)), (FP32, 1, 1, (6, 5, 24)), (FP32DEV, 1, 0, (1, 11, 40))],
    ids=["multipass-d3q19", "multipass-d2q9", "threepass-d3q19", "threepass-d2q9"])
def test_mass_with_populations_above_the_density(precision, schedule, lattice, shape, nc, tau, width, trace, speed):
    c = seeded_mixture(500 + nc, nc, lattice, shape, Tfac=1.2)
    rho = smooth_rho(500 + nc, c, shape, 0.1, 0.3)
    few = np.arange(shape[2]) // width % 2 == 0
    rho[1:, :, :, few] *= trace
    u = np.zeros((2 + lattice,) + shape)
    u[0] = speed
    with gpu_problem(c, lattice, shape, tau=tau, precision=precision, schedule=schedule) as gp:
        gp.init_fields(rho, u)
        before = gp.mass()
        gp.step(1)
        g = gp.get_state()
        after = gp.mass()
    assert np.isfinite(g).all()
    moving = np.abs(g[:, 1:]).max(axis=1)
    assert (moving[1:][..., few] > 1e3 * rho[1:][..., few]).any()  # the case is met
    N = rho[0].size
    bound = 256 * 2.0**-48 * N * np.maximum(rho.reshape(nc, -1).max(axis=1), np.abs(g).reshape(nc, -1).max(axis=1))
    assert (np.abs(after - before) <= bound).all(), (after - before, bound)
