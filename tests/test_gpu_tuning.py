"""What the launch-geometry tuners remember: a choice serves the problems that run the
same kernel at the same load, and no others.  Trials are launches, which are counted."""
from __future__ import annotations

import numpy as np
import pytest

from helpers import gpu_problem, seeded_mixture, smooth_rho

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [2, 1], ids=["fp32", "fp32dev"])
def test_batch_tuner_knows_kernel_and_load(precision):
    from paper_2306_10652_gb300 import lbmfug
    nc, shape = 2, (1, 3, 37 + precision)
    c = seeded_mixture(510, nc, 0, shape)
    rho = smooth_rho(510, c, shape)[:, 0]

    def trials(njobs, tau):
        with lbmfug.Batch(c["a"], c["b"], c["omega"], c["kij"], tau, [(c["T"], rho)] * njobs, precision=precision) as b:
            return b.info()["launches"]

    for njobs, tau in ((8, 1.0), (700, 1.0), (8, 0.8), (700, 0.8)):  # one job per SM, and four or more
        assert trials(njobs, tau) > 0, (njobs, tau)
        assert trials(njobs, tau) == 0, (njobs, tau)


@pytest.mark.parametrize("precision,launches", [(2, 1), (1, 2)], ids=["fp32", "fp32dev"])
def test_step_tuner_knows_the_kernel(precision, launches):
    nc, shape = 3, (1, 22, 150 + precision)
    c = seeded_mixture(515, nc, 0, shape, Tfac=1.2)
    rho = smooth_rho(515, c, shape)

    def first_step(tau):
        with gpu_problem(c, 0, shape, tau=tau, precision=precision, schedule=2) as gp:
            gp.init_fields(rho)
            n = gp.launch_count()
            gp.step(1)
            return gp.launch_count() - n, gp.get_state()

    for tau in (1.0, 0.8):
        n, tuned = first_step(tau)
        assert n > launches, tau
        n, again = first_step(tau)
        assert n == launches and np.array_equal(tuned, again), tau


@pytest.mark.parametrize("nc", [3, 6])
def test_batch_returns_to_the_tuned_size(nc):
    from paper_2306_10652_gb300 import lbmfug
    shape = (1, 4, 200)
    c = seeded_mixture(520 + nc, nc, 0, shape, Tfac=1.2)
    rho = smooth_rho(520 + nc, c, shape)[:, 0]
    with lbmfug.Batch(c["a"], c["b"], c["omega"], c["kij"], 1.0, [(c["T"], rho)] * 300) as b:
        tuned = b.info()
        for threads in (128, 256, 512):
            b.set_threads(threads)
            assert b.info()["threads"] == threads
            b.set_threads(tuned["threads"])
            assert {k: b.info()[k] for k in ("threads", "ctas")} == {k: tuned[k] for k in ("threads", "ctas")}
        for threads in (64, 100, 2048):
            with pytest.raises(lbmfug.LbmError):
                b.set_threads(threads)
        b.run(max_steps=10, check_every=10, tol=0.0)
        assert np.isfinite(b.state(0)["rho"]).all()
