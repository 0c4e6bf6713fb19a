"""Device memory of a handle, through the allocation hooks: what a box of Nc components
takes per node, odd and even Nc alike, and that the estimate of the served form covers it."""
from __future__ import annotations

import ctypes

import numpy as np
import pytest

from helpers import gpu_problem, seeded_mixture

pytestmark = pytest.mark.gpu

FP64, FP32DEV, FP32 = 0, 1, 2
AUTO, FUSED, MULTIPASS = 0, 2, 3


def node_bytes(lattice, precision, schedule, nc):
    """State (two buffers), densities and ln f, psi, lap psi and momentum in binary64; mu and
    psi (LBM_FP32DEV) and the sums of the departures in binary32: the most that a node
    may take."""
    D, Q = ((2, 9), (3, 19))[lattice]
    if precision == FP64:
        return 2 * nc * Q * 8 + 16 * nc + 8 * (2 + D)
    b = 2 * nc * ((Q - 1) * 4 + 8) + 16 * nc + 8 * (2 + D) + 8 * nc
    if precision == FP32DEV:
        b += 8 * nc + (8 if schedule == MULTIPASS else 0)
    return b


@pytest.mark.parametrize("nc", [1, 2, 3, 7])
@pytest.mark.parametrize("precision,schedule,lattice,shape", [
    (FP32, FUSED, 0, (1, 512, 510)), (FP32DEV, FUSED, 0, (1, 512, 510)), (FP32DEV, MULTIPASS, 0, (1, 512, 510)),
    (FP32DEV, MULTIPASS, 1, (64, 64, 62)), (FP64, AUTO, 0, (1, 512, 510)), (FP64, AUTO, 1, (64, 64, 62)),
    (FP32, AUTO, 1, (64, 64, 62))],
    ids=["fp32-fused", "fp32dev-fused", "multipass-d2q9", "multipass-d3q19", "fp64-d2q9", "fp64-d3q19", "fp32-d3q19"])
def test_bytes_of_a_handle(precision, schedule, lattice, shape, nc):
    import torch
    from paper_2306_10652_gb300 import lbmfug
    held = {}

    @lbmfug.ALLOC_FN
    def alloc(n, _):
        t = torch.empty(n, dtype=torch.uint8, device="cuda")
        held[t.data_ptr()] = t
        return t.data_ptr()

    @lbmfug.FREE_FN
    def free(ptr, n, _):
        assert held.pop(ptr).numel() == n

    c = seeded_mixture(530 + nc, nc, lattice, shape, Tfac=1.2)
    N = int(np.prod(shape))
    rho = np.full((nc,) + shape, 0.2 / nc) / np.asarray(c["b"])[:, None, None, None]
    u = np.zeros(((2, 3)[lattice],) + shape)
    with gpu_problem(c, lattice, shape, precision=precision, schedule=schedule, tune=0) as gp:
        opt = lbmfug.lbm_options()
        lbmfug._lib.lbm_options_default(ctypes.byref(opt))
        opt.precision, opt.schedule, opt.tune, opt.alloc, opt.free = precision, schedule, 0, alloc, free
        assert lbmfug._lib.lbm_set_options(gp._h, ctypes.byref(opt)) == 0
        gp.init_fields(rho, u)
        gp.step(2)
        m = gp.moments()
        total = sum(t.numel() for t in held.values())
    assert not held
    assert np.abs(m["rho"] / rho - 1).max() < 1e-6 and np.abs(m["u"]).max() < 1e-6
    # tables, partial sums and flags: below 512 KB
    assert total <= node_bytes(lattice, precision, schedule, nc) * N + (1 << 19), total / N
    est = ctypes.c_size_t()
    assert lbmfug._lib.lbm_server_estimate_bytes(lattice, shape[2], shape[1], shape[0], nc, precision,
                                                 ctypes.byref(est)) == 0
    assert total <= est.value
