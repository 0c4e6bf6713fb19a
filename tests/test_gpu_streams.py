"""Problems that share a stream: captured chunks of steps, and captured rounds of the
batched form, hold the work of their own handle and nothing else, whatever other
threads enqueue on the stream meanwhile.

Every result is bitwise that of the same calls alone: a node's arithmetic depends
neither on the stream nor on what runs beside it.
"""
from __future__ import annotations

import ctypes
import threading

import numpy as np
import pytest

from helpers import gpu_problem, seeded_mixture, smooth_rho

pytestmark = pytest.mark.gpu

FP64, FP32DEV, FP32 = 0, 1, 2
NC, SHAPE, PARTS = 3, (1, 20, 33), (48, 20, 33, 48)
FORMS = [(FP64, 1), (FP32DEV, 3), (FP32, 2)]


def mixture():
    c = seeded_mixture(480, NC, 0, SHAPE, Tfac=1.2)
    return c, smooth_rho(480, c, SHAPE)


def run(c, rho, form, stream, start=None):
    """Runs of lbm_step and lbm_step_graph, each the first of its kind on the handle."""
    with gpu_problem(c, 0, SHAPE, precision=form[0], schedule=form[1], tune=0, stream=stream) as gp:
        gp.init_fields(rho)
        if start is not None:
            start.wait()
        for k, n in enumerate(PARTS):
            (gp.step_graph if k % 2 else gp.step)(n)
        assert gp.step_count() == sum(PARTS)
        return gp.get_state()


def together(calls):
    out, errors = [None] * len(calls), []

    def body(k):
        try:
            out[k] = calls[k]()
        except Exception as e:  # reported by the main thread
            errors.append(e)

    threads = [threading.Thread(target=body, args=(k,)) for k in range(len(calls))]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
    return out


def test_two_handles_of_one_stream_in_two_threads():
    import torch
    c, rho = mixture()
    alone = {f: run(c, rho, f, None) for f in FORMS}
    st = torch.cuda.Stream()
    for _ in range(4):
        for f in FORMS:
            for g in FORMS:
                start = threading.Barrier(2)
                a, b = together([lambda: run(c, rho, f, st.cuda_stream, start),
                                 lambda: run(c, rho, g, st.cuda_stream, start)])
                assert np.array_equal(a, alone[f]) and np.array_equal(b, alone[g])


@pytest.mark.parametrize("tau", [1.0, 0.8])
def test_two_batches_of_one_stream_in_two_threads(tau):
    import torch
    from paper_2306_10652_gb300 import lbmfug
    c, _ = mixture()
    shapes = [(4, 64), (3, 50), (20, 33)]
    rho = [smooth_rho(490 + k, c, (1,) + s)[:, 0] for k, s in enumerate(shapes)]

    def batch(order, stream, start=None):
        with lbmfug.Batch(c["a"], c["b"], c["omega"], c["kij"], tau, [(c["T"], rho[k]) for k in order],
                          stream=stream) as bt:
            if start is not None:
                start.wait()
            for n in (3, 5, 4):  # each another round: captured anew
                bt.run(max_steps=n, check_every=n, tol=0.0)
            return {k: bt.state(i)["rho"] for i, k in enumerate(order)}

    alone = batch((0, 1, 2), None)
    st = torch.cuda.Stream()
    for _ in range(4):
        start = threading.Barrier(2)
        for got in together([lambda: batch((0, 1), st.cuda_stream, start),
                             lambda: batch((2, 1, 0), st.cuda_stream, start)]):
            for k, r in got.items():
                assert np.array_equal(r, alone[k]), k


def test_other_work_on_the_stream_runs_once_and_where_it_was_enqueued():
    import torch
    c, rho = mixture()
    form = FORMS[0]
    alone = run(c, rho, form, None)
    st = torch.cuda.Stream()
    x = torch.zeros(1000, device="cuda")
    torch.cuda.synchronize()
    adds = 2000

    def other(start):
        start.wait()
        with torch.cuda.stream(st):
            for _ in range(adds):
                x.add_(1.0)

    for k in range(3):
        start = threading.Barrier(2)
        a, _ = together([lambda: run(c, rho, form, st.cuda_stream, start), lambda: other(start)])
        assert np.array_equal(a, alone)
        st.synchronize()
        assert (x == float(adds * (k + 1))).all()


@pytest.mark.parametrize("form", FORMS, ids=["fp64", "fp32dev", "fp32"])
def test_chunks_on_a_stream_ordered_with_the_legacy_stream(form):
    import torch
    c, rho = mixture()
    h = ctypes.c_void_p()
    rt = torch.cuda.cudart()
    torch.cuda.check_error(rt.cudaStreamCreate(ctypes.addressof(h)))
    try:
        got = run(c, rho, form, h.value)
    finally:
        torch.cuda.check_error(rt.cudaStreamDestroy(h.value))
    assert np.array_equal(got, run(c, rho, form, None))
