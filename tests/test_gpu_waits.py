"""Bounded device waits give up with a status instead of hanging.

The tensor-core correlator kernel hands stages between its warp roles through
mbarrier waits, each limited to a number of polls.  With the limit set to zero
every wait gives up at once: no MMA is issued, every role runs out its loops,
the tensor memory is freed and the kernel returns normally; the context's
device flag makes qsg_read_correlators report QSG_ERR_TIMEOUT.  Nothing waits
on anything that cannot arrive, and no fault is raised.
"""
from __future__ import annotations

import numpy as np
import pytest

torch = pytest.importorskip("torch")

import oracle  # noqa: E402
from paper_2310_07486_gb300 import qsg as Q  # noqa: E402

pytestmark = pytest.mark.gpu


def _run(shape, lad, seed, wait_limit=None):
    ctx = Q.Context([shape])
    ctx.qsg_init_samples(seed, [lad])
    ctx.qsg_set_option(Q.OPT_CORR_KERNEL, Q.CORR_TENSOR)
    if wait_limit is not None:
        ctx.qsg_set_option(Q.OPT_WAIT_LIMIT, wait_limit)
    ctx.qsg_sweep(2)
    ctx.qsg_measure_correlators()
    return ctx


def test_wait_that_gives_up_reports_timeout_and_the_next_context_works():
    shape = Q.Shape(8, 256, 64, 2, 1, Q.HEATBATH, Q.PBC)
    lad = np.array([0.3])
    ctx = _run(shape, lad, 7, wait_limit=0)
    with pytest.raises(Q.QSGError) as e:
        ctx.qsg_read_correlators()
    assert e.value.status == -4
    # the flag stays set for that context
    with pytest.raises(Q.QSGError) as e:
        ctx.qsg_read_correlators()
    assert e.value.status == -4
    # the device and a fresh context are unaffected
    ctx.qsg_sweep(1)
    torch.cuda.synchronize()
    good = _run(shape, lad, 7)
    orc = oracle.OracleGroup(shape.L, shape.Ltau, shape.n_samples, shape.n_replicas, shape.n_k,
                             algo=shape.algo, boundary=shape.boundary)
    orc.init(7, lad)
    orc.sweep(2)
    orc.measure()
    got, ref = good.qsg_read_correlators(raw=True), orc.read()
    for key in ("C_raw", "Q2_raw", "q2_raw"):
        assert np.array_equal(got[key], ref[key]), key


def test_wait_limit_is_validated():
    shape = Q.Shape(8, 16, 64, 1, 1)
    ctx = Q.Context([shape])
    for bad in (-1, 1 << 31):
        with pytest.raises(Q.QSGError):
            ctx.qsg_set_option(Q.OPT_WAIT_LIMIT, bad)
    ctx.qsg_set_option(Q.OPT_WAIT_LIMIT, 1 << 22)


def test_asynchronous_read_reports_the_flag_when_waited_for():
    """qsg_read_correlators_async queues its copies without checking the
    device flag; qsg_wait_correlators reports it once the copies are done,
    and a context whose waits never gave up reports nothing."""
    shape = Q.Shape(8, 256, 64, 2, 1, Q.HEATBATH, Q.PBC)
    lad = np.array([0.3])
    copy_stream = torch.cuda.Stream()
    bad = _run(shape, lad, 7, wait_limit=0)
    bad.qsg_read_correlators_async(bad.correlator_buffers(pinned=True), copy_stream)
    with pytest.raises(Q.QSGError) as e:
        bad.qsg_wait_correlators()
    assert e.value.status == -4
    good = _run(shape, lad, 7)
    out = good.correlator_buffers(pinned=True)
    good.qsg_read_correlators_async(out, copy_stream)
    good.qsg_wait_correlators()
    ref = good.qsg_read_correlators()
    for key in ("C", "Q2", "q2"):
        assert np.array_equal(out[key], ref[key]), key


def _spins_on_device(ctx, shape):
    out = torch.empty(shape.slots * shape.Ltau * shape.L ** 2, dtype=torch.int64, device=ctx.device)
    ctx.qsg_get_spins_device(0, out)
    return out


@pytest.mark.parametrize("L,Ltau,R,variant", [(8, 48, 9, 0), (6, 32, 9, 1), (6, 820, 2, 1), (10, 6, 3, 1), (16, 512, 3, 1),
                                              (24, 256, 2, 1)])
@pytest.mark.parametrize("graph", [False, True])
def test_sweep_whose_waits_give_up_leaves_the_spins_and_the_counters(L, Ltau, R, variant, graph):
    """The resident form and chunks of one and of several planes per step: no spin
    changes, every block ends, the device flag is set, and sweeps with the limit put
    back are those of a context that never gave up."""
    if graph and Ltau % 16:
        pytest.skip("graphs need L_tau to be a multiple of 16")
    shape = Q.Shape(L, Ltau, 70, R, 2, Q.HEATBATH, Q.APBC)
    lad = np.array([0.25, 0.3])
    ctx, plain = Q.Context([shape]), Q.Context([shape])
    for c in (ctx, plain):
        c.qsg_init_samples(7, [lad])
    try:
        ctx.qsg_set_option(Q.OPT_WAVEFRONT_VARIANT, variant)
        if graph:
            ctx.qsg_set_option(Q.OPT_GRAPH, 2)
        ctx.qsg_set_option(Q.OPT_WAIT_LIMIT, 0)
        before = _spins_on_device(ctx, shape)
        ctx.qsg_sweep(2)
        assert torch.equal(_spins_on_device(ctx, shape), before)
        with pytest.raises(Q.QSGError) as e:
            ctx.qsg_read_correlators()
        assert e.value.status == -4
        ctx.qsg_set_option(Q.OPT_WAIT_LIMIT, 1 << 22)
        ctx.qsg_set_counters(0, 0)
        ctx.qsg_sweep(4)
        plain.qsg_set_option(Q.OPT_SWEEP_KERNEL, Q.SWEEP_REFERENCE)
        plain.qsg_sweep(4)
        assert torch.equal(_spins_on_device(ctx, shape), _spins_on_device(plain, shape))
    finally:
        ctx.qsg_set_option(Q.OPT_WAVEFRONT_VARIANT, 0)


@pytest.mark.parametrize("what", ["sweep", "measurement"])
def test_every_read_of_results_reports_the_flag(what):
    """Energies, accepted swaps, one-time sums, overlaps and spins as the correlators,
    more than once; a context whose waits never gave up reads all of them."""
    shape = Q.Shape(8, 256, 64, 3, 2, Q.HEATBATH, Q.PBC)
    reads = ("qsg_get_spins", "qsg_read_energies", "qsg_read_accepts", "qsg_read_onetime", "qsg_read_pair_overlaps",
             "qsg_read_correlators", "qsg_get_spins", "qsg_read_energies")
    for limit in (0, 1 << 22):
        ctx = Q.Context([shape])
        ctx.qsg_init_samples(7, [np.array([0.25, 0.3])])
        ctx.qsg_read_energies()  # the flag read before the wait that gives up
        if what == "sweep":
            ctx.qsg_set_option(Q.OPT_WAIT_LIMIT, limit)
            ctx.qsg_sweep(1)
        ctx.qsg_tempering_swap()
        ctx.qsg_set_option(Q.OPT_WAIT_LIMIT, limit)
        ctx.qsg_measure_correlators()
        for name in reads:
            if limit:
                getattr(ctx, name)()
                continue
            with pytest.raises(Q.QSGError) as e:
                getattr(ctx, name)()
            assert e.value.status == -4, name
