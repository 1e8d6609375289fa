"""What the tuner's choice depends on: a choice made for one kind of parameters or
tolerance is not taken over for another, and what it chose for one kind is dropped when
the context gets parameters of the other.  The launch that an untuned context takes is
among the candidates."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SMS = 152


def _km(n, dual=False, **tol):
    km = (W.km_dual if dual else W.km)(1, n, n_phases=2, pa_max=0.6e5, f_min=2e5)
    ph = km["phys"]
    ph["pA1"][:] = np.linspace(0.2e5, 0.6e5, n)
    if dual:
        ph["pA2"][:] = 0.5 * ph["pA1"]
    C = ens.ens_km_coefficients(*[ph[k] for k in ("pA1", "f1", "pA2", "f2", "theta", "RE")], km["liquid"])
    return C, km["y0"], ens.make_tol(**{**dict(rtol=1e-7, atol=1e-7, n_phases=2), **tol})


def _create(C, y0, tol):
    return ens.ens_create(ens.ENS_SYS_KELLER_MIKSIS, C.shape[1], C, y0, (0.0, 1.0), ens.ENS_RKCK45, tol)


def _shapes(ctx):
    keys = ("mode", "block", "blocks_per_sm", "cost_order", "systems_per_thread")
    return [tuple(r["launch"][k] for k in keys) for r in ens.ens_autotune_table(ctx)]


def _spt2(shapes):
    return [s for s in shapes if s[4] == 2]


def test_choices_are_kept_per_kind_of_parameters_and_tolerance():
    n = 65 * SMS + 3
    C, y0, tol = _km(n)
    other = C.copy()
    other[10] = 4.0
    contexts = [_create(C, y0, tol), _create(other, y0, tol), _create(*_km(n, dual=True))]
    try:
        tables = []
        for ctx in contexts:
            ens.ens_autotune(ctx)
            tables.append(_shapes(ctx))
            ens.ens_solve(ctx)                 # a kernel for these parameters runs
            assert ens.ens_sync(ctx) == ens.ENS_OK
        assert _spt2(tables[0]) and not _spt2(tables[1]) and not _spt2(tables[2])
        relay = (ens.ENS_LAUNCH_PERSISTENT, 32, 1, 1, 1)
        assert relay in tables[0] and relay not in tables[1] and relay in tables[2]
        # another tolerance is timed for itself, the same one is looked up
        times = [r["ms"] for r in ens.ens_autotune_table(contexts[0])]
        for tol2, same in ((ens.make_tol(rtol=1e-5, atol=1e-7, n_phases=2), False),
                           (ens.make_tol(rtol=1e-7, atol=1e-5, n_phases=2), False), (tol, True)):
            ctx = _create(C, y0, tol2)
            contexts.append(ctx)
            ens.ens_autotune(ctx)
            assert ([r["ms"] for r in ens.ens_autotune_table(ctx)] == times) == same
    finally:
        for ctx in contexts:
            ens.ens_destroy(ctx)


@pytest.mark.parametrize("use_graph", [0, 1])
def test_a_tuned_launch_goes_with_the_parameters_it_was_made_for(use_graph):
    n = 300 * SMS + 1
    C, y0, tol = _km(n)
    D, _, _ = _km(n, dual=True)
    ctx, fresh = _create(C, y0, tol), _create(D, y0, tol)
    try:
        default = ens.ens_get_launch(ctx)
        default.use_graph = use_graph
        ens.ens_set_launch(ctx, default)
        tuned = ens.ens_autotune(ctx).as_dict()
        assert tuned["use_graph"] == use_graph
        ens.ens_set_inputs(ctx, C, y0)
        assert ens.ens_get_launch(ctx).as_dict() == tuned
        ens.ens_set_inputs(ctx, D, y0)
        assert ens.ens_get_launch(ctx).as_dict() == {**ens.ens_get_launch(fresh).as_dict(), "use_graph": use_graph}
        for c in (ctx, fresh):
            ens.ens_solve(c)
            assert ens.ens_sync(c) == ens.ENS_OK
        for w in (ens.ENS_STATE, ens.ENS_ACC, ens.ENS_NSTEPS):
            assert np.array_equal(ens.ens_read(ctx, w), ens.ens_read(fresh, w))
        # a launch that the caller sets stays, tuned context or not
        ens.ens_set_launch(ctx, ens.make_launch(block=96, blocks_per_sm=1))
        ens.ens_set_inputs(ctx, C, y0)
        assert ens.ens_get_launch(ctx).block == 96
    finally:
        ens.ens_destroy(ctx)
        ens.ens_destroy(fresh)


@pytest.mark.parametrize("case,prec,n", [("valve", ens.ENS_FP64, 500), ("valve", ens.ENS_FP32X2, 500),
                                         ("km", ens.ENS_FP64, 500), ("km", ens.ENS_FP64, 1300 * SMS),
                                         ("km", ens.ENS_FP64, 1700 * SMS), ("km", ens.ENS_FP64, 150 * SMS),
                                         ("km", ens.ENS_FP32_COMP, 500), ("km", ens.ENS_FP32_COMP, 1300 * SMS),
                                         ("km", ens.ENS_FP32X2, 200 * SMS), ("km", ens.ENS_FP32X2, 1300 * SMS)])
def test_the_untuned_launch_is_a_candidate(case, prec, n):
    if case == "valve":
        w = W.prv(n, t1=2.0)
        t = w["tol"]
        ctx = ens.ens_create(ens.ENS_SYS_RELIEF_VALVE, n, w["params"], w["y0"], (0.0, 2.0), ens.ENS_RKCK45,
                             ens.make_tol(rtol=1e-7, atol=1e-7, dt0=t.dt0, dt_max=t.dt_max, event_tol=t.event_tol,
                                          prec=prec))
    else:
        C, y0, tol = _km(n, n_phases=1, rtol=1e-5, atol=1e-5, prec=prec)
        ctx = _create(C, y0, tol)
    try:
        d = ens.ens_get_launch(ctx)
        untuned = (d.mode, d.block, d.blocks_per_sm, d.cost_order, 1)
        ens.ens_autotune(ctx)
        rows = ens.ens_autotune_table(ctx)
        first = [s for s, r in zip(_shapes(ctx), rows) if r["horizon_frac"] == rows[0]["horizon_frac"]]
        assert untuned in first and len(set(first)) == len(first)      # none of them twice
    finally:
        ens.ens_destroy(ctx)
