"""The valve kernel that spreads a trial over four warps gives the bits of the one-warp
kernel: at the edges of a warp of systems, with one and several of them per SM, for lanes
that claim further systems, for impacts, sticking and rejections, and for systems that
are retired early."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SMS = 152
READ = (ens.ENS_STATE, ens.ENS_ACC, ens.ENS_STATUS, ens.ENS_NSTEPS, ens.ENS_NREJ, ens.ENS_NRHS, ens.ENS_TIME,
        ens.ENS_DT)
ONE_WARP = dict(mode=ens.ENS_LAUNCH_PLAIN, block=64, blocks_per_sm=0)
RELAY = dict(mode=ens.ENS_LAUNCH_PLAIN, block=32, blocks_per_sm=0)


def _claiming(per_sm, order=0):
    return dict(mode=ens.ENS_LAUNCH_PERSISTENT, block=32, blocks_per_sm=per_sm, cost_order=order)


def _solve(ctx, **launch):
    ens.ens_set_launch(ctx, ens.make_launch(**launch))
    ens.ens_solve(ctx)
    return [ens.ens_sync(ctx)] + [ens.ens_read(ctx, w) for w in READ]


def _compare(n, launch, t1=6.0, t0=0.0, acc=0.0, **tol):
    w = W.prv(n, t1=t1)
    rng = np.random.default_rng(n)
    w["params"][0][:] = rng.uniform(0.05, 10.0, n)        # q: from sticking and chattering to no impact
    w["y0"][0][:] = rng.uniform(0.0, 0.4, n)
    t = w["tol"]
    kw = dict(rtol=t.rtol, atol=t.atol, dt0=t.dt0, dt_min=t.dt_min, dt_max=t.dt_max, event_tol=t.event_tol,
              acc_t_start=acc)
    ctx = ens.ens_create(ens.ENS_SYS_RELIEF_VALVE, n, w["params"], w["y0"], (t0, t1), ens.ENS_RKCK45,
                         ens.make_tol(**{**kw, **tol}))
    try:
        ref, got = _solve(ctx, **ONE_WARP), _solve(ctx, **launch)
    finally:
        ens.ens_destroy(ctx)
    assert ref[0] == got[0]
    for k, a, b in zip(READ, ref[1:], got[1:]):
        assert np.array_equal(a, b, equal_nan=True), k
    return ref


@pytest.mark.parametrize("n,launch", [
    (1, RELAY), (32, RELAY), (33, RELAY), (32 * SMS + 1, RELAY), (128 * SMS, RELAY),
    (128 * SMS + 1, RELAY),                       # more than four per SM: the one-warp kernel
    (20000, _claiming(1)), (20000, _claiming(2, 1)), (300, _claiming(4)),
])
def test_relays_give_the_one_warp_bits(n, launch):
    ref = _compare(n, launch)
    if n > 1000:
        assert ref[2][-1].max() > 0 and ref[2][-2].max() > 0       # impacts and maxima


@pytest.mark.parametrize("kw", [
    dict(t0=1.5, acc=3.0),
    dict(max_steps=37), dict(max_steps=1),               # retired early
    dict(dt_min=1e-2, dt0=0.1),                          # step-size underflow after a rejection
    dict(rtol=1e-4, atol=1e-4, dt0=0.5, dt_max=0.5),     # many rejections
    dict(event_tol=1e-12),                               # events that take many retries
])
def test_relays_keep_events_budgets_and_rejections(kw):
    for launch in (RELAY, _claiming(1)):
        ref = _compare(700, launch, **kw)
        if "max_steps" in kw or "dt_min" in kw:
            assert ref[0] == ens.ENS_ESYSTEM
