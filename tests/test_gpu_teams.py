"""The Keller-Miksis kernels with teams of warps (FP64: three, double-float: two)
give the bits of the one-warp kernels: at the edges of its warps and blocks, for both pairs and one or
two frequencies, with a phase that does not start at tau = 0 or last one period
(the drive then differs between a phase's end and the next one's start), and for
systems that are retired early."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

READ = (ens.ENS_STATE, ens.ENS_ACC, ens.ENS_STATUS, ens.ENS_NSTEPS, ens.ENS_NREJ, ens.ENS_NRHS, ens.ENS_TIME,
        ens.ENS_DT)
PLAIN, PERSISTENT = ens.ENS_LAUNCH_PLAIN, ens.ENS_LAUNCH_PERSISTENT
ONE_WARP = dict(mode=PLAIN, block=256, blocks_per_sm=0)        # FP64 blocks above 160 threads: no teams


def _solve(ctx, **launch):
    ens.ens_set_launch(ctx, ens.make_launch(**launch))
    ens.ens_solve(ctx)
    return [ens.ens_sync(ctx)] + [ens.ens_read(ctx, w) for w in READ]


def _compare(n, launch, solver=ens.ENS_RKCK45, dual=False, t0=0.0, **tol):
    km = (W.km_dual if dual else W.km)(1, n, pa_max=1e5)
    km["phys"]["pA1"][:] = np.random.default_rng(n).uniform(0.0, 1.2e5, n)
    ph = km["phys"]
    if dual:
        ph["pA2"][:] = 0.5 * ph["pA1"]
    C = ens.ens_km_coefficients(*[ph[k] for k in ("pA1", "f1", "pA2", "f2", "theta", "RE")], km["liquid"])
    assert np.any(C[6]) == dual
    t = ens.make_tol(**{**dict(rtol=1e-8, atol=1e-8, n_phases=3), **tol})
    # the double-float one-warp kernel takes launches of more than 8 warps per SM
    copies = -(-40000 // n) if t.prec == ens.ENS_FP32X2 else 1
    out = []
    for reps, shape in ((copies, ONE_WARP), (1, launch)):
        ctx = ens.ens_create(ens.ENS_SYS_KELLER_MIKSIS, n * reps, np.tile(C, (1, reps)), np.tile(km["y0"], (1, reps)),
                             (t0, t0 + 1.0), solver, t)
        try:
            r = _solve(ctx, **shape)
        finally:
            ens.ens_destroy(ctx)
        out.append([r[0]] + [a[..., :n] for a in r[1:]])
    ref, got = out
    assert ref[0] == got[0]
    for w, a, b in zip(READ, ref[1:], got[1:]):
        assert np.array_equal(a, b, equal_nan=True), w
    return ref


@pytest.mark.parametrize("solver", [ens.ENS_RKCK45, ens.ENS_DOPRI5])
@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("n,launch", [
    (1, dict(mode=PLAIN, block=32, blocks_per_sm=0)),
    (33, dict(mode=PLAIN, block=32, blocks_per_sm=0)),
    (161, dict(mode=PLAIN, block=160, blocks_per_sm=0)),
    (1000, dict(mode=PERSISTENT, block=96, blocks_per_sm=1, cost_order=0)),
    (23000, dict(mode=PERSISTENT, block=128, blocks_per_sm=1, cost_order=0)),      # lanes claim a second system
    (60000, dict(mode=PERSISTENT, block=160, blocks_per_sm=1, cost_order=1)),      # ranked first claims
    (30000, dict(mode=PERSISTENT, block=64, blocks_per_sm=2, cost_order=1)),
])
def test_teams_give_the_one_warp_bits(n, launch, solver, dual):
    _compare(n, launch, solver=solver, dual=dual)


@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("n,launch", [
    (1, dict(mode=PLAIN, block=32, blocks_per_sm=0)),
    (193, dict(mode=PLAIN, block=192, blocks_per_sm=0)),
    (257, dict(mode=PLAIN, block=256, blocks_per_sm=0)),
    (23000, dict(mode=PERSISTENT, block=128, blocks_per_sm=1, cost_order=0)),
    (60000, dict(mode=PERSISTENT, block=224, blocks_per_sm=1, cost_order=1)),
    (60000, dict(mode=PERSISTENT, block=192, blocks_per_sm=1, cost_order=1)),
    (30000, dict(mode=PERSISTENT, block=64, blocks_per_sm=3, cost_order=1)),
])
def test_double_float_teams_give_the_one_warp_bits(n, launch, dual):
    _compare(n, launch, dual=dual, prec=ens.ENS_FP32X2)


SMALL = dict(mode=PERSISTENT, block=64, blocks_per_sm=1, cost_order=1)


@pytest.mark.parametrize("solver,prec", [(ens.ENS_RKCK45, ens.ENS_FP64), (ens.ENS_DOPRI5, ens.ENS_FP64),
                                         (ens.ENS_RKCK45, ens.ENS_FP32X2)])
@pytest.mark.parametrize("kw", [
    dict(t0=0.3, phase_len=0.7),                       # the phase start's drive has other bits than its end's
    dict(n_phases=5, n_transient=4),
    dict(max_steps=37),                                # retired in mid-phase
    dict(dt_min=3e-3, dt0=0.1),                        # step-size underflow after a rejection
    dict(rtol=1e-4, atol=1e-4, dt0=0.5, dt_max=0.5),   # many rejections
])
def test_teams_keep_phases_budgets_and_rejections(kw, solver, prec):
    ref = _compare(700, SMALL, solver=solver, prec=prec, **kw)
    if "max_steps" in kw or "dt_min" in kw:
        assert ref[0] == ens.ENS_ESYSTEM


@pytest.mark.parametrize("prec", [ens.ENS_FP64, ens.ENS_FP32X2])
def test_teams_stop_at_the_wall_clock_budget(prec):
    """Systems that a 1 us budget catches are flagged; the call returns and says so."""
    n = 700
    km = W.km(1, n, pa_max=1e5)
    ph = km["phys"]
    C = ens.ens_km_coefficients(*[ph[k] for k in ("pA1", "f1", "pA2", "f2", "theta", "RE")], km["liquid"])
    ctx = ens.ens_create(ens.ENS_SYS_KELLER_MIKSIS, n, C, km["y0"], (0.0, 1.0), ens.ENS_RKCK45,
                         ens.make_tol(n_phases=64, timeout_s=1e-6, prec=prec))
    try:
        got = _solve(ctx, mode=PLAIN, block=32, blocks_per_sm=0)
    finally:
        ens.ens_destroy(ctx)
    assert got[0] == ens.ENS_ETIMEOUT and np.all(got[3] == ens.ENS_SYS_TIMEOUT)
    assert np.isnan(got[2][-1]).all()                  # the phases not reached
