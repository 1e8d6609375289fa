"""Launches that pick their kernel by size, against the one-warp kernel: the default launch of
small ensembles, the allocation-free entry point on both sides of its lines and with an
exponent the team kernels do not have, and the valve relay's wall-clock budget."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SMS = 152
READ = (ens.ENS_STATE, ens.ENS_ACC, ens.ENS_STATUS, ens.ENS_NSTEPS, ens.ENS_NREJ, ens.ENS_NRHS, ens.ENS_TIME,
        ens.ENS_DT)
ONE_WARP = ens.make_launch(mode=ens.ENS_LAUNCH_PLAIN, block=256, blocks_per_sm=0)


def _km(n, dual=False, **liquid):
    km = (W.km_dual if dual else W.km)(1, n, n_phases=1, f_min=1e5)
    ph = km["phys"]
    ph["pA1"][:] = np.random.default_rng(n).uniform(0.0, 1e5, n)
    if dual:
        ph["pA2"][:] = 0.5 * ph["pA1"]
    C = ens.ens_km_coefficients(*[ph[k] for k in ("pA1", "f1", "pA2", "f2", "theta", "RE")], {**km["liquid"], **liquid})
    return C, km["y0"]


def _solve(C, y0, tol, launch=None):
    ctx = ens.ens_create(ens.ENS_SYS_KELLER_MIKSIS, C.shape[1], C, y0, (0.0, 1.0), ens.ENS_RKCK45, tol)
    try:
        if launch is not None:
            ens.ens_set_launch(ctx, launch)
        ens.ens_solve(ctx)
        return [ens.ens_sync(ctx)] + [ens.ens_read(ctx, w) for w in READ]
    finally:
        ens.ens_destroy(ctx)


@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("prec,n", [(ens.ENS_FP64, 1), (ens.ENS_FP64, 33), (ens.ENS_FP64, 64 * SMS),
                                    (ens.ENS_FP64, 64 * SMS + 1), (ens.ENS_FP32X2, 33), (ens.ENS_FP32X2, 64 * SMS)])
def test_default_launches_of_small_ensembles(prec, n, dual):
    C, y0 = _km(n, dual)
    tol = ens.make_tol(rtol=1e-7, atol=1e-7, n_phases=1, prec=prec)
    got = _solve(C, y0, tol)
    # double-float launches take the one-warp kernel above 8 warps of systems per SM
    reps = -(-60000 // n) if prec == ens.ENS_FP32X2 else 1
    ref = _solve(np.tile(C, (1, reps)), np.tile(y0, (1, reps)), tol, ONE_WARP)
    assert got[0] == ref[0]
    for w, a, b in zip(READ, got[1:], ref[1:]):
        assert np.array_equal(a, b[..., :n], equal_nan=True), w


@pytest.mark.parametrize("n,cost_order,dual,liquid", [
    (260 * SMS - 1, 0, False, {}), (260 * SMS, 0, False, {}),          # relays, teams
    (410 * SMS - 1, 1, False, {}), (410 * SMS, 1, False, {}),
    (260 * SMS, 0, True, {}),
    (300, 0, False, dict(gamma=1.33)), (260 * SMS, 1, False, dict(gamma=1.33)),     # the one-warp kernel
])
def test_noalloc_kernels_give_the_one_warp_bits(n, cost_order, dual, liquid):
    import torch
    C, y0 = _km(n, dual, **liquid)
    tol = ens.make_tol(rtol=1e-6, atol=1e-6, n_phases=1)
    ref = _solve(C, y0, tol, ONE_WARP)[1:]
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a)).cuda()
    f64 = lambda *s: torch.empty(s, dtype=torch.float64, device="cuda")
    i64 = lambda: torch.empty(n, dtype=torch.int64, device="cuda")
    y, t, dt, acc, nacc, nrej, nrhs = f64(2, n), f64(n), f64(n), f64(2, n), i64(), i64(), i64()
    status = torch.empty(n, dtype=torch.int32, device="cuda")
    for _ in range(2):
        ens.ens_solve_noalloc(ens.ENS_SYS_KELLER_MIKSIS, n, dev(C), dev(y0), (0.0, 1.0), tol, y, t, dt, acc, status,
                              nacc, nrej, nrhs, cost_order)
        torch.cuda.synchronize()
        for w, a, b in zip(READ, (y, acc, status, nacc, nrej, nrhs, t, dt), ref):
            assert np.array_equal(a.cpu().numpy(), b, equal_nan=True), w


@pytest.mark.parametrize("launch", [dict(mode=ens.ENS_LAUNCH_PLAIN, block=32, blocks_per_sm=0),
                                    dict(mode=ens.ENS_LAUNCH_PERSISTENT, block=32, blocks_per_sm=1)])
def test_valve_relays_stop_at_the_wall_clock_budget(launch):
    """Valves that a 1 us budget catches are flagged, those not claimed yet among them."""
    n = 33 * SMS
    w = W.prv(n, t1=64.0)
    t = w["tol"]
    ctx = ens.ens_create(ens.ENS_SYS_RELIEF_VALVE, n, w["params"], w["y0"], (0.0, 64.0), ens.ENS_RKCK45,
                         ens.make_tol(rtol=t.rtol, atol=t.atol, dt0=t.dt0, dt_min=t.dt_min, dt_max=t.dt_max,
                                      event_tol=t.event_tol, timeout_s=1e-6))
    try:
        ens.ens_set_launch(ctx, ens.make_launch(**launch))
        ens.ens_solve(ctx)
        assert ens.ens_sync(ctx) == ens.ENS_ETIMEOUT
        assert np.all(ens.ens_read(ctx, ens.ENS_STATUS) == ens.ENS_SYS_TIMEOUT)
        assert np.all(ens.ens_read(ctx, ens.ENS_TIME) < 64.0)
    finally:
        ens.ens_destroy(ctx)
