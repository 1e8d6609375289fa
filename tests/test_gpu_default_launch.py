"""The launch a context picks when its caller sets none: results are those of a
plain launch, bit for bit, on both sides of each line of the rule."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SMS = 152


def _solve(ctx):
    ens.ens_solve(ctx)
    status = ens.ens_sync(ctx)
    return [ens.ens_read(ctx, w) for w in (ens.ENS_STATE, ens.ENS_ACC, ens.ENS_NSTEPS, ens.ENS_STATUS)] + [status]


def _same(ctx):
    default = ens.ens_get_launch(ctx).as_dict()
    a = _solve(ctx)
    ens.ens_set_launch(ctx, ens.make_launch(mode=ens.ENS_LAUNCH_PLAIN, block=64, blocks_per_sm=0))
    b = _solve(ctx)
    for u, v in zip(a, b):
        assert np.array_equal(u, v, equal_nan=True) if isinstance(u, np.ndarray) else u == v
    return default


@pytest.mark.parametrize("prec,n", [(ens.ENS_FP64, 1), (ens.ENS_FP64, 64 * SMS), (ens.ENS_FP64, 64 * SMS + 1),
                                    (ens.ENS_FP64, 145 * SMS), (ens.ENS_FP64, 410 * SMS), (ens.ENS_FP64, 480 * SMS),
                                    (ens.ENS_FP64, 600 * SMS), (ens.ENS_FP64, 1300 * SMS),
                                    (ens.ENS_FP32_COMP, 128 * SMS), (ens.ENS_FP32_COMP, 700 * SMS),
                                    (ens.ENS_FP32_COMP, 128 * SMS + 1), (ens.ENS_FP32_COMP, 1300 * SMS),
                                    (ens.ENS_FP32_COMP, 2600 * SMS), (ens.ENS_FP32X2, 33),
                                    (ens.ENS_FP32X2, 64 * SMS + 1), (ens.ENS_FP32X2, 320 * SMS),
                                    (ens.ENS_FP32X2, 440 * SMS), (ens.ENS_FP32X2, 710 * SMS)])
@pytest.mark.parametrize("dual", [False, True])
def test_keller_miksis_default_launch(prec, n, dual):
    """One short period; the dual-frequency runs also take the split-precision
    claim-order pilot through its second forcing."""
    km = (W.km_dual if dual else W.km)(1, n, n_phases=1, pa_max=0.6e5, f_min=2e5)
    ph = km["phys"]
    ph["pA1"][:] = np.linspace(0.2e5, 0.6e5, n)
    if dual:
        ph["pA2"][:] = 0.5 * ph["pA1"]
    C = ens.ens_km_coefficients(*[ph[k] for k in ("pA1", "f1", "pA2", "f2", "theta", "RE")], km["liquid"])
    tol = ens.make_tol(rtol=1e-7, atol=1e-7, n_phases=1, prec=prec)
    ctx = ens.ens_create(ens.ENS_SYS_KELLER_MIKSIS, n, C, km["y0"], (0.0, 1.0), ens.ENS_RKCK45, tol)
    try:
        default = _same(ctx)
        once = 64 if prec == ens.ENS_FP64 or (dual and prec == ens.ENS_FP32X2) else 128   # all start at once
        assert (default["mode"] == ens.ENS_LAUNCH_PLAIN) == (n <= once * SMS)
    finally:
        ens.ens_destroy(ctx)


@pytest.mark.parametrize("prec", [ens.ENS_FP64, ens.ENS_FP32X2])
@pytest.mark.parametrize("n", [1, 512 * SMS - 1, 512 * SMS])
def test_valve_default_launch(prec, n):
    w = W.prv(n, t1=1.0)
    t = w["tol"]
    tol = ens.make_tol(rtol=1e-8, atol=1e-8, dt0=t.dt0, dt_max=t.dt_max, event_tol=t.event_tol, prec=prec)
    ctx = ens.ens_create(ens.ENS_SYS_RELIEF_VALVE, n, w["params"], w["y0"], (0.0, 1.0), ens.ENS_RKCK45, tol)
    try:
        assert _same(ctx)["mode"] == ens.ENS_LAUNCH_PLAIN
    finally:
        ens.ens_destroy(ctx)


def test_default_launch_follows_the_parameters():
    """A context that only ever had the default changes it with the exponent that
    decides on the team kernels; one whose caller chose keeps the choice."""
    n = 64 * SMS + 1
    km = W.km(1, n, n_phases=1, pa_max=0.6e5)
    ph = km["phys"]
    C = ens.ens_km_coefficients(*[ph[k] for k in ("pA1", "f1", "pA2", "f2", "theta", "RE")], km["liquid"])
    other = C.copy()
    other[10] = 4.0
    ctx = ens.ens_create(ens.ENS_SYS_KELLER_MIKSIS, n, C, km["y0"], (0.0, 1.0), ens.ENS_RKCK45, ens.make_tol(n_phases=1))
    try:
        mode = lambda: ens.ens_get_launch(ctx).mode
        assert mode() == ens.ENS_LAUNCH_PERSISTENT
        ens.ens_set_inputs(ctx, other, km["y0"])
        assert mode() == ens.ENS_LAUNCH_PLAIN
        ens.ens_set_inputs(ctx, C, km["y0"])
        assert mode() == ens.ENS_LAUNCH_PERSISTENT
        ens.ens_set_launch(ctx, ens.make_launch(mode=ens.ENS_LAUNCH_PERSISTENT, block=96, blocks_per_sm=1))
        ens.ens_set_inputs(ctx, other, km["y0"])
        assert ens.ens_get_launch(ctx).block == 96
    finally:
        ens.ens_destroy(ctx)
