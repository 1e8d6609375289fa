"""Keller-Miksis launches of a caller's own shape whose ensemble the GPU holds at once:
all systems start together, so no shape takes much longer than one whose blocks all fit.
A launch that runs in two waves takes up to twice as long."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

PLAIN, PERSISTENT = ens.ENS_LAUNCH_PLAIN, ens.ENS_LAUNCH_PERSISTENT


def _plain(block):
    return dict(mode=PLAIN, block=block, blocks_per_sm=0)


def _persistent(block, per_sm):
    return dict(mode=PERSISTENT, block=block, blocks_per_sm=per_sm)


def _context(n, prec, dual):
    km = (W.km_dual if dual else W.km)(1, n, n_phases=1)
    ph = km["phys"]
    rng = np.random.default_rng(n)
    ph["pA1"][:] = rng.uniform(0.0, 2e5, n)
    ph["f1"][:] = rng.permutation(ph["f1"])
    if dual:
        ph["pA2"][:] = 0.5 * ph["pA1"]
    C = ens.ens_km_coefficients(*[ph[k] for k in ("pA1", "f1", "pA2", "f2", "theta", "RE")], km["liquid"])
    return ens.ens_create(ens.ENS_SYS_KELLER_MIKSIS, n, C, km["y0"], (0.0, 1.0), ens.ENS_RKCK45,
                          ens.make_tol(rtol=1e-9, atol=1e-9, n_phases=1, prec=prec))


def _best_ms(ctx, launch, runs=3):
    ens.ens_set_launch(ctx, ens.make_launch(**launch))
    best = float("inf")
    for _ in range(runs):
        ens.ens_solve(ctx)
        ens.ens_sync(ctx)
        best = min(best, ens.ens_kernel_ms(ctx))
    return best


@pytest.mark.parametrize("prec,dual,n,fits,launches", [
    (ens.ENS_FP64, False, 16000, _plain(32), [_plain(96)]),
    (ens.ENS_FP64, False, 20000, _plain(32), [_plain(64), _plain(96), _plain(128), _persistent(128, 2)]),
    (ens.ENS_FP64, True, 24320, _plain(32), [_plain(64), _plain(128), _persistent(128, 2)]),
    (ens.ENS_FP32X2, False, 37000, _persistent(256, 1), [_plain(64), _plain(224), _plain(256), _persistent(224, 2)]),
])
def test_no_shape_runs_in_two_waves(prec, dual, n, fits, launches):
    ctx = _context(n, prec, dual)
    try:
        ref = _best_ms(ctx, fits)
        times = [(launch, _best_ms(ctx, launch)) for launch in launches]
    finally:
        ens.ens_destroy(ctx)
    print(n, round(ref, 2), [(t[0]["block"], round(t[1], 2)) for t in times])
    assert all(ms < 1.3 * ref for _, ms in times), (ref, times)
