"""The double-float one-warp kernel with unrolled stages, which launches of few warps per SM
take, gives the bits of the rolled one: at once and with lanes that claim further systems,
on both sides of its lines."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SMS = 152
N = 700
READ = (ens.ENS_STATE, ens.ENS_ACC, ens.ENS_STATUS, ens.ENS_NSTEPS, ens.ENS_NREJ, ens.ENS_NRHS, ens.ENS_TIME,
        ens.ENS_DT)
PLAIN, PERSISTENT = ens.ENS_LAUNCH_PLAIN, ens.ENS_LAUNCH_PERSISTENT


def _run(total, dual, launch, **tol):
    """N systems over and over, `total` in all; the first and the last N of the results."""
    km = (W.km_dual if dual else W.km)(1, N, n_phases=2)
    ph = km["phys"]
    ph["pA1"][:] = np.random.default_rng(3).uniform(0.0, 1.2e5, N)
    if dual:
        ph["pA2"][:] = 0.5 * ph["pA1"]
    C = ens.ens_km_coefficients(*[ph[k] for k in ("pA1", "f1", "pA2", "f2", "theta", "RE")], km["liquid"])
    pick = np.arange(total) % N
    ctx = ens.ens_create(ens.ENS_SYS_KELLER_MIKSIS, total, np.ascontiguousarray(C[:, pick]),
                         np.ascontiguousarray(km["y0"][:, pick]), (0.0, 1.0), ens.ENS_RKCK45,
                         ens.make_tol(**{**dict(rtol=1e-8, atol=1e-8, n_phases=2, prec=ens.ENS_FP32X2), **tol}))
    try:
        ens.ens_set_launch(ctx, ens.make_launch(**launch))
        ens.ens_solve(ctx)
        status = ens.ens_sync(ctx)
        out = [ens.ens_read(ctx, w) for w in READ]
    finally:
        ens.ens_destroy(ctx)
    order = np.argsort(pick[-N:])
    return status, [a[..., :N] for a in out], [a[..., -N:][..., order] for a in out]


@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("kw", [dict(), dict(max_steps=37), dict(rtol=1e-4, atol=1e-4, dt0=0.5, dt_max=0.5)])
def test_unrolled_stages_give_the_rolled_bits(dual, kw):
    rolled = _run(320 * SMS + 1, dual, dict(mode=PLAIN, block=128, blocks_per_sm=0), **kw)
    for total, launch in ((192 * SMS + 1, dict(mode=PLAIN, block=64, blocks_per_sm=0)),
                          (320 * SMS, dict(mode=PLAIN, block=256, blocks_per_sm=0)),
                          (320 * SMS, dict(mode=PERSISTENT, block=96, blocks_per_sm=3, cost_order=1)),
                          (1024 * SMS, dict(mode=PERSISTENT, block=128, blocks_per_sm=2)),
                          (1024 * SMS + 1, dict(mode=PERSISTENT, block=128, blocks_per_sm=2, cost_order=1))):
        got = _run(total, dual, launch, **kw)
        assert got[0] == rolled[0]
        for side in got[1:]:
            for w, a, b in zip(READ, rolled[1], side):
                assert np.array_equal(a, b, equal_nan=True), (total, w)
