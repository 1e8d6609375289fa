"""The Keller-Miksis kernel that spreads a trial over eight warps gives the bits of
the one-warp kernel: at the edges of a warp of systems, with one and two of them per
SM, for lanes that claim further systems, for phases that do not start at tau = 0 or
last one period, and for systems that are retired early."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from test_gpu_teams import PERSISTENT, PLAIN, _compare, _solve

pytestmark = pytest.mark.gpu

SMS = 152
RELAY = dict(mode=PLAIN, block=32, blocks_per_sm=0)


def _claiming(per_sm, order):
    return dict(mode=PERSISTENT, block=32, blocks_per_sm=per_sm, cost_order=order)


@pytest.mark.parametrize("solver", [ens.ENS_RKCK45, ens.ENS_DOPRI5])
@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("n,launch", [
    (32, RELAY), (65, RELAY), (32 * SMS + 1, RELAY), (64 * SMS, RELAY),
    (64 * SMS + 1, RELAY),                       # one more than two per SM: teams
    (9000, _claiming(1, 1)),                     # ranked first claims, a second system per lane
    (20000, _claiming(2, 0)), (300, _claiming(2, 1)),
])
def test_relays_give_the_one_warp_bits(n, launch, solver, dual):
    _compare(n, launch, solver=solver, dual=dual)


@pytest.mark.parametrize("solver", [ens.ENS_RKCK45, ens.ENS_DOPRI5])
@pytest.mark.parametrize("dual", [False, True])
@pytest.mark.parametrize("kw", [
    dict(t0=0.3, phase_len=0.7),                       # the phase start's drive has other bits than its end's
    dict(n_phases=5, n_transient=4),
    dict(max_steps=37), dict(max_steps=1),             # retired in mid-phase
    dict(dt_min=3e-3, dt0=0.1),                        # step-size underflow after a rejection
    dict(rtol=1e-4, atol=1e-4, dt0=0.5, dt_max=0.5),   # many rejections
])
def test_relays_keep_phases_budgets_and_rejections(kw, solver, dual):
    for launch in (RELAY, _claiming(1, 0)):
        ref = _compare(700, launch, solver=solver, dual=dual, **kw)
        if "max_steps" in kw or "dt_min" in kw:
            assert ref[0] == ens.ENS_ESYSTEM
