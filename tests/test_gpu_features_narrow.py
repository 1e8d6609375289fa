"""Screening features of narrow ranges around 1 and elsewhere: the float is the rounded
formula, whatever the factor 2 / (l1 - l0) that takes the logarithm's error with it.  The
formula in FP64 is within 2^-50 of its terms of the exact value, and the float it rounds
to within half an ulp of that."""
import math

import numpy as np
import pytest

import paper_2011_01740_gb300 as ens

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("centre,width", [(1.0, w) for w in (1e-2, 1e-3, 1e-5, 1e-6, 1e-7, 1e-8, 1e-10, 1e-12, 1e-14)]
                         + [(1.0, 0.3), (1.5, 1e-6), (1e5, 1e-6), (1e-3, 1e-9)])
def test_narrow_ranges_round_the_formula(centre, width):
    import torch
    n = 1 << 18
    lo, hi = centre * (1 - width), centre * (1 + width)
    rng = np.random.default_rng(5)
    v = np.stack([rng.uniform(lo, hi, n), np.exp(rng.uniform(math.log(lo), math.log(hi), n))])
    v[:, :3] = lo, hi, centre
    x = torch.empty((n, 2), dtype=torch.float32, device="cuda")
    ens.ens_km_features(n, torch.from_numpy(v[0].copy()).cuda(), torch.from_numpy(v[1].copy()).cuda(), (lo, hi, lo, hi), x)
    got = x.cpu().numpy().T
    a, b = math.log(lo), math.log(hi)
    log_v = np.log(v)
    ref = 2.0 * (log_v - a) / (b - a) - 1.0
    terms = 2.0 * (np.abs(log_v) + abs(a)) / (b - a) + 2.0
    want = ref.astype(np.float32)
    half_ulp = 0.5 * np.spacing(np.maximum(np.abs(got), np.abs(want))).astype(np.float64)
    assert (np.abs(got - ref) <= half_ulp + 2.0 ** -50 * terms).all()
