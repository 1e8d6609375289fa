"""Screening features against the FP64 formula in torch: over the screened ranges, for
features near zero, at the ends, and for values without a logarithm.  Either side takes
a logarithm within an ulp and rounds three times more, 2^-50 of its terms in all, so
the floats they round to are at most a float ulp apart beyond that, and the same for
all but few."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rng4", [W.KM_FEATURE_RANGE, (1.0, 2.0, 1e-9, 1e9), (1e-300, 1e300, 3.0, 3.0000001)])
def test_features_are_those_of_the_formula(rng4):
    import torch
    n = 1 << 21
    gen = torch.Generator(device="cuda").manual_seed(7)
    lo = [float(np.log(v)) for v in rng4]

    def values(a, b):
        mid = 0.5 * (a + b)
        u = torch.rand(n, generator=gen, device="cuda", dtype=torch.float64)
        v = torch.exp(a + (b - a) * u)
        k = torch.logspace(-12, -1, n // 4, device="cuda", dtype=torch.float64)
        v[: n // 4] = torch.exp(mid + (b - a) * k * (2 * u[: n // 4] - 1))      # features towards zero
        v[-12:] = torch.tensor([np.exp(a), np.exp(b), 1.0, 2.0 ** 0.5, 0.0, -0.0, -1.0, np.inf, -np.inf, np.nan,
                                5e-324, 2.0 ** -1022], dtype=torch.float64)
        return v

    pa, f = values(lo[0], lo[1]), values(lo[2], lo[3])
    x = torch.empty((n, 2), dtype=torch.float32, device="cuda")
    ens.ens_km_features(n, pa, f, rng4, x)
    ref = torch.stack([2.0 * (torch.log(v) - a) / (b - a) - 1.0
                       for v, a, b in ((pa, lo[0], lo[1]), (f, lo[2], lo[3]))], 1)
    terms = torch.stack([2.0 * (torch.log(v).abs() + abs(a)) / (b - a) + 2.0
                         for v, a, b in ((pa, lo[0], lo[1]), (f, lo[2], lo[3]))], 1)
    special = ~torch.isfinite(ref)
    want = ref.to(torch.float32)
    assert torch.equal(torch.isnan(x), torch.isnan(want))
    assert torch.equal(x[special & ~torch.isnan(want)], want[special & ~torch.isnan(want)])      # infinities
    err = (x.double() - want.double()).abs()[~special]
    ulp = torch.nextafter(want.abs(), torch.full_like(want, float("inf"))).double() - want.abs().double()
    assert (err <= ulp[~special] + 2.0 ** -50 * terms[~special]).all()
    ordinary = (want.abs() > 2.0 ** -10) & ~special
    assert (x != want)[ordinary].double().mean() < 1e-4
