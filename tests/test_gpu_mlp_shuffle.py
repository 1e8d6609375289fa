"""The shuffles of training: draws on the device, swaps on the host, buffers kept
from run to run.  Same samples in the same order give the same weights, bit for bit."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

MEMBERS, SHIFT, U64 = 2, 0x51ed2701, (1 << 64) - 1


def _hash(x):
    x = (x + 0x9e3779b97f4a7c15) & U64
    x = ((x ^ (x >> 30)) * 0xbf58476d1ce4e5b9) & U64
    x = ((x ^ (x >> 27)) * 0x94d049bb133111eb) & U64
    return x ^ (x >> 31)


def _shuffle(n, seed, epoch):
    ctr = ((seed + SHIFT * (epoch + 1)) << 20) & U64
    p = list(range(n))
    for k, i in enumerate(range(n - 1, 0, -1)):
        j = _hash((ctr + k) & U64) % (i + 1)
        p[i], p[j] = p[j], p[i]
    return np.array(p)


def _weights(m, runs):
    """Weights after runs of (x, y, config) from one start."""
    import torch
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float32)).cuda()
    w0 = ens.ens_mlp_get_params(m, torch.empty((MEMBERS, W.MLP_PARAMS), dtype=torch.float32, device="cuda")).clone()
    for x, y, cfg in runs:
        ens.ens_mlp_train(m, len(x), dev(x), dev(y), cfg, MEMBERS)
    w = ens.ens_mlp_get_params(m, torch.empty_like(w0)).clone()
    ens.ens_mlp_set_params(m, w0)
    return w.cpu().numpy()


def test_shuffles():
    m = ens.ens_mlp_create(MEMBERS, W.SEED)
    cfg = lambda seed, epochs: ens.make_train_cfg(epochs=epochs, batch=300, lr=1e-3, seed=seed)
    try:
        for n in (1000, 3001, 1, 2, 700):      # the buffers grow, then serve smaller runs
            x, y = W.mlp_batch(n, seed=n)
            # the same samples in the same order through two different shuffles
            pa, pb = _shuffle(n, 5, 0), _shuffle(n, 99, 0)
            q = np.empty(n, dtype=np.int64)
            q[pb] = pa
            a = _weights(m, [(x, y, cfg(5, 1))])
            assert np.array_equal(a, _weights(m, [(x[q], y[q], cfg(99, 1))])), n
            # several epochs in one call, and in calls of one epoch
            many = _weights(m, [(x, y, cfg(5, 4))])
            assert np.array_equal(many, _weights(m, [(x, y, cfg(5 + e * SHIFT, 1)) for e in range(4)])), n
            assert n == 1 or not np.array_equal(a, many)
    finally:
        ens.ens_mlp_destroy(m)
