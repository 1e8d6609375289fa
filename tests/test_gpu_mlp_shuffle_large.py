"""Training runs over more samples than the network keeps shuffle buffers for, whose host
buffers are pageable and given back: several epochs in one call are those of calls of one
epoch, and a smaller run after it finds buffers of its own."""
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

SHIFT, N = 0x51ed2701, (1 << 24) + 3


def test_shuffles_of_a_large_run():
    import torch
    m = ens.ens_mlp_create(1, W.SEED)
    out = lambda: ens.ens_mlp_get_params(m, torch.empty((1, W.MLP_PARAMS), dtype=torch.float32, device="cuda"))
    cfg = lambda seed, epochs: ens.make_train_cfg(epochs=epochs, batch=1 << 20, lr=1e-3, seed=seed)
    try:
        w0 = out().clone()

        def weights(runs):
            for x, y, c in runs:
                ens.ens_mlp_train(m, len(x), x, y, c, 1)
            w = out().clone()
            ens.ens_mlp_set_params(m, w0)
            return w

        gen = torch.Generator(device="cuda").manual_seed(3)
        x = torch.rand((N, 2), generator=gen, device="cuda") * 2 - 1
        y = torch.rand((N, 2), generator=gen, device="cuda")
        many = weights([(x, y, cfg(5, 2))])
        singly = [(x, y, cfg(5 + e * SHIFT, 1)) for e in range(2)]
        assert torch.equal(many, weights(singly))
        assert not torch.equal(many, weights(singly[:1]))
        small = weights([(x[:1000], y[:1000], cfg(5, 2))])
        assert torch.equal(small, weights([(x[:1000], y[:1000], cfg(5 + e * SHIFT, 1)) for e in range(2)]))
    finally:
        ens.ens_mlp_destroy(m)
