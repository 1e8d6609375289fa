"""The tcgen05 kernels of the surrogate network at the edges of their tiles,
slices and CTA rounds, against the mma.sync kernels."""
import numpy as np
import pytest

import paper_2011_01740_gb300 as ens
from paper_2011_01740_gb300 import workloads as W

pytestmark = pytest.mark.gpu

# Both implementations round the same operands to BF16 and accumulate in FP32;
# another order of the FP32 sums can round an activation to the neighbouring
# BF16 value, 2^-8 of it, and with it at most that share of an output or of a
# gradient block (the targets lie about 3 from the outputs, so the residuals do
# not amplify it).
TOL = 2.0 ** -8


def _dev(a):
    import torch
    return torch.from_numpy(np.ascontiguousarray(a)).cuda()


def _both(members, call):
    out = []
    for impl in (1, 0):
        m = ens.ens_mlp_create(members, 3)
        try:
            ens.ens_mlp_set_params(m, W.mlp_params(members, seed=3))
            ens.ens_mlp_set_train_impl(m, impl)
            out.append(call(m))
            assert ens.ens_mlp_set_train_impl(m, impl) == 0          # no expired tensor-core wait
        finally:
            ens.ens_mlp_destroy(m)
    return out


# tiles of 128, slices of a multiple of 64 samples (8 from 1,024 samples on; at
# 1,100 two of them lie past the end), two rounds of tiles per CTA at 8,192 and
# up to 17 at 20,001 samples and 8 members
@pytest.mark.parametrize("n,members", [(1, 1), (64, 2), (65, 1), (127, 3), (128, 4), (129, 8), (192, 2), (1024, 1),
                                       (1025, 4), (1100, 3), (8192, 4), (20001, 8)])
def test_gradient_tiles_and_slices(n, members):
    x, y = W.mlp_batch(n, seed=n)
    y[:, 0] += 3.0
    xd, yd = _dev(x), _dev(y)

    def call(m):
        import torch
        grad = torch.full((members, W.MLP_PARAMS), float("nan"), device="cuda")
        return ens.ens_mlp_loss_grad(m, n, xd, yd, members, grad), grad.cpu().numpy().astype(np.float64)

    (l1, g1), (l0, g0) = _both(members, call)
    np.testing.assert_allclose(l1, l0, rtol=TOL)
    offs = np.cumsum([0] + [s for s, _ in W.MLP_FAN_IN])
    for k in range(members):
        for a, b in zip(offs[:-1], offs[1:]):
            assert np.linalg.norm(g1[k, a:b] - g0[k, a:b]) <= TOL * np.linalg.norm(g0[k, a:b]), (k, a)


@pytest.mark.parametrize("n,members", [(1, 1), (127, 2), (129, 8), (9728, 8), (9729, 8), (77825, 1), (20001, 5)])
def test_forward_tiles_and_rounds(n, members):
    x, _ = W.mlp_batch(n, seed=n)
    xd = _dev(x)

    def call(m):
        import torch
        out = torch.full((members, n, 2), float("nan"), device="cuda")
        ens.ens_mlp_forward(m, n, xd, out)
        return out.cpu().numpy()

    o1, o0 = _both(members, call)
    assert np.abs(o1 - o0).max() <= TOL * np.abs(o0).max()


def test_training_on_a_shuffled_ragged_set_matches_a_batch_at_a_time():
    """Rows picked through the shuffle, the last batch ragged: one epoch of two
    batches moves the loss as two gradients of the same rows do."""
    n, members = 1300, 2
    x, y = W.mlp_batch(n, seed=5)

    def call(m):
        return ens.ens_mlp_train(m, n, _dev(x), _dev(y), ens.make_train_cfg(epochs=3, batch=900, lr=1e-3), members)

    h1, h0 = _both(members, call)
    np.testing.assert_allclose(h1, h0, rtol=TOL)
