"""Surrogate network at the edges of its tiles: widths that fill half a 128-row tile, batches that end
inside a 64-row stage of the weight-gradient contraction, and the batch sizes around the small-batch
form of inference (32 rows)."""
import numpy as np
import pytest
import torch

import paper_1610_01071_gb300 as pe
from oracle import mlp as omlp
from paper_1610_01071_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _net(dims, max_batch, seed):
    X, Y = inputs.regression_set(600, dims[0], dims[-1], seed + 1)
    p = inputs.random_mlp_params(dims, seed)
    net = pe.MLP(dims, max_batch=max_batch, device=DEV)
    net.init(0)
    net.set_params(_dev(p))
    net.fit_norm(_dev(X), _dev(Y))
    Ws, bs = omlp.unflatten(p, dims)
    Ws = [omlp.bf16_round(W) for W in Ws]
    (mu, sd), (mo, so) = omlp.zscore_stats(X), omlp.zscore_stats(Y)
    return net, X, Y, Ws, bs, (X - mu) / sd, (Y - mo) / so, mo, so


# BF16 activations and gradients (relative rounding 2^-9) through up to three layers: within 2e-2
@pytest.mark.parametrize("dims,B", [([64, 64], 32), ([64, 192, 64], 96), ([192, 64, 320], 160), ([320, 128, 64, 192], 544)])
def test_gradients_at_tile_edges(dims, B):
    net, X, Y, Ws, bs, x, t, _, _ = _net(dims, B, 11)
    loss = net.grad(_dev(X), _dev(Y), rows=_dev(np.arange(B, dtype=np.int32)))
    L, dWs, dbs = omlp.loss_and_grads(Ws, bs, x[:B], t[:B])
    assert loss == pytest.approx(L, rel=2e-2)
    gW, gb = omlp.unflatten(net.grads().cpu().numpy(), dims)
    for l in range(len(dims) - 1):
        for got, want in ((gW[l], dWs[l]), (gb[l], dbs[l])):
            assert np.linalg.norm(got - want) <= 2e-2 * np.linalg.norm(want), l
    assert net.sync_status() == 0


@pytest.mark.parametrize("dims", [[64, 64], [64, 192, 64], [640, 128, 192]])
def test_small_and_large_batches_give_the_same_rows(dims):
    net, X, _, Ws, bs, x, _, mo, so = _net(dims, 64, 21)
    full = net.forward(_dev(X[:64]))
    want = omlp.forward(Ws, bs, x[:64])[0]
    got = (full.cpu().numpy() - mo) / so
    assert np.linalg.norm(got - want) <= 2e-2 * np.linalg.norm(want)
    for B in (1, 31, 32, 33):  # 32 and below: the exchanged product, whose sums run in the same order
        assert torch.equal(net.forward(_dev(X[:B])), full[:B]), B
    assert net.sync_status() == 0
