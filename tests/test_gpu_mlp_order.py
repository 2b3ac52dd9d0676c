"""Evaluations queued behind weight updates on one stream, through the C entry points and with nothing
between them that synchronises: the same results as when the host waits after every update. The
network is large enough that an update takes tens of microseconds."""
import numpy as np
import pytest
import torch

import paper_1610_01071_gb300 as pe
from paper_1610_01071_gb300 import _binding as pb
from paper_1610_01071_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")
DIMS, B, ROUNDS = [512, 1024, 1024, 512], 128, 200


def _dev(x):
    return torch.from_numpy(np.ascontiguousarray(x)).to(DEV)


def _rounds(how, rows, wait):
    lib, s = pe.load(), torch.cuda.Stream(DEV)
    X, Y = (_dev(a) for a in inputs.regression_set(512, DIMS[0], DIMS[-1], 3))
    x = X[:rows].contiguous()
    y = torch.full((ROUNDS, rows, DIMS[-1]), float("nan"), device=DEV)
    torch.cuda.synchronize()
    net = pe.MLP(DIMS, max_batch=B, device=DEV, stream=s)
    net.init(5)
    net.fit_norm(X, Y)
    h = net._h
    for r in range(ROUNDS):
        if how == "adam":
            pb.check(lib.pe_mlp_grad(h, pb._ptr(X), pb._ptr(Y), X.shape[0], None, B, None), "grad")
            pb.check(lib.pe_mlp_adam(h, 1e-2, 0.9, 0.999, 1e-8), "adam")
        else:  # one step runs eagerly, without a graph
            pb.check(lib.pe_mlp_train(h, pb._ptr(X), pb._ptr(Y), X.shape[0], B, 0, 9, 1, 1e-2, None), "train")
        if wait:
            s.synchronize()
        pb.check(lib.pe_mlp_forward(h, pb._ptr(x), 0, rows, pb._ptr(y[r]), 0), "forward")
    s.synchronize()
    assert net.sync_status() == 0
    return y


@pytest.mark.parametrize("rows", [1, 32, 33])  # 32 and below: the form that loads its weights early
@pytest.mark.parametrize("how", ["adam", "train"])
def test_evaluations_read_the_updated_weights(how, rows):
    queued, waited = _rounds(how, rows, False), _rounds(how, rows, True)
    assert torch.equal(queued, waited)
    assert not torch.equal(waited[0], waited[-1])  # the updates do change the outputs
