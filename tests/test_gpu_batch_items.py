"""Work list of a batched pass: realisations from a handful of ions to several chunks, none a multiple of
a chunk, must give the coarse states of each realisation advanced alone (1e-8 of its largest component:
the batch partitions its field solves differently), through the eager, captured and replayed step."""
import numpy as np
import pytest
import torch

import paper_1610_01071_gb300 as pe

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def make(i, ncell, N, slab):
    cfg = pe.make_config(ncell, 16, 5, N, 0.5 * ncell, 0.1, 1.0, seed=40 + i, newton_tol=1e-10, newton_maxit=80,
                         boundary="absorbing" if slab else "periodic")
    ctx = pe.Context(cfg, device=DEV)
    if slab:
        ctx.load_initial(profile="slab")
    else:
        ctx.load_initial(0.1 + 0.05 * i)
    return ctx


@pytest.mark.parametrize("sizes", [[(64, 64 * 64, False)],
                                   [(64, 64 * 65, False), (128, 128 * 777, False), (256, 256 * 33, True)],
                                   [(512, 512 * 391, True), (64, 64 * 67, False), (1024, 1024 * 129, False)]])
def test_uneven_realisations_match_lone_contexts(sizes):
    alone = [make(i, *s) for i, s in enumerate(sizes)]
    group = [make(i, *s) for i, s in enumerate(sizes)]
    batch = pe.Batch(group)
    for _ in range(3):
        batch.step()
        for a, b in zip(alone, group):
            a.step()
            x, y = a.get_coarse().cpu().numpy(), b.get_coarse().cpu().numpy()
            assert np.max(np.abs(x - y)) <= 1e-8 * np.max(np.abs(x))
    for c in group:
        assert c.sync_status() == 0
