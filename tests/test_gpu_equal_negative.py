"""Equal-weight loading of a profile with negative densities, whose cumulative mass does not ascend: several
cells then hold a point. The one taken is the last that the walk forward from the cell found for the
smallest point of the slot's group of four reaches (the slot's own point in the ragged end), as a host
evaluation of that rule gives it. Masses are small integers and their sum a power of two, so the table
is exact."""
import numpy as np
import pytest
import torch

import paper_1610_01071_gb300 as pe

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


def _points(n):
    s = np.arange(n, dtype=np.int64)
    rev = np.array([int(f"{k:012b}"[::-1], 2) for k in range(4096)], dtype=np.int64)
    return np.where((s | 4095) < n, (s & ~4095) | rev[s & 4095], s)


def _cells(prof, n):
    m = (prof[:-1] + prof[1:]) / 2.0
    C = np.concatenate([[0.0], np.cumsum(m)])
    first = np.clip(np.ceil(C * (n / C[-1]) - 0.5), 0, n).astype(np.int64)
    first[-1] = n
    ncl = len(m)
    pts = _points(n)
    start = pts.copy()
    full = n & ~3
    start[:full] = pts[:full].reshape(-1, 4).min(1).repeat(4)
    out = np.empty(n, np.int32)
    for k, (a, b) in enumerate(zip(start, pts)):
        lo, hi = 0, ncl
        while hi - lo > 1:
            mid = (lo + hi) >> 1
            lo, hi = (mid, hi) if first[mid] <= a else (lo, mid)
        while lo < ncl - 1 and first[lo + 1] <= b:
            lo += 1
        out[k] = lo
    return out


@pytest.mark.parametrize("ncell", [8, 64, 1024])
@pytest.mark.parametrize("n", [7, 4095, 4097, 20003])
def test_cells_of_a_table_that_does_not_ascend(ncell, n):
    rng = np.random.default_rng(ncell)
    prof = rng.integers(-2, 5, ncell).astype(np.float64) * 2.0
    total = 2.0 ** np.ceil(np.log2(max(8.0, prof.sum())))  # the masses sum to this
    prof[ncell // 2] += total - (prof.sum() - (prof[0] + prof[-1]) / 2.0)
    assert (prof < 0).any() and (prof[:-1] + prof[1:]).sum() / 2 == total
    p = torch.from_numpy(prof.astype(np.float32)).to(DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    cell, theta, _, w, rho = pe.quiet_start_equal(n, ncell, p, torch.zeros_like(p), 1.0, 3, 8, status=st)
    assert int(st.item()) == 0
    assert np.array_equal(cell.cpu().numpy(), _cells(prof, n))
    assert bool((w == np.float32(total / n)).all())
    assert torch.equal(rho, pe.deposit(cell, theta, w, ncell, 8))
