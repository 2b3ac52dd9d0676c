"""Field solve at the edges of its launch shapes: blocks below a full warp, one warp, one block,
clusters of blocks of one warp up to the largest grid; charges below and beyond 2^53 (their
conversion rounds), empty nodes, and a start far enough away to be damped."""
import numpy as np
import pytest
import torch

import oracle as orc
import paper_1610_01071_gb300 as pe
from paper_1610_01071_gb300 import inputs

pytestmark = pytest.mark.gpu
DEV = torch.device("cuda:0")


@pytest.mark.parametrize("walls", [False, True])
@pytest.mark.parametrize("ncell,s_w,start", [(8, 30, 0.0), (16, 20, -4.0), (32, 30, 3.0), (64, 8, 0.0), (256, 30, -4.0),
                                             (512, 20, 0.0), (1024, 30, 3.0), (8192, 30, -4.0)])
def test_field_shapes_match_oracle(ncell, s_w, start, walls):
    dx = 0.5
    n = inputs.random_density(ncell, seed=ncell + 1, amp=0.4)
    n[:: max(4, ncell // 8)] = 0.0
    rho = np.rint(n * 2.0 ** (s_w + 24)).astype(np.int64)
    dens = rho * 2.0 ** -(s_w + 24)
    solve = orc.newton_pb_walls if walls else orc.newton_pb
    phi_o, _, fail = solve(dens, dx, phi0=np.zeros(ncell), tol=1e-12, maxit=80)
    assert fail == 0
    E_o = (orc.efield_walls if walls else orc.efield)(phi_o, dx)
    phi = torch.full((ncell,), start, dtype=torch.float64, device=DEV)
    st = torch.zeros(1, dtype=torch.int32, device=DEV)
    E, Ef, diag = pe.field(torch.from_numpy(rho).to(DEV), ncell, dx, s_w, phi, tol=1e-12, maxit=80, status=st,
                           boundary="absorbing" if walls else "periodic")
    assert int(st.item()) == 0 and int(diag[1]) == 1
    # both are Newton solutions to 1e-12; the FP64 residuals differ by rounding (a few 2^-52 / dx^2)
    assert np.max(np.abs(phi.cpu().numpy() - phi_o)) < 1e-9
    scale = np.max(np.abs(E_o))
    assert np.max(np.abs(E.cpu().numpy() - E_o)) < 1e-8 * scale
    assert np.max(np.abs(Ef.cpu().numpy() - E_o)) < 1e-6 * scale
