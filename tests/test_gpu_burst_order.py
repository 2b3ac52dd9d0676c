"""Bursts and plain steps as chains of dependent launches against the same launches one at a time: a child
process under CUDA_LAUNCH_BLOCKING=1 (the host waits for every launch, so none starts under another)
returns the same bits. Covers the passes that begin before the field solve in front of them has ended
(moments, nodal moments, three moments, both phase-space forms), bounded grids, the electrons' push beside
the ions', the energy sample between a solve and a push, and the sample that ends a burst. What both
could share, a charge grid cleared at the wrong time, is checked against a deposit of the particles."""
import os
import subprocess
import sys

import pytest
import torch

import paper_1610_01071_gb300 as pe

pytestmark = pytest.mark.gpu
ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

KINETIC = dict(electrons="kinetic", coarse="phase_space", n_v=32)
FORMS = {
    "moments": (512, 200, {}),
    "nodal": (1024, 90, dict(wavelet="d4")),
    "pressure": (256, 130, dict(coarse="moments_pressure")),
    "phase": (512, 200, dict(coarse="phase_space", n_v=32)),
    "wavelet": (256, 150, dict(coarse="phase_space", n_v=128, n_v_coarse=32, wavelet="coif4")),
    "walls": (512, 200, dict(boundary="absorbing")),
    "walls_phase": (512, 200, dict(boundary="absorbing", coarse="phase_space", n_v=32)),
    "kinetic": (256, 150, KINETIC),
    "kinetic_large": (8192, 40, KINETIC),
    "kinetic_energy": (128, 200, dict(KINETIC, te_active=True)),
}


def _run(form):
    ncell, ppc, kw = FORMS[form]
    kin = kw.get("electrons") == "kinetic"
    dt, K = 0.005 if kin else 0.1, 7
    cfg = pe.make_config(ncell, max(8, ncell // 16), K, ncell * ppc, (0.28 if kin else 0.5) * ncell, dt, 5 * K * dt,
                         v_th=0.3 if kin else 1.0, seed=11, newton_tol=1e-10, newton_maxit=80, **kw)
    ctx = pe.Context(cfg, device="cuda", stream=torch.cuda.Stream())
    ctx.load_initial(profile="slab") if kw.get("boundary") == "absorbing" else ctx.load_initial(0.3)
    out = []
    for _ in range(3):
        ctx.step()
        ctx.stream.synchronize()
        out += [ctx.get_coarse(), ctx.get_slope()]
    ctx.pic_steps(5)
    ctx.stream.synchronize()
    assert ctx.sync_status() == 0
    species = ["ions"] + (["electrons"] if kin else [])
    for sp in species:
        out += list(ctx.particles(species=sp))
    rho = ctx.view("rho", torch.int64, ncell)
    c, t, _, w = ctx.particles()
    assert torch.equal(rho, pe.deposit(c, t, w, ncell, ctx.diagnostics().s_w))
    out += [rho, ctx.view("E", torch.float64, ncell)]
    torch.cuda.synchronize()
    return [torch.as_tensor(x).cpu().clone() for x in out]


@pytest.fixture(scope="module")
def blocking(tmp_path_factory):
    path = str(tmp_path_factory.mktemp("blocking") / "out.pt")
    env = dict(os.environ, CUDA_LAUNCH_BLOCKING="1", PYTHONPATH=ROOT + os.pathsep + os.path.dirname(os.path.abspath(__file__)))
    r = subprocess.run([sys.executable, os.path.abspath(__file__), path], env=env, capture_output=True, text=True, timeout=300)
    assert r.returncode == 0, r.stderr[-2000:]
    return torch.load(path)


@pytest.mark.parametrize("form", list(FORMS))
def test_chains_equal_launches_one_at_a_time(form, blocking):
    want = blocking[form]
    for _ in range(2):
        got = _run(form)
        assert len(got) == len(want)
        for k, (x, y) in enumerate(zip(got, want)):
            assert torch.equal(x, y), k


if __name__ == "__main__":
    torch.save({f: _run(f) for f in FORMS}, sys.argv[1])
