"""The time step in other units of length and mass: the wall pressures' sums have to hold
where the kernel's constant times a pressure is far outside float32's range (a channel of
0.8 micrometres in metres and picograms: W(0) 2e20, pressures 2e19)."""
import numpy as np
import pytest

import scenes
from oracle import step as ostep
from sph_testutil import torch_cuda
from test_gpu_step import _params, _perturb, _stepper

pytestmark = pytest.mark.gpu


def _scaled(s, dx, rho0):
    """The scene with spacing dx and density rho0; velocities as they are."""
    f, m = dx / s.dx, rho0 / 1000.0
    s = s.copy()
    s.pos = s.pos.copy()
    s.pos[:, :3] *= np.float32(f)
    s.pos[:, 3] *= np.float32(f ** 3 * m)
    s.rho = (s.rho * np.float64(m)).astype(np.float32)
    s.mu = np.full_like(s.mu, 1e-6 * rho0)
    s.lo, s.hi = np.asarray(s.lo) * f, np.asarray(s.hi) * f
    s.h, s.dx = float(np.float32(s.h * f)), dx
    p = s.pos[:, :3]
    for ax in range(3):   # float32 coordinates inside the box
        if s.periodic[ax]:
            p[:, ax] = np.where(p[:, ax] >= s.hi[ax], np.float32(s.lo[ax]), p[:, ax])
            p[:, ax] = np.maximum(p[:, ax], np.nextafter(np.float32(s.lo[ax]), np.float32(np.inf)))
    return s


@pytest.mark.parametrize("kernel", [0, 1])
@pytest.mark.parametrize("dx,rho0,mu,dt", [(1e-9, 1000.0, 1e-8, 1e-5), (0.01, 1000.0, 1.0, 1e-4), (1e6, 1e-20, 1e-6, 1e2)])
def test_operator_matches_oracle_in_any_units(dx, rho0, mu, dt, kernel):
    """A(dt) where 2 dt / h^5 alone is beyond float32's range though its quotient by rho is
    not (nanometres in SI units), as it is, and far on the other side.  Bounds as in
    test_gpu_tiles: 1e-5 for the float32 apply, 1e-12 for the residual."""
    torch = torch_cuda()
    from sph_testutil import lib_build, oracle_system, params_for, rel_l2

    s = _scaled(scenes.couette(1, nx=13, ny=12, nz=13, layers=4 if kernel else 3, kernel=kernel), dx, rho0)
    s.mu, s.dt = np.full_like(s.mu, mu), dt
    nb, _ = lib_build(s, 320)
    _, _, A = oracle_system(s)
    rng = np.random.default_rng(3)
    v = np.zeros((s.n, 4), np.float32)
    v[:, :3] = rng.normal(size=(s.n, 3))
    y = torch.empty((s.n, 4), device="cuda")
    nb.apply(params_for(s), torch.from_numpy(v).cuda(), y)
    assert rel_l2(y.cpu().numpy()[:, :3], A @ v[:, :3].astype(np.float64)) < 1e-5
    x, b = rng.normal(size=(s.n, 3)), rng.normal(size=(s.n, 3))
    r = torch.empty((s.n, 3), dtype=torch.float64, device="cuda")
    nb.residual(params_for(s), torch.from_numpy(x).cuda(), torch.from_numpy(b).cuda(), r)
    scale = np.linalg.norm(b) + np.linalg.norm(abs(A) @ abs(x))
    assert np.linalg.norm(r.cpu().numpy() - (b - A @ x)) < 1e-12 * scale


@pytest.mark.parametrize("dx,rho0,c0,dt", [(1e-7, 1e18, 100.0, 3e-10), (0.01, 1000.0, 20.0, 2e-4), (1e4, 1e-3, 1e3, 3.0)])
def test_one_step_matches_oracle_in_any_units(dx, rho0, c0, dt):
    """Bounds as in test_gpu_step.test_one_step_matches_oracle."""
    torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = _perturb(_scaled(scenes.couette(1, nx=10, ny=8, nz=10), dx, rho0), 1)
    prm = dict(dt=dt, rho0=rho0, c0=c0, zeta=7.0, g=(0.5, -2.0, 0.0))
    st, t = _stepper(s)
    rep = st.step(_params(s, prm), binding.solve_opts(rtol=1e-10, eps_inner=1e-3))
    st.close()
    assert rep["status"] == 0, rep
    new, info = ostep.step(s, prm)
    fl = s.ptype == scenes.FLUID
    u = t["vel"].cpu().numpy()[:, :3].astype(np.float64)
    assert np.linalg.norm(u[fl] - info["u_new"][fl]) < 1e-5 * np.linalg.norm(info["u_new"][fl])
    np.testing.assert_allclose(t["rho"].cpu().numpy().astype(np.float64), new.rho.astype(np.float64), rtol=2e-6)
