"""Tiles of eight slices (1,800 slices and more): lists, apply, residual, the cooperative
solve and the time step, against the oracle.  That a scene has them, and that its solve is
the cooperative kernel, is asserted from the apply's grid (one block per tile) and the
number of launches, so a change of the rules cannot empty these tests.

Tolerances as in test_gpu_tiles and test_gpu_step."""
import numpy as np
import pytest

import scenes
from oracle import operator as oop, step as ostep
from sph_testutil import lib_build, oracle_system, params_for, rel_l2, torch_cuda
from test_gpu_step import _params, _perturb, _stepper

pytestmark = pytest.mark.gpu

CASES = {
    "wendland": (lambda: scenes.lava_box(4, n=35), 128),                       # 63,878 rows, ragged last tile
    "gaussian": (lambda: scenes.lava_box(5, n=32, layers=4, kernel=1), 320),   # 57,600 rows of up to ~250
    "dynamic": (lambda: scenes.couette(6, nx=41, ny=30, nz=40, boundary=scenes.BC_DYNAMIC), 128),
}


def _slices_per_tile(nb, s):
    grid = nb.profile_read()["apply_grid"][0]
    return -(-(-(-s.n // 32)) // grid)


@pytest.mark.parametrize("name", sorted(CASES))
def test_lists_apply_residual_and_cooperative_solve(name):
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    make, maxnb = CASES[name]
    s = make()
    nb, _ = lib_build(s, maxnb)
    off, idx, A = oracle_system(s)
    o, i = nb.export()
    np.testing.assert_array_equal(o.cpu().numpy(), off)
    np.testing.assert_array_equal(i.cpu().numpy(), idx)
    rng = np.random.default_rng(11)
    v = np.zeros((s.n, 4), np.float32)
    v[:, :3] = rng.normal(size=(s.n, 3))
    y = torch.empty((s.n, 4), device="cuda")
    nb.apply(params_for(s), torch.from_numpy(v).cuda(), y)
    assert rel_l2(y.cpu().numpy()[:, :3], A @ v[:, :3].astype(np.float64)) < 1e-5
    x = rng.normal(size=(s.n, 3))
    r = torch.empty((s.n, 3), dtype=torch.float64, device="cuda")
    nb.residual(params_for(s), torch.from_numpy(x).cuda(), torch.from_numpy(s.b).cuda(), r)
    scale = np.linalg.norm(s.b) + np.linalg.norm(abs(A) @ abs(x))
    assert np.linalg.norm(r.cpu().numpy() - (s.b - A @ x)) < 1e-12 * scale
    b, xs = torch.from_numpy(s.b).cuda(), []
    for profiled in (False, True):   # the cooperative kernel, then the launched loop
        nb.profile(profiled)
        xt = torch.from_numpy(s.x0).cuda()
        before = binding.launch_count()
        rep = nb.solve(params_for(s), binding.solve_opts(rtol=1e-10), b, xt)
        launches = binding.launch_count() - before
        assert rep["status"] == 0 and rep["true_rel_res"] <= 1e-10
        assert (launches < rep["iters"]) == (not profiled), (launches, rep)
        assert _slices_per_tile(nb, s) == 8
        xs.append(xt.cpu().numpy())
        assert oop.true_residual(A, xs[-1], s.b)[0] <= 1.1e-10
    assert rel_l2(xs[0], xs[1]) < 1e-7


@pytest.mark.parametrize("boundary", [scenes.BC_DUMMY, scenes.BC_DYNAMIC])
def test_step(boundary):
    torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = _perturb(scenes.couette(1, nx=41, ny=30, nz=40, boundary=boundary), 1)
    nb, _ = lib_build(s)
    z = torch_cuda().zeros((s.n, 3), dtype=torch_cuda().float64, device="cuda")
    nb.solve(params_for(s), binding.solve_opts(), z, z.clone())
    assert _slices_per_tile(nb, s) == 8
    prm = dict(dt=2e-4, rho0=1000.0, c0=20.0, zeta=7.0, g=(0.5, -2.0, 0.0))
    st, t = _stepper(s)
    rep = st.step(_params(s, prm), binding.solve_opts(rtol=1e-10, eps_inner=1e-3))
    st.close()
    assert rep["status"] == 0, rep
    new, info = ostep.step(s, prm)
    fl = s.ptype == scenes.FLUID
    u = t["vel"].cpu().numpy()[:, :3].astype(np.float64)
    assert np.linalg.norm(u[fl] - info["u_new"][fl]) < 1e-5 * np.linalg.norm(info["u_new"][fl])
    np.testing.assert_allclose(t["rho"].cpu().numpy().astype(np.float64), new.rho.astype(np.float64), rtol=2e-6)
