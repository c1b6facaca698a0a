"""Everything that runs on a set without tiles (one tile that does not fit sends a set to
32-bit rows): solves with every form and reduction, CG, all-float64, time step, viscosity
pass, wall closure and features, against the oracle.  The scenes are ordinary ones beside a
spray of scattered particles; that they have no tiles is asserted.

Tolerances as in the tests of the same calls on sets with tiles."""
import numpy as np
import pytest

import scenes
from oracle import operator as oop, rheology, step as ostep, warmstart as ows
from sph_testutil import lib_build, oracle_system, params_for, rel_l2, torch_cuda
from test_gpu_list_rows import has_tiles, with_spray
from test_gpu_step import _params, _perturb, _stepper

pytestmark = pytest.mark.gpu

H = 0.013


def _box(boundary=scenes.BC_DUMMY):
    return with_spray(scenes.random_box(9, nf=900, mu_spread=4.0, mass_spread=0.2, boundary=boundary), H)[1]


def _built(s):
    nb, t = lib_build(s)
    assert not has_tiles(nb, s)
    return nb, t


@pytest.mark.parametrize("opts", [dict(), dict(merged_reductions=1), dict(launch_mode=1), dict(precision=1),
                                  dict(apply_form=1), dict(apply_form=5), dict(apply_form=6)],
                         ids=lambda o: "-".join(f"{k}{v}" for k, v in o.items()) or "default")
def test_solve(opts):
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = _box()
    nb, _ = _built(s)
    _, _, A = oracle_system(s)
    x = torch.from_numpy(s.x0).cuda()
    rep = nb.solve(params_for(s), binding.solve_opts(rtol=1e-9, **opts), torch.from_numpy(s.b).cuda(), x)
    assert rep["status"] == 0, rep
    assert oop.true_residual(A, x.cpu().numpy(), s.b)[0] <= 1.1e-9


@pytest.mark.parametrize("jacobi", [0, 1])
def test_cg(jacobi):
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = _box(scenes.BC_DYNAMIC)
    nb, _ = _built(s)
    _, _, A = oracle_system(s)
    x = torch.from_numpy(s.x0).cuda()
    rep = nb.solve(params_for(s), binding.solve_opts(rtol=1e-9, method=binding.SPH_SOLVER_CG, jacobi=jacobi),
                   torch.from_numpy(s.b).cuda(), x)
    assert rep["status"] == 0, rep
    assert oop.true_residual(A, x.cpu().numpy(), s.b)[0] <= 1.1e-9


@pytest.mark.parametrize("boundary", [scenes.BC_DUMMY, scenes.BC_DYNAMIC])
def test_step(boundary):
    torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = with_spray(scenes.couette(1, nx=10, ny=8, nz=10, boundary=boundary), H)[1]
    s = _perturb(s, 1)
    nb, _ = _built(s)
    nb.close()
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


def test_viscosity_pass():
    torch = torch_cuda()
    s = _box()
    rng = np.random.default_rng(4)
    s.vel = s.vel.copy()
    s.vel[:900, :3] = rng.normal(size=(900, 3))
    s.rheology = (100.0, 1000.0, 0.02)
    nb, _ = _built(s)
    off, idx, _ = oracle_system(s)
    want, _ = rheology.mu_pass(s, off, idx)
    out = torch.empty(s.n, device="cuda")
    nb.mu_papanastasiou(torch.from_numpy(s.vel).cuda(), torch.from_numpy(s.wall_vel).cuda(), *s.rheology, out)
    fl = s.ptype == scenes.FLUID
    assert (np.abs(out.cpu().numpy()[fl] - want[fl]) / want[fl]).max() < 1e-4


def test_wall_closure_and_features():
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    a, s = with_spray(scenes.random_box(9, nf=900, mu_spread=4.0), H)
    v = np.zeros((s.n, 4), np.float32)
    v[:, :3] = np.random.default_rng(5).normal(size=(s.n, 3))
    v[s.ptype != scenes.FLUID, :3] = s.vel[s.ptype != scenes.FLUID, :3]
    v[a.n:] = 0.0
    nb, t = _built(s)
    _, _, A = oracle_system(s)
    b = torch.from_numpy(s.b).cuda()
    x0 = torch.empty_like(b)
    binding.warm_start(nb, params_for(s), None, torch.from_numpy(v).cuda(), t["ptype"], b, x0)
    got, ref, fl = x0.cpu().numpy(), ows.start(A, s.b, v, None, s.ptype, 1.0), s.ptype == scenes.FLUID
    np.testing.assert_array_equal(got[fl], v[fl, :3].astype(np.float64))
    assert rel_l2(got[~fl], ref[~fl]) <= 1e-5
    # the features of the rows away from the spray are those of the set without it: their
    # sums run along the same 32-bit rows, the applies over another form (bf16 results)
    feats = []
    for sc, velocity in ((s, v), (a, v[:a.n])):
        h, _ = lib_build(sc)
        f = torch.empty((sc.n, 16), dtype=torch.int16, device="cuda")
        binding.mlp_features(h, params_for(sc), torch.from_numpy(np.ascontiguousarray(velocity)).cuda(), f)
        feats.append(f[:a.n].view(torch.bfloat16).float().cpu().numpy())
    # (the common scale of the features counts the spray's resting particles; compare directions)
    for c in range(16):
        x, y = feats[0][:, c], feats[1][:, c]
        nx, ny = np.linalg.norm(x), np.linalg.norm(y)
        assert (nx == 0) == (ny == 0)
        if nx > 0:
            assert np.linalg.norm(x / nx - y / ny) < 0.02
