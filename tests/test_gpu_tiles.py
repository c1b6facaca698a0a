"""The tile form of the lists and of A(dt): every tile size, both search regions, rows of
more than 255 entries, ragged ends and the fall-back to 32-bit rows, against the oracle.

Tolerances: neighbour sets bit for bit; the float32 apply 1e-5 relative L2 (sums of ~80
difference terms, a few ulp each); the float64 residual 1e-12 of ||b|| + |||A||x||
(coefficients to a few 2^-45)."""
import numpy as np
import pytest

import scenes
from oracle import operator as oop
from sph_testutil import lib_build, oracle_system, params_for, rel_l2, torch_cuda

pytestmark = pytest.mark.gpu


def _with_h(s, h, kernel=0):
    s.h, s.kernel = float(np.float32(h)), kernel
    return s


CASES = {
    # 64-row tiles: fewer than 1,100 slices; n mod 32 = 1, 31 and a single row
    "one_row": (lambda: scenes.random_box(1, nf=1, nw_layers=0, periodic=(0, 0, 0)), 128),
    "ragged_1": (lambda: scenes.random_box(5, nf=640 + 1, nw_layers=0, mu_spread=5.0, mass_spread=0.3), 128),
    "ragged_31": (lambda: scenes.random_box(6, nf=96 + 31, nw_layers=0, periodic=(0, 0, 0)), 128),
    "dynamic": (lambda: scenes.couette(2, nx=21, ny=9, nz=11, boundary=scenes.BC_DYNAMIC), 128),
    "gaussian": (lambda: scenes.couette(3, nx=12, ny=13, nz=15, layers=4, kernel=1), 320),
    # ~390 entries per row (16-bit counters of the plan)
    "wide_rows": (lambda: _with_h(scenes.random_box(7, nf=4000, mu_spread=3.0), 0.0221), 640),
    # 125 particles per cell: the large search region
    "large_region": (lambda: scenes.poiseuille(inv_dp=16, h_factor=2.5), 700),
    # about one particle per cell: too many cells for a tile, the global scan
    "sparse": (lambda: _with_h(scenes.random_box(8, nf=6000), 0.0045), 128),
    # 256-row tiles, ragged last tile; 128-row tiles (rows of ~250)
    "tiles_256": (lambda: scenes.lava_box(4, n=33), 128),
    "tiles_128": (lambda: scenes.lava_box(5, n=27, layers=4, kernel=1), 320),
}


@pytest.mark.parametrize("name", sorted(CASES))
def test_lists_apply_and_residual(name):
    torch = torch_cuda()
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
    vt = torch.from_numpy(v).cuda()
    yt = torch.full_like(vt, 7.0)
    nb.apply(params_for(s), vt, yt)
    y = yt.cpu().numpy()
    assert rel_l2(y[:, :3], A @ v[:, :3].astype(np.float64)) < 1e-5
    np.testing.assert_array_equal(y[:, 3], 0.0)
    x = rng.normal(size=(s.n, 3))
    rt = torch.empty((s.n, 3), dtype=torch.float64, device="cuda")
    nb.residual(params_for(s), torch.from_numpy(x).cuda(), torch.from_numpy(s.b).cuda(), rt)
    scale = np.linalg.norm(s.b) + np.linalg.norm(abs(A) @ abs(x))
    assert np.linalg.norm(rt.cpu().numpy() - (s.b - A @ x)) < 1e-12 * scale


def test_infinite_values_stay_in_their_rows():
    """A non-finite velocity reaches its own row and its neighbours' rows only (the
    filling of a row's last group of four reads no other row)."""
    torch = torch_cuda()
    s = scenes.couette(4, nx=13, ny=8, nz=9)
    nb, _ = lib_build(s)
    off, idx, A = oracle_system(s)
    for bad, value in ((0, np.inf), (s.n - 1, -np.inf), (s.n // 2, np.nan)):
        v = np.ones((s.n, 4), np.float32)
        v[bad, 1] = value
        yt = torch.empty((s.n, 4), device="cuda")
        nb.apply(params_for(s), torch.from_numpy(v).cuda(), yt)
        touched = np.zeros(s.n, bool)
        touched[A[:, bad].nonzero()[0]] = True
        y = yt.cpu().numpy()
        assert np.isfinite(y[~touched]).all() and np.isfinite(y[:, [0, 2]]).all()
        assert not np.isfinite(y[touched, 1]).any()


def test_forms_follow_each_other():
    """The 32-bit rows made on demand (forced apply form) and the tile form give one
    operator, before and after a change of dt and of the viscosity."""
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = scenes.random_box(9, nf=700, mu_spread=4.0)
    nb, t = lib_build(s)
    b = torch.from_numpy(s.b).cuda()
    for dt, scale in ((s.dt, 1.0), (2 * s.dt, 1.0), (2 * s.dt, 3.0)):
        nb.set_viscosity(t["mu"] * scale)
        xs = []
        for form in (0, 2, 0):
            x = torch.from_numpy(s.x0).cuda()
            rep = nb.solve(params_for(s, dt), binding.solve_opts(rtol=1e-9, apply_form=form), b, x)
            assert rep["status"] == 0
            xs.append(x.cpu().numpy())
        off, idx, _ = oracle_system(s)
        A = oop.assemble(s, off, idx, dt=dt, mu=s.mu * np.float32(scale))
        for x in xs:
            res, _ = oop.true_residual(A, x, s.b)
            assert res <= 1.1e-9


@pytest.mark.parametrize("name", ["one_row", "ragged_1", "gaussian", "large_region", "tiles_256", "tiles_128"])
def test_cooperative_solve_equals_the_launched_loop(name):
    """The one-kernel solve against the launched loop (which runs while the applies are
    profiled) and the oracle's matrix: both reach the same true residual, and at 1e-10 the
    two solutions agree to the residual times the system's conditioning (below 1e3 here)."""
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    make, maxnb = CASES[name]
    s = make()
    nb, _ = lib_build(s, maxnb)
    _, _, A = oracle_system(s)
    b = torch.from_numpy(s.b).cuda()
    xs = []
    for profiled in (False, True):
        nb.profile(profiled)
        x = torch.from_numpy(s.x0).cuda()
        rep = nb.solve(params_for(s), binding.solve_opts(rtol=1e-10), b, x)
        assert rep["status"] == 0 and rep["true_rel_res"] <= 1e-10
        xs.append(x.cpu().numpy())
        res, _ = oop.true_residual(A, xs[-1], s.b)
        assert res <= 1.1e-10
    assert rel_l2(xs[0], xs[1]) < 1e-7


def test_cooperative_solve_limits_and_stalls():
    """maxit, max_refine, a zero right-hand side and an exact start end the one-kernel solve
    as they end the loop."""
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = scenes.couette(5)
    nb, _ = lib_build(s)
    b = torch.from_numpy(s.b).cuda()
    for kw, status in ((dict(maxit=3), 6), (dict(max_refine=1, rtol=1e-10), 6), (dict(), 0)):
        reps = []
        for profiled in (False, True):
            nb.profile(profiled)
            x = torch.from_numpy(s.x0).cuda()
            reps.append(nb.solve(params_for(s), binding.solve_opts(**kw), b, x))
        assert [r["status"] for r in reps] == [status, status]
        if "maxit" in kw:
            assert reps[0]["iters"] == reps[1]["iters"] == 3
        if "max_refine" in kw:
            assert reps[0]["refinements"] == reps[1]["refinements"] == 1
    nb.profile(False)
    zero = torch.zeros_like(b)
    x = torch.zeros_like(b)
    rep = nb.solve(params_for(s), binding.solve_opts(), zero, x)
    assert rep["status"] == 0 and rep["iters"] == 0 and float(x.abs().max()) == 0.0


@pytest.mark.parametrize("make,maxnb", [
    # either side of the one-slice rule: 151 and 152 slices (fewer tiles than SMs, or not)
    (lambda: scenes.random_box(11, nf=151 * 32 - 5, nw_layers=0, mu_spread=3.0), 128),
    (lambda: scenes.random_box(12, nf=152 * 32 - 5, nw_layers=0, mu_spread=3.0), 128),
    # two slices per tile with walls, and with rows of ~250
    (lambda: scenes.couette(13, nx=20, ny=16, nz=19), 128),
    (lambda: scenes.couette(14, nx=18, ny=23, nz=18, layers=4, kernel=1), 320)])
def test_one_and_two_slice_tiles(make, maxnb):
    """Lists, apply, residual and a solve where the rule turns from one slice per tile to
    two; tolerances as above, the solve's true residual by the oracle's matrix."""
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = make()
    nb, _ = lib_build(s, maxnb)
    off, idx, A = oracle_system(s)
    o, i = nb.export()
    np.testing.assert_array_equal(o.cpu().numpy(), off)
    np.testing.assert_array_equal(i.cpu().numpy(), idx)
    v = np.zeros((s.n, 4), np.float32)
    v[:, :3] = np.random.default_rng(15).normal(size=(s.n, 3))
    yt = torch.empty((s.n, 4), device="cuda")
    nb.apply(params_for(s), torch.from_numpy(v).cuda(), yt)
    assert rel_l2(yt.cpu().numpy()[:, :3], A @ v[:, :3].astype(np.float64)) < 1e-5
    x = torch.from_numpy(s.x0).cuda()
    rep = nb.solve(params_for(s), binding.solve_opts(rtol=1e-8), torch.from_numpy(s.b).cuda(), x)
    assert rep["status"] == 0, rep
    assert oop.true_residual(A, x.cpu().numpy(), s.b)[0] <= 1.1e-8


def test_region_sizes_follow_each_other_on_one_handle():
    """A handle rebuilt on sets that need the small, the largest and again the small search
    region (it starts with the size of its last rebuild), and the global scan in between."""
    first = scenes.couette(2, nx=21, ny=9, nz=11)
    nb, _ = lib_build(first)
    for make, maxnb in (CASES["large_region"], (lambda: first, 128), CASES["sparse"], (lambda: first, 128), CASES["gaussian"]):
        s = make()
        t = _tensors(s)
        nb.rebuild(t["pos"], t["rho"], t["mu"], t["ptype"], s.lo, s.hi, s.periodic, s.h, maxnb,
                   kernel=getattr(s, "kernel", 0))
        off, idx, _ = oracle_system(s)
        o, i = nb.export()
        np.testing.assert_array_equal(o.cpu().numpy(), off)
        np.testing.assert_array_equal(i.cpu().numpy(), idx)


def _tensors(s):
    from paper_2206_14780_gb300 import binding

    return binding.scene_tensors(s)
