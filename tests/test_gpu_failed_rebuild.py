"""A rebuild that fails leaves the handle without lists: every call that would read them is
refused on the host (nothing is launched), and the next successful build restores the handle."""
import numpy as np
import pytest

import scenes
from sph_testutil import gpu_solve, lib_build, oracle_system, params_for, rel_l2, torch_cuda

pytestmark = pytest.mark.gpu


def _args(s, t):
    return t["pos"], t["rho"], t["mu"], t["ptype"], s.lo, s.hi, s.periodic, s.h


@pytest.mark.parametrize("why", ["capacity", "crowded_cell", "position", "density"])
def test_calls_after_a_failed_rebuild_are_refused(why):
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    first, second = scenes.couette(2, nx=21, ny=9, nz=11), scenes.random_box(9, nf=2500, mu_spread=4.0)
    nb, _ = lib_build(first)
    params = params_for(second)
    t = binding.scene_tensors(second)
    bad = {k: v.clone() for k, v in t.items()}
    capacity, code = 128, "NONFINITE"
    if why == "capacity":
        capacity, code = 20, "CAPACITY"
    elif why == "crowded_cell":      # more than 64 (max_neighbors + 1) particles in one cell
        capacity, code = 1, "CAPACITY"
        bad["pos"][:400, :3] = bad["pos"][0, :3]
    elif why == "position":
        bad["pos"][5, 1] = float("nan")
    else:
        bad["rho"][7] = -1.0
    with pytest.raises(binding.SphError, match=code):
        nb.rebuild(*_args(second, bad), capacity)
    n = second.n
    vel = torch.zeros((n, 4), device="cuda")
    out = torch.zeros((n, 4), device="cuda")
    d3 = torch.zeros((n, 3), dtype=torch.float64, device="cuda")
    one = torch.ones(n, device="cuda")
    nb.n = n
    calls = {
        "export": lambda: binding._check(binding._lib.sph_neighbors_export(
            nb.handle, binding._ptr(torch.zeros(n + 1, dtype=torch.int64, device="cuda")),
            binding._ptr(torch.zeros(1 << 20, dtype=torch.int32, device="cuda")), binding._stream(None))),
        "viscosity": lambda: nb.set_viscosity(one),
        "setup": lambda: nb.setup(params),
        "apply": lambda: nb.apply(params, vel, out),
        "apply_otf": lambda: nb.apply_otf(params, vel, out),
        "apply_noalloc": lambda: nb.apply_noalloc(params, vel, out),
        "residual": lambda: nb.residual(params, d3, d3.clone(), d3.clone()),
        "solve": lambda: nb.solve(params, binding.solve_opts(), d3, d3.clone()),
        "solve64": lambda: nb.solve(params, binding.solve_opts(precision=binding.SPH_PREC_FP64), d3, d3.clone()),
        "row_norms": lambda: nb.row_norms(params, one.clone()),
        "mu": lambda: nb.mu_papanastasiou(vel, vel, 1.0, 1.0, 10.0, one.clone()),
        "warm": lambda: binding.warm_start(nb, params, None, vel, t["ptype"], d3, d3.clone()),
        "batch": lambda: binding.Batch([nb], [params]),
        "shard": lambda: binding.Shard(nb, params, 2),
    }
    launched = binding.launch_count()
    for name, call in calls.items():
        with pytest.raises(binding.SphError, match="INVALID"):
            call()
    assert binding.launch_count() == launched
    nb.rebuild(*_args(second, t), 128)
    off, idx, A = oracle_system(second)
    o, i = nb.export()
    np.testing.assert_array_equal(o.cpu().numpy(), off)
    np.testing.assert_array_equal(i.cpu().numpy(), idx)
    v = np.random.default_rng(1).normal(size=(n, 4)).astype(np.float32)
    nb.apply(params, torch.from_numpy(v).cuda(), out)
    assert rel_l2(out.cpu().numpy()[:, :3], A @ v[:, :3].astype(np.float64)) < 1e-5
    x, rep = gpu_solve(nb, second)
    assert rep["status"] == 0


def test_a_refused_argument_keeps_the_lists():
    """Arguments that are refused before the build begins leave the handle as it was."""
    torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = scenes.couette(2, nx=21, ny=9, nz=11)
    nb, t = lib_build(s)
    with pytest.raises(binding.SphError, match="INVALID"):
        nb.rebuild(*_args(s, t), 2000)
    x, rep = gpu_solve(nb, s)
    assert rep["status"] == 0
