"""A batch against handles that change after it was made: the solve refuses on the host what
it was not made for (no kernel is launched), and follows a set-up that was changed and
changed back."""
import numpy as np
import pytest

import scenes
from oracle import operator as oop
from sph_testutil import lib_build, oracle_system, params_for, torch_cuda

pytestmark = pytest.mark.gpu


def _args(s, t):
    return t["pos"], t["rho"], t["mu"], t["ptype"], s.lo, s.hi, s.periodic, s.h


def _ensemble():
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    ens = [scenes.couette(0), scenes.lava_box(1, n=10, nu=3.0, dt=2e-4)]
    built = [lib_build(s) for s in ens]
    nbs, ts = [b[0] for b in built], [b[1] for b in built]
    batch = binding.Batch(nbs, [params_for(s) for s in ens])

    def solve():
        xs = [torch.from_numpy(s.x0).cuda() for s in ens]
        st, reps = batch.solve(binding.solve_opts(rtol=1e-8), [torch.from_numpy(s.b).cuda() for s in ens], xs)
        return st, [x.cpu().numpy() for x in xs]

    return binding, torch, ens, nbs, ts, solve


def _refused(binding, solve):
    launched = binding.launch_count()
    with pytest.raises(binding.SphError, match="INVALID"):
        solve()
    assert binding.launch_count() == launched


@pytest.mark.parametrize("then", ["apply", "setup", "solve"])
def test_a_rebuilt_handle_is_refused(then):
    """Also once the rebuilt handle has been set up again: the unions of the new lists may
    be larger than the shared memory the batch asks for."""
    binding, torch, ens, nbs, ts, solve = _ensemble()
    assert solve()[0] == 0
    s, t = ens[1], ts[1]
    moved = t["pos"].clone()
    moved[:, :3] += 1e-4 * (torch.rand(moved[:, :3].shape, device="cuda") - 0.5)
    nbs[1].rebuild(moved, *_args(s, t)[1:])
    _refused(binding, solve)
    params = params_for(s)
    v = torch.zeros((s.n, 4), device="cuda")
    if then == "apply":
        nbs[1].apply(params, v, torch.empty_like(v))
    elif then == "setup":
        nbs[1].setup(params)
    else:
        nbs[1].solve(params, binding.solve_opts(), torch.from_numpy(s.b).cuda(), torch.from_numpy(s.x0).cuda())
    _refused(binding, solve)


def test_other_parameters_are_refused_and_the_first_ones_followed():
    """A set-up for another dt or boundary changes A(dt) on the handle; after the set-up
    for the batch's own parameters it solves its own systems again, wherever the arrays
    lie now."""
    binding, torch, ens, nbs, ts, solve = _ensemble()
    st, first = solve()
    assert st == 0
    other = 1 - ens[0].boundary
    for params in (params_for(ens[0], 3.0 * ens[0].dt), binding.visc_params(ens[0].dt, other, ens[0].mean)):
        nbs[0].setup(params)
        _refused(binding, solve)
    nbs[0].setup(params_for(ens[0]))
    st, again = solve()
    assert st == 0
    for s, x, y in zip(ens, first, again):
        np.testing.assert_array_equal(x, y)
        _, _, A = oracle_system(s)
        assert oop.true_residual(A, y, s.b)[0] <= 1.1e-8
