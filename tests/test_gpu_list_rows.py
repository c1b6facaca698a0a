"""The 32-bit rows of the lists are the same, entry by entry, whether the neighbour search
ran over tiles or over global memory: everything that sums along them gives the same bits."""
import numpy as np
import pytest

import scenes
from sph_testutil import lib_build, torch_cuda

pytestmark = pytest.mark.gpu


def with_spray(s, h, n_spray=22000, seed=5):
    """The scene in a box grown beyond the support radius along y, and a scattering of
    particles there at about one per cell, which no tile can hold.  Returns (the scene in
    the larger box, the same with the scattered particles after its own)."""
    import copy

    rng = np.random.default_rng(seed)
    cell = 2.0 * h
    lo, hi = np.array(s.lo, float), np.array(s.hi, float)
    area = (hi[0] - lo[0]) * (hi[2] - lo[2])
    height = n_spray * cell ** 3 / area
    a = copy.deepcopy(s)
    a.hi = np.array([hi[0], hi[1] + 3 * cell + height, hi[2]])
    a.h = float(np.float32(h))
    p = rng.uniform(size=(n_spray, 3)) * np.array([hi[0] - lo[0], height, hi[2] - lo[2]]) + np.array(
        [lo[0], hi[1] + 3 * cell, lo[2]])
    b = copy.deepcopy(a)
    extra = np.concatenate([p, np.full((n_spray, 1), s.pos[0, 3])], axis=1)
    b.pos = np.concatenate([a.pos, extra]).astype(a.pos.dtype)
    for name, value in (("rho", s.rho[0]), ("mu", s.mu[0]), ("ptype", 0)):
        old = getattr(a, name)
        setattr(b, name, np.concatenate([old, np.full(n_spray, value, old.dtype)]))
    for name in ("b", "x0", "vel", "wall_vel"):
        old = getattr(a, name)
        setattr(b, name, np.concatenate([old, np.zeros((n_spray,) + old.shape[1:], old.dtype)]))
    return a, b


def has_tiles(nb, s):
    """Whether the solves on this handle run over tiles (sph_profile_counters.apply_variant 6)."""
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding
    from sph_testutil import params_for

    zero = torch.zeros((s.n, 3), dtype=torch.float64, device="cuda")
    nb.solve(params_for(s), binding.solve_opts(), zero, zero.clone())
    return nb.profile_read()["apply_variant"][0] == 6


@pytest.mark.parametrize("nf", [700, 14000])
def test_rows_of_tiles_and_of_the_global_scan(nf):
    torch = torch_cuda()
    from sph_testutil import params_for

    a, b = with_spray(scenes.random_box(9, nf=nf, mu_spread=4.0, mass_spread=0.3), 0.013)
    got = []
    for s, tiles in ((a, True), (b, False)):
        nb, _ = lib_build(s)
        assert has_tiles(nb, s) == tiles
        v = np.zeros((s.n, 4), np.float32)
        v[:a.n, :3] = np.random.default_rng(2).normal(size=(a.n, 3))
        y, norms = torch.empty((s.n, 4), device="cuda"), torch.empty(s.n, device="cuda")
        nb.apply_otf(params_for(s), torch.from_numpy(v).cuda(), y)
        nb.row_norms(params_for(s), norms)
        got.append((y[:a.n].cpu().numpy(), norms[:a.n].cpu().numpy()))
    (y0, norms0), (y1, norms1) = got
    assert np.isfinite(y0).all() and np.isfinite(norms0).all()
    np.testing.assert_array_equal(y0, y1)
    # the row norms run along the operator's own form: sums of at most ~100 positive float32
    # terms in another order, 100 half-units of float32's last place
    np.testing.assert_allclose(norms0, norms1, rtol=100 * 2.0 ** -24)
