"""What a rebuild remembers of the last one on its handle: the size of the tiles' search
region, down as well as up, and that a set has no tiles.  Seen in the number of kernels a
rebuild launches; the lists are the oracle's throughout."""
import numpy as np
import pytest

import scenes
from sph_testutil import lib_build, oracle_system, torch_cuda
from test_gpu_list_rows import has_tiles, with_spray

pytestmark = pytest.mark.gpu


def _rebuild(nb, s, maxnb):
    """Kernels launched by the rebuild."""
    from paper_2206_14780_gb300 import binding

    t = binding.scene_tensors(s)
    before = binding.launch_count()
    nb.rebuild(t["pos"], t["rho"], t["mu"], t["ptype"], s.lo, s.hi, s.periodic, s.h, maxnb,
               kernel=getattr(s, "kernel", 0))
    return binding.launch_count() - before


def _lists_are_the_oracles(nb, s):
    off, idx, _ = oracle_system(s)
    o, i = nb.export()
    np.testing.assert_array_equal(o.cpu().numpy(), off)
    np.testing.assert_array_equal(i.cpu().numpy(), idx)


def test_region_size_goes_down_again():
    torch_cuda()
    large, small = scenes.poiseuille(inv_dp=16, h_factor=2.5), scenes.couette(2, nx=21, ny=9, nz=11)
    nb, _ = lib_build(small)
    twice = _rebuild(nb, large, 700)          # searched with the smaller region first
    once = _rebuild(nb, large, 700)
    assert once < twice
    _lists_are_the_oracles(nb, large)
    assert _rebuild(nb, small, 128) <= once
    assert _rebuild(nb, large, 700) == twice  # the small set's region is the smaller one again
    _lists_are_the_oracles(nb, large)


def test_a_set_without_tiles_is_remembered_and_tried_again():
    torch_cuda()
    tiled, spray = with_spray(scenes.random_box(9, nf=700, mu_spread=4.0), 0.013)
    nb, _ = lib_build(spray)
    assert not has_tiles(nb, spray)
    again = _rebuild(nb, spray, 128)
    fresh, _ = lib_build(tiled)
    assert _rebuild(fresh, spray, 128) > again      # one failed search, then none
    _lists_are_the_oracles(nb, spray)
    # another set on the handle: tiles at once
    _rebuild(nb, tiled, 128)
    assert has_tiles(nb, tiled)
    # the same shape moved together: tiles within the next 33 rebuilds
    _rebuild(nb, spray, 128)
    import copy

    packed = copy.deepcopy(spray)
    rng = np.random.default_rng(3)
    n = packed.n
    k, d = np.arange(n), 0.01                       # 9 x 9 columns of the box's cross-section
    at = np.stack([k % 9, k // 81, k // 9 % 9], axis=1) + 0.5 + 0.2 * (rng.random((n, 3)) - 0.5)
    packed.pos[:, :3] = np.array(packed.lo) + at * d
    for tries in range(1, 40):
        _rebuild(nb, packed, 128)
        if has_tiles(nb, packed):
            break
    assert 1 < tries <= 33
    _lists_are_the_oracles(nb, packed)
