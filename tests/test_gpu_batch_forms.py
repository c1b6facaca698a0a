"""Which form a batch runs on, and that each gives the oracle's solutions: row loops for
ensembles of small scenes and where a scene has no tiles, the tile form where large scenes
(8-slice tiles, with 4- and 1-slice ones beside them) or long rows prevail.

Tolerance: the 1e-8 true residual that the solve is asked for, by the oracle's matrix (its
float64 sums and the library's differ by a few 1e-15 of the right-hand side)."""
import numpy as np
import pytest

import scenes
from oracle import operator as oop
from sph_testutil import lib_build, oracle_system, params_for, torch_cuda
from test_gpu_list_rows import with_spray

pytestmark = pytest.mark.gpu


def _gauss(seed, **kw):
    return scenes.couette(seed, layers=4, kernel=1, **kw)


ENSEMBLES = {
    "small_scenes": (lambda: [scenes.couette(0), scenes.lava_box(1, n=10, nu=3.0, dt=2e-4), scenes.lava_box(4, n=14)],
                     128, False),
    "long_rows": (lambda: [_gauss(1, nx=12, ny=12, nz=13), _gauss(2, nx=18, ny=23, nz=18),
                           scenes.lava_box(3, n=12, layers=4, kernel=1)], 320, True),
    # 1,998, 1,021 and 100 slices
    "large_scenes": (lambda: [scenes.lava_box(4, n=35), scenes.lava_box(5, n=27), scenes.couette(6)], 128, True),
    "one_without_tiles": (lambda: [with_spray(scenes.random_box(9, nf=700, mu_spread=4.0), 0.013)[1],
                                   scenes.lava_box(5, n=12)], 128, False),
    "none_with_tiles": (lambda: [with_spray(scenes.random_box(k, nf=300 * k, mu_spread=4.0), 0.013)[1]
                                 for k in (3, 4)], 128, False),
}


@pytest.mark.parametrize("name", sorted(ENSEMBLES))
def test_batch_form(name):
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    make, maxnb, tiles = ENSEMBLES[name]
    ens = make()
    nbs = [lib_build(s, maxnb)[0] for s in ens]
    batch = binding.Batch(nbs, [params_for(s) for s in ens])
    bs = [torch.from_numpy(s.b).cuda() for s in ens]
    for _ in range(2):   # the tuning solve and a replayed one
        xs = [torch.from_numpy(s.x0).cuda() for s in ens]
        st, reps = batch.solve(binding.solve_opts(rtol=1e-8), bs, xs)
        assert st == 0, reps
    # the tile form has one variant; the row loops are timed in all eight
    tune = np.array(batch.info()["tune_ms"])
    assert (tune[1:] > 0).all() != tiles and (tune[1:] == 0).all() == tiles
    for s, x in zip(ens, xs):
        _, _, A = oracle_system(s)
        assert oop.true_residual(A, x.cpu().numpy(), s.b)[0] <= 1.1e-8, s.name
    batch.close()
