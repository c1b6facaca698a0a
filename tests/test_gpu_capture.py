"""What a handle counts as made stays true across streams and stream captures: the operator
is not set up inside a capture, 32-bit rows expanded inside one are made again outside, and
rows made on one stream are complete for every other."""
import os

import numpy as np
import pytest

import scenes
from oracle import operator as oop
from sph_testutil import lib_build, oracle_system, params_for, rel_l2, torch_cuda

pytestmark = pytest.mark.gpu


def _velocity(s, seed=1):
    torch = torch_cuda()
    v = np.zeros((s.n, 4), np.float32)
    v[:, :3] = np.random.default_rng(seed).normal(size=(s.n, 3))
    return torch.from_numpy(v).cuda()


def _captured(call):
    """(graph, the call's error or None)"""
    torch = torch_cuda()
    g, error = torch.cuda.CUDAGraph(), None
    torch.cuda.synchronize()
    with torch.cuda.stream(torch.cuda.Stream()):
        g.capture_begin()
        try:
            call()
        except RuntimeError as e:
            error = e
        finally:
            g.capture_end()
    torch.cuda.synchronize()
    return g, error


def test_set_up_inside_a_capture_is_refused():
    torch = torch_cuda()
    s = scenes.random_box(9, nf=2500, mu_spread=4.0)
    nb, _ = lib_build(s)
    v, y = _velocity(s), torch.zeros((s.n, 4), device="cuda")
    _, error = _captured(lambda: nb.apply(params_for(s), v, y))
    assert error is not None and "CUDA" in str(error)
    _, _, A = oracle_system(s)
    nb.apply(params_for(s), v, y)      # set up here, not taken for done
    want = A @ v.cpu().numpy()[:, :3].astype(np.float64)
    assert rel_l2(y.cpu().numpy()[:, :3], want) < 1e-5
    y.zero_()
    g, error = _captured(lambda: nb.apply(params_for(s), v, y))
    assert error is None
    g.replay()
    torch.cuda.synchronize()
    assert rel_l2(y.cpu().numpy()[:, :3], want) < 1e-5


def test_row_norms_are_captured_after_a_set_up():
    torch = torch_cuda()
    s = scenes.lava_box(1, n=12)
    nb, _ = lib_build(s)
    nb.setup(params_for(s))
    got, want = torch.zeros(s.n, device="cuda"), torch.zeros(s.n, device="cuda")
    g, error = _captured(lambda: nb.row_norms(params_for(s), got))
    assert error is None
    g.replay()
    nb.row_norms(params_for(s), want)
    torch.cuda.synchronize()
    np.testing.assert_array_equal(got.cpu().numpy(), want.cpu().numpy())
    _, _, A = oracle_system(s)
    np.testing.assert_allclose(got.cpu().numpy(), oop.row_norms2(A), rtol=2e-5)


def test_calls_are_captured_on_either_form_of_the_operator():
    """After an all-float64 solve the operator is set up along 32-bit rows only."""
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = scenes.lava_box(1, n=12)
    nb, t = lib_build(s)
    x, b = torch.from_numpy(s.x0).cuda(), torch.from_numpy(s.b).cuda()
    rep = nb.solve(params_for(s), binding.solve_opts(precision=binding.SPH_PREC_FP64), b, x)
    assert rep["status"] == 0
    v, y, norms = _velocity(s), torch.zeros((s.n, 4), device="cuda"), torch.zeros(s.n, device="cuda")
    nb.apply_noalloc(params_for(s), v, y)
    want = y.clone()

    def calls():
        nb.apply_noalloc(params_for(s), v, y)
        nb.row_norms(params_for(s), norms)

    y.zero_()
    g, error = _captured(calls)
    assert error is None
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(y.cpu().numpy(), want.cpu().numpy())
    _, _, A = oracle_system(s)
    np.testing.assert_allclose(norms.cpu().numpy(), oop.row_norms2(A), rtol=2e-5)


def test_rows_expanded_inside_a_capture():
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = scenes.lava_box(1, n=12)
    nb, t = lib_build(s)
    with np.load(os.path.join(os.path.dirname(binding.__file__), "weights", "scale_head_mlp.npz")) as w:
        mlp = binding.Mlp(w["params"])
    v, params = _velocity(s), params_for(s)
    want, got = torch.zeros(s.n, device="cuda"), torch.zeros(s.n, device="cuda")
    binding.mlp_row_scale(nb, params, mlp, v, want)
    nb.rebuild(t["pos"], t["rho"], t["mu"], t["ptype"], s.lo, s.hi, s.periodic, s.h)
    nb.setup(params)
    g, error = _captured(lambda: binding.mlp_row_scale(nb, params, mlp, v, got))
    assert error is None
    off, idx, _ = oracle_system(s)     # the graph has not run yet: the rows are made here
    o, i = nb.export()
    np.testing.assert_array_equal(o.cpu().numpy(), off)
    np.testing.assert_array_equal(i.cpu().numpy(), idx)
    g.replay()
    torch.cuda.synchronize()
    np.testing.assert_array_equal(got.cpu().numpy(), want.cpu().numpy())


def test_rows_made_on_one_stream_are_read_on_another():
    torch = torch_cuda()
    from paper_2206_14780_gb300 import binding

    s = scenes.lava_box(2, n=30)
    off, idx, _ = oracle_system(s)
    nb, t = lib_build(s)
    v, y = _velocity(s), torch.zeros((s.n, 4), device="cuda")
    first, second = torch.cuda.Stream(), torch.cuda.Stream()
    busy = torch.zeros((8192, 8192), device="cuda", dtype=torch.bfloat16)
    for _ in range(5):
        nb.rebuild(t["pos"], t["rho"], t["mu"], t["ptype"], s.lo, s.hi, s.periodic, s.h)
        torch.cuda.synchronize()
        with torch.cuda.stream(first):
            for _ in range(20):     # the rows are not made yet when the other stream asks
                busy @ busy
            nb.apply_otf(params_for(s), v, y)
        with torch.cuda.stream(second):
            o, i = nb.export()
        np.testing.assert_array_equal(o.cpu().numpy(), off)
        np.testing.assert_array_equal(i.cpu().numpy(), idx)
        torch.cuda.synchronize()
