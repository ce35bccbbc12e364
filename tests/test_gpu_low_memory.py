"""Calls whose cluster-tree workspace the device has no room for run the direct kernels, as they do by
ISW_PARAM_WAIT_POLLS: the same bits.  The loop sums of lightcone_adjoint do without stored terms.  The rest of the device's memory is held by one tensor meanwhile."""
import contextlib

import numpy as np
import pytest

from test_gpu_tree import _samples, isw  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
LEFT = 24 << 20


@contextlib.contextmanager
def _little_memory():
    torch.cuda.synchronize()
    torch.cuda.empty_cache()
    hold = torch.empty(torch.cuda.mem_get_info()[0] - LEFT, dtype=torch.uint8, device="cuda")
    try:
        yield
    finally:
        del hold
        torch.cuda.empty_cache()


def _calls(isw, n, ctx):  # noqa: F811
    S = torch.from_numpy(_samples(n, 31)).cuda()
    pix = torch.arange(13000, device="cuda")
    g = torch.randn(13000, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    out = {k: torch.empty(13000, dtype=torch.float64, device="cuda") for k in ("f32c", "f64")}
    flat = {k: torch.empty(64, 64, dtype=torch.float64, device="cuda") for k in ("f32c", "f64")}
    grad = torch.empty(6, n, dtype=torch.float64, device="cuda")
    return {
        "map32": lambda: isw.isw_map(64, S, pix=pix, prec="f32c", out=out["f32c"], ctx=ctx),
        "map64": lambda: isw.isw_map(64, S, pix=pix, prec="f64", out=out["f64"], ctx=ctx),
        "adjoint32": lambda: isw.isw_map_adjoint(64, S, g, prec="f32c", pix=pix, out=grad, ctx=ctx),
        "adjoint64": lambda: isw.isw_map_adjoint(64, S, g, prec="f64", pix=pix, out=grad, ctx=ctx),
        "flat32": lambda: isw.isw_map_patch(np.eye(3), 64, 0.1, S, prec="f32c", approx=isw.FLATSKY, out=flat["f32c"], ctx=ctx),
        "flat64": lambda: isw.isw_map_patch(np.eye(3), 64, 0.1, S, prec="f64", approx=isw.FLATSKY, out=flat["f64"], ctx=ctx),
    }


@pytest.mark.parametrize("name", ["map32", "map64", "adjoint32", "adjoint64", "flat32", "flat64"])
def test_no_room_for_the_tree(isw, name):  # noqa: F811
    ctx = isw.Context()
    try:
        call = _calls(isw, 400000, ctx)[name]
        ctx.set_param(isw.PARAM_WAIT_POLLS, 2**22 - 1)
        want = call().clone()
        ctx.timing()
        ctx.set_param(isw.PARAM_WAIT_POLLS, -1)
        with _little_memory():
            got = call()
        direct = ctx.timing()[2]
        assert ctx.check_status()[0] == isw.OK
        assert torch.equal(got, want)
        call()                             # with room
        assert ctx.timing()[2] != direct
    finally:
        ctx.close()


def test_no_room_for_the_loop_terms(isw):  # noqa: F811
    nloops, nodes = 900, 512
    n = nloops * nodes
    rng = np.random.default_rng(2)
    P = rng.uniform(0.01, 0.1, (17, nloops))
    P[0:3], P[3:12] = rng.normal(size=(3, nloops)), np.eye(3).ravel()[:, None]
    P[13:15] = rng.integers(1, 6, (2, nloops))
    X = np.zeros((10, n))
    X[0], X[1] = np.repeat(np.arange(nloops), nodes), rng.uniform(0.0, 0.1, n)
    P, X = torch.from_numpy(P).cuda(), torch.from_numpy(X).cuda()
    gen = torch.Generator("cuda").manual_seed(1)
    tau, gs = (torch.randn(s, dtype=torch.float64, device="cuda", generator=gen) for s in ((n,), (9, n)))
    gn, gl = torch.empty(10, n, dtype=torch.float64, device="cuda"), torch.empty(17, nloops, dtype=torch.float64, device="cuda")
    ctx = isw.Context()
    try:
        call = lambda: isw.lightcone_adjoint(isw.BURDEN, X, tau, gs, loop_params=P, out=gn, out_loops=gl, ctx=ctx)  # noqa: E731
        call()
        want = gn.clone(), gl.clone()
        gl.zero_()
        ctx.close()
        ctx = isw.Context()
        with _little_memory():
            call()
        assert torch.equal(gn, want[0]) and torch.equal(gl, want[1]) and gl.abs().sum() > 0
        ctx.check_status()
    finally:
        ctx.close()
