"""The checks of test_gpu_tree.py at the sizes from which calls run over the cluster tree, and that they do: many of
that module's own sizes lie below the thresholds by now and compare the direct kernels with themselves."""
import numpy as np
import pytest

import test_gpu_tree as tree
from test_gpu_tree import TOL32, TOL64, _adjoint, _check, _samples, isw  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SKY32 = [(4, 5209), (9, 1100), (16, 331), (32, 8139), (49, 4097), (100, 1000), (257, 127)]
SKY64 = [(20, 18755), (33, 6913), (64, 1857), (65, 1823), (96, 833), (100, 769), (257, 127)]
RINGS64 = [80, 95, 96, 97, 128, 130]
PATCH = [("f32c", 111, 8200), ("f32c", 160, 4000), ("f64", 222, 1300), ("f64", 256, 1000)]
FLAT = [("f32c", TOL32, 33, 0.1, 826500), ("f32c", TOL32, 64, 0.3, 219800), ("f32c", TOL32, 100, 0.05, 90001), ("f32c", TOL32, 512, 0.13, 3457),
        ("f32c", TOL32, 543, 0.2, 3073), ("f64", TOL64, 33, 0.1, 45953), ("f64", TOL64, 64, 0.3, 12225), ("f64", TOL64, 100, 0.05, 5001)]
ADJOINT32 = [(32, 65201, 6, {}), (33, 61313, 10, {}), (47, 30209, 9, dict(spot=0.05, mixed=True)), (64, 16321, 6, dict(spot=1e-3)),
             (100, 6703, 10, {}), (257, 1023, 6, {})]
ADJOINT64 = [(32, 501, 6, {}), (45, 263, 9, {}), (64, 407, 6, {}), (65, 448, 10, {}), (257, 63, 9, {})]


@pytest.mark.parametrize("nside,n", SKY64)
def test_sky_f64(isw, nside, n):  # noqa: F811
    _check(isw, nside, _samples(n, nside), "f64", TOL64)


@pytest.mark.parametrize("nside", RINGS64)
def test_rings_f64(isw, nside):  # noqa: F811
    tree.test_tree_rings_f64(isw, nside)


@pytest.mark.parametrize("npix,n", [(49153, 1900), (4097, 22001)])
def test_lists_and_ranges_f64(isw, npix, n):  # noqa: F811
    tree.test_tree_lists_and_ranges(isw, "f64", TOL64, npix, n)


@pytest.mark.parametrize("prec,tol,M,width,n", FLAT)
def test_flat(isw, prec, tol, M, width, n):  # noqa: F811
    tree.test_flat_tree(isw, M=M, width=width, n=n, prec=prec, tol=tol)


@pytest.mark.parametrize("nside,n,ngrad,kw", ADJOINT32)
def test_adjoint(isw, nside, n, ngrad, kw):  # noqa: F811
    tree.test_adjoint_tree(isw, nside, n, ngrad, kw)


def test_adjoint_f64(isw):  # noqa: F811
    tree.test_adjoint_tree_f64(isw, 45, 263, 9, {})


@pytest.mark.parametrize("prec,tol,nside,npix,n", [("f32c", 1e-6, 256, 12301, 163000), ("f64", 1e-12, 256, 12301, 501),
                                                   ("f64", 1e-12, 32, 12288, 501)])
def test_adjoint_lists(isw, prec, tol, nside, npix, n):  # noqa: F811
    S = torch.from_numpy(_samples(n, 12)).cuda()
    pix = torch.randint(12 * nside * nside, (npix,), device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    g = torch.randn(npix, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    for kw in (dict(pix=pix), dict(pix0=0 if nside == 32 else 1234, npix=npix)):   # the range at N_side 32 is the sky
        got = _adjoint(isw, nside, S, g, prec, 6, **kw)
        ref = _adjoint(isw, nside, S, g, "f64", 6, split=4, **kw)
        for b in (slice(0, 3), slice(3, 6)):
            assert ((got - ref)[b].abs().max() / ref[b].abs().max()).item() <= tol
    assert isw.default_context().check_status()[0] == isw.OK


TAKEN = ([("sky", "f32c", *k, None) for k in SKY32] + [("sky", "f64", *k, None) for k in SKY64 + [(k, 1300) for k in RINGS64] + [(64, 4001), (64, 4500)]]
         + [("list", "f32c", 256, 24600, 12289), ("list", "f64", 256, 1900, 49153), ("list", "f64", 256, 22001, 4097)]
         + [("patch", *k, None) for k in PATCH] + [("flat", p, M, n, w) for p, _, M, w, n in FLAT] + [("flat", "f64", 512, 129, 0.1), ("flat", "f64", 543, 1000, 0.1)]
         + [("adjoint", "f32c", *k[:2], None) for k in ADJOINT32] + [("adjoint", "f64", *k[:2], None) for k in ADJOINT64]
         + [("adjoint", "f32c", 256, 163000, 12301), ("adjoint", "f64", 256, 501, 12301)])
DIRECT = [("sky", "f32c", 4, 5208, None), ("sky", "f64", 64, 1831, None), ("sky", "f64", 18, 40000, None), ("list", "f32c", 256, 24000, 12289),
          ("list", "f64", 256, 1800, 49153), ("flat", "f32c", 64, 219000, 0.1), ("flat", "f64", 100, 4990, 0.1), ("patch", "f64", 222, 1200, None), ("adjoint", "f32c", 64, 16200, None),
          ("adjoint", "f64", 44, 9000, None), ("adjoint", "f64", 33, 9000, None), ("adjoint", "f32c", 256, 160000, 12301)]


@pytest.mark.parametrize("kind,prec,side,n,arg,taken", [(*k, True) for k in TAKEN] + [(*k, False) for k in DIRECT])
def test_route(isw, kind, prec, side, n, arg, taken):  # noqa: F811
    """A call of these sizes makes more launches than with the direct kernels asked for, or, below the thresholds,
    the same."""
    S = torch.from_numpy(_samples(n, 3)).cuda()
    if kind == "sky":
        call = lambda: isw.isw_map(side, S, prec=prec)  # noqa: E731
    elif kind == "list":
        call = lambda: isw.isw_map(side, S, pix0=77, npix=arg, prec=prec)  # noqa: E731
    elif kind == "adjoint":
        g = torch.ones(arg or 12 * side * side, dtype=torch.float64, device="cuda")
        call = lambda: isw.isw_map_adjoint(side, S, g, pix0=0, npix=arg, prec=prec)  # noqa: E731
    else:
        approx = isw.FLATSKY if kind == "flat" else isw.FULLSKY
        call = lambda: isw.isw_map_patch(np.eye(3), side, arg or 0.2, S, prec=prec, approx=approx)  # noqa: E731
    ctx, launches = isw.default_context(), []
    try:
        for polls in (-1, 2**22 - 1):
            ctx.set_param(isw.PARAM_WAIT_POLLS, polls)
            ctx.timing()
            call()
            launches.append(ctx.timing()[2])
    finally:
        ctx.set_param(isw.PARAM_WAIT_POLLS, -1)
    ctx.check_status()
    assert launches[0] > launches[1] if taken else launches[0] == launches[1]
