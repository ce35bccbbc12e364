"""Lists and ranges of pixels over the cluster tree where a cluster is out of the ordinary: leaves without
one valid pixel (indices out of range sort last).  The tolerances are those of test_gpu_tree.py, whose direct
kernels are the reference."""
import numpy as np
import pytest

from test_gpu_tree import TOL32, TOL64, _adjoint, _direct, _samples, isw  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _bad_list(nside, good, bad):
    """good valid pixels with bad indices out of range among them, and the places of the valid ones"""
    rng = np.random.default_rng(good + bad)
    pix = np.concatenate([rng.integers(0, 12 * nside * nside, good), rng.choice([-1, 12 * nside * nside, -(2**62), 2**62], bad)])
    pix = torch.from_numpy(rng.permutation(pix)).cuda()
    return pix, (pix >= 0) & (pix < 12 * nside * nside)


LISTS32 = [(12288, 1), (12544, 1), (12544, 2), (12545, 255), (49920, 81), (12800, 700), (256, 13000)]
LISTS64 = [(12288, 1), (49152, 1), (50176, 2), (50176, 2500), (1024, 49000)]


@pytest.mark.parametrize("prec,tol,good,bad", [("f32c", TOL32, *k) for k in LISTS32] + [("f64", TOL64, *k) for k in LISTS64])
def test_map_list_with_empty_leaves(isw, prec, tol, good, bad):  # noqa: F811
    """Indices out of range fill whole leaves, alone under their parent or next to leaves of valid pixels: the
    valid pixels keep their values, the others are reported and left alone."""
    nside, pairs = 256, 3.01e8 if prec == "f32c" else 6.01e7
    S = torch.from_numpy(_samples(int(pairs / (good + bad)) + 1, 8)).cuda()
    pix, ok = _bad_list(nside, good, bad)
    ctx = isw.default_context()
    ctx.check_status()
    out = torch.full((good + bad,), 7.0, dtype=torch.float64, device="cuda")
    isw.isw_map(nside, S, pix=pix, prec=prec, out=out)
    assert ctx.check_status()[0] == isw.EINVAL
    assert (out[~ok] == 7.0).all()
    ref = _direct(isw, nside, S, pix=pix[ok])
    assert ((out[ok] - ref).abs().max() / ref.square().mean().sqrt()).item() <= tol
    ctx.check_status()


@pytest.mark.parametrize("prec,tol,good,bad", [("f32c", 1e-6, *k) for k in LISTS32] + [("f64", 1e-12, *k) for k in LISTS64])
def test_adjoint_list_with_empty_leaves(isw, prec, tol, good, bad):  # noqa: F811
    nside, pairs = 256, 3.01e8 if prec == "f32c" else 6.1e6
    n = int(pairs / (good + bad)) + 1
    S = torch.from_numpy(_samples(n, 12)).cuda()
    pix, ok = _bad_list(nside, good, bad)
    g = torch.randn(good + bad, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    ctx = isw.default_context()
    ctx.check_status()
    got = _adjoint(isw, nside, S, g, prec, 9, pix=pix)
    assert ctx.check_status()[0] == isw.EINVAL
    ref = _adjoint(isw, nside, S, g[ok], "f64", 9, split=1, pix=pix[ok])
    for a in (0, 3, 6):
        assert ((got - ref)[a : a + 3].abs().max() / ref[a : a + 3].abs().max()).item() <= tol
    ctx.check_status()
