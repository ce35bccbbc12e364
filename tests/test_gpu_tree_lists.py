"""Lists and ranges of pixels over the cluster tree where a cluster is out of the ordinary: leaves without
one valid pixel (indices out of range sort last), and leaves wider than a hemisphere.  The tolerances are those of test_gpu_tree.py, whose direct
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
    nside, pairs = 256, 3.01e8 if prec == "f32c" else 9.01e7
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
    nside, pairs = 256, 2.01e9 if prec == "f32c" else 6.1e6
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


@pytest.mark.parametrize("nside", [49, 51, 52, 58, 59, 61, 62, 63])
def test_map_equator_ring(isw, nside):  # noqa: F811
    """One leaf around the whole equator: its mean direction is zero (49 to 58) or the rounding of its sum, with
    a pixel at the antipode of the centre for odd N_side."""
    S = torch.from_numpy(_samples(int(3.001e8 / (4 * nside)) + 1, nside)).cuda()
    ring = dict(pix0=2 * nside * (nside - 1) + 4 * nside * nside, npix=4 * nside)
    got, ref = isw.isw_map(nside, S, **ring), _direct(isw, nside, S, **ring)
    assert ((got - ref).abs().max() / ref.square().mean().sqrt()).item() <= TOL32
    assert isw.default_context().check_status()[0] == isw.OK


def _antipodes(isw, nside, count, seed):  # noqa: F811
    p = torch.randint(12 * nside * nside, (count // 2,), device="cuda", generator=torch.Generator("cuda").manual_seed(seed))
    return torch.cat([p, isw.hp_vec2pix_ring(nside, -isw.hp_pix2vec_ring(nside, pix=p))])


@pytest.mark.parametrize("prec,tol,count", [("f32c", TOL32, 192), ("f32c", TOL32, 260), ("f32c", TOL32, 1000), ("f64", TOL64, 4096),
                                            ("f64", TOL64, 4100)])
def test_map_antipodal_pairs(isw, prec, tol, count):  # noqa: F811
    """Scattered pixels with their antipodes in few leaves; and the N_side 2 sky repeated."""
    S = torch.from_numpy(_samples(int((3.001e8 if prec == "f32c" else 9.001e7) / count) + 1, 21)).cuda()
    sky2 = torch.arange(48, device="cuda").repeat(count // 48 + 1)[:count]
    for nside, pix in ((64, _antipodes(isw, 64, count, count)), (2, sky2)):
        got, ref = isw.isw_map(nside, S, pix=pix, prec=prec), _direct(isw, nside, S, pix=pix)
        assert ((got - ref).abs().max() / ref.square().mean().sqrt()).item() <= tol
    assert isw.default_context().check_status()[0] == isw.OK


@pytest.mark.parametrize("prec,tol,count", [("f32c", 1e-6, 12288), ("f64", 1e-12, 12288)])
def test_adjoint_antipodal_pairs(isw, prec, tol, count):  # noqa: F811
    S = torch.from_numpy(_samples(int((2.01e9 if prec == "f32c" else 6.1e6) / count) + 1, 22)).cuda()
    g = torch.randn(count, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    for nside, pix in ((64, _antipodes(isw, 64, count, 2)), (2, torch.arange(48, device="cuda").repeat(count // 48))):
        got = _adjoint(isw, nside, S, g, prec, 9, pix=pix)
        ref = _adjoint(isw, nside, S, g, "f64", 9, split=1, pix=pix)
        for a in (0, 3, 6):
            assert ((got - ref)[a : a + 3].abs().max() / ref[a : a + 3].abs().max()).item() <= tol
    assert isw.default_context().check_status()[0] == isw.OK


@pytest.mark.parametrize("prec,tol,tola", [("f32c", TOL32, 1e-6), ("f64", TOL64, 1e-12)])
@pytest.mark.parametrize("one", [6200, 12200])
def test_two_opposite_points(isw, prec, tol, tola, one):  # noqa: F811
    """A list of two opposite pixels, over and over: compact leaves but for the one that holds both."""
    nside, count = 64, 12400
    a = torch.tensor([20011], device="cuda")
    b = isw.hp_vec2pix_ring(nside, -isw.hp_pix2vec_ring(nside, pix=a))
    pix = torch.cat([a.expand(one), b.expand(count - one)])[torch.randperm(count, device="cuda", generator=torch.Generator("cuda").manual_seed(1))]
    S = torch.from_numpy(_samples(int((2.01e9 if prec == "f32c" else 9.1e7) / count) + 1, 23)).cuda()
    got, ref = isw.isw_map(nside, S, pix=pix, prec=prec), _direct(isw, nside, S, pix=pix)
    assert ((got - ref).abs().max() / ref.square().mean().sqrt()).item() <= tol
    g = torch.randn(count, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(5))
    got = _adjoint(isw, nside, S, g, prec, 9, pix=pix)
    ref = _adjoint(isw, nside, S, g, "f64", 9, split=1, pix=pix)
    for k in (0, 3, 6):
        assert ((got - ref)[k : k + 3].abs().max() / ref[k : k + 3].abs().max()).item() <= tola
    assert isw.default_context().check_status()[0] == isw.OK
