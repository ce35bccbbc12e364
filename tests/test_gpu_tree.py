"""Maps over the cluster tree against the direct kernels (ISW_PARAM_SPLIT forces those), at sizes where
the tree can go wrong: sides at and around multiples of the 16-pixel leaf, sample counts around the
64-sample tiles, samples on one spot, in the beams, on pixel centres, skipped ones, weights of both
signs.  Tolerances: the truncation of the 8 x 8 interpolation is below 4e-7 of the rms next to the
strings (rate 5^-8 at a near radius of 3.5 half-sizes) and FP32 pair rounding adds up to 1.2e-6 where
samples spread over the sky; where thousands of terms of both signs meet in a few pixels FP32 gives
3e-6 in either kind of kernel, and the bar is the FP32 maps' 1e-5."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL32 = 2e-6
BAR32 = 1e-5


@pytest.fixture(scope="module")
def isw():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    import paper_1204_5041_gb300 as m

    m.build()
    return m


def _samples(n, seed, spot=None, cusp=False, mixed=False):
    """Samples with X.Xdot free, Xdot.X' = 0 and |Xdot|^2 + |X'|^2 = 1."""
    rng = np.random.default_rng(seed)
    x = rng.normal(size=(3, n))
    if spot is not None:
        x = np.array([0.3, -0.5, 0.4])[:, None] + spot * x
    x *= rng.uniform(0.3, 0.6, n) / np.linalg.norm(x, axis=0)
    u = rng.normal(size=(3, n))
    u /= np.linalg.norm(u, axis=0)
    p = rng.normal(size=(3, n))
    p -= (p * u).sum(0) * u
    p /= np.linalg.norm(p, axis=0)
    v = 1.0 - 10.0 ** rng.uniform(-8, -1, n) if cusp else rng.uniform(0.0, 0.95, n)
    S = np.empty((10, n))
    S[0:3], S[3:6], S[6:9] = x, v * u, np.sqrt(1 - v * v) * p
    S[9] = 1e-3 * (rng.choice([-1.0, 1.0], n) if mixed else 1.0)
    return S


def _direct(isw, nside, S, prec="f64", **kw):
    ctx = isw.default_context()
    ctx.set_param(isw.PARAM_SPLIT, 1)
    try:
        return isw.isw_map(nside, S, prec=prec, **kw)
    finally:
        ctx.set_param(isw.PARAM_SPLIT, 0)


def _check(isw, nside, S, prec, tol):
    ctx = isw.default_context()
    Sd = torch.from_numpy(np.ascontiguousarray(S)).cuda()
    ctx.check_status()
    got = isw.isw_map(nside, Sd, prec=prec)
    status, counts = ctx.check_status()
    launches = ctx.timing()[2]
    ref = _direct(isw, nside, Sd)
    status_d, counts_d = ctx.check_status()
    assert status == status_d and counts["skipped_samples"] == counts_d["skipped_samples"]
    assert counts["zero_pairs"] == counts_d["zero_pairs"]
    err = ((got - ref).abs().max() / ref.square().mean().sqrt()).item()
    print(f"nside {nside} n {S.shape[1]} {prec}: max err {err:.2e}, launches {launches}")
    assert err <= tol
    return got, ref


@pytest.mark.parametrize("nside,n", [(32, 8139), (33, 8192), (47, 8191), (48, 8193), (49, 4097), (100, 1000), (257, 127)])
def test_tree_sizes(isw, nside, n):
    _check(isw, nside, _samples(n, nside), "f32c", TOL32)


@pytest.mark.parametrize("kw", [dict(spot=1e-3), dict(spot=0.0), dict(cusp=True), dict(mixed=True), dict(spot=0.05, mixed=True)])
def test_tree_sample_layouts(isw, kw):
    _check(isw, 64, _samples(4001, 3, **kw), "f32c", BAR32)


def test_tree_skipped_zero_pairs_accumulate(isw):
    nside = 64
    S = _samples(4500, 5)
    centre = isw.hp_pix2vec_ring(nside).cpu().numpy()
    S[0:3, 7] = centre[:, 12345]              # on a pixel's line of sight
    S[3:6, 100] = [0.6, 0.8, 0.0]             # |Xdot| = 1
    got, ref = _check(isw, nside, S, "f32c", TOL32)
    Sd = torch.from_numpy(S).cuda()
    base = torch.full_like(got, 2.0)
    isw.isw_map(nside, Sd, prec="f32c", accumulate=True, out=base)
    rms = ref.square().mean().sqrt()
    assert ((base - 2.0 - got).abs().max() / rms).item() <= 1e-14
    again = isw.isw_map(nside, Sd, prec="f32c")
    assert torch.equal(again, got)            # reproducible
    isw.default_context().check_status()


def test_tree_near_pairs_and_observer(isw):
    """The FP64 near pairs are those of the direct kernels; an observer away from the origin."""
    S = torch.from_numpy(_samples(9000, 6)).cuda()
    ctx = isw.default_context()
    ctx.check_status()
    for x_obs in (None, (0.02, -0.01, 0.03)):
        got = isw.isw_map(64, S, prec="f32c", x_obs=x_obs)
        near = ctx.check_status()[1]["near_pairs"]
        _direct(isw, 64, S, "f32c", x_obs=x_obs)
        assert abs(near - ctx.check_status()[1]["near_pairs"]) <= 2   # |d| = rho to rounding
        ref = _direct(isw, 64, S, x_obs=x_obs)
        assert ((got - ref).abs().max() / ref.square().mean().sqrt()).item() <= TOL32
