"""Maps over the cluster tree against the direct kernels (ISW_PARAM_SPLIT forces those), at sizes where
the tree can go wrong: sides at and around multiples of the 16-pixel leaf, sample counts around the
64-sample tiles, samples on one spot, in the beams, on pixel centres, skipped ones, weights of both
signs.  Tolerances: the truncation of the 8 x 8 interpolation is below 4e-7 of the rms next to the
strings (rate 5^-8 at a near radius of 3.5 half-sizes) and FP32 pair rounding adds up to 1.2e-6 where
samples spread over the sky; where thousands of terms of both signs meet in a few pixels FP32 gives
3e-6 in either kind of kernel, and the bar is the FP32 maps' 1e-5.  FP64: truncation below 1e-16 and
rounding of 2e-15 of the rms against the maps' bar of 1e-12."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu
TOL32 = 2e-6
BAR32 = 1e-5
TOL64 = 1e-12


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


@pytest.mark.parametrize("nside,n", [(4, 5209), (9, 1100), (16, 331), (32, 8139), (33, 8192), (47, 8191), (48, 8193), (49, 4097), (100, 1000), (257, 127)])
def test_tree_sizes(isw, nside, n):
    _check(isw, nside, _samples(n, nside), "f32c", TOL32)


@pytest.mark.parametrize("nside,n", [(20, 12545), (33, 4609), (64, 1281), (65, 1217), (96, 1025), (100, 577), (257, 77)])
def test_tree_sizes_f64(isw, nside, n):
    _check(isw, nside, _samples(n, nside), "f64", TOL64)


@pytest.mark.parametrize("nside", [64, 65, 95, 130])
def test_tree_rings_f64(isw, nside):
    """Samples and beams at the poles, on the border of the polar caps and at azimuths where faces meet: the
    pixels' ring and azimuth forms have their edges there."""
    S = _samples(1300, nside + 1)
    k = 0
    for z in (1.0, -1.0, 2 / 3, -2 / 3, 0.0, 1 - 1e-12, 0.6666):
        for phi in np.arange(8) * np.pi / 4:
            s = np.sqrt(1 - z * z)
            v = np.array([s * np.cos(phi), s * np.sin(phi), z]) if abs(z) < 1 else np.array([0.0, 0.0, z])
            S[0:3, k] = 0.4 * v
            t = np.cross(v, [0.3, 0.5, 0.8])
            t /= np.linalg.norm(t)
            S[3:6, k + 1], S[6:9, k + 1] = -0.999 * v, np.sqrt(1 - 0.999**2) * t
            k += 2
    _check(isw, nside, S, "f64", TOL64)


@pytest.mark.parametrize("prec,tol", [("f32c", BAR32), ("f64", TOL64)])
@pytest.mark.parametrize("kw", [dict(spot=1e-3), dict(spot=0.0), dict(cusp=True), dict(mixed=True), dict(spot=0.05, mixed=True)])
def test_tree_sample_layouts(isw, kw, prec, tol):
    _check(isw, 64, _samples(4001, 3, **kw), prec, tol)


@pytest.mark.parametrize("prec,tol", [("f32c", TOL32), ("f64", TOL64)])
def test_tree_skipped_zero_pairs_accumulate(isw, prec, tol):
    nside = 64
    S = _samples(4500, 5)
    centre = isw.hp_pix2vec_ring(nside).cpu().numpy()
    S[0:3, 7] = centre[:, 12345]              # on a pixel's line of sight
    S[3:6, 100] = [0.6, 0.8, 0.0]             # |Xdot| = 1
    got, ref = _check(isw, nside, S, prec, tol)
    Sd = torch.from_numpy(S).cuda()
    base = torch.full_like(got, 2.0)
    isw.isw_map(nside, Sd, prec=prec, accumulate=True, out=base)
    rms = ref.square().mean().sqrt()
    assert ((base - 2.0 - got).abs().max() / rms).item() <= 1e-14
    again = isw.isw_map(nside, Sd, prec=prec)
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


@pytest.mark.parametrize("prec,tol,npix,n", [("f32c", TOL32, 12289, 24600), ("f64", TOL64, 49153, 1300)])
def test_tree_lists_and_ranges(isw, prec, tol, npix, n):
    """Pixels of a list (random, with repeats; an index out of range is reported and left alone) and of a
    range, summed in spatial order and written to their own places."""
    nside = 256
    S = torch.from_numpy(_samples(n, 8)).cuda()
    g = torch.Generator("cuda").manual_seed(4)
    pix = torch.randint(12 * nside * nside, (npix,), device="cuda", generator=g)
    pix[5] = pix[4]
    ctx = isw.default_context()
    ctx.check_status()
    for kw in (dict(pix=pix), dict(pix0=77, npix=npix)):
        got = isw.isw_map(nside, S, prec=prec, **kw)
        ref = _direct(isw, nside, S, **kw)
        assert ((got - ref).abs().max() / ref.square().mean().sqrt()).item() <= tol
    assert ctx.check_status()[0] == isw.OK
    pix[9] = 12 * nside * nside
    out = torch.full((npix,), 7.0, dtype=torch.float64, device="cuda")
    isw.isw_map(nside, S, pix=pix, prec=prec, out=out)
    assert ctx.check_status()[0] == isw.EINVAL and out[9].item() == 7.0
    ref = _direct(isw, nside, S, pix=pix[10:])
    assert ((out[10:] - ref).abs().max() / ref.square().mean().sqrt()).item() <= tol
    ctx.check_status()


@pytest.mark.parametrize("prec,tol,M,n", [("f32c", TOL32, 111, 8200), ("f32c", TOL32, 160, 4000), ("f64", TOL64, 222, 1300),
                                          ("f64", TOL64, 256, 1000)])
def test_tree_patch(isw, prec, tol, M, n):
    S = torch.from_numpy(_samples(n, M, spot=0.1)).cuda()
    e3 = S[0:3, 0].cpu().numpy() / np.linalg.norm(S[0:3, 0].cpu().numpy())
    e1 = np.cross(e3, [0.0, 0.0, 1.0])
    e1 /= np.linalg.norm(e1)
    frame = np.stack([e1, np.cross(e3, e1), e3])
    ctx = isw.default_context()
    got = isw.isw_map_patch(frame, M, 0.2, S, prec=prec)
    ctx.set_param(isw.PARAM_SPLIT, 1)
    try:
        ref = isw.isw_map_patch(frame, M, 0.2, S, prec="f64")
    finally:
        ctx.set_param(isw.PARAM_SPLIT, 0)
    assert ctx.check_status()[0] == isw.OK
    assert ((got - ref).abs().max() / ref.square().mean().sqrt()).item() <= tol


@pytest.mark.parametrize("prec,tol", [("f32c", TOL32), ("f64", TOL64)])
@pytest.mark.parametrize("M,width,n", [(33, 0.1, 30000), (64, 0.3, 8191), (100, 0.05, 3000), (512, 0.13, 129), (543, 0.2, 1000)])
def test_flat_tree(isw, prec, tol, M, width, n):
    """Flat-sky patches over the series tree against the direct kernel: both leaf sizes, ragged sides,
    samples in the field, beyond it and behind its plane, one exactly on a pixel.  The flat sky has no FP64
    near field: a pixel next to a sample is one term of any size, good to FP32's few ulp of itself, so the
    FP32 bound is tol * rms + 1e-6 of the value."""
    S = _samples(n, M, spot=0.1)
    S[0:3, : n // 8] = _samples(n // 8, M + 1)[0:3]        # all over the sky: half of these behind
    e3 = np.array([0.3, -0.5, 0.4]) / np.sqrt(0.5)
    e1 = np.cross(e3, [0.0, 0.0, 1.0])
    e1 /= np.linalg.norm(e1)
    frame = np.stack([e1, np.cross(e3, e1), e3])
    i, j = M // 2, M // 3
    S[0:3, 1] = 0.5 * (e3 + (i + 0.5 - 0.5 * M) * width / M * e1 + (j + 0.5 - 0.5 * M) * width / M * np.cross(e3, e1))
    Sd = torch.from_numpy(S).cuda()
    ctx = isw.default_context()
    got = isw.isw_map_patch(frame, M, width, Sd, prec=prec, approx=isw.FLATSKY)
    base = torch.full_like(got, 3.0)
    isw.isw_map_patch(frame, M, width, Sd, prec=prec, approx=isw.FLATSKY, accumulate=True, out=base)
    ctx.set_param(isw.PARAM_SPLIT, 1)
    try:
        ref = isw.isw_map_patch(frame, M, width, Sd, prec="f64", approx=isw.FLATSKY)
    finally:
        ctx.set_param(isw.PARAM_SPLIT, 0)
    assert ctx.check_status()[0] == isw.OK
    keep = torch.ones_like(ref, dtype=torch.bool)
    keep[j, i] = False       # 1 / |d| of a rounding error: any value
    rms = ref[keep].square().mean().sqrt()
    own = 1e-6 if prec == "f32c" else 1e-13
    assert ((got - ref).abs() <= tol * rms + own * ref.abs())[keep].all()
    assert ((base - 3.0 - got).abs() <= 1e-13 * (rms + ref.abs()))[keep].all()


def _adjoint(isw, nside, S, g, prec, ngrad, split=0, **kw):
    ctx = isw.default_context()
    ctx.set_param(isw.PARAM_SPLIT, split)
    try:
        return isw.isw_map_adjoint(nside, S, g, prec=prec, ngrad=ngrad, **kw)
    finally:
        ctx.set_param(isw.PARAM_SPLIT, 0)


@pytest.mark.parametrize("nside,n,ngrad,kw", [(32, 24539, 6, {}), (33, 24577, 10, {}), (47, 12000, 9, dict(spot=0.05, mixed=True)),
                                              (64, 6145, 6, dict(spot=1e-3)), (100, 2900, 10, {}), (257, 383, 6, {})])
def test_adjoint_tree(isw, nside, n, ngrad, kw):
    """FP32 gradients over the tree against the direct FP64 kernel, per block of rows, relative to the
    block's largest entry (the adjoint's bar, 1e-6); skipped samples get zero rows; reproducible."""
    S = _samples(n, nside, **kw)
    S[3:6, n // 2] = [0.0, 0.6, 0.8]
    Sd = torch.from_numpy(S).cuda()
    g = torch.randn(12 * nside * nside, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    ctx = isw.default_context()
    ctx.check_status()
    got = _adjoint(isw, nside, Sd, g, "f32c", ngrad)
    status, counts = ctx.check_status()
    ref = _adjoint(isw, nside, Sd, g, "f64", ngrad, split=4)
    assert status == isw.EDOMAIN and counts["skipped_samples"] == 1 and ctx.check_status()[1]["skipped_samples"] == 1
    assert (got[:, n // 2] == 0).all()
    used = torch.arange(n, device="cuda") != n // 2
    for a in range(0, ngrad, 3):
        b = (slice(a, min(a + 3, ngrad)), used)
        assert ((got - ref)[b].abs().max() / ref[b].abs().max()).item() <= 1e-6
    assert torch.equal(got, _adjoint(isw, nside, Sd, g, "f32c", ngrad))
    ctx.check_status()


def test_adjoint_tree_list(isw):
    nside, npix, n = 256, 12301, 24600
    S = torch.from_numpy(_samples(n, 12)).cuda()
    pix = torch.randint(12 * nside * nside, (npix,), device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    g = torch.randn(npix, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    for kw in (dict(pix=pix), dict(pix0=1234, npix=npix)):
        got = _adjoint(isw, nside, S, g, "f32c", 6, **kw)
        ref = _adjoint(isw, nside, S, g, "f64", 6, split=4, **kw)
        for b in (slice(0, 3), slice(3, 6)):
            assert ((got - ref)[b].abs().max() / ref[b].abs().max()).item() <= 1e-6
    assert isw.default_context().check_status()[0] == isw.OK


@pytest.mark.parametrize("nside,n,ngrad,kw", [(64, 407, 6, {}), (65, 448, 10, {}), (67, 449, 9, dict(spot=0.05, mixed=True)),
                                              (96, 4001, 6, dict(spot=1e-3)), (100, 1001, 10, dict(cusp=True)), (257, 63, 9, {})])
def test_adjoint_tree_f64(isw, nside, n, ngrad, kw):
    """FP64 gradients over the tree against the direct FP64 kernel, per block of rows relative to the block's
    largest entry; samples on the line of sight of a pixel, at a pole, skipped.  Bound: the two sum ~1e5 terms of
    either sign in different orders, 1e-15 of the largest terms, and a beam with 1 - |Xdot| = 1e-8 magnifies the
    rounding of B by up to 1e-16 / 1e-8 against the largest entry's own size; hence 1e-12 (1e-7 with cusps)."""
    S = _samples(n, nside, **kw)
    S[3:6, n // 2] = [0.0, 0.6, 0.8]
    S[0:3, 3] = [0.0, 0.0, 0.5]
    S[0:3, 7] = isw.hp_pix2vec_ring(nside).cpu().numpy()[:, 12345]
    Sd = torch.from_numpy(S).cuda()
    g = torch.randn(12 * nside * nside, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    ctx = isw.default_context()
    ctx.check_status()
    got = _adjoint(isw, nside, Sd, g, "f64", ngrad)
    status, counts = ctx.check_status()
    ref = _adjoint(isw, nside, Sd, g, "f64", ngrad, split=4)
    status_d, counts_d = ctx.check_status()
    assert status == status_d and counts["skipped_samples"] == counts_d["skipped_samples"] == 1
    assert counts["zero_pairs"] == counts_d["zero_pairs"]
    assert (got[:, n // 2] == 0).all()
    used = torch.arange(n, device="cuda") != n // 2
    for a in range(0, ngrad, 3):
        b = (slice(a, min(a + 3, ngrad)), used)
        assert ((got - ref)[b].abs().max() / ref[b].abs().max()).item() <= (1e-7 if "cusp" in kw else 1e-12)
    assert torch.equal(got, _adjoint(isw, nside, Sd, g, "f64", ngrad))
    ctx.check_status()


def test_adjoint_tree_list_f64(isw):
    nside, npix, n = 256, 49153, 500
    S = torch.from_numpy(_samples(n, 12)).cuda()
    pix = torch.randint(12 * nside * nside, (npix,), device="cuda", generator=torch.Generator("cuda").manual_seed(2))
    g = torch.randn(npix, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    for kw in (dict(pix=pix), dict(pix0=1234, npix=npix)):
        got = _adjoint(isw, nside, S, g, "f64", 6, **kw)
        ref = _adjoint(isw, nside, S, g, "f64", 6, split=4, **kw)
        for b in (slice(0, 3), slice(3, 6)):
            assert ((got - ref)[b].abs().max() / ref[b].abs().max()).item() <= 1e-12
    assert isw.default_context().check_status()[0] == isw.OK


@pytest.mark.parametrize("nside", [32, 33, 63, 64, 130])
def test_sky_table_bits(isw, nside):
    """The pixel directions of a full-sky map are those of a list of all pixels, bit for bit: one sample of
    weight, every pair in FP64, so a map value is one term of the pixel's direction."""
    npix = 12 * nside * nside
    S = _samples(300_000_000 // npix + 1, 9)
    S[9, 1:] = 0.0
    S = torch.from_numpy(S).cuda()
    pix = torch.arange(npix, device="cuda")
    ctx = isw.default_context()
    near_k = ctx.get_param(isw.PARAM_NEAR_K)
    ctx.set_param(isw.PARAM_NEAR_K, 1e5)
    try:
        sky, lst = isw.isw_map(nside, S), isw.isw_map(nside, S, pix=pix)
    finally:
        ctx.set_param(isw.PARAM_NEAR_K, near_k)
    assert (sky != 0).all() and torch.equal(sky, lst)
    ctx.check_status()
