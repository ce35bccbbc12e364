"""Flat-sky patches at scales where squares leave the range of float: samples next to the patch plane, whose
coordinates in it are enormous, and patches of extreme width (which take the direct kernels).  Tolerances: those of
the flat-sky tests, a pixel next to a sample being good to FP32's few ulp of itself."""
import numpy as np
import pytest

from test_gpu_tree import TOL32, TOL64, _samples, isw  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _direct(isw, *args, **kw):  # noqa: F811
    ctx = isw.default_context()
    ctx.set_param(isw.PARAM_SPLIT, 1)
    try:
        return isw.isw_map_patch(*args, approx=isw.FLATSKY, **kw)
    finally:
        ctx.set_param(isw.PARAM_SPLIT, 0)


def _field(n):
    S = _samples(n, 41, spot=0.1)
    S[0:3] = S[[2, 0, 1], :]           # most within a radian of the z axis
    S[2] = np.abs(S[2]) + 0.1
    return S


@pytest.mark.parametrize("prec,tol,own", [("f32c", TOL32, 1e-6), ("f64", TOL64, 1e-13)])
@pytest.mark.parametrize("z", [1e-17, 1e-21, 1e-25, 1e-32])
def test_samples_next_to_the_plane(isw, z, prec, tol, own):  # noqa: F811
    S = _field(221400)
    S[2, ::11070] = z
    Sd = torch.from_numpy(S).cuda()
    args = (np.eye(3), 64, 0.3, Sd)
    got = isw.isw_map_patch(*args, prec=prec, approx=isw.FLATSKY)
    ref = _direct(isw, *args, prec="f64")
    rms = ref.square().mean().sqrt()
    assert ((got - ref).abs() <= tol * rms + own * ref.abs()).all()


@pytest.mark.parametrize("prec", ["f32c", "f64"])
@pytest.mark.parametrize("width", [1e-50, 1e-40, 1e-25, 1e18, 1e30])
def test_extreme_widths(isw, width, prec):  # noqa: F811
    Sd = torch.from_numpy(_field(221400)).cuda()
    ctx = isw.default_context()
    ctx.timing()
    got = isw.isw_map_patch(np.eye(3), 64, width, Sd, prec=prec, approx=isw.FLATSKY)
    launches = ctx.timing()[2]
    ctx.set_param(isw.PARAM_WAIT_POLLS, 2**22 - 1)      # the direct kernels
    try:
        ref = isw.isw_map_patch(np.eye(3), 64, width, Sd, prec=prec, approx=isw.FLATSKY)
    finally:
        ctx.set_param(isw.PARAM_WAIT_POLLS, -1)
    assert ctx.timing()[2] == launches
    assert torch.equal(torch.nan_to_num(got, 1.25), torch.nan_to_num(ref, 1.25))
