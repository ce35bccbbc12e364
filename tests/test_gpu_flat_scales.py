"""Flat-sky patches at scales where squares leave the range of float: patches of extreme width take the direct
kernels."""
import numpy as np
import pytest

from test_gpu_tree import _samples, isw  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _field(n):
    S = _samples(n, 41, spot=0.1)
    S[0:3] = S[[2, 0, 1], :]           # most within a radian of the z axis
    S[2] = np.abs(S[2]) + 0.1
    return S


@pytest.mark.parametrize("prec", ["f32c", "f64"])
@pytest.mark.parametrize("width", [1e-50, 1e-40, 1e-25, 1e18, 1e30])
def test_extreme_widths(isw, width, prec):  # noqa: F811
    Sd = torch.from_numpy(_field(8200)).cuda()
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
