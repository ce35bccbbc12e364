"""Tunables and the cluster tree: those that the tree does not have ask for the direct kernels."""
import pytest

from test_gpu_tree import _samples, isw  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("kind", ["map", "adjoint"])
@pytest.mark.parametrize("value", [0.1, 4.0])
def test_far_field_distance(isw, kind, value):  # noqa: F811
    """ISW_PARAM_D_FAR takes effect on FP32 calls of every size: the bits are those of the direct kernels."""
    S = torch.from_numpy(_samples(17000, 3)).cuda()
    g = torch.randn(12 * 64 * 64, dtype=torch.float64, device="cuda")
    call = {"map": lambda: isw.isw_map(64, S, prec="f32c"), "adjoint": lambda: isw.isw_map_adjoint(64, S, g, prec="f32c")}[kind]
    ctx = isw.default_context()
    default, out = ctx.get_param(isw.PARAM_D_FAR), []
    try:
        for polls in (-1, 2**22 - 1):
            ctx.set_param(isw.PARAM_D_FAR, value)
            ctx.set_param(isw.PARAM_WAIT_POLLS, polls)
            out.append(call())
    finally:
        ctx.set_param(isw.PARAM_D_FAR, default)
        ctx.set_param(isw.PARAM_WAIT_POLLS, -1)
    assert torch.equal(out[0], out[1])
    assert not torch.equal(out[0], call())     # default settings: the tree


def test_variant_of_the_last_map(isw):  # noqa: F811
    S = torch.from_numpy(_samples(2000, 3)).cuda()
    ctx = isw.Context()
    try:
        assert ctx.get_param(isw.PARAM_VARIANT) == -1
        isw.isw_map(4, S, prec="f32c", ctx=ctx)            # 384,000 pairs: the direct kernels
        assert ctx.get_param(isw.PARAM_VARIANT) == 0
        isw.isw_map(64, S, prec="f32c", ctx=ctx)
        assert ctx.get_param(isw.PARAM_VARIANT) == -1
        isw.isw_map(64, S, prec="f64", ctx=ctx)
        ctx.set_param(isw.PARAM_VARIANT, 1)
        isw.isw_map(64, S, prec="f32c", ctx=ctx)
        assert ctx.get_param(isw.PARAM_VARIANT) == 1
    finally:
        ctx.close()


@pytest.mark.parametrize("value", [0.0, 1e-3, 1.0])
def test_far_field_distance_of_the_f64_adjoint(isw, value):  # noqa: F811
    """Samples on and next to the pixels' lines of sight keep their gradients at any ISW_PARAM_D_FAR."""
    nside = 64
    S = _samples(3000, 3)
    centre = isw.hp_pix2vec_ring(nside).cpu().numpy()
    S[0:3, :300] = 0.5 * centre[:, 1000:1300]
    S[0:3, 300:600] = 0.5 * centre[:, 2000:2300] + 1e-9
    S = torch.from_numpy(S).cuda()
    g = torch.randn(12 * nside * nside, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(1))
    ctx = isw.default_context()
    default, out = ctx.get_param(isw.PARAM_D_FAR), {}
    try:
        for polls in (-1, 2**22 - 1):
            ctx.set_param(isw.PARAM_D_FAR, value)
            ctx.set_param(isw.PARAM_WAIT_POLLS, polls)
            out[polls] = isw.isw_map_adjoint(nside, S, g, prec="f64", ngrad=9)
    finally:
        ctx.set_param(isw.PARAM_D_FAR, default)
        ctx.set_param(isw.PARAM_WAIT_POLLS, -1)
    got, ref = out.values()
    for a in (0, 3, 6):
        # relative to each sample's own gradient: those on a line of sight are 1e12 times the others
        scale = ref[a : a + 3].norm(dim=0) + ref[a : a + 3].norm(dim=0).median()
        assert (((got - ref)[a : a + 3].norm(dim=0)) / scale).max().item() <= 1e-11
    ctx.check_status()
