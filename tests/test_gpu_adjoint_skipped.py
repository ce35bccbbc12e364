"""Skipped samples (|Xdot| >= 1, zero weight) get zero gradient rows from the direct kernels, too, where the last
pixel tile is padded."""
import pytest

from test_gpu_tree import _adjoint, _samples, isw  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32c", "f64"])
@pytest.mark.parametrize("nside,n,ngrad", [(3, 1, 6), (5, 130, 9), (9, 1000, 10), (16, 300, 6)])
def test_skipped_rows_are_zero(isw, prec, nside, n, ngrad):  # noqa: F811
    S = _samples(n, 5)
    skipped = slice(0, n, 7)
    S[3:6, skipped] = [[0.0], [0.6], [0.8]]
    g = torch.randn(12 * nside * nside, dtype=torch.float64, device="cuda", generator=torch.Generator("cuda").manual_seed(n))
    Sd = torch.from_numpy(S).cuda()
    ctx = isw.default_context()
    ctx.check_status()
    for pix in (None, torch.arange(11 * nside * nside, device="cuda")):
        got = _adjoint(isw, nside, Sd, g if pix is None else g[: len(pix)], prec, ngrad, split=1, pix=pix)
        assert ctx.check_status()[0] == isw.EDOMAIN
        used = torch.ones(n, dtype=torch.bool, device="cuda")
        used[skipped] = False
        assert (got[:, ~used] == 0).all() and torch.isfinite(got[:, used]).all()
        # the other samples' rows are those of a call without the skipped ones
        if used.any():
            alone = _adjoint(isw, nside, Sd[:, used].contiguous(), g if pix is None else g[: len(pix)], prec, ngrad, split=1, pix=pix)
            assert ((got[:, used] - alone).abs().max() / alone.abs().max()).item() <= 1e-6
            ctx.check_status()
