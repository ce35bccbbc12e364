"""The launch counts that isw_get_timing reports against the kernel nodes of a capture of the same call."""
import ctypes

import numpy as np
import pytest

from test_gpu_tree import _samples, isw  # noqa: F401

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu


def _kernel_nodes(call):
    """Kernels of one call, captured on a stream of its own."""
    rt = ctypes.CDLL(f"libcudart.so.{torch.version.cuda.split('.')[0]}")
    stream, graph, count = torch.cuda.Stream(), ctypes.c_void_p(), ctypes.c_size_t()
    with torch.cuda.stream(stream):
        h = ctypes.c_void_p(stream.cuda_stream)
        assert rt.cudaStreamBeginCapture(h, 2) == 0
        try:
            call()
        finally:
            assert rt.cudaStreamEndCapture(h, ctypes.byref(graph)) == 0
    assert rt.cudaGraphGetNodes(graph, None, ctypes.byref(count)) == 0
    nodes, kind, kernels = (ctypes.c_void_p * count.value)(), ctypes.c_int(), 0
    assert rt.cudaGraphGetNodes(graph, nodes, ctypes.byref(count)) == 0
    for n in nodes:
        assert rt.cudaGraphNodeGetType(ctypes.c_void_p(n), ctypes.byref(kind)) == 0
        kernels += kind.value == 0
    assert rt.cudaGraphDestroy(graph) == 0
    return kernels


CALLS = ["sky32", "sky64", "list32", "list64", "range32", "patch32", "patch64", "flat32", "flat64", "flat32_512", "adjoint32", "adjoint64",
         "adjoint32_list", "adjoint64_list", "cl"]


@pytest.mark.parametrize("direct", [False, True])
@pytest.mark.parametrize("name", CALLS)
def test_launch_counts(isw, name, direct):  # noqa: F811
    kind, prec = name.split("_")[0].rstrip("0123456789"), "f64" if "64" in name else "f32c"
    nside, n = 64, 230000
    S = torch.from_numpy(_samples(n, 3)).cuda()
    pix = torch.randint(12 * nside * nside, (12800,), device="cuda")
    M = 512 if "512" in name else 64
    g = torch.randn(12 * nside * nside, dtype=torch.float64, device="cuda")
    out, grad = torch.empty_like(g), torch.empty(6, n, dtype=torch.float64, device="cuda")
    patch = torch.empty(M, M, dtype=torch.float64, device="cuda")
    sel = pix if name.endswith("list") else None
    call = {
        "sky": lambda: isw.isw_map(nside, S, prec=prec, out=out),
        "list": lambda: isw.isw_map(nside, S, pix=pix, prec=prec, out=out[:12800]),
        "range": lambda: isw.isw_map(nside, S, pix0=5, npix=12800, prec=prec, out=out[:12800]),
        "patch": lambda: isw.isw_map_patch(np.eye(3), M, 0.1, S, prec=prec, out=patch),
        "flat": lambda: isw.isw_map_patch(np.eye(3), M, 0.1, S, prec=prec, approx=isw.FLATSKY, out=patch),
        "adjoint": lambda: isw.isw_map_adjoint(nside, S, g[: 12800 if sel is not None else None], pix=sel, prec=prec, out=grad),
        "cl": lambda: isw.isw_map_cl(nside, g, 128),
    }[kind]
    ctx = isw.default_context()
    ctx.set_param(isw.PARAM_WAIT_POLLS, 2**22 - 1 if direct else -1)
    try:
        call()                  # sizes the workspace
        torch.cuda.synchronize()
        ctx.timing()
        kernels = _kernel_nodes(call)
        assert ctx.timing()[2] == kernels
    finally:
        ctx.set_param(isw.PARAM_WAIT_POLLS, -1)
    ctx.check_status()
