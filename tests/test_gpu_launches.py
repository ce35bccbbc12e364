"""The launch counts that isw_get_timing reports against the kernel nodes of a capture of the same call, and the
route of the calls that the cluster-tree tests make."""
import ctypes

import numpy as np
import pytest

import test_gpu_tree as tree
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
    nside, n = 64, 25000
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


def _sizes(test):
    """The arguments of a parametrised test, by name."""
    marks = [m for m in test.pytestmark if m.name == "parametrize"]
    cases = [{}]
    for m in marks:
        names = [a.strip() for a in m.args[0].split(",")]
        cases = [dict(c, **dict(zip(names, v if len(names) > 1 else (v,)))) for c in cases for v in m.args[1]]
    return cases


def _tree_calls():
    """(name, prec, call arguments) of the calls that test_gpu_tree.py makes over the tree"""
    for c in _sizes(tree.test_tree_sizes):
        yield "sky", "f32c", c["nside"], c["n"], None
    for c in _sizes(tree.test_tree_sizes_f64):
        yield "sky", "f64", c["nside"], c["n"], None
    for c in _sizes(tree.test_tree_rings_f64):
        yield "sky", "f64", c["nside"], 1300, None
    for prec in ("f32c", "f64"):
        for n in (4001, 4500):
            yield "sky", prec, 64, n, None
    for c in _sizes(tree.test_tree_lists_and_ranges):
        yield "list", c["prec"], 256, c["n"], c["npix"]
    for c in _sizes(tree.test_tree_patch):
        yield "patch", c["prec"], c["M"], c["n"], None
    for c in _sizes(tree.test_flat_tree):
        yield "flat", c["prec"], c["M"], c["n"], c["width"]
    for c in _sizes(tree.test_adjoint_tree):
        yield "adjoint", "f32c", c["nside"], c["n"], None
    for c in _sizes(tree.test_adjoint_tree_f64):
        yield "adjoint", "f64", c["nside"], c["n"], None
    yield "adjoint", "f32c", 256, 24600, 12301
    yield "adjoint", "f64", 256, 500, 49153


@pytest.mark.parametrize("kind,prec,side,n,arg", list(_tree_calls()))
def test_tree_is_taken(isw, kind, prec, side, n, arg):  # noqa: F811
    """A call of the sizes of test_gpu_tree.py takes another route than with the direct kernels asked for, so
    that these tests do not compare the direct kernels with themselves."""
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
    assert launches[0] > launches[1]
