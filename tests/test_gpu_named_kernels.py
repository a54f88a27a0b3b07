"""A step kernel asked for by name is the one that is launched, whatever the size of the grid; the
library's own choice (LB_KERNEL_AUTO, or a request that does not apply) takes one node per thread where that
is faster.  The launch is read from a captured graph.  And the two-node kernels give the bits of the
one-node kernel above the sizes at which the library's own choice takes them, with partial last blocks, and
with the paper's literal equilibrium."""
import ctypes

import pytest
import torch

from helpers import TORCH_DTYPE
from paper_1909_08406_gb300 import lb
from paper_1909_08406_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

ONE, ROWS, PAIRS, TMA, WS = "6k_stepI", "7k_step2I", "8k_step2xI", "10k_step_tmaI", "9k_step_wsI"


class _KernelNode(ctypes.Structure):  # CUDA_KERNEL_NODE_PARAMS_v2
    _fields_ = [("func", ctypes.c_void_p), ("dims", ctypes.c_uint * 7), ("params", ctypes.c_void_p),
                ("extra", ctypes.c_void_p), ("kern", ctypes.c_void_p), ("ctx", ctypes.c_void_p)]


def _launched(ctx, stream):
    """Mangled names of the kernels that one step launches, from a captured graph."""
    cu = ctypes.CDLL("libcuda.so.1")

    def call(f, *args):
        assert f(*args) == 0, f.__name__

    graph, count, names = ctypes.c_void_p(), ctypes.c_size_t(), []
    call(cu.cuStreamBeginCapture_v2, ctypes.c_void_p(stream), 1)
    lb.lb_step(ctx, 1)
    call(cu.cuStreamEndCapture, ctypes.c_void_p(stream), ctypes.byref(graph))
    call(cu.cuGraphGetNodes, graph, None, ctypes.byref(count))
    nodes = (ctypes.c_void_p * count.value)()
    call(cu.cuGraphGetNodes, graph, nodes, ctypes.byref(count))
    for n in nodes:
        kind, p, name = ctypes.c_int(), _KernelNode(), ctypes.c_char_p()
        call(cu.cuGraphNodeGetType, ctypes.c_void_p(n), ctypes.byref(kind))
        if kind.value != 0:  # CU_GRAPH_NODE_TYPE_KERNEL
            continue
        call(cu.cuGraphKernelNodeGetParams_v2, ctypes.c_void_p(n), ctypes.byref(p))
        if p.func:
            call(cu.cuFuncGetName, ctypes.byref(name), ctypes.c_void_p(p.func))
        else:
            call(cu.cuKernelGetName, ctypes.byref(name), ctypes.c_void_p(p.kern))
        names.append(name.value.decode())
    call(cu.cuGraphDestroy, graph)
    return names


CASES = [((33, 18, 20), "f32", lb.LB_KERNEL_DIRECT1, ONE), ((33, 18, 20), "f32", lb.LB_KERNEL_DIRECT2, ROWS),
         ((33, 18, 20), "f16", lb.LB_KERNEL_DIRECT2R, ROWS), ((6, 3, 5), "f16", lb.LB_KERNEL_DIRECT2X, PAIRS),
         ((6, 3, 5), "bf16", lb.LB_KERNEL_DIRECT2XL, PAIRS), ((160, 62, 5), "f32", lb.LB_KERNEL_DIRECT2, ROWS),
         ((150, 66, 5), "f32", lb.LB_KERNEL_DIRECT2, ROWS), ((128, 2, 2), "f32", lb.LB_KERNEL_STAGED, TMA),
         ((128, 2, 2), "f16", lb.LB_KERNEL_WARPSPEC, WS),
         # the library's choice: two nodes per thread from a size on, FP32 rows of whole lines only
         ((32, 18, 20), "f32", lb.LB_KERNEL_AUTO, ONE), ((160, 62, 5), "f32", lb.LB_KERNEL_AUTO, ROWS),
         ((150, 66, 5), "f32", lb.LB_KERNEL_AUTO, ONE), ((32, 18, 20), "f16", lb.LB_KERNEL_AUTO, ONE),
         ((150, 66, 5), "f16", lb.LB_KERNEL_AUTO, PAIRS), ((151, 66, 5), "bf16", lb.LB_KERNEL_AUTO, ROWS),
         # requests that do not apply
         ((32, 18, 20), "f32", lb.LB_KERNEL_STAGED, ONE), ((33, 17, 20), "f32", lb.LB_KERNEL_DIRECT2, ONE),
         ((160, 62, 5), "f32", lb.LB_KERNEL_DIRECT2X, ROWS)]


@pytest.mark.parametrize("shape,prec,kernel,want", CASES)
def test_launched_kernel(shape, prec, kernel, want):
    stream = torch.cuda.Stream()
    ctx = lb.lb_init(shape, 0.4, prec, stream=stream.cuda_stream)
    try:
        lb.lb_set_step_kernel(ctx, kernel)
        names = _launched(ctx, stream.cuda_stream)
    finally:
        lb.lb_destroy(ctx)
    assert len(names) == 1 and want in names[0], names


@pytest.mark.parametrize("shape,kernel,want", [((16, 6, 5), lb.LB_KERNEL_AUTO, ONE), ((16, 6, 5), lb.LB_KERNEL_DIRECT2XL, PAIRS),
                                               ((16, 6, 5), lb.LB_KERNEL_DIRECT2X, PAIRS), ((13, 6, 5), lb.LB_KERNEL_DIRECT2XL, ONE),
                                               ((150, 66, 5), lb.LB_KERNEL_AUTO, PAIRS), ((150, 66, 5), lb.LB_KERNEL_STAGED, PAIRS)])
def test_launched_kernel_of_the_stochastic_store(shape, kernel, want):
    stream = torch.cuda.Stream()
    ctx = lb.lb_init(shape, 0.4, "bf16", stream=stream.cuda_stream)
    try:
        lb.lb_set_step_kernel(ctx, kernel)
        lb.lb_set_stochastic_rounding(ctx, 5)
        names = _launched(ctx, stream.cuda_stream)
    finally:
        lb.lb_destroy(ctx)
    assert len(names) == 1 and want in names[0], names


def _run(shape, prec, kernel, fields, steps, flags, seed=None):
    ctx = lb.lb_init(shape, 0.3, prec, flags=flags)
    try:
        lb.lb_set_step_kernel(ctx, kernel)
        if seed is not None:
            lb.lb_set_stochastic_rounding(ctx, seed)
        lb.lb_set_fields(ctx, *fields)
        lb.lb_step(ctx, steps)
        raw = torch.empty((2, 41, shape[2], shape[1], shape[0]), dtype=TORCH_DTYPE[prec], device="cuda")
        lb.lb_get_state(ctx, raw)
        lb.lb_sync(ctx)
    finally:
        lb.lb_destroy(ctx)
    return raw


@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", [(2, 70, 150), (150, 66, 5), (160, 62, 5), (151, 66, 5), (6, 3, 5), (62, 4, 5)])
@pytest.mark.parametrize("flags", [0, lb.LB_FLAG_PAPER_LITERAL])
def test_two_node_kernels_give_the_one_node_bits(shape, prec, flags):
    amp = 0.02
    fl = wl.random_fields(*shape, lb.lb_theta0(), seed=9, du=amp, drho=amp, dtheta=amp)
    fields = [fl[k].cuda() for k in ("rho", "u", "theta")]
    want = _run(shape, prec, lb.LB_KERNEL_DIRECT1, fields, 10, flags)
    for k in (lb.LB_KERNEL_AUTO, lb.LB_KERNEL_DIRECT2, lb.LB_KERNEL_DIRECT2R, lb.LB_KERNEL_DIRECT2X):
        assert torch.equal(_run(shape, prec, k, fields, 10, flags), want), (shape, prec, k)


@pytest.mark.parametrize("shape", [(2, 2, 2), (16, 6, 5), (62, 4, 5), (262, 3, 2), (130, 9, 16)])
def test_the_stochastic_pairs_give_the_one_node_bits(shape):
    """Below the size from which the library takes x pairs: one node per thread (which
    test_gpu_stochastic_rounding.py compares with the oracle there) against the pairs by name."""
    fl = wl.random_fields(*shape, lb.lb_theta0(), seed=4, du=0.02, drho=0.02, dtheta=0.02)
    fields = [fl[k].cuda() for k in ("rho", "u", "theta")]
    want = _run(shape, "bf16", lb.LB_KERNEL_AUTO, fields, 10, 0, seed=77)
    assert torch.equal(_run(shape, "bf16", lb.LB_KERNEL_DIRECT2XL, fields, 10, 0, seed=77), want)
