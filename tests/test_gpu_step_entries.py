"""The direct step kernels number their work (nodes, pairs of rows, x pairs) linearly over the grid: at
sizes where a warp crosses rows, planes and the sub-lattices, where the grid is smaller than a block
and where the last block is partial, every kernel that applies gives the same bits (their arithmetic
rounds alike: products and multiply-adds are written out; tests/test_gpu_parity.py compares each with
the oracle).  A captured graph of steps replays to the eager result (the launches carry the
programmatic attribute)."""
import pytest
import torch

from helpers import TORCH_DTYPE
from paper_1909_08406_gb300 import lb
from paper_1909_08406_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(2, 1, 1), (2, 2, 1), (1, 2, 3), (5, 2, 2), (6, 3, 5), (34, 2, 3), (62, 4, 5), (33, 18, 20), (150, 6, 4)]
TAU = 0.3
AMPLITUDE = {"f32": 0.05, "f16": 0.02, "bf16": 0.02}


def _run(shape, prec, kernel, fields, steps):
    ctx = lb.lb_init(shape, TAU, prec)
    try:
        lb.lb_set_step_kernel(ctx, kernel)
        used = lb.lb_step_variant(ctx)
        lb.lb_set_fields(ctx, *fields)
        lb.lb_step(ctx, steps)
        raw = torch.empty((2, 41, shape[2], shape[1], shape[0]), dtype=TORCH_DTYPE[prec], device="cuda")
        lb.lb_get_state(ctx, raw)
        lb.lb_sync(ctx)
    finally:
        lb.lb_destroy(ctx)
    return used, raw


@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", SHAPES)
def test_entry_kinds_give_the_same_bits(shape, prec):
    amp = AMPLITUDE[prec]
    fl = wl.random_fields(*shape, lb.lb_theta0(), seed=9, du=amp, drho=amp, dtheta=amp)
    fields = [fl[k].cuda() for k in ("rho", "u", "theta")]
    steps = 20
    _, ref = _run(shape, prec, lb.LB_KERNEL_DIRECT1, fields, steps)
    for k in (lb.LB_KERNEL_AUTO, lb.LB_KERNEL_DIRECT2, lb.LB_KERNEL_DIRECT2R, lb.LB_KERNEL_DIRECT2X, lb.LB_KERNEL_DIRECT2XL):
        used, raw = _run(shape, prec, k, fields, steps)
        assert torch.equal(raw, ref), (shape, prec, k, used)


@pytest.mark.parametrize("prec,shape", [("f32", (33, 6, 5)), ("f16", (30, 5, 7)), ("f64", (9, 4, 3))])
def test_captured_steps_replay(prec, shape):
    fl = wl.random_fields(*shape, lb.lb_theta0(), seed=3, du=0.02, drho=0.02, dtheta=0.02)
    fields = [fl[k].cuda() for k in ("rho", "u", "theta")]
    _, want = _run(shape, prec, lb.LB_KERNEL_AUTO, fields, 4)
    stream = torch.cuda.Stream()
    ctx = lb.lb_init(shape, TAU, prec, stream=stream.cuda_stream)
    start = torch.empty_like(want)
    out = torch.empty_like(want)
    try:
        lb.lb_set_fields(ctx, *fields)
        lb.lb_get_state(ctx, start)
        lb.lb_sync(ctx)
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            lb.lb_set_state(ctx, start)  # a copy node, then four step launches (an even number: the same buffers)
            lb.lb_step(ctx, 4)
            lb.lb_get_state(ctx, out)
        for _ in range(2):
            out.zero_()
            torch.cuda.synchronize()
            g.replay()
            torch.cuda.synchronize()
            assert torch.equal(out, want)
    finally:
        lb.lb_destroy(ctx)
