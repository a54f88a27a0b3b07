"""Steps launched with programmatic overlap: a step's blocks may be resident while the previous step's
kernel still writes, and every load of populations and fields must stay behind the wait for it.  Many
steps queued in one call therefore give the bits of the same steps taken one by one with a
synchronisation after each, in every storage type and in every mode whose passes overlap.  Likewise
the persistent batch kernel, whose loads must stay behind its grid barrier, and one launch per step."""
import pytest
import torch

from helpers import TORCH_DTYPE
from paper_1909_08406_gb300 import lb
from paper_1909_08406_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

STEPS = 40
SMALL, PAIRS = (33, 18, 20), (64, 34, 20)  # one node per thread; two nodes per thread
CASES = [(prec, shape, "plain") for prec in ("f64", "f32", "f16", "bf16") for shape in (SMALL, PAIRS)]
CASES += [("bf16", PAIRS, "stochastic"), ("f16", PAIRS, "nonideal"), ("f16", SMALL, "nonideal"),
          ("f16", PAIRS, "walls"), ("bf16", SMALL, "walls")]


def _context(shape, prec, mode):
    amp = 0.01
    fl = wl.random_fields(*shape, lb.lb_theta0(), seed=21, du=amp, drho=amp, dtheta=amp)
    ctx = lb.lb_init(shape, 0.4, prec)
    lb.lb_set_fields(ctx, *[fl[k].cuda() for k in ("rho", "u", "theta")])
    th0 = lb.lb_theta0()
    if mode == "walls":
        lb.lb_set_walls(ctx, (0.0, 0.0, th0), (0.01, 0.0, th0))
    elif mode == "nonideal":
        a, b = lb.lb_nonideal_constants("vdw", 1.1)
        lb.lb_set_nonideal(ctx, a, b, 0.02, 0.5, eos="vdw")
    elif mode == "stochastic":
        lb.lb_set_stochastic_rounding(ctx, 77)
    lb.lb_sync(ctx)
    return ctx


def _state(ctx, shape, prec):
    nx, ny, nz = shape
    raw = torch.empty((2, 41, nz, ny, nx), dtype=TORCH_DTYPE[prec], device="cuda")
    lb.lb_get_state(ctx, raw)
    lb.lb_sync(ctx)
    return raw


@pytest.mark.parametrize("prec,shape,mode", CASES)
def test_queued_steps_equal_synchronised_steps(prec, shape, mode):
    ctx = _context(shape, prec, mode)
    try:
        for _ in range(STEPS):
            lb.lb_step(ctx, 1)
            lb.lb_sync(ctx)
        want = _state(ctx, shape, prec)
    finally:
        lb.lb_destroy(ctx)
    ctx = _context(shape, prec, mode)
    try:
        lb.lb_step(ctx, STEPS)
        got = _state(ctx, shape, prec)
    finally:
        lb.lb_destroy(ctx)
    assert torch.equal(got, want)


@pytest.mark.parametrize("prec", ["f16", "bf16"])
def test_persistent_steps_equal_separate_launches(prec):
    shapes = [SMALL, (24, 24, 24), (40, 22, 18)]

    def run(calls, steps):
        b = lb.lb_batch_init(shapes, [0.4] * len(shapes), prec)
        try:
            for k, shape in enumerate(shapes):
                fl = wl.random_fields(*shape, lb.lb_theta0(), seed=k, du=0.01, drho=0.01, dtheta=0.01)
                lb.lb_set_fields(lb.lb_batch_sim(b, k), *[fl[n].cuda() for n in ("rho", "u", "theta")])
            for _ in range(calls):
                lb.lb_batch_step(b, steps, lb.LB_BATCH_PERSISTENT)
                torch.cuda.synchronize()
            return [_state(lb.lb_batch_sim(b, k), shape, prec) for k, shape in enumerate(shapes)]
        finally:
            lb.lb_batch_destroy(b)

    for got, want in zip(run(1, STEPS), run(STEPS, 1)):
        assert torch.equal(got, want)
