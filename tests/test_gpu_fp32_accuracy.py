"""Error of the stored deviation h = f / w - 1 in FP32 over many steps of a small grid, where nothing is
averaged out: relative 2-norm against the FP64 oracle from the same fields.

Bound: unbiased rounding adds up like a random walk.  A step rounds each stored value once (up to half
a unit, 2^-24 relative, 0.58 of that in the mean square) after sums and a relaxation of the same size, at
most 2.4 x 2^-24 together, and damps part of it; 100 steps give 10 x 2.4 x 2^-24 = 1.43e-6.  A bias of
one part in 10^8 per step (as the approximate reciprocal has near 1) adds up linearly and exceeds it."""
import math

import numpy as np
import pytest
import torch

import oracle
from helpers import lib_to_oracle_perm, to_lib_order
from paper_1909_08406_gb300 import lb
from paper_1909_08406_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

STEPS = 100
BOUND = math.sqrt(STEPS) * 2.4 * 2.0 ** -24


def _fields(nx, ny, nz, theta0, seed):
    """A density pulse, shear waves and a Fourier box of temperature (deviations of 4e-3 to 1e-2)."""
    r = np.random.default_rng(seed)
    pos = wl.node_positions(nx, ny, nz)
    r2 = 0
    for p, n in zip(pos, (nx, ny, nz)):
        d = p - r.uniform(0, n)
        r2 = r2 + (d - n * torch.round(d / n)) ** 2
    rho = 1.0 + 8e-3 * torch.exp(-r2 / 72.0)
    u = torch.stack([4e-3 * torch.sin(2 * math.pi * pos[(a + 1) % 3] / (nx, ny, nz)[(a + 1) % 3] + a) for a in range(3)])
    theta = theta0 * (1.0 + 1e-3 * wl.fourier_box_field(nx, ny, nz, seed + 7, kmax=4))
    return [x.contiguous() for x in (rho, u, theta)]


@pytest.mark.parametrize("shape,tau", [((21, 95, 12), 0.5793), ((33, 18, 20), 0.3), ((64, 32, 20), 0.3)])
@pytest.mark.parametrize("kernel", [lb.LB_KERNEL_DIRECT1, lb.LB_KERNEL_DIRECT2])
def test_error_of_many_steps(shape, tau, kernel):
    nx, ny, nz = shape
    fields = _fields(nx, ny, nz, lb.lb_theta0(), 11)
    ctx = lb.lb_init(shape, tau, "f32")
    try:
        lb.lb_set_step_kernel(ctx, kernel)
        lb.lb_set_fields(ctx, *[f.cuda() for f in fields])
        lb.lb_step(ctx, STEPS)
        got = torch.empty((2, 41, nz, ny, nx), dtype=torch.float32)
        lb.lb_get_state(ctx, got)
        lb.lb_sync(ctx)
    finally:
        lb.lb_destroy(ctx)
    w = np.asarray(lb.lb_velocity_set()[1])[None, :, None, None, None]
    f = oracle.step(oracle.init_fields(*[x.numpy() for x in fields]), tau, STEPS)
    want = to_lib_order(f, lib_to_oracle_perm()) / w - 1.0
    err = np.linalg.norm(got.numpy().astype(np.float64) - want) / np.linalg.norm(want)
    assert err <= BOUND, (shape, tau, err)
