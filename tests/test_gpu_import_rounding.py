"""Rounding of the FP64 population import: the stored value of f is (f - w) / w, formed in two FP32 terms
to 2^-20 of an FP32 spacing, rounded to FP32 and then, for 16-bit storage, to the storage type.  So it lies
within 1/2 + 2^-20 spacings of the exact quotient (FP32) or within half a spacing of the storage type
plus half an FP32 one, 2^-13 (FP16) and 2^-16 (BF16) of it."""
import numpy as np
import pytest
import torch

from helpers import STORE_SCALE, TORCH_DTYPE
from paper_1909_08406_gb300 import lb

pytestmark = pytest.mark.gpu

DIGITS = {"f32": 24, "f16": 11, "bf16": 8}          # of the significand
SMALLEST = {"f32": -149, "f16": -24, "bf16": -133}  # exponent of the smallest spacing
SLACK = {"f32": 2.0 ** -20, "f16": 2.0 ** -13, "bf16": 2.0 ** -16}


@pytest.mark.parametrize("prec", ["f32", "f16", "bf16"])
@pytest.mark.parametrize("spread", [1e-6, 1e-3, 0.2])
def test_import_is_rounded_once(prec, spread):
    shape = (40, 18, 7)
    w = np.asarray(lb.lb_velocity_set()[1])[None, :, None, None, None]
    r = np.random.default_rng(8)
    f = w * (1.0 + spread * r.standard_normal((2, 41, *shape[::-1])))
    ctx = lb.lb_init(shape, 0.4, prec)
    try:
        lb.lb_set_populations(ctx, torch.from_numpy(f).cuda())
        raw = torch.empty((2, 41, *shape[::-1]), dtype=TORCH_DTYPE[prec], device="cuda")
        lb.lb_get_state(ctx, raw)
        lb.lb_sync(ctx)
    finally:
        lb.lb_destroy(ctx)
    want = (f - w) / w * STORE_SCALE[prec]  # to 2^-52 relative
    exponent = np.floor(np.log2(np.maximum(np.abs(want), 1e-300)))
    spacing = 2.0 ** np.maximum(exponent - DIGITS[prec] + 1, SMALLEST[prec])
    off = np.abs(raw.cpu().to(torch.float64).numpy() - want) / spacing
    assert off.max() <= 0.5 + SLACK[prec], (prec, spread, off.max(), (off > 0.5 + SLACK[prec]).mean())
