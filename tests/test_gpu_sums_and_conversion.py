"""Global sums and the FP64 import / export of the stored populations at the sizes where their
loads change form: planes with an odd number of nodes (one node per load), pairs, a base that is
not aligned to a pair, grids below one block, and host transfers whose chunks split a plane.

Tolerances.  Export: f = w (1 + h) of the stored h in one fused FP64 multiply-add, 2^-53 relative
to the exact value.  Import: (f - w) / w is formed to about 2^-44 relative and then rounded to FP32
and to the storage type, so a stored value differs from the doubly rounded FP64 quotient only where
that lies within 2^-40 of a rounding boundary: at most one spacing, in a fraction below 1e-4 of
the values.  Sums: each node's FP32 moments (41 terms, rounding below 41 2^-24 sum |d|) added in
FP64."""
import numpy as np
import pytest
import torch

from helpers import STORE_SCALE, TORCH_DTYPE
from paper_1909_08406_gb300 import lb
from paper_1909_08406_gb300 import workloads as wl

pytestmark = pytest.mark.gpu

SHAPES = [(1, 1, 1), (3, 1, 5), (7, 5, 3), (6, 4, 5), (33, 18, 20), (64, 6, 11)]


def _populations(shape, seed):
    _, w = lb.lb_velocity_set()
    return wl.random_populations(*shape, w, seed, spread=0.05), np.asarray(w)


def _raw(ctx, shape, prec):
    raw = torch.empty((2, 41, shape[2], shape[1], shape[0]), dtype=TORCH_DTYPE[prec], device="cuda")
    lb.lb_get_state(ctx, raw)
    return raw


def _check_import(raw, f, w, prec):
    q = (f - w[None, :, None, None, None]) / w[None, :, None, None, None] * STORE_SCALE[prec]
    want = torch.from_numpy(q).to(torch.float32).to(TORCH_DTYPE[prec])
    got = raw.cpu()
    differ = got != want
    assert differ.double().mean() < 1e-4
    a, b = got[differ].double(), want[differ].double()
    assert bool(((a - b).abs() <= 2 ** -7 * b.abs()).all())


@pytest.mark.parametrize("prec", ["f64", "f32", "f16", "bf16"])
@pytest.mark.parametrize("shape", SHAPES)
def test_import_export_and_sums(shape, prec):
    f, w = _populations(shape, 3)
    ctx = lb.lb_init(shape, 0.4, prec)
    try:
        lb.lb_set_populations(ctx, torch.from_numpy(f).cuda())
        raw = _raw(ctx, shape, prec)
        out = torch.empty(f.shape, dtype=torch.float64, device="cuda")
        lb.lb_get_populations(ctx, out)
        sums = np.array(lb.lb_conserved(ctx))
    finally:
        lb.lb_destroy(ctx)
    stored = raw.cpu().to(torch.float64).numpy()
    if prec == "f64":
        assert np.array_equal(stored, f)
        back = f
    else:
        _check_import(raw, f, w, prec)
        back = w[None, :, None, None, None] * (1.0 + stored / STORE_SCALE[prec])
    assert np.max(np.abs(out.cpu().numpy() - back) / back) <= 2.0 ** -51
    c = np.asarray(lb.lb_velocity_set()[0], dtype=np.float64) / 2
    n = f[:, 0].size
    want = [back.sum()] + [(back * c[None, :, k, None, None, None]).sum() for k in range(3)]
    want.append(0.5 * (back * (c * c).sum(1)[None, :, None, None, None]).sum())
    tol = (1e-13 if prec == "f64" else 41 * 2.0 ** -24 * 0.05 * 4) * n
    assert np.max(np.abs(sums - np.array(want))) <= tol
    # the same sums from a copy of the state that starts one element into its allocation
    off = torch.empty(raw.numel() + 1, dtype=raw.dtype, device="cuda")[1:]
    off.copy_(raw.reshape(-1))
    got = torch.empty(5, dtype=torch.float64, device="cuda")
    lb.lb_conserved_noalloc(off, shape, prec, got)
    assert np.max(np.abs(got.cpu().numpy() - sums)) <= 1e-13 * max(n, 1) + (0 if prec == "f64" else tol)


@pytest.mark.parametrize("prec", ["f32", "f16"])
def test_extreme_values_import(prec):
    """Zero deviations, the smallest and largest finite ones, infinities and NaN take the same
    values as the FP64 quotient rounded to the storage type."""
    shape = (5, 2, 1)
    f, w = _populations(shape, 4)
    specials = np.array([0.0, 1e-300, -1e-300, 1e-30, 5e-22, -5e-22, 1e17, 1e19, np.inf, np.nan])
    f[0, :, 0] = w[:, None, None] + specials.reshape(2, 5)
    f[1, :, 0, 0, 0] = w * (1 + 2.0 ** -60)
    ctx = lb.lb_init(shape, 0.4, prec)
    try:
        lb.lb_set_populations(ctx, torch.from_numpy(f).cuda())
        got = _raw(ctx, shape, prec).cpu()
    finally:
        lb.lb_destroy(ctx)
    q = (f - w[None, :, None, None, None]) / w[None, :, None, None, None] * STORE_SCALE[prec]
    with np.errstate(over="ignore"):
        want = torch.from_numpy(q.astype(np.float32)).to(TORCH_DTYPE[prec])
    assert bool((torch.isnan(got) == torch.isnan(want)).all())
    fine = ~torch.isnan(want)
    same = got[fine] == want[fine]
    close = (got[fine].double() - want[fine].double()).abs() <= 2.0 ** -9 * want[fine].double().abs()
    assert bool((same | close).all())


def test_host_chunks_that_split_a_plane():
    """Host arrays go through a staging buffer of 64 Mi values: the second chunk starts inside a
    plane."""
    shape = (96, 97, 90)
    f, w = _populations(shape, 5)
    assert f.size > 1 << 26 and (1 << 26) % (shape[0] * shape[1] * shape[2]) != 0
    ctx = lb.lb_init(shape, 0.4, "f16")
    try:
        lb.lb_set_populations(ctx, f)
        raw = _raw(ctx, shape, "f16")
        back = np.empty_like(f)
        lb.lb_get_populations(ctx, back)
    finally:
        lb.lb_destroy(ctx)
    _check_import(raw, f, w, "f16")
    want = w[None, :, None, None, None] * (1.0 + raw.cpu().to(torch.float64).numpy() / STORE_SCALE["f16"])
    assert np.max(np.abs(back - want) / want) <= 2.0 ** -51
