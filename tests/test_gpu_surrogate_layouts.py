"""sg_conv3d_fwd_to: the convolution whose result is written in another d-layout is, bit for bit, the
convolution followed by sg_relabel, for both kernels, every pair of layouts, with and without the
residual, the added tensor and the kept pre-activation; and the activation's backward pass at element
counts and alignments that leave its four-element path."""
import pytest
import torch

from paper_1909_08406_gb300 import sg

pytestmark = pytest.mark.gpu

D = (1, 2, 4, 8)


@pytest.mark.parametrize("impl", [sg.CONV_TCGEN05, sg.CONV_MMA_SYNC])
@pytest.mark.parametrize("cin,cout,act,res,add", [(16, 32, sg.ACT_GELU, False, False), (32, 32, sg.ACT_GELU, True, True),
                                                  (32, 16, sg.ACT_NONE, False, True)])
def test_output_layout_equals_relabel(impl, cin, cout, act, res, add):
    nat = (2, 8, 32, 64)
    g = torch.Generator(device="cuda").manual_seed(cin + cout)
    vol = torch.randn(nat + (cin,), device="cuda", generator=g).to(torch.bfloat16)
    w = (torch.randn((cout, 27, cin), device="cuda", generator=g) / 20).to(torch.bfloat16)
    b = torch.randn(cout, device="cuda", generator=g)
    extra = torch.randn(nat + (cout,), device="cuda", generator=g).to(torch.bfloat16) if add else None
    prev = sg.set_conv_impl(impl)
    try:
        for df in D:
            x = vol if df == 1 else sg.relabel(vol, 1, df, nat + (cin,))
            ef = extra if extra is None or df == 1 else sg.relabel(extra, 1, df, nat + (cout,))
            z0 = torch.empty(x.shape[:-1] + (cout,), device="cuda")
            y0 = sg.conv3d_fwd(x, w, b, act=act, res_in=res, add=ef, z_out=z0, xper=64 // df)
            for dt in D:
                et = extra if extra is None or dt == 1 else sg.relabel(extra, 1, dt, nat + (cout,))
                z1 = torch.empty_like(z0)
                y1 = sg.conv3d_fwd_to(x, w, b, act, res, nat + (cin,), df, dt, add=et, z_out=z1)
                want = y0 if dt == df else sg.relabel(y0, df, dt, nat + (cout,))
                assert torch.equal(y1, want) and torch.equal(z1, z0), (df, dt)
        sg.status()
    finally:
        sg.set_conv_impl(prev)


def test_output_layout_rejects_bad_layouts():
    x = torch.zeros((1, 8, 32, 64, 16), dtype=torch.bfloat16, device="cuda")
    w = torch.zeros((32, 27, 16), dtype=torch.bfloat16, device="cuda")
    for df, dt in ((1, 3), (3, 1), (1, 16), (2, 1)):  # (2, 1): one item is not the 2-layout of a volume
        with pytest.raises((RuntimeError, ZeroDivisionError)):
            sg.conv3d_fwd_to(x, w, None, sg.ACT_NONE, False, tuple(x.shape), df, dt)


@pytest.mark.parametrize("n", [1, 3, 4, 5, 1023, 1025, 4097])
@pytest.mark.parametrize("act", [sg.ACT_NONE, sg.ACT_GELU])
def test_act_backward_remainders_and_alignment(n, act):
    g = torch.Generator(device="cuda").manual_seed(n)
    dy, z = torch.randn(n + 3, device="cuda", generator=g), torch.randn(n + 3, device="cuda", generator=g)
    want = None
    for off in (0, 1, 2):  # the same values behind aligned and unaligned pointers
        a, b = torch.empty(n + 3, device="cuda")[off:off + n], torch.empty(n + 3, device="cuda")[off:off + n]
        a.copy_(dy[:n])
        b.copy_(z[:n])
        got = sg.act_backward(a, b, act)
        want = got if want is None else want
        assert torch.equal(got, want)
    d, zz = dy[:n].double(), z[:n].double()
    if act == sg.ACT_GELU:
        d = d * (0.5 * (1 + torch.erf(zz / 2 ** 0.5)) + zz * torch.exp(-0.5 * zz * zz) / (2 * torch.pi) ** 0.5)
    # one BF16 rounding (2^-8 of spacing) of an FP32 value within a few 1e-7
    assert bool(((want.double() - d).abs() <= 2.0 ** -8 * d.abs() + 1e-6).all())
