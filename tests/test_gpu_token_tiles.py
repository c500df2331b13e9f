"""Sparse forward and input gradient: the few-token kernel where it does not split and on either side of its line, the 256-row
tiles at every width (32 ... 224 in steps of 32) and the 512-row tiles at the widths that are chosen for them (96 ... 224), ragged last
tiles and row tiles that are half empty, with and without adapters; the fused forward against the separate calls.

The reference is the fp64 product of the bf16 operands the kernels read (T as written), so outputs are rounded
once: 1.7e-3 relative on Gaussian data, 5e-3 allowed, and parity_error's bound per element."""
import numpy as np
import pytest

from paper_2608_24070_b200 import inputs as si
from helpers import REL_TOL, GpuLayer, parity_error, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b,d_in,d_out,r", [
    (1, 128, 384, 0),            # few-token kernel without a split: one k-block, one token
    (5, 128, 256, 16),
    (16, 256, 19200, 0),         # more slabs than SMs
    # tile rows x width of the forward / the input gradient
    (17, 128, 640, 64),          # 256x32 / 256x32
    (128, 256, 512, 32),         # 256x32 / 256x32
    (129, 256, 384, 0),          # 256x32 / 256x32, last row tile half empty
    (161, 1024, 256, 16),        # 256x32 / 256x64
    (250, 640, 1920, 0),         # 256x64 / 256x32
    (353, 512, 4096, 48),        # 256x128 / 256x32
    (449, 768, 2304, 0),         # 256x96 / 256x32
    (500, 4096, 1152, 64),       # 256x64 / 256x128
    (673, 384, 2176, 256),       # 256x128 / 256x32
    (1000, 768, 2304, 16),       # 256x128 / 256x64
    (1345, 1152, 640, 0),        # 256x96 / 256x128
    (2048, 1024, 4096, 32),      # 256x160 / 256x128
    (5000, 2048, 1408, 0),       # 512x224, several waves / 256x192
    (1782, 128, 896, 32),        # 256x224 / 256x64
    (458, 1152, 6400, 48),       # 512x96 / 256x64
    (496, 1152, 6528, 0),        # 512x128 / 256x64
    (1826, 1024, 2560, 16),      # 512x160 / 256x128
    (3974, 1024, 1408, 0),       # 512x192 / 256x224
    (15257, 512, 3968, 0),       # 31 row blocks: in the last 512-row tile one CTA has rows for one sub-tile only
])
def test_token_tiles_match_fp64(b, d_in, d_out, r):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    Wb = si.gaussian_bf16((d_out, d_in), 0.02, 51)
    layer = GpuLayer(Wb, fused_setup=True)
    Xb, dYb = si.gaussian_bf16((b, d_in), 1.0, 52), si.gaussian_bf16((b, d_out), 1.0, 53)
    X, dY = B.bf16_from_bits(Xb), B.bf16_from_bits(dYb)
    bits = lambda m: np.unpackbits(m.cpu().numpy(), axis=1, bitorder="little").astype(bool)
    fW = to_f64(Wb)
    ref_Y, ref_dX = to_f64(Xb) @ (fW * bits(layer.mask1)).T, to_f64(dYb) @ (fW * bits(layer.mask2))
    g = lambda t: to_f64(B.bits_from_bf16(t))
    nan = lambda *shape: torch.full(shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    Y, dX = nan(b + 1, d_out), nan(b + 1, d_in)                 # a spare row: nothing behind the last token
    T = dT = L = R = None
    if r:
        Lb, Rb = si.gaussian_bf16((d_in, r), 0.1, 54), si.gaussian_bf16((r, d_out), 0.1, 55)
        L, R = B.bf16_from_bits(Lb), B.bf16_from_bits(Rb)
        T, dT = layer.adapter_T(X, L), nan(b, r)
        B.slope_adapter_fwd_bwd(2, None, dY, None, R, b, d_out, d_in, r, dT=dT)
        ref_Y, ref_dX = ref_Y + g(T) @ to_f64(Rb), ref_dX + g(dT) @ to_f64(Lb).T
        T1, Y1 = nan(b, r), nan(b, d_out)
        B.slope_linear_fwd_adapter(X, layer.Wc_vals, layer.Wc_meta, d_out, L, R, T1, Y1)
        assert torch.equal(T1.view(torch.int16), T.view(torch.int16))
        assert parity_error(g(Y1), ref_Y) <= REL_TOL
    B.slope_linear_fwd(X, layer.Wc_vals, layer.Wc_meta, d_out, Y[:b], T, R)
    B.slope_linear_bwd_dx(dY, layer.WTc_vals, layer.WTc_meta, d_in, dX[:b], dT, L)
    layer.poll()
    assert torch.isnan(Y[b]).all() and torch.isnan(dX[b]).all()
    assert parity_error(g(Y[:b]), ref_Y) <= REL_TOL
    assert parity_error(g(dX[:b]), ref_dX) <= REL_TOL


@pytest.mark.parametrize("b,before", [(1, 16), (7, 16), (13, 16), (17, 64), (63, 64), (65, 128), (127, 128)])
def test_few_tokens_do_not_see_what_an_earlier_launch_left_in_shared_memory(b, before):
    """Activation tiles are loaded for as many tokens as there are; the MMAs also read the rows behind them."""
    _leftovers_are_not_seen(b, before, 2048)


@pytest.mark.parametrize("b,before", [(33, 64), (66, 128), (127, 128)])
def test_few_tokens_on_long_reductions_do_not_see_them_either(b, before):
    _leftovers_are_not_seen(b, before, 6144)                     # (127 tokens take the few-token kernel on long reductions only)


def _leftovers_are_not_seen(b, before, d_in):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    d_out, r = 1024, 32
    layer = GpuLayer(si.gaussian_bf16((d_out, d_in), 0.02, 56), fused_setup=True)
    L, R = (B.bf16_from_bits(si.gaussian_bf16(s, 0.1, 57)) for s in ((d_in, r), (r, d_out)))
    X = B.bf16_from_bits(si.gaussian_bf16((b, d_in), 1.0, 58))
    out = []
    for fill in (0.0, float("nan")):
        noise, T0, Y0 = (torch.full((before, n), fill, dtype=torch.bfloat16, device="cuda") for n in (d_in, r, d_out))
        for _ in range(3):                                       # on every SM
            B.slope_linear_fwd(noise, layer.Wc_vals, layer.Wc_meta, d_out, Y0, T0, R)
        T, Y = (torch.empty((b, n), dtype=torch.bfloat16, device="cuda") for n in (r, d_out))
        B.slope_linear_fwd_adapter(X, layer.Wc_vals, layer.Wc_meta, d_out, L, R, T, Y)
        out.append((T, Y))
    (T, Y), (T1, Y1) = out
    assert torch.isfinite(Y).all() and torch.equal(Y.view(torch.int16), Y1.view(torch.int16))
    assert torch.equal(T.view(torch.int16), T1.view(torch.int16))
    assert B.slope_poll_status() == 0


@pytest.mark.parametrize("b,d_in,d_out,r", [
    (17, 1152, 256, 0), (17, 896, 256, 16),          # either side of the few-token kernel's line, 17 tokens
    (64, 2304, 1280, 64), (65, 1792, 1280, 0),       # its 64- and 128-token tiles
    (128, 4096, 512, 256), (127, 3456, 640, 0),
    (40, 7808, 5632, 0), (40, 5888, 5760, 32),       # 44 row slabs and 45
])
def test_few_token_kernel_on_either_side_of_its_line(b, d_in, d_out, r):
    test_token_tiles_match_fp64(b, d_in, d_out, r)
