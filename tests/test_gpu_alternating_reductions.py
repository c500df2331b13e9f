"""Long reductions.  The weight gradient (masked, dense, with the adapter gradients) from 5632 tokens on: CTA pairs work on two tiles in
turn and take them from alternating ends.  The sparse 512-row tiles where a raster group's weights are more than L2 keeps.  Ragged last
k-blocks, last row tiles that are half empty, more than one raster group (the second one runs backwards), halved items of the last wave.

The reference is the fp64 product on sampled rows; outputs are rounded once (1.7e-3 relative on Gaussian data, 5e-3 allowed, and
parity_error's bound per element), dL and dR from bf16 T and dT."""
import numpy as np
import pytest

from paper_2608_24070_b200 import inputs as si
from helpers import REL_TOL, GpuLayer, parity_error, to_f64

pytestmark = pytest.mark.gpu


def _bits(mask):
    return np.unpackbits(mask.cpu().numpy(), axis=1, bitorder="little").astype(bool)


@pytest.mark.parametrize("b,d_in,d_out,r", [
    (5631, 2304, 2560, 0),       # a token short of it
    (5632, 2304, 2560, 0),
    (8128, 2304, 2560, 0),
    (6000, 4352, 1664, 0),       # seven tile rows, the last one half empty
    (8192, 2304, 2560, 0),       # 10 x 9 tiles: two raster groups, 16 tiles of the last wave halved
    (8193, 2432, 2432, 16),      # a last k-block of one token, last row and column of tiles half empty
    (8200, 3328, 3072, 64),      # 13 x 12 tiles, fused with the adapter gradients; 8 of them halved
])
def test_weight_gradient(b, d_in, d_out, r):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    layer = GpuLayer(si.gaussian_bf16((d_out, d_in), 0.02, 61), fused_setup=True)
    Xb, dYb = si.gaussian_bf16((b, d_in), 1.0, 62), si.gaussian_bf16((b, d_out), 1.0, 63)
    X, dY = B.bf16_from_bits(Xb), B.bf16_from_bits(dYb)
    nan = lambda *shape: torch.full(shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    dWc, dW = layer.dw(dY, X), nan(d_out, d_in)
    B.slope_dense_linear_bwd_dw(dY, X, dW)
    g = lambda t: to_f64(B.bits_from_bf16(t))
    rows = si.sample_indices(d_out, 96, 64)
    ref = to_f64(dYb[:, rows]).T @ to_f64(Xb)
    assert parity_error(g(dW)[rows], ref) <= REL_TOL
    assert parity_error(g(dWc)[rows], ref[_bits(layer.mask1)[rows]].reshape(len(rows), d_in // 2)) <= REL_TOL
    if r:
        T, dT = B.bf16_from_bits(si.gaussian_bf16((b, r), 1.0, 65)), B.bf16_from_bits(si.gaussian_bf16((b, r), 1.0, 66))
        dWc2, dL, dR = nan(d_out, d_in // 2), nan(d_in, r), nan(r, d_out)
        ws = torch.empty(B.slope_bwd_dw_adapter_workspace_bytes(b, d_out, d_in, r), dtype=torch.uint8, device="cuda")
        B.slope_linear_bwd_dw_adapter(dY, X, T, dT, layer.mask1, dWc2, dL, dR, ws)
        assert torch.equal(dWc.view(torch.int16), dWc2.view(torch.int16))
        assert parity_error(g(dR)[:, rows], g(T).T @ to_f64(dYb[:, rows])) <= REL_TOL
        cols = si.sample_indices(d_in, 96, 67)
        assert parity_error(g(dL)[cols], to_f64(Xb[:, cols]).T @ g(dT)) <= REL_TOL
    layer.poll()


def test_carriers_in_a_ragged_reversed_group():
    """9 x 13 tiles, in one launch with the adapter gradients: the second group of tile rows is a single row, half empty, and runs
    backwards, so that the first carrier of its dR is the half-empty last column tile."""
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    b, d_in, d_out, r = 8193, 3200, 2176, 64
    gen = torch.Generator("cuda").manual_seed(68)
    new = lambda *shape: torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16)
    nan = lambda *shape: torch.full(shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    X, dY, T, dT = new(b, d_in), new(b, d_out), new(b, r), new(b, r)
    vals, meta, mask = B.alloc_compressed(d_out, d_in)
    B.slope_prune_24(new(d_out, d_in), vals, meta, mask)
    dWc, dWc2, dL, dR = nan(d_out, d_in // 2), nan(d_out, d_in // 2), nan(d_in, r), nan(r, d_out)
    ws = torch.empty(B.slope_bwd_dw_adapter_workspace_bytes(b, d_out, d_in, r), dtype=torch.uint8, device="cuda")
    ws.view(torch.float32).fill_(float("nan"))             # (a carrier that skips its share leaves this in the sums)
    B.slope_linear_bwd_dw_masked(dY, X, mask, dWc)
    launches = B.slope_launch_count()
    B.slope_linear_bwd_dw_adapter(dY, X, T, dT, mask, dWc2, dL, dR, ws)
    assert B.slope_launch_count() - launches == 2          # the fused one and the sum of its shares
    assert B.slope_poll_status() == 0
    assert torch.equal(dWc.view(torch.int16), dWc2.view(torch.int16))
    g = lambda t: to_f64(B.bits_from_bf16(t))
    assert parity_error(g(dR), g(T).T @ g(dY)) <= REL_TOL
    assert parity_error(g(dL), g(X).T @ g(dT)) <= REL_TOL


@pytest.mark.parametrize("b,d_in,d_out,r", [
    (5001, 13824, 2560, 64),     # 5 row tiles of 512, the weights of all of them in one group
    (4500, 11008, 3968, 0),      # 31 row blocks: one CTA of the last row tile has rows for one sub-tile only
])
def test_sparse_forward(b, d_in, d_out, r):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    Wb = si.gaussian_bf16((d_out, d_in), 0.02, 71)
    layer = GpuLayer(Wb, fused_setup=True)
    Xb = si.gaussian_bf16((b, d_in), 1.0, 72)
    X, T, R = B.bf16_from_bits(Xb), None, None
    rows = np.unique(np.concatenate([si.sample_indices(b, 96, 73), np.arange(b - 40, b)]))
    ref = to_f64(Xb[rows]) @ (to_f64(Wb) * _bits(layer.mask1)).T
    if r:
        Lb, Rb = si.gaussian_bf16((d_in, r), 0.1, 74), si.gaussian_bf16((r, d_out), 0.1, 75)
        R, T = B.bf16_from_bits(Rb), layer.adapter_T(X, B.bf16_from_bits(Lb))
        ref += to_f64(B.bits_from_bf16(T))[rows] @ to_f64(Rb)
    Y = torch.full((b + 1, d_out), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.slope_linear_fwd(X, layer.Wc_vals, layer.Wc_meta, d_out, Y[:b], T, R)
    layer.poll()
    assert torch.isnan(Y[b]).all()
    assert parity_error(to_f64(B.bits_from_bf16(Y[:b]))[rows], ref) <= REL_TOL
