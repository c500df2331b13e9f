"""Weight-gradient and dense GEMM epilogues at the edges of their tiles: the one-CTA kernel and every width of the CTA-pair
kernel (64, 128, 192, 256), halved items of the last wave, last tiles that are partly empty in either dimension, few tokens
(one k-block, a ragged one).

The reference is the fp64 product of the same bf16 operands; outputs are rounded once (2^-9 / sqrt(3) ~ 1.7e-3
relative on Gaussian data, 5e-3 allowed, and parity_error's bound per element)."""
import pytest

from paper_2608_24070_b200 import inputs as si
from helpers import REL_TOL, parity_error, to_f64

pytestmark = pytest.mark.gpu


def _operands(b, d_in, d_out):
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    bits = [si.gaussian_bf16((b, d_in), 1.0, 41), si.gaussian_bf16((b, d_out), 1.0, 42),
            si.gaussian_bf16((d_out, d_in), 0.02, 43)]
    return B, [B.bf16_from_bits(x) for x in bits], [to_f64(x) for x in bits]


@pytest.mark.parametrize("b,d_in,d_out", [
    (1, 128, 128),               # one-CTA kernel, one tile, one token
    (65, 384, 640),              # one-CTA kernel, a k-block and one token
    (200, 1152, 1920),           # one-CTA kernel, 135 tiles
    (70, 2176, 2432),            # 128 wide, last row tile half empty
    (200, 3200, 2688),           # 256 wide, half empty in both dimensions
    (90, 4096, 4096),            # 256 tiles: the last wave's are halved
    (2049, 128, 128),            # 64 wide, row tile half empty, 33 k-blocks, the last with one token
    (2111, 512, 512),            # 64 wide
    (2100, 384, 384),            # 64 wide, last row tile half empty
    (2200, 1152, 1920),          # 128 wide, last row tile half empty
])
def test_masked_weight_gradient(b, d_in, d_out):
    import numpy as np
    import torch

    B, (X, dY, W), (fX, fdY, _) = _operands(b, d_in, d_out)
    vals, meta, mask = B.alloc_compressed(d_out, d_in)
    B.slope_prune_24(W, vals, meta, mask)
    dWc = torch.full((d_out, d_in // 2), float("nan"), dtype=torch.bfloat16, device="cuda")
    B.slope_linear_bwd_dw_masked(dY, X, mask, dWc)
    assert B.slope_poll_status() == 0
    kept = np.unpackbits(mask.cpu().numpy(), axis=1, bitorder="little").astype(bool)
    ref = (fdY.T @ fX)[kept].reshape(d_out, d_in // 2)
    assert parity_error(to_f64(B.bits_from_bf16(dWc)), ref) <= REL_TOL


@pytest.mark.parametrize("b,d_in,d_out", [(1, 128, 128), (130, 256, 384), (300, 1152, 640), (513, 384, 2176),
                                        (700, 2048, 4224), (600, 3200, 2688),
                                        (3000, 256, 4992),
                                        (1000, 1024, 1024),      # one-CTA kernel in all three, last row tile partly empty
                                        (777, 1024, 1280)])      # and beside a 128-wide input gradient
def test_dense_layer(b, d_in, d_out):
    import torch

    B, (X, dY, W), (fX, fdY, fW) = _operands(b, d_in, d_out)
    nan = lambda *shape: torch.full(shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    Y, dX, dW = nan(b + 1, d_out), nan(b + 1, d_in), nan(d_out, d_in)       # a spare row: nothing behind the last token
    B.slope_dense_linear_fwd(X, W, Y[:b])
    B.slope_dense_linear_bwd_dx(dY, W, dX[:b])
    B.slope_dense_linear_bwd_dw(dY, X, dW)
    assert B.slope_poll_status() == 0
    assert torch.isnan(Y[b]).all() and torch.isnan(dX[b]).all()
    g = lambda t: to_f64(B.bits_from_bf16(t))
    for got, ref in ((Y[:b], fX @ fW.T), (dX[:b], fdY @ fW), (dW, fdY.T @ fX)):
        assert parity_error(g(got), ref) <= REL_TOL


@pytest.mark.parametrize("b,d_in,d_out", [(1, 640, 8320), (9, 8320, 640),     # one-CTA tiles in the forward / the input gradient
                                          (2, 2304, 640), (127, 1024, 3840)])
def test_few_tokens_do_not_see_what_an_earlier_launch_left_in_shared_memory(b, d_in, d_out):
    """Boxes hold as many token rows as there are; the MMAs also read the rows behind them."""
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    gen = torch.Generator("cuda").manual_seed(44)
    new = lambda *shape: torch.randn(shape, generator=gen, dtype=torch.bfloat16, device="cuda")
    X, dY, W = new(b, d_in), new(b, d_out), new(d_out, d_in)
    out = []
    for fill in (0.0, float("nan")):
        for tokens in (128, 4000):                               # both kernels, on every SM
            noise = lambda n: torch.full((tokens, n), fill, dtype=torch.bfloat16, device="cuda")
            B.slope_dense_linear_fwd(noise(d_in), W, noise(d_out))
            B.slope_dense_linear_bwd_dx(noise(d_out), W, noise(d_in))
        Y, dX = (torch.full((b, n), float("nan"), dtype=torch.bfloat16, device="cuda") for n in (d_out, d_in))
        B.slope_dense_linear_fwd(X, W, Y)
        B.slope_dense_linear_bwd_dx(dY, W, dX)
        out.append((Y, dX))
    for x, y in zip(*out):
        assert torch.isfinite(x).all() and torch.equal(x.view(torch.int16), y.view(torch.int16))
    assert B.slope_poll_status() == 0
