"""Few tokens through tall weights with adapters: the T launch has further CTAs that ask L2 for the forward's weights.  Sizes on
either side of the line (16384 rows, 40 MB of compressed weights; at wide ranks no more than 1.5 slabs per SM), one and two CTAs per SM in the forward, T in one and in several
column tiles, repeated calls behind the kernel that writes the activations.

The reference is the fp64 product with T as written, on sampled features; outputs are rounded once (1.7e-3 relative on
Gaussian data, 5e-3 allowed, and parity_error's bound per element)."""
import numpy as np
import pytest

from paper_2608_24070_b200 import inputs as si
from helpers import REL_TOL, parity_error, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b,d_in,d_out,r", [
    (1, 2304, 16384, 16),        # 42 MB, 18 k-blocks
    (16, 2176, 16384, 64),       # 40.1 MB, 17 k-blocks
    (16, 2048, 16384, 64),       # below the line
    (7, 2432, 16256, 32),        # 127 slabs: below the line
    (8, 2560, 16512, 256),       # 129 slabs, widest rank
    (3, 4096, 22016, 64),        # 172 slabs, two CTAs per SM
    (17, 2304, 16384, 16),       # a token more than the line
    (5, 640, 65536, 32),         # T in clusters of four
    (2, 2048, 28160, 256),       # widest rank, 220 slabs: as many as are served beside it
    (2, 1536, 29696, 256),       # 232 slabs: more
])
def test_forward_with_adapter(b, d_in, d_out, r):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    gen = torch.Generator("cuda").manual_seed(81)
    new = lambda *shape, sigma=1.0: torch.randn(shape, generator=gen, dtype=torch.bfloat16, device="cuda").mul_(sigma)
    nan = lambda *shape: torch.full(shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    W, source, L, R = new(d_out, d_in, sigma=0.02), new(b, d_in), new(d_in, r, sigma=0.1), new(r, d_out, sigma=0.1)
    vals, meta, mask = B.alloc_compressed(d_out, d_in)
    B.slope_prune_24(W, vals, meta, mask)
    X, T, T0, Y = nan(b, d_in), nan(b, r), nan(b, r), nan(b + 1, d_out)        # a spare row: nothing behind the last token
    launches = B.slope_launch_count()
    for k in range(3):
        torch.mul(source, 2.0 ** k, out=X)
        B.slope_linear_fwd_adapter(X, vals, meta, d_out, L, R, T, Y[:b])
    assert B.slope_launch_count() - launches == 6
    B.slope_adapter_fwd_bwd(0, X, None, L, None, b, d_out, d_in, r, T=T0)
    assert B.slope_poll_status() == 0
    assert torch.isnan(Y[b]).all() and torch.equal(T.view(torch.int16), T0.view(torch.int16))
    g = lambda t: to_f64(B.bits_from_bf16(t))
    feats = si.sample_indices(d_out, 512, 82)
    kept = np.unpackbits(mask[torch.as_tensor(feats, device="cuda")].cpu().numpy(), axis=1, bitorder="little").astype(bool)
    ref = g(X) @ (g(W[torch.as_tensor(feats, device="cuda")]) * kept).T + g(T) @ g(R)[:, feats]
    assert parity_error(g(Y[:b])[:, feats], ref) <= REL_TOL
