"""Equal token rows of one call give equal bits, wherever in the batch they stand: every tile of a product takes the sums of a row in the
same order.  Long reductions on many token blocks (several tiles per CTA pair), ragged last tiles, where a kernel could gain from
taking some of its tiles from another end."""
import pytest

pytestmark = pytest.mark.gpu

PERIOD = 61              # no divisor of a tile's rows: each of the distinct rows comes up at every position of a tile


def _rows(b, d, seed):
    import torch

    gen = torch.Generator("cuda").manual_seed(seed)
    return torch.randn((PERIOD, d), generator=gen, device="cuda", dtype=torch.bfloat16).repeat(-(-b // PERIOD), 1)[:b].contiguous()


def _assert_equal_rows(out):
    import torch

    bits = out.view(torch.int16)
    assert torch.isfinite(out).all()
    assert torch.equal(bits[PERIOD:], bits[:-PERIOD])


@pytest.mark.parametrize("b,k,m,r", [
    (5001, 13824, 2560, 64),     # 5 row tiles of 512 in one raster group, a CTA pair works on two token blocks
    (4500, 11008, 3968, 0),      # 31 row blocks, 168 tiles
    (9000, 4096, 4096, 16),      # weights that stay in L2
    (700, 11008, 2048, 0),       # 256-row tiles
    (128, 11008, 512, 64),       # the few-token kernel, its reduction split over clusters
])
def test_sparse_products(b, k, m, r):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    gen = torch.Generator("cuda").manual_seed(91)
    new = lambda *shape, sigma: torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16).mul_(sigma)
    vals, meta, _ = B.alloc_compressed(m, k)
    B.slope_prune_24(new(m, k, sigma=0.02), vals, meta, None)
    act = _rows(b, k, 92)
    low, R, L = (_rows(b, r, 93), new(r, m, sigma=0.1), new(m, r, sigma=0.1)) if r else (None, None, None)
    Y, dX = (torch.full((b, m), float("nan"), device="cuda", dtype=torch.bfloat16) for _ in range(2))
    B.slope_linear_fwd(act, vals, meta, m, Y, low, R)
    B.slope_linear_bwd_dx(act, vals, meta, m, dX, low, L)
    assert B.slope_poll_status() == 0
    _assert_equal_rows(Y)
    _assert_equal_rows(dX)
    if not r:
        assert torch.equal(Y, dX)      # without adapters the two calls are one product


@pytest.mark.parametrize("b,d,r", [(300, 4096, 64), (4097, 2048, 256), (16384, 768, 16)])
def test_adapter_products(b, d, r):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    gen = torch.Generator("cuda").manual_seed(96)
    L, R = (torch.randn(shape, generator=gen, device="cuda", dtype=torch.bfloat16) for shape in ((d, r), (r, d)))
    X = _rows(b, d, 97)
    T, dT = (torch.full((b, r), float("nan"), device="cuda", dtype=torch.bfloat16) for _ in range(2))
    B.slope_adapter_fwd_bwd(0, X, None, L, None, b, d, d, r, T=T)
    ws = torch.empty(max(16, B.slope_adapter_workspace_bytes(b, d, d, r)), dtype=torch.uint8, device="cuda")
    dL, dR = (torch.empty(shape, device="cuda", dtype=torch.bfloat16) for shape in ((d, r), (r, d)))
    B.slope_adapter_fwd_bwd(1, X, X, L, R, b, d, d, r, T=T, dT=dT, dL=dL, dR=dR, workspace=ws)
    assert B.slope_poll_status() == 0
    _assert_equal_rows(T)
    _assert_equal_rows(dT)


@pytest.mark.parametrize("b,k,m,backward", [
    (4100, 8320, 4096, False),   # 17 x 16 tiles of 256 x 256, two in turn; a last row tile of four tokens
    (2500, 8192, 5120, True),    # 10 x 20, the second raster group backwards
    (1793, 8192, 4992, True),    # eight rows of tiles, the last one with one token; the last wave's tiles halved
    (1792, 8192, 4992, True),    # seven
    (1536, 8192, 5120, True),    # six: one tile after the other
    (4100, 5632, 4096, False),   # the shortest reduction
    (4100, 5504, 4096, False),   # shorter: one tile after the other
])
def test_dense_products(b, k, m, backward):
    import torch
    from paper_2608_24070_b200 import binding as B, build
    from helpers import REL_TOL, parity_error, to_f64

    build.build()
    gen = torch.Generator("cuda").manual_seed(94)
    W = torch.randn((k, m) if backward else (m, k), generator=gen, device="cuda", dtype=torch.bfloat16).mul_(0.02)
    act = _rows(b, k, 95)
    out = torch.full((b + 1, m), float("nan"), device="cuda", dtype=torch.bfloat16)
    (B.slope_dense_linear_bwd_dx if backward else B.slope_dense_linear_fwd)(act, W, out[:b])
    assert B.slope_poll_status() == 0
    assert torch.isnan(out[b]).all()
    _assert_equal_rows(out[:b])
    g = lambda t: to_f64(B.bits_from_bf16(t))
    assert parity_error(g(out[:PERIOD]), g(act[:PERIOD]) @ (g(W) if backward else g(W).T)) <= REL_TOL
