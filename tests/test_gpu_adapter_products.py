"""The adapter's low-rank products at the edges of their kernel: every column tile (64, 128, 256) and every
reduction split (1, 2, 4, 8) that the estimate gives them, one and two CTAs per SM, ragged last tiles and k-blocks;
operands whose boxes are not full; gradients that take the place of operands.

The reference is the fp64 product of the same bf16 operands (dL is checked from the dT the call wrote), so
an output is rounded once: 2^-9 / sqrt(3) ~ 1.7e-3 relative on Gaussian data, 5e-3 allowed, and
parity_error's bound per element."""
import pytest

from paper_2608_24070_b200 import inputs as si
from helpers import REL_TOL, parity_error, to_f64

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("b,d_in,d_out,r", [
    (1, 128, 128, 16),           # one token, two k-blocks of T, one of dL: no split
    (63, 256, 384, 16),          # boxes of 63 and of 16 rows, no split
    (130, 4096, 1152, 64),       # ragged second row tile, T and dT split in eight
    (257, 128, 2176, 48),        # dT split in eight; ragged k-block in dL / dR, columns past r in the 64-wide tile
    (1000, 768, 2304, 256),      # widest rank on few tiles: four column tiles; dT split in four
    (1100, 640, 256, 176),       # rank between the column tiles
    (4096, 1024, 512, 128),      # dL / dR split in four
    (9500, 512, 640, 256),       # 75 row tiles: 256-wide tiles; dL / dR on 128-wide ones, split in four
    (19100, 128, 256, 80),       # more row tiles than SMs: two CTAs per SM on 128-wide tiles
    (40000, 128, 128, 16),       # several waves; 625 k-blocks for two row tiles, split in eight
])
def test_adapter_products_match_fp64(b, d_in, d_out, r):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    bits = {"X": si.gaussian_bf16((b, d_in), 1.0, 31), "dY": si.gaussian_bf16((b, d_out), 1.0, 32),
            "L": si.gaussian_bf16((d_in, r), 0.01, 33), "R": si.gaussian_bf16((r, d_out), 0.01, 34)}
    X, dY, L, R = (B.bf16_from_bits(bits[k]) for k in ("X", "dY", "L", "R"))
    f = {k: to_f64(v) for k, v in bits.items()}
    nan = lambda *shape: torch.full(shape, float("nan"), dtype=torch.bfloat16, device="cuda")
    T, dT2 = nan(b + 1, r), nan(b + 1, r)                       # a spare row each: nothing may be written behind the last token
    B.slope_adapter_fwd_bwd(0, X, None, L, None, b, d_out, d_in, r, T=T[:b])
    B.slope_adapter_fwd_bwd(2, None, dY, None, R, b, d_out, d_in, r, dT=dT2[:b])
    dT, dL, dR = nan(b, r), nan(d_in, r), nan(r, d_out)
    ws = torch.empty(B.slope_adapter_workspace_bytes(b, d_out, d_in, r), dtype=torch.uint8, device="cuda")
    B.slope_adapter_fwd_bwd(1, X, dY, L, R, b, d_out, d_in, r, T=T[:b], dT=dT, dL=dL, dR=dR, workspace=ws)
    assert B.slope_poll_status() == 0
    assert torch.isnan(T[b]).all() and torch.isnan(dT2[b]).all()
    assert torch.equal(dT.view(torch.int16), dT2[:b].view(torch.int16))
    g = lambda t: to_f64(B.bits_from_bf16(t))
    errs = {"T": parity_error(g(T[:b]), f["X"] @ f["L"]), "dT": parity_error(g(dT), f["dY"] @ f["R"].T),
            "dL": parity_error(g(dL), f["X"].T @ g(dT)), "dR": parity_error(g(dR), g(T[:b]).T @ f["dY"])}
    assert all(v <= REL_TOL for v in errs.values()), errs


@pytest.mark.parametrize("b,d_in,d_out,r", [
    # T: column tile / split, in two CTAs per SM where it says shared
    (1090, 1536, 128, 256),      # 64 / 2
    (9558, 1664, 128, 16),       # 64 / 2 shared
    (2974, 1536, 128, 80),       # 64 / 4 shared
    (1531, 1024, 128, 80),       # 64 / 8 shared
    (2102, 3584, 128, 256),      # 128 / 2
    (1067, 2816, 128, 208),      # 128 / 4
    (150, 4992, 128, 240),       # 128 / 8
    (2032, 2560, 128, 112),      # 128 / 8 shared
    (2785, 5376, 384, 256),      # 256 / 2
    (1328, 5888, 128, 240),      # 256 / 4
    # dT
    (1047, 128, 2176, 240),      # 64 / 2
    (2197, 128, 7168, 48),       # 64 / 8 shared
    (2387, 128, 5504, 208),      # 128 / 2
    (1055, 128, 4864, 208),      # 128 / 4
    # dL and dR
    (1989, 1024, 128, 208),      # 64 / 2
    (260, 4864, 128, 256),       # 128 / 1
    (6391, 128, 2176, 240),      # 128 / 2
    (8983, 256, 256, 224),       # 128 / 8
    (13715, 1664, 512, 208),     # 256 / 4
    (28495, 384, 768, 208),      # 256 / 8
])
def test_tiles_and_splits(b, d_in, d_out, r):
    test_adapter_products_match_fp64(b, d_in, d_out, r)


@pytest.mark.parametrize("b,d_in,d_out,r", [(1, 1024, 896, 16), (5, 640, 1152, 48), (17, 4096, 640, 80), (127, 768, 2304, 256)])
def test_rows_that_are_not_loaded_are_not_seen(b, d_in, d_out, r):
    """Boxes hold as many rows of the tokens and of R as there are; the MMAs also read the rows behind them."""
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    gen = torch.Generator("cuda").manual_seed(36)
    new = lambda *shape: torch.randn(shape, generator=gen, dtype=torch.bfloat16, device="cuda")
    full = lambda v, *shape: torch.full(shape, v, dtype=torch.bfloat16, device="cuda")
    X, dY, L, R, wide = new(b, d_in), new(b, d_out), new(d_in, r), new(r, d_out), 256
    out = []
    for fill in (0.0, float("nan")):
        for _ in range(3):                                       # on every SM
            B.slope_adapter_fwd_bwd(0, full(fill, 20000, d_in), None, full(fill, d_in, wide), None, 20000, d_out, d_in, wide,
                                    T=full(0, 20000, wide))
            B.slope_adapter_fwd_bwd(2, None, full(fill, 20000, d_out), None, full(fill, wide, d_out), 20000, d_out, d_in, wide,
                                    dT=full(0, 20000, wide))
        T, dT = full(float("nan"), b, r), full(float("nan"), b, r)
        B.slope_adapter_fwd_bwd(0, X, None, L, None, b, d_out, d_in, r, T=T)
        B.slope_adapter_fwd_bwd(2, None, dY, None, R, b, d_out, d_in, r, dT=dT)
        out.append((T, dT))
    for x, y in zip(*out):
        assert torch.isfinite(x).all() and torch.equal(x.view(torch.int16), y.view(torch.int16))
    assert B.slope_poll_status() == 0


def _gradient_operands(b, d_in, d_out, r):
    import torch
    from paper_2608_24070_b200 import binding as B, build

    build.build()
    gen = torch.Generator("cuda").manual_seed(35)
    new = lambda *shape: torch.randn(shape, generator=gen, dtype=torch.bfloat16, device="cuda")
    o = {"X": new(b, d_in), "dY": new(b, d_out), "R": new(r, d_out), "T": new(b, r), "dT": new(b, r)}
    fresh = lambda: {k: v.clone() for k, v in o.items()} | {
        "dL": torch.empty((d_in, r), dtype=torch.bfloat16, device="cuda"), "dR": torch.empty((r, d_out), dtype=torch.bfloat16, device="cuda")}
    return B, fresh


def _same_gradients(fresh, run, d_in, d_out, r, places):
    """run(o) with gradients of their own against the same call with dL / dR at the start of an operand's memory."""
    import torch

    o = fresh()
    run(o)
    for dL_in, dR_in in places:
        q = fresh()
        if dL_in:
            q["dL"] = q[dL_in].view(-1)[:d_in * r].view(d_in, r)
        if dR_in:
            q["dR"] = q[dR_in].view(-1)[:r * d_out].view(r, d_out)
        run(q)
        for k in ("dL", "dR"):
            assert torch.equal(o[k].view(torch.int16), q[k].view(torch.int16)), (dL_in, dR_in, k)


@pytest.mark.parametrize("b,d_in,d_out,r", [(700, 256, 384, 128), (1000, 768, 2304, 16), (4096, 1024, 2560, 256), (2500, 128, 128, 64)])
def test_gradients_may_take_the_place_of_operands(b, d_in, d_out, r):
    B, fresh = _gradient_operands(b, d_in, d_out, r)
    ws = B.torch.empty(B.slope_adapter_workspace_bytes(b, d_out, d_in, r), dtype=B.torch.uint8, device="cuda")
    run = lambda o: B.slope_adapter_fwd_bwd(1, o["X"], o["dY"], None, o["R"], b, d_out, d_in, r, T=o["T"], dT=o["dT"], dL=o["dL"],
                                            dR=o["dR"], workspace=ws)
    _same_gradients(fresh, run, d_in, d_out, r, [(None, "R"), ("X", "dY"), ("dY", "X"), ("T", "R") if b >= d_in else ("X", "R")])
    assert B.slope_poll_status() == 0


@pytest.mark.parametrize("b,d_in,d_out,r", [(1000, 768, 2304, 16), (700, 256, 384, 128), (600, 4096, 4096, 32)])
def test_gradients_beside_the_weight_gradient_may_take_the_place_of_operands(b, d_in, d_out, r):
    B, fresh = _gradient_operands(b, d_in, d_out, r)
    W = B.torch.randn((d_out, d_in), dtype=B.torch.bfloat16, device="cuda")
    v, m, mask = B.alloc_compressed(d_out, d_in)
    B.slope_prune_24(W, v, m, mask)
    dWc = B.torch.empty_like(v)
    ws = B.torch.empty(B.slope_bwd_dw_adapter_workspace_bytes(b, d_out, d_in, r), dtype=B.torch.uint8, device="cuda")
    run = lambda o: B.slope_linear_bwd_dw_adapter(o["dY"], o["X"], o["T"], o["dT"], mask, dWc, o["dL"], o["dR"], ws)
    _same_gradients(fresh, run, d_in, d_out, r, [("X", None), (None, "dY"), ("dY", "X")])
    assert B.slope_poll_status() == 0


@pytest.mark.parametrize("b,d_in,d_out,r", [(1000, 768, 128, 16), (300, 256, 128, 256), (2000, 1024, 128, 256)])
def test_noalloc_gradient_may_take_the_place_of_an_operand(b, d_in, d_out, r):
    B, fresh = _gradient_operands(b, d_in, d_out, r)
    run = lambda o: B.slope_adapter_dl_noalloc(o["X"], o["dT"], o["dL"])
    o = fresh()
    run(o)
    for place in ("X", "dT"):
        q = fresh()
        if q[place].numel() < d_in * r:
            continue
        q["dL"] = q[place].view(-1)[-d_in * r:].view(d_in, r)
        run(q)
        assert B.torch.equal(o["dL"].view(B.torch.int16), q["dL"].view(B.torch.int16)), place
    assert B.slope_poll_status() == 0
